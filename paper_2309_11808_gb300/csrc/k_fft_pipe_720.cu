// The pipelined block DFT for nfft = 720 (fft_pipe.cuh).
#include "fft_pipe.cuh"

namespace spod {

PipeLen pipe_len_720() { return pipe_len<720>(); }

}  // namespace spod
