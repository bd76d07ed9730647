// The pipelined block DFT for nfft = 256 (fft_pipe.cuh).
#include "fft_pipe.cuh"

namespace spod {

PipeLen pipe_len_256() { return pipe_len<256>(); }

}  // namespace spod
