// The pipelined block DFT for nfft = 512 (fft_pipe.cuh).
#include "fft_pipe.cuh"

namespace spod {

PipeLen pipe_len_512() { return pipe_len<512>(); }

}  // namespace spod
