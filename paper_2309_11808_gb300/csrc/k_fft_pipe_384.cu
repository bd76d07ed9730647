// The pipelined block DFT for nfft = 384 (fft_pipe.cuh).
#include "fft_pipe.cuh"

namespace spod {

PipeLen pipe_len_384() { return pipe_len<384>(); }

}  // namespace spod
