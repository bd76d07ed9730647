// Selection and launch of the pipelined block DFT (fft_pipe.cuh): the compiled
// lengths, the tile width of a plan and of a launch.
#include "spod_internal.cuh"

namespace spod {
namespace {

// the entry points of a compiled length, or none
PipeLen pipe_len_of(int nfft) {
  switch (nfft) {
    case 256: return pipe_len_256();
    case 384: return pipe_len_384();
    case 512: return pipe_len_512();
    case 720: return pipe_len_720();
    default: return PipeLen{};
  }
}

}  // namespace

// Whether the pipelined kernel has a form with tp-point tiles (16 or 32) for the
// plan's nfft and input type.
bool fft_pipe_has(const spod_plan_s& p, int tp) {
  const PipeLen e = pipe_len_of(p.nfft);
  return e.has && (tp == 16 || tp == 32) && e.has(p, tp);
}

// Tile choice of a plan: 32 points (or wider, see fft_pipe_width) when that form
// exists, else 16.
int fft_pipe_tile(const spod_plan_s& p) { return fft_pipe_has(p, 32) ? 32 : 16; }

// Points per tile, and per row of an X box, of a launch over the given points.
int fft_pipe_width(const spod_plan_s& p, int64_t points) { return pipe_len_of(p.nfft).width(p, points); }

bool fft_pipe_usable(const spod_plan_s& p) {
  if (p.f64 || p.ring_boxr <= 0) return false;
  const size_t el = p.desc.in_dtype == SPOD_F64 || p.desc.in_dtype == SPOD_C64 ? 8
                   : p.desc.in_dtype == SPOD_C128                              ? 16
                   : p.desc.in_dtype == SPOD_F32                               ? 4
                                                                               : 2;
  if ((p.M * (int64_t)el) % 16 != 0) return false;          // TMA row stride
  if (p.nfft % p.ring_boxr != 0 || p.step % p.ring_boxr != 0) return false;
  return fft_pipe_has(p, p.pipe_tp);
}

cudaError_t launch_fft_pipe_chunk(const spod_plan_s& p, const CUtensorMap& xmap, int width, const void* d_X, int64_t m0,
                                  int64_t mcount, cudaStream_t s, int* nlaunch) {
  return pipe_len_of(p.nfft).launch(p, xmap, width, d_X, m0, mcount, s, nlaunch);
}

}  // namespace spod
