// Persistent block DFT (Eqs. blocks, blocks-ft, blocks-k) for the nfft values
// with a compiled form (256, 384, 512, 720): the kernel template, instantiated
// for one nfft per translation unit (k_fft_pipe_256.cu ..).
//
// Complex data (CPLX) runs through the same ring and passes as an array of
// 2M interleaved real components: a column of the transform then holds one
// complex point (its real and imaginary parts) instead of two real points,
// and the output phase keeps all nfft bins with no separation.
//
// Persistent CTAs walk tiles of TP spatial points (TP / 2 complex columns);
// each CTA transforms the Welch blocks l = 0 .. nb-1 of its tile in order.  The
// tile's time rows arrive by TMA into a ring of exactly nfft rows: block 0
// loads nfft rows, each later block only its step new rows, written over the
// rows the previous block no longer needs, so every sample of X is read from
// HBM once and the request for block l+1 is in flight while block l is
// transformed.
//
// A transform is the Stockham pass sequence of the length (8-8-4, 8-8-2-3,
// 8-2-3-3-5, 8-8-8; a 16 x 16 x 2 form for real data at nfft = 512), taken in three
// stages of one or two passes each in registers.  After passes of product Ns an
// element is (g, k), k < Ns, g < N / Ns; a pass of radix R combines the groups
// g' + r N / (Ns R) of one k (twiddle W_N^(r k N / (Ns R))) into k + q Ns of group
// g':
//   stage A  thread (column, g'') takes its RA samples from the ring (mean
//            removed as a double-float pair, window c w_n) and stores its RA
//            outputs;
//   stage B  thread (column, k, g'') takes RBB = RB / RC values and stores its
//            outputs over them (in place: no second buffer is needed for it);
//   stage C  the last RC-point transforms, taken by the output phase: a thread
//            takes one k and its mirror Ns - k, which together hold every X[f]
//            and X[N - f] it needs to separate the two real spectra packed in
//            each complex column; sqrt(W) is folded in and the planar rows
//            Q[f][l][m] (re) and Q[f][nb+l][m] (im) are stored.
// Per element one ring read, two shared-memory writes and two reads, whatever the
// number of passes, and the arithmetic of the passes as such.  With two buffers
// used in turn a block costs two barriers; with one a third, before stage A's
// stores.
//
// What bounds it: instruction issue and the shared-memory pipe together (the
// HBM traffic alone would take half the time).  Hence three stages instead of a
// pass over shared memory per radix, and wide tiles: a 128-byte line of the
// blocked BF16 layout holds 64 points of one row, so a 64-point tile stores whole
// lines.  bf16x3 with the mean inside, against Stockham passes through generic
// shared-memory pointers (an integer round trip in the alignment of the dynamic
// array had cost the compiler the address space): 512 x 256 x 3 points, nt = 10 000,
// nfft 512, 12.6 -> 11.2 ms; 361 x 720 x 2 points, nt = 4380, nfft 384, 10.0 -> 6.7;
// nt = 2920, nfft 720, 9.8 -> 5.1; BF16 input and output, nfft 256, 8.0 -> 5.1 (6.8 TB/s
// of X and Qhat would take 7.0 / 3.9 / 2.6 / 2.0 ms).
#pragma once

#include <algorithm>
#include <type_traits>

#include "fft_common.cuh"
#include "tc_common.cuh"

namespace spod {
namespace {

using namespace fft;

// Stages of the compiled lengths: the radices of stage A (A1, A2), B (B1, B2) and
// C (C1, C2), 1: none.  N = RA RB, RB = RBB RC.  TPT: threads per point (pipe_tpt); WMAX:
// points of the widest tile.
template <int N, bool CPLX> struct Stages;
template <bool CPLX> struct Stages<256, CPLX> {
  static constexpr int A1 = 8, A2 = 1, B1 = 8, B2 = 1, C1 = 4, C2 = 1, TPT = 8, WMAX = 32;
};
template <bool CPLX> struct Stages<384, CPLX> {
  static constexpr int A1 = 8, A2 = 1, B1 = 8, B2 = 1, C1 = 2, C2 = 3, TPT = 8, WMAX = 64;
};
template <> struct Stages<512, true> {
  static constexpr int A1 = 8, A2 = 1, B1 = 8, B2 = 1, C1 = 8, C2 = 1, TPT = 16, WMAX = 32;
};
// 16 x 16 x 2, decimated in time: stage A is one 16-point DFT (n = 32 n1 + n2),
// stage B the two 16-point DFTs (n2 = 2 m + h) of each k1, C their radix-2 step
template <> struct Stages<512, false> {
  static constexpr int A1 = 16, A2 = 1, B1 = 16, B2 = 1, C1 = 2, C2 = 1, TPT = 16, WMAX = 32;
};
template <bool CPLX> struct Stages<720, CPLX> {
  static constexpr int A1 = 8, A2 = 2, B1 = 3, B2 = 3, C1 = 5, C2 = 1, TPT = 16, WMAX = 32;
};

// Threads per point of a form: the length's, but 16 in tiles of 16 points (small grids:
// one tile an SM, so the threads are all the latency hiding there is) and for 8-byte
// input at nfft 384 (whose 32-point ring leaves room for one CTA).  With 8 and 16 threads
// (nb = 10): F32, 2048 points, nfft 256, bf16x3 28.1 and 24.9 us, F64 41.7 and 32.9; F64,
// 16 384 points, nfft 384, FP32 221 and 193, bf16x3 275 and 230.
template <typename Tin, int N, int TP, bool CPLX> constexpr int pipe_tpt() {
  return TP == 16 || (sizeof(Tin) == 8 && N == 384) ? 16 : Stages<N, CPLX>::TPT;
}

// Tile geometry: TP points, TPT threads each.
template <int N, int TP, bool CPLX, int TPT>
struct Geo {
  using F = Stages<N, CPLX>;
  static constexpr int RA = F::A1 * F::A2, RB = N / RA, RBB = F::B1 * F::B2, RC = RB / RBB;
  static constexpr int NSC = RA * RBB;             // Ns before stage C
  static_assert(RC == F::C1 * F::C2, "the stages' radices multiply to N");
  static constexpr int PTP = TP;                   // points per tile
  static constexpr int PC = TP / 2;                // complex columns (point pairs)
  static constexpr int THREADS = TPT * TP;
  static constexpr int BSTEP = THREADS / PC;       // threads per column
  static constexpr int NA = (RB + BSTEP - 1) / BSTEP;   // stage-A tasks per thread
  static constexpr int OUTCP = PC / 2;             // column pairs per tile
  static constexpr int OUTFSTEP = THREADS / OUTCP; // output items between a thread's consecutive ones
};
// Partial sums per column of the folded mean (fixed, so that the sums do not
// depend on the tile)
constexpr int kPart = 32;

struct PipeArgs {
  int64_t m0, mcount, chunk;
  int64_t tile0, ntiles;             // the launch's tiles [tile0, ntiles)
  int64_t xoff;                      // column of X's first TMA column (tiled data)
  int step, nb, nf, boxr;
  int subtract_mean;
  int qrows;                         // Qhat rows per frequency (blocked layout)
  // time mean folded into the transform (FOLD, real data): a provisional centre
  // c (the mean of kCentreSamples evenly spaced snapshots of the column) is
  // subtracted instead of the mean, the sum of x - c over all nt snapshots
  // accumulated, mu = c + mean(x - c) written to mu_out and
  // rho = sqrt(W) mean(x - c) to Qhat row 2 nb of every frequency
  int64_t nt, tail0;                 // snapshots; first snapshot in no block
  const void* xg;                    // X itself (tail samples), row stride xld, column of point lm: xc0 + lm
  int64_t xld, xc0;
  double* mu_out;
};

// Snapshots that give the provisional centre of a column when the mean is
// folded: the closer c is to mu, the smaller the rank-one correction and the
// cancellation it brings to the low bins (the centre's offset from mu enters
// the uncorrected spectra times sum_n w_n)
constexpr int kCentreSamples = 128;

// Compensated (Kahan) FP32 sum: s + (-c) carries the running total to about
// one rounding of the result.  The folded mean's sums use it instead of FP64
// adds, which run at a small fraction of the FP32 rate on this part.
__device__ __forceinline__ void kahan_add(float& s, float& c, float v) {
  const float y = v - c;
  const float t = s + y;
  c = (t - s) - y;
  s = t;
}

struct PipeHdr {
  uint64_t full;
  int abort;
};

template <typename Tin> struct PairLoad;
template <> struct PairLoad<float> {
  static __device__ __forceinline__ float2 get(const float* p) { return *reinterpret_cast<const float2*>(p); }
};
template <> struct PairLoad<__nv_bfloat16> {
  static __device__ __forceinline__ float2 get(const __nv_bfloat16* p) {
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
  }
};
template <> struct PairLoad<double> {
  static __device__ __forceinline__ float2 get(const double* p) {
    const double2 d = *reinterpret_cast<const double2*>(p);
    return make_float2((float)d.x, (float)d.y);
  }
};

__device__ __forceinline__ uint32_t pack_bf16x2(float a, float b) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&h);
}
__device__ __forceinline__ float bf16_lo_f(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi_f(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

// 16-point forward DFT in registers (radix 4 x 4).
__device__ __forceinline__ void dft16(float2* v) {
  constexpr float c1 = 0.92387953251128675613f, s1 = 0.38268343236508977173f, r2 = 0.70710678118654752440f;
  float2 a[4][4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    float2 t[4] = {v[q], v[q + 4], v[q + 8], v[q + 12]};
    dft_small<4, float2, float>(t);
#pragma unroll
    for (int r = 0; r < 4; ++r) a[q][r] = t[r];
  }
  // a[q][r] *= W16^(q r)
  const float2 w1 = make_float2(c1, -s1), w3 = make_float2(s1, -c1), w9 = make_float2(-c1, s1);
  a[1][1] = cmul(a[1][1], w1);
  a[1][2] = make_float2(r2 * (a[1][2].x + a[1][2].y), r2 * (a[1][2].y - a[1][2].x));   // W^2
  a[1][3] = cmul(a[1][3], w3);
  a[2][1] = make_float2(r2 * (a[2][1].x + a[2][1].y), r2 * (a[2][1].y - a[2][1].x));   // W^2
  a[2][2] = mul_mi(a[2][2]);                                                            // W^4
  a[2][3] = make_float2(r2 * (a[2][3].y - a[2][3].x), -r2 * (a[2][3].x + a[2][3].y));  // W^6
  a[3][1] = cmul(a[3][1], w3);
  a[3][2] = make_float2(r2 * (a[3][2].y - a[3][2].x), -r2 * (a[3][2].x + a[3][2].y));  // W^6
  a[3][3] = cmul(a[3][3], w9);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float2 t[4] = {a[0][r], a[1][r], a[2][r], a[3][r]};
    dft_small<4, float2, float>(t);
#pragma unroll
    for (int q = 0; q < 4; ++q) v[r + 4 * q] = t[q];
  }
}


// A twiddle product with its FMAs fixed (left to the compiler, which product of the
// imaginary part is rounded first depends on the code around it): a.x b.y first
// (XFIRST) or a.y b.x.
template <bool XFIRST>
__device__ __forceinline__ float2 cmul_fma(float2 a, float2 b) {
  const float re = __fmaf_rn(a.x, b.x, -__fmul_rn(a.y, b.y));
  return make_float2(re, XFIRST ? __fmaf_rn(a.y, b.x, __fmul_rn(a.x, b.y)) : __fmaf_rn(a.x, b.y, __fmul_rn(a.y, b.x)));
}

// One pass, or two, in registers: v[r1 + R1 r2] holds the element of group
// g'' + (r2 + R2 r1) (N / (Ns R1 R2)) at k; on return v[q1 + R1 q2] is the one at
// k + Ns (q1 + R1 q2).
template <int N, int NS, int R1, int R2>
__device__ __forceinline__ void passes(float2* v, int k, const float2* __restrict__ tw) {
#pragma unroll
  for (int r2 = 0; r2 < R2; ++r2) {
    if constexpr (NS > 1) {
#pragma unroll
      for (int r1 = 1; r1 < R1; ++r1) v[r1 + R1 * r2] = cmul_fma<true>(v[r1 + R1 * r2], tw[r1 * k * (N / (NS * R1))]);
    }
    dft_small<R1, float2, float>(v + R1 * r2);
  }
  if constexpr (R2 > 1) {
#pragma unroll
    for (int q1 = 0; q1 < R1; ++q1) {
      float2 u[R2];
#pragma unroll
      for (int r2 = 0; r2 < R2; ++r2) {
        u[r2] = v[q1 + R1 * r2];
        if (r2 > 0) u[r2] = cmul_fma<(NS > 1)>(u[r2], tw[r2 * (k + q1 * NS) * (N / (NS * R1 * R2))]);
      }
      dft_small<R2, float2, float>(u);
#pragma unroll
      for (int r2 = 0; r2 < R2; ++r2) v[q1 + R1 * r2] = u[r2];
    }
  }
}

// Stage A of the task g'' = n2 of this thread's column, into v (stored by the
// caller).  With FOLD the samples n = n2 + RB n1 with n1 >= n1thr (a block-uniform
// bound) are also summed into acc0 / acc1.
template <typename Tin, int N, int TP, bool CPLX, bool FOLD>
__device__ __forceinline__ void stage_a(const Tin* __restrict__ ring, int rb, int n2, float2* v,
                                        const float* __restrict__ wsm, const float2* __restrict__ tw, float mhi0,
                                        float mlo0, float mhi1, float mlo1, int n1thr, float& acc0, float& acc1) {
  using G = Geo<N, TP, CPLX, pipe_tpt<Tin, N, TP, CPLX>()>;
  using F = Stages<N, CPLX>;
  constexpr int RA = G::RA, RB = G::RB;
  const int col = threadIdx.x % G::PC;
  const int s0 = rb + n2;
#pragma unroll
  for (int n1 = 0; n1 < RA; ++n1) {
    const int n = RB * n1 + n2;
    int slot = s0 + RB * n1;
    if constexpr ((N & (N - 1)) == 0) slot &= N - 1;
    else if (slot >= N) slot -= N;
    const float2 x = PairLoad<Tin>::get(ring + slot * G::PTP + 2 * col);
    const float wn = wsm[n];
    // (the folded mean's centre is one float: known at compile time, 720 takes
    // 5.09 ms for 5.32, 384 6.71 for 6.94, 256 with BF16 5.10 for 5.29)
    const float d0 = FOLD ? x.x - mhi0 : (x.x - mhi0) - mlo0, d1 = FOLD ? x.y - mhi1 : (x.y - mhi1) - mlo1;
    if (FOLD && n1 >= n1thr) {           // a snapshot no earlier block held
      acc0 += d0;
      acc1 += d1;
    }
    // a rounded product where N is not a power of two (elsewhere it may contract
    // into the first butterfly's sum): the spectra keep their last bits
    v[n1 / F::A2 + F::A1 * (n1 % F::A2)] =
        (N & (N - 1)) ? make_float2(__fmul_rn(d0, wn), __fmul_rn(d1, wn)) : make_float2(d0 * wn, d1 * wn);
  }
  if constexpr (F::A1 == 16) {
    dft16(v);
#pragma unroll
    for (int k1 = 1; k1 < RA; ++k1) v[k1] = cmul(v[k1], tw[n2 * k1]);
  } else {
    passes<N, 1, F::A1, F::A2>(v, 0, tw);
  }
}

// Stage B, in place: task j = (k, g'').
template <int N, int TP, bool CPLX, int TPT>
__device__ __forceinline__ void stage_b(float2* __restrict__ buf, const float2* __restrict__ tw) {
  using G = Geo<N, TP, CPLX, TPT>;
  using F = Stages<N, CPLX>;
  constexpr int RA = G::RA, RBB = G::RBB, RC = G::RC, PC = G::PC, STEP = G::BSTEP;
  const int col = threadIdx.x % PC;
#pragma unroll
  for (int i = 0; i < (RA * RC + STEP - 1) / STEP; ++i) {
    const int j = threadIdx.x / PC + i * STEP;
    if (RA * RC % STEP != 0 && j >= RA * RC) break;
    const int k = j / RC, g = j - k * RC;
    float2* const p = buf + (k * G::RB + g) * PC + col;
    float2 v[RBB];
#pragma unroll
    for (int m = 0; m < RBB; ++m) v[m / F::B2 + F::B1 * (m % F::B2)] = p[RC * m * PC];
    if constexpr (F::B1 == 16) dft16(v);
    else passes<N, RA, F::B1, F::B2>(v, k, tw);
#pragma unroll
    for (int m = 0; m < RBB; ++m) p[RC * m * PC] = v[m];
  }
}

// Store the one-sided spectra of the four points of column pair cp at bin f
// from z = X[f] and zc = X[N - f] of its two complex columns (float4 = two
// columns): the even point of a column is (z + conj zc) / 2, the odd one
// (z - conj zc) / 2i; sw carries sqrt(W) / 2.
template <int OUTK>
__device__ __forceinline__ void store_bin4(const float4 z, const float4 zc, const float (&sw)[4], const PipeArgs& a,
                                           int64_t o, void* __restrict__ qout, void* __restrict__ qlo) {
  const float r0 = (z.x + zc.x) * sw[0], i0 = (z.y - zc.y) * sw[0];
  const float r1 = (z.y + zc.y) * sw[1], i1 = (zc.x - z.x) * sw[1];
  const float r2 = (z.z + zc.z) * sw[2], i2 = (z.w - zc.w) * sw[2];
  const float r3 = (z.w + zc.w) * sw[3], i3 = (zc.z - z.z) * sw[3];
  if constexpr (OUTK == OUT_NATIVE) {
    float* q = static_cast<float*>(qout);
    *reinterpret_cast<float4*>(q + o) = make_float4(r0, r1, r2, r3);
    *reinterpret_cast<float4*>(q + o + (int64_t)a.nb * a.chunk) = make_float4(i0, i1, i2, i3);
  } else {
    const int64_t imoff = (int64_t)a.nb * kQBlock;
    __nv_bfloat16* qh = static_cast<__nv_bfloat16*>(qout);
    const uint32_t hr01 = pack_bf16x2(r0, r1), hr23 = pack_bf16x2(r2, r3);
    const uint32_t hi01 = pack_bf16x2(i0, i1), hi23 = pack_bf16x2(i2, i3);
    *reinterpret_cast<uint2*>(qh + o) = make_uint2(hr01, hr23);
    *reinterpret_cast<uint2*>(qh + o + imoff) = make_uint2(hi01, hi23);
    if constexpr (OUTK == OUT_BF16X3) {
      __nv_bfloat16* ql = static_cast<__nv_bfloat16*>(qlo);
      const uint32_t lr01 = pack_bf16x2(r0 - bf16_lo_f(hr01), r1 - bf16_hi_f(hr01));
      const uint32_t lr23 = pack_bf16x2(r2 - bf16_lo_f(hr23), r3 - bf16_hi_f(hr23));
      const uint32_t li01 = pack_bf16x2(i0 - bf16_lo_f(hi01), i1 - bf16_hi_f(hi01));
      const uint32_t li23 = pack_bf16x2(i2 - bf16_lo_f(hi23), i3 - bf16_hi_f(hi23));
      *reinterpret_cast<uint2*>(ql + o) = make_uint2(lr01, lr23);
      *reinterpret_cast<uint2*>(ql + o + imoff) = make_uint2(li01, li23);
    }
  }
}

__device__ __forceinline__ float4 c2add(float4 a, float4 b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); }
__device__ __forceinline__ float4 c2sub(float4 a, float4 b) { return make_float4(a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w); }
// both complex columns of a float4 times w
__device__ __forceinline__ float4 c2mul(float4 a, float2 w) {
  return make_float4(a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x, a.z * w.x - a.w * w.y, a.z * w.y + a.w * w.x);
}

// Complex data: store bin f of the two points of a column pair.
template <int OUTK>
__device__ __forceinline__ void store_bin2c(const float4 z, const float (&sw)[4], const PipeArgs& a, int64_t o,
                                            void* __restrict__ qout, void* __restrict__ qlo) {
  const int64_t imoff = (int64_t)a.nb * (OUTK != OUT_NATIVE ? (int64_t)kQBlock : a.chunk);
  const float r0 = z.x * sw[0], i0 = z.y * sw[0];
  const float r1 = z.z * sw[1], i1 = z.w * sw[1];
  if constexpr (OUTK == OUT_NATIVE) {
    float* q = static_cast<float*>(qout);
    *reinterpret_cast<float2*>(q + o) = make_float2(r0, r1);
    *reinterpret_cast<float2*>(q + o + imoff) = make_float2(i0, i1);
  } else {
    __nv_bfloat16* qh = static_cast<__nv_bfloat16*>(qout);
    const uint32_t hr = pack_bf16x2(r0, r1), hi = pack_bf16x2(i0, i1);
    *reinterpret_cast<uint32_t*>(qh + o) = hr;
    *reinterpret_cast<uint32_t*>(qh + o + imoff) = hi;
    if constexpr (OUTK == OUT_BF16X3) {
      __nv_bfloat16* ql = static_cast<__nv_bfloat16*>(qlo);
      *reinterpret_cast<uint32_t*>(ql + o) = pack_bf16x2(r0 - bf16_lo_f(hr), r1 - bf16_hi_f(hr));
      *reinterpret_cast<uint32_t*>(ql + o + imoff) = pack_bf16x2(i0 - bf16_lo_f(hi), i1 - bf16_hi_f(hi));
    }
  }
}

// Stage C of one k for the two columns of a pair: X[k + NSC q], q < RC, of column
// 2 cp (u) and 2 cp + 1 (w).
template <int N, int TP, bool CPLX, int TPT>
__device__ __forceinline__ void stage_c(const float4* __restrict__ U4, int k, const float2* __restrict__ tw, float2* u,
                                        float2* w) {
  using G = Geo<N, TP, CPLX, TPT>;
  using F = Stages<N, CPLX>;
  const float4* const p = U4 + ((k % G::RA) * G::RB + (k / G::RA) * G::RC) * G::OUTCP;
#pragma unroll
  for (int g = 0; g < G::RC; ++g) {
    const float4 z = p[g * G::OUTCP];
    u[g / F::C2 + F::C1 * (g % F::C2)] = make_float2(z.x, z.y);
    w[g / F::C2 + F::C1 * (g % F::C2)] = make_float2(z.z, z.w);
  }
  passes<N, G::NSC, F::C1, F::C2>(u, k, tw);
  passes<N, G::NSC, F::C1, F::C2>(w, k, tw);
}

__device__ __forceinline__ float4 pair4(float2 a, float2 b) { return make_float4(a.x, a.y, b.x, b.y); }

// Output phase: a thread takes one column pair (four points; complex data: two).
// Complex data: item k < NSC, the bins k + NSC q.  Real data: item j < NSC / 2,
// k = j and its mirror NSC - j (X[N - k - NSC q] is entry RC - 1 - q of the mirror);
// item 0 takes k = 0 and k = NSC / 2, each its own mirror.
template <int OUTK, int TP, int N, bool CPLX, int TPT>
__device__ __forceinline__ void output_phase(const float2* __restrict__ U, const float2* __restrict__ tw,
                                             const PipeArgs& a, int l, int64_t lm0, const float (&sw)[4],
                                             void* __restrict__ qout, void* __restrict__ qlo) {
  using G = Geo<N, TP, CPLX, TPT>;
  constexpr int kCp = G::OUTCP, kStep = G::OUTFSTEP, RC = G::RC, NSC = G::NSC;
  const int cp = threadIdx.x % kCp;
  const float4* const U4 = reinterpret_cast<const float4*>(U) + cp;
  // FP32 planes are planar [nf][2 nb][chunk]; BF16 planes are blocked by 64
  // points, [chunk / 64][nf][qrows][64] (see qhat_blocked_offset)
  constexpr bool BLK = OUTK != OUT_NATIVE;
  const int64_t lm = CPLX ? lm0 / 2 + 2 * cp : lm0 + 4 * cp;
  const int64_t o0 = BLK ? qhat_blocked_offset(a.nf, a.qrows, 0, l, lm) : (int64_t)l * a.chunk + lm;
  const int64_t fstep = BLK ? (int64_t)a.qrows * kQBlock : (int64_t)2 * a.nb * a.chunk;
  constexpr int kItems = CPLX ? NSC : NSC / 2;
  if constexpr (N == 512 && !CPLX) {
    // X[f] = U_0 + W32^k2 U_1 and X[256 + f] = U_0 - W32^k2 U_1 with
    // (k1, k2) = (f mod 16, f / 16); items f in [0, 128] with the partner
    // (k1', k2') = ((16 - k1) mod 16, k1 ? 15 - k2 : (16 - k2) mod 16), which gives
    // X[N - f] and X[256 - f] (the signs swap at f = 0, where the partner is the
    // item itself): an item stores bins f and 256 - f.
    for (int j = threadIdx.x / kCp; j <= 128; j += kStep) {
      const int k1 = j & 15, k2 = j >> 4;
      const int k1p = (16 - k1) & 15;
      const int k2p = k1 ? 15 - k2 : (16 - k2) & 15;
      const float4 u0 = U4[(k1 * 32 + 2 * k2) * kCp];
      const float4 u1 = c2mul(U4[(k1 * 32 + 2 * k2 + 1) * kCp], tw[16 * k2]);
      const float4 v0 = U4[(k1p * 32 + 2 * k2p) * kCp];
      const float4 v1 = c2mul(U4[(k1p * 32 + 2 * k2p + 1) * kCp], tw[16 * k2p]);
      const float4 xf = c2add(u0, u1);                 // X[f]
      const float4 xf256 = c2sub(u0, u1);              // X[256 + f]
      const float4 xnf = j ? c2sub(v0, v1) : c2add(v0, v1);     // X[N - f]
      const float4 xg = j ? c2add(v0, v1) : c2sub(v0, v1);      // X[256 - f]
      store_bin4<OUTK>(xf, xnf, sw, a, o0 + j * fstep, qout, qlo);
      if (j != 128) store_bin4<OUTK>(xg, xf256, sw, a, o0 + (256 - j) * fstep, qout, qlo);
    }
  } else {
    for (int j = threadIdx.x / kCp; j < kItems; j += kStep) {
      float2 u[RC], w[RC];
      stage_c<N, TP, CPLX, TPT>(U4, j, tw, u, w);
      if constexpr (CPLX) {
#pragma unroll
        for (int q = 0; q < RC; ++q) store_bin2c<OUTK>(pair4(u[q], w[q]), sw, a, o0 + (j + q * NSC) * fstep, qout, qlo);
      } else {
        const int jm = j ? NSC - j : NSC / 2;
        float2 um[RC], wm[RC];
        stage_c<N, TP, CPLX, TPT>(U4, jm, tw, um, wm);
        if (j) {
#pragma unroll
          for (int q = 0; q < (RC + 1) / 2; ++q)
            store_bin4<OUTK>(pair4(u[q], w[q]), pair4(um[RC - 1 - q], wm[RC - 1 - q]), sw, a, o0 + (j + q * NSC) * fstep,
                             qout, qlo);
#pragma unroll
          for (int q = 0; q < RC / 2; ++q)
            store_bin4<OUTK>(pair4(um[q], wm[q]), pair4(u[RC - 1 - q], w[RC - 1 - q]), sw, a,
                             o0 + (jm + q * NSC) * fstep, qout, qlo);
        } else {
#pragma unroll
          for (int q = 0; q <= RC / 2; ++q)
            store_bin4<OUTK>(pair4(u[q], w[q]), pair4(u[(RC - q) % RC], w[(RC - q) % RC]), sw, a, o0 + q * NSC * fstep,
                             qout, qlo);
#pragma unroll
          for (int q = 0; q <= (RC - 1) / 2; ++q)
            store_bin4<OUTK>(pair4(um[q], wm[q]), pair4(um[RC - 1 - q], wm[RC - 1 - q]), sw, a,
                             o0 + (jm + q * NSC) * fstep, qout, qlo);
        }
      }
    }
  }
}

constexpr size_t kPipeSmemMax = 227 * 1024;

// Shared-memory layout (bytes from the 1024-aligned base).
template <typename Tin, int TP, int N, bool CPLX, int NBUF>
struct PipeBytes {
  static constexpr size_t hdr = 0;
  static constexpr size_t ring = 128;
  static constexpr size_t buf0 = ring + (size_t)N * TP * sizeof(Tin);
  static constexpr size_t buf1 = buf0 + (size_t)(NBUF - 1) * N * (TP / 2) * sizeof(float2);
  static constexpr size_t tw = buf1 + (size_t)N * (TP / 2) * sizeof(float2);
  static constexpr size_t win = tw + (size_t)N * sizeof(float2);
  // folded mean (kept out of the registers the passes need and of the pass
  // buffers): the compensated partial sums of x - c, (s0, c0, s1, c1) [kPart][TP / 2];
  // the partial sums of the next tile's centre samples [kPart][TP]; the
  // centres and the rho values of a tile [TP] each; the centre sample rows
  static constexpr size_t acc = (win + (size_t)N * sizeof(float) + 15) / 16 * 16;
  static constexpr size_t cred = acc + (size_t)kPart * (TP / 2) * sizeof(float4);
  static constexpr size_t cen = cred + (size_t)kPart * TP * sizeof(float);
  static constexpr size_t rho = cen + (size_t)TP * sizeof(float);
  static constexpr size_t crow = rho + (size_t)TP * sizeof(float);
  static constexpr size_t end = crow + (size_t)kCentreSamples * sizeof(int);
  static constexpr size_t dyn = end + 1024;                    // alignment slack
};
// CTAs per SM aimed at: 512 threads at 128 registers
template <typename Tin, int TP, int N, bool CPLX> constexpr int pipe_ctas() {
  return pipe_tpt<Tin, N, TP, CPLX>() * TP <= 256 ? 2 : 1;
}
// two transform buffers where they fit beside that many CTAs, else one
template <typename Tin, int TP, int N, bool CPLX> constexpr int pipe_nbuf() {
  return PipeBytes<Tin, TP, N, CPLX, 2>::dyn + 1024 <= kPipeSmemMax / pipe_ctas<Tin, TP, N, CPLX>() ? 2 : 1;
}
template <typename Tin, int TP, int N, bool CPLX>
struct PipeLayout : PipeBytes<Tin, TP, N, CPLX, pipe_nbuf<Tin, TP, N, CPLX>()> {
  static constexpr int NBUF = pipe_nbuf<Tin, TP, N, CPLX>();
  static constexpr bool fits = PipeBytes<Tin, TP, N, CPLX, NBUF>::dyn <= kPipeSmemMax &&
                               TP <= Stages<N, CPLX>::WMAX;
};

template <typename Tin, int OUTK, int TP, int N, bool CPLX, bool FOLD>
__global__ void __launch_bounds__(pipe_tpt<Tin, N, TP, CPLX>() * TP, pipe_ctas<Tin, TP, N, CPLX>()) k_fft_pipe(const __grid_constant__ CUtensorMap xmap,
                                                          const float* __restrict__ win,
                                                          const float2* __restrict__ tw_g,
                                                          const float* __restrict__ sqrtW,
                                                          const double* __restrict__ mu, void* __restrict__ qout,
                                                          void* __restrict__ qlo, PipeArgs a,
                                                          unsigned* __restrict__ gflags) {
  using namespace tc;
  using L = PipeLayout<Tin, TP, N, CPLX>;
  constexpr int TPT = pipe_tpt<Tin, N, TP, CPLX>();
  using G = Geo<N, TP, CPLX, TPT>;
  constexpr int PTP = G::PTP, PC = G::PC, PTHREADS = G::THREADS;
  extern __shared__ unsigned char smem_raw[];
  uint8_t* sm = smem_align1024(smem_raw);
  PipeHdr* hdr = reinterpret_cast<PipeHdr*>(sm + L::hdr);
  Tin* ring = reinterpret_cast<Tin*>(sm + L::ring);
  float2* buf0 = reinterpret_cast<float2*>(sm + L::buf0);
  float2* buf1 = reinterpret_cast<float2*>(sm + L::buf1);
  float2* tw = reinterpret_cast<float2*>(sm + L::tw);
  float* wsm = reinterpret_cast<float*>(sm + L::win);
  const int tid = threadIdx.x;
  float4* const acc_all = reinterpret_cast<float4*>(sm + L::acc);
  float* const cred = reinterpret_cast<float*>(sm + L::cred);
  float* const cen = reinterpret_cast<float*>(sm + L::cen);
  float* const rhos = reinterpret_cast<float*>(sm + L::rho);
  int* const crow = reinterpret_cast<int*>(sm + L::crow);
  const uint32_t bar = smem_u32(&hdr->full);
  volatile int* abort_flag = &hdr->abort;

  if (tid == 0) {
    mbar_init(bar, 1);
    hdr->abort = 0;
    fence_mbar_init();
  }
  for (int i = tid; i < N; i += PTHREADS) {
    tw[i] = tw_g[i];
    wsm[i] = win[i];
  }
  // folded mean: the centre's sample rows t_k = floor((2k + 1) nt / (2 nc))
  const int ncen = (int)(a.nt < kCentreSamples ? a.nt : kCentreSamples);
  if (tid < ncen) crow[tid] = (int)(((int64_t)(2 * tid + 1) * a.nt) / (2 * ncen));
  __syncthreads();

  const int64_t t_first = a.tile0 + blockIdx.x;
  const int64_t t_step = gridDim.x;
  if (t_first >= a.ntiles) return;
  constexpr uint32_t row_bytes = PTP * sizeof(Tin);

  // TMA boxes for time rows [r0, r0 + nrows) of tile t; row r lands in ring slot r mod N
  auto issue = [&](int64_t t, int r0, int nrows) {
    mbar_arrive_expect_tx(bar, (uint32_t)nrows * row_bytes);
    const int x = (int)(a.m0 - a.xoff + t * PTP);
    for (int r = r0; r < r0 + nrows; r += a.boxr) tma_load_2d(smem_u32(ring + (size_t)(r % N) * PTP), &xmap, x, r, bar);
  };
  // L2 prefetch of time rows [r0, r0 + nrows) of tile t: the rows of block
  // l + 2 are requested from HBM while block l + 1's rows travel to the ring,
  // so the ring's load (one block ahead, all the shared memory allows) finds
  // them in L2
  auto prefetch = [&](int64_t t, int r0, int nrows) {
    const int x = (int)(a.m0 - a.xoff + t * PTP);
    for (int r = r0; r < r0 + nrows; r += a.boxr) tma_prefetch_2d(&xmap, x, r);
  };
  if (tid == 0) {
    prefetch_tmap(&xmap);
    issue(t_first, 0, N);
    if (a.nb > 1) prefetch(t_first, N, a.step);
  }

  const int col = tid % PC;
  uint32_t phase = 0;
  bool last_ok = true;               // thread 0: its last wait saw the copy land
  int par = 0;                       // buffer roles of the current block

  // Folded mean (real data, BF16 / BF16X3 output): the provisional centre c
  // of a column is the mean of its ncen snapshots at rows crow[k]; partial sum b
  // of a column takes k = b, b + kPart, ...  The loads for tile t + t_step are issued
  // while tile t runs (pc0 / pc1) and reduced at its end.
  static_assert(!FOLD || (!CPLX && OUTK != OUT_NATIVE), "the mean is folded for real data and BF16 output");
  constexpr bool fold = FOLD;
  constexpr int PB = G::BSTEP;
  const int b0 = tid / PC;
  const Tin* const xg = static_cast<const Tin*>(a.xg);
  // partial sums v (of thread b0: entries b0 + v PB of the column's kPart)
  static_assert(PB <= G::RB, "a stage-A task for every thread");
  constexpr int NV = kPart / PB;
  static_assert(kPart % PB == 0, "whole partial sums per thread");
  auto centre_partial = [&](int64_t t, float (&c0)[NV], float (&c1)[NV]) {
#pragma unroll
    for (int v = 0; v < NV; ++v) c0[v] = c1[v] = 0.f;
    if (t >= a.ntiles) return;
    const int64_t lmA = t * PTP + 2 * col;
    const Tin* base = xg + a.xc0 + lmA;
#pragma unroll
    for (int v = 0; v < NV; ++v) {
#pragma unroll 1
      for (int k = b0 + v * PB; k < ncen; k += kPart) {
        const Tin* row = base + (int64_t)crow[k] * a.xld;
        if (lmA < a.mcount) c0[v] += to_f32<Tin>(row[0]);
        if (lmA + 1 < a.mcount) c1[v] += to_f32<Tin>(row[1]);
      }
    }
  };
  auto put_centre = [&](const float (&c0)[NV], const float (&c1)[NV]) {
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      cred[(b0 + v * PB) * PTP + 2 * col] = c0[v];
      cred[(b0 + v * PB) * PTP + 2 * col + 1] = c1[v];
    }
  };
  auto centre_of = [&](int p) {
    float sm = 0.f;
#pragma unroll 1
    for (int q = 0; q < kPart; ++q) sm += cred[q * PTP + p];
    return sm / (float)ncen;
  };
  auto clear_acc = [&]() {
#pragma unroll
    for (int v = 0; v < NV; ++v) acc_all[(b0 + v * PB) * PC + col] = make_float4(0.f, 0.f, 0.f, 0.f);
  };
  float cen0 = 0.f, cen1 = 0.f;      // this thread's column pair: centres of the current tile
  float pc0[NV], pc1[NV];            // partial centre sums of the next tile
  float swr = 0.f, cme = 0.f;        // threads < TP: sqrt(W) and centre of point tid of the tile
  if constexpr (fold) {
    centre_partial(t_first, pc0, pc1);
    put_centre(pc0, pc1);
    __syncthreads();
    if (tid < PTP) cen[tid] = centre_of(tid);
    __syncthreads();
    cen0 = cen[2 * col];
    cen1 = cen[2 * col + 1];
    if (tid < PTP) cme = cen[tid];
    clear_acc();
    centre_partial(t_first + t_step, pc0, pc1);
  }
  for (int64_t t = t_first; t < a.ntiles; t += t_step) {
    const int64_t lm0 = t * PTP;
    const int64_t gm0 = a.m0 + lm0;
    float mhi0 = 0.f, mlo0 = 0.f, mhi1 = 0.f, mlo1 = 0.f;
    float sw[4];                     // 0.5 sqrt(W) of the output phase's four points (zero past mcount);
                                     // complex data: sqrt(W) of its two points
    {
      const int64_t lm = lm0 + 2 * col;
      if (a.subtract_mean && !fold && lm < a.mcount) {
        const double d = mu[gm0 + 2 * col]; mhi0 = (float)d; mlo0 = (float)(d - (double)mhi0);
      }
      if (a.subtract_mean && !fold && lm + 1 < a.mcount) {
        const double d = mu[gm0 + 2 * col + 1]; mhi1 = (float)d; mlo1 = (float)(d - (double)mhi1);
      }
      const int cp = tid % G::OUTCP;
      if constexpr (CPLX) {          // components -> points
        const int64_t lp = lm0 / 2 + 2 * cp, gp = gm0 / 2 + 2 * cp;
#pragma unroll
        for (int q = 0; q < 4; ++q) sw[q] = (q < 2 && 2 * (lp + q) < a.mcount) ? sqrtW[gp + q] : 0.f;
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          sw[q] = (lm0 + 4 * cp + q < a.mcount) ? 0.5f * sqrtW[gm0 + 4 * cp + q] : 0.f;
      }
    }
    if constexpr (fold) {
      mhi0 = cen0;
      mhi1 = cen1;
      if (tid < PTP) swr = lm0 + tid < a.mcount ? sqrtW[gm0 + tid] : 0.f;
    }
    int rb = 0;                      // ring slot of the block's first row
    for (int l = 0; l < a.nb; ++l) {
      last_ok = mbar_wait(bar, phase & 1, abort_flag, gflags);
      ++phase;
      float2* const buf = L::NBUF == 2 && par ? buf1 : buf0;
      {
        // with the folded mean the centre c replaces mu (mlo = 0) and the
        // snapshots no earlier block held (all of block 0, the last step rows
        // of the others) are summed: FP32 runs of a thread's samples, then
        // compensated FP32 running sums
        // The new snapshots are n >= N - step; when N - step is a multiple of
        // RB (50 % overlap, none, 75 %, ...) they are the samples
        // n1 >= (N - step) / RB of every stage-A task, otherwise a separate
        // loop re-reads them from the ring.
        constexpr int RA = G::RA, RB = G::RB, NA = G::NA;
        const int nnew0 = !fold ? N : l == 0 ? 0 : N - a.step;
        const bool in_pass = nnew0 % RB == 0;
        const int rthr = fold && in_pass ? nnew0 / RB : RA;
        float s0[NV], s1[NV];
#pragma unroll
        for (int v = 0; v < NV; ++v) s0[v] = s1[v] = 0.f;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
          const int n2 = b0 + i * PB;
          if (RB % PB == 0 || n2 < RB) {
            float2 v[RA];
            stage_a<Tin, N, TP, CPLX, FOLD>(ring, rb, n2, v, wsm, tw, mhi0, mlo0, mhi1, mlo1, rthr, s0[i % NV],
                                             s1[i % NV]);
            // one buffer: the previous block's output phase must be done reading
            // it (every thread has a first task: PB <= RB)
            if (i == 0 && L::NBUF == 1) __syncthreads();
#pragma unroll
            for (int k1 = 0; k1 < RA; ++k1) buf[(k1 * RB + n2) * PC + col] = v[k1];
          }
        }
        if constexpr (fold) {
#pragma unroll
          for (int vv = 0; vv < NV; ++vv) {
            if (!in_pass) {
              for (int n = nnew0 + b0 + vv * PB; n < N; n += kPart) {
                int slot = rb + n;
                if (slot >= N) slot -= N;
                const float2 x = PairLoad<Tin>::get(ring + slot * PTP + 2 * col);
                s0[vv] += x.x - mhi0;
                s1[vv] += x.y - mhi1;
              }
            }
            float4* const pa = acc_all + (b0 + vv * PB) * PC + col;
            float4 ac = *pa;
            kahan_add(ac.x, ac.y, s0[vv]);
            kahan_add(ac.z, ac.w, s1[vv]);
            *pa = ac;
          }
        }
      }
      __syncthreads();
      if (hdr->abort) break;
      // the ring rows of this block are consumed: request the next rows
      if (tid == 0) {
        if (l + 1 < a.nb) {
          issue(t, l * a.step + N, a.step);
          if (l + 2 < a.nb) prefetch(t, (l + 1) * a.step + N, a.step);   // rows of block l + 2 (< nt)
        } else if (t + t_step < a.ntiles) {
          issue(t + t_step, 0, N);
          if (a.nb > 1) prefetch(t + t_step, N, a.step);
        }
      }
      stage_b<N, TP, CPLX, TPT>(buf, tw);
      __syncthreads();
      // two buffers: the next block's stage A writes the other one, which nobody
      // reads since the barrier after its own block's stage A
      output_phase<OUTK, TP, N, CPLX, TPT>(buf, tw, a, l, lm0, sw, qout, qlo);
      par ^= 1;
      rb += a.step;
      if (rb >= N) rb -= N;
    }
    if (hdr->abort) break;
    if constexpr (fold) {
      // the snapshots in no block (the tail): partial sum b of a column takes t = tail0 + b + kPart k
      const int64_t lmA = lm0 + 2 * col;
#pragma unroll
      for (int v = 0; v < NV; ++v) {
        float4* const pa = acc_all + (b0 + v * PB) * PC + col;
        float4 ac = *pa;
        for (int64_t tt = a.tail0 + b0 + v * PB; tt < a.nt; tt += kPart) {
          const Tin* row = xg + tt * a.xld + a.xc0 + lmA;
          if (lmA < a.mcount) kahan_add(ac.x, ac.y, to_f32<Tin>(row[0]) - mhi0);
          if (lmA + 1 < a.mcount) kahan_add(ac.z, ac.w, to_f32<Tin>(row[1]) - mhi1);
        }
        *pa = ac;
      }
      put_centre(pc0, pc1);
      __syncthreads();
      if (tid < PTP) {
        // point tid: its column's kPart compensated partials in a fixed order,
        // mu = c + sum / nt, rho = sqrt(W) (mu - c)
        const int c = tid >> 1, h = tid & 1;
        float ss = 0.f, sc = 0.f, cc = 0.f;
#pragma unroll 1
        for (int q = 0; q < kPart; ++q) {
          const float4 v = acc_all[q * PC + c];
          kahan_add(ss, sc, h ? v.z : v.x);
          cc += h ? v.w : v.y;
        }
        // each partial is s - c; the total (ss - sc) - sum of the c
        const double mup = ((double)ss - (double)sc - (double)cc) / (double)a.nt;
        float rho = 0.f;
        if (lm0 + tid < a.mcount) {
          a.mu_out[gm0 + tid] = (double)cme + mup;
          rho = (float)(mup * (double)swr);
        }
        rhos[tid] = rho;
      } else if (tid < 2 * PTP) {
        // the next tile's centre of point tid - TP
        const int p = tid - PTP;
        cen[p] = centre_of(p);
      }
      __syncthreads();
      // rho into Qhat row 2 nb of every frequency (two points per word)
      for (int it = tid; it < a.nf * (PTP / 2); it += PTHREADS) {
        const int f = it / (PTP / 2), j = it - f * (PTP / 2);
        const int64_t o = qhat_blocked_offset(a.nf, a.qrows, f, 2 * a.nb, lm0 + 2 * j);
        const uint32_t hw = pack_bf16x2(rhos[2 * j], rhos[2 * j + 1]);
        *reinterpret_cast<uint32_t*>(static_cast<__nv_bfloat16*>(qout) + o) = hw;
        if constexpr (OUTK == OUT_BF16X3)
          *reinterpret_cast<uint32_t*>(static_cast<__nv_bfloat16*>(qlo) + o) =
              pack_bf16x2(rhos[2 * j] - bf16_lo_f(hw), rhos[2 * j + 1] - bf16_hi_f(hw));
      }
      cen0 = cen[2 * col];
      cen1 = cen[2 * col + 1];
      if (tid < PTP) cme = cen[tid];
      clear_acc();
      centre_partial(t + 2 * t_step, pc0, pc1);
      // cen and rhos are next written after the next tile's first barrier,
      // by which time every thread has read them
    }
  }
  // a request issued before an abort must land before the CTA exits
  if (tid == 0 && !last_ok) mbar_drain(bar, (phase - 1) & 1, gflags);
}

// Welch blocks a CTA transforms per launch, about.  CTAs that walk many tiles drift
// apart, and with them the rows of X that neighbouring tiles read from the same
// DRAM pages and L2 lines: 512 x 256 x 3 points, nt = 10 000 (81 tiles of 38 blocks
// per CTA) took 13.5 ms in one launch and takes 11.1 in launches of 3 to 40 tiles
// per CTA, while a quarter of the grid runs the same either way (2.84 ms).
constexpr int64_t kBlocksPerLaunch = 1024;

// Complex data (CPLX): m0 and mcount count points; the ring, the mean and the
// tiles work on the 2M interleaved components.  Adds its launches to *nlaunch.
template <typename Tin, int OUTK, int TP, int N, bool CPLX, bool FOLD = false>
cudaError_t launch_pipe_n(const spod_plan_s& p, const CUtensorMap& xmap, const void* d_X, int64_t m0,
                          int64_t mcount, cudaStream_t s, int* nlaunch) {
  constexpr int PTHREADS = pipe_tpt<Tin, N, TP, CPLX>() * TP;
  constexpr int64_t K = CPLX ? 2 : 1;          // components per point
  PipeArgs a;
  a.m0 = K * m0; a.mcount = K * mcount; a.chunk = p.chunk_points;
  a.xoff = K * p.x_off;
  const int64_t mpad = K * std::min<int64_t>(p.chunk_points, (mcount + 63) / 64 * 64);
  const int64_t ntiles = mpad / TP;
  a.step = p.step; a.nb = p.nb; a.nf = p.nf;
  a.boxr = p.ring_boxr;
  a.subtract_mean = p.desc.subtract_mean;
  a.qrows = p.qrows;
  a.nt = p.nt;
  a.tail0 = (int64_t)(p.nb - 1) * p.step + p.nfft;
  a.xg = d_X;
  a.xld = K * (p.x_ld ? p.x_ld : p.M);
  a.xc0 = a.m0 - a.xoff;
  a.mu_out = p.d_mu;
  const size_t smem = PipeLayout<Tin, TP, N, CPLX>::dyn;
  auto kern = k_fft_pipe<Tin, OUTK, TP, N, CPLX, FOLD>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 1;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, PTHREADS, smem);
  per_sm = std::max(1, per_sm);
  const int64_t grid = std::min<int64_t>(ntiles, (int64_t)(p.num_sms > 0 ? p.num_sms : 148) * per_sm);
  if (grid <= 0) return cudaSuccess;
  const int64_t per = std::max<int64_t>(1, kBlocksPerLaunch / p.nb) * grid;
  for (a.tile0 = 0; a.tile0 < ntiles; a.tile0 += per) {
    a.ntiles = std::min<int64_t>(ntiles, a.tile0 + per);
    kern<<<(unsigned)grid, PTHREADS, smem, s>>>(xmap, static_cast<const float*>(p.d_win),
                                                static_cast<const float2*>(p.d_tw),
                                                static_cast<const float*>(p.d_sqrtW), p.d_mu, p.d_qhat, p.d_qlo, a,
                                                p.d_flags);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    ++*nlaunch;
  }
  return cudaSuccess;
}

// Width of the tiles a launch takes (the box width of its X map): up to the
// plan's choice -- 16 points, or 32 and the widest form there is -- the widest for
// which every SM has a tile (2048 points, nfft 256: 0.037 ms with 16-point tiles,
// 0.042 with 32); a choice that was set is not narrowed below 32.  C64 data takes 32
// components as soon as 16 would give some SM a second tile (nb = 10, 1300 points, bf16x3:
// nfft 256 31.2 us with 16, 24.9 with 32, nfft 512 57.6 and 42.8; 1200 points 20.8 and
// 24.8, 35.8 and 42.9).  WMAX: at nfft 384
// one CTA of 64 points takes 6.9 ms where two of 32 take 8.5 (361 x 720 x 2 points), at
// nfft 256 two CTAs of 32 points 5.3 and one of 64 5.7 (their ring and buffers leave
// room for two buffers, so one CTA's barriers overlap the other's passes).
template <typename Tin, int N, bool CPLX>
int pipe_width_n(const spod_plan_s& p, int64_t points, int sms) {
  if (p.pipe_tp < 32) return 16;
  if constexpr (PipeLayout<Tin, 64, N, CPLX>::fits) {
    if (points >= (int64_t)64 * sms) return 64;
  }
  if constexpr (PipeLayout<Tin, 32, N, CPLX>::fits) {
    const int64_t from = CPLX && sizeof(Tin) == 4 ? (int64_t)16 * sms + 1 : (int64_t)32 * sms;
    if (p.pipe_tp_set || points >= from) return 32;
  }
  return 16;
}

// Whether there is a form of the tile choice (16 or 32).
template <typename Tin, int N, bool CPLX>
bool pipe_has(int tp) {
  return tp == 32 ? PipeLayout<Tin, 32, N, CPLX>::fits : PipeLayout<Tin, 16, N, CPLX>::fits;
}

template <typename Tin, int OUTK, int TP, bool CPLX, int N>
cudaError_t launch_pipe_f(const spod_plan_s& p, const CUtensorMap& xmap, const void* d_X, int64_t m0, int64_t mcount,
                          cudaStream_t s, int* nlaunch) {
  if constexpr (!CPLX && OUTK != OUT_NATIVE) {
    if (p.mean_fold) return launch_pipe_n<Tin, OUTK, TP, N, CPLX, true>(p, xmap, d_X, m0, mcount, s, nlaunch);
  }
  return launch_pipe_n<Tin, OUTK, TP, N, CPLX>(p, xmap, d_X, m0, mcount, s, nlaunch);
}

template <typename Tin, int OUTK, bool CPLX, int N>
cudaError_t launch_pipe_t(const spod_plan_s& p, const CUtensorMap& xmap, int width, const void* d_X, int64_t m0,
                          int64_t mcount, cudaStream_t s, int* nlaunch) {
  if constexpr (PipeLayout<Tin, 64, N, CPLX>::fits) {
    if (width == 64) return launch_pipe_f<Tin, OUTK, 64, CPLX, N>(p, xmap, d_X, m0, mcount, s, nlaunch);
  }
  if constexpr (PipeLayout<Tin, 32, N, CPLX>::fits) {
    if (width == 32) return launch_pipe_f<Tin, OUTK, 32, CPLX, N>(p, xmap, d_X, m0, mcount, s, nlaunch);
  }
  if (width != 16) return cudaErrorInvalidValue;
  return launch_pipe_f<Tin, OUTK, 16, CPLX, N>(p, xmap, d_X, m0, mcount, s, nlaunch);
}

template <typename Tin, bool CPLX, int N>
cudaError_t launch_pipe_in(const spod_plan_s& p, const CUtensorMap& xmap, int width, const void* d_X, int64_t m0,
                           int64_t mcount, cudaStream_t s, int* nlaunch) {
  if (p.desc.precision == SPOD_PREC_BF16X3)
    return launch_pipe_t<Tin, OUT_BF16X3, CPLX, N>(p, xmap, width, d_X, m0, mcount, s, nlaunch);
  if (p.desc.precision == SPOD_PREC_BF16)
    return launch_pipe_t<Tin, OUT_BF16, CPLX, N>(p, xmap, width, d_X, m0, mcount, s, nlaunch);
  return launch_pipe_t<Tin, OUT_NATIVE, CPLX, N>(p, xmap, width, d_X, m0, mcount, s, nlaunch);
}

// The entry points of one compiled length (PipeLen).
template <int N>
PipeLen pipe_len() {
  PipeLen e;
  e.has = [](const spod_plan_s& p, int tp) {
    switch (p.desc.in_dtype) {
      case SPOD_F64: return pipe_has<double, N, false>(tp);
      case SPOD_F32: return pipe_has<float, N, false>(tp);
      case SPOD_C64: return pipe_has<float, N, true>(tp);
      case SPOD_C128: return pipe_has<double, N, true>(tp);
      default: return pipe_has<__nv_bfloat16, N, false>(tp);
    }
  };
  e.width = [](const spod_plan_s& p, int64_t points) {
    const int64_t pts = p.cplx ? 2 * points : points;       // components
    const int sms = p.num_sms > 0 ? p.num_sms : 148;
    switch (p.desc.in_dtype) {
      case SPOD_F64: return pipe_width_n<double, N, false>(p, pts, sms);
      case SPOD_F32: return pipe_width_n<float, N, false>(p, pts, sms);
      case SPOD_C64: return pipe_width_n<float, N, true>(p, pts, sms);
      case SPOD_C128: return pipe_width_n<double, N, true>(p, pts, sms);
      default: return pipe_width_n<__nv_bfloat16, N, false>(p, pts, sms);
    }
  };
  e.launch = [](const spod_plan_s& p, const CUtensorMap& xmap, int width, const void* d_X, int64_t m0, int64_t mcount,
                cudaStream_t s, int* nlaunch) {
    switch (p.desc.in_dtype) {
      case SPOD_F64: return launch_pipe_in<double, false, N>(p, xmap, width, d_X, m0, mcount, s, nlaunch);
      case SPOD_F32: return launch_pipe_in<float, false, N>(p, xmap, width, d_X, m0, mcount, s, nlaunch);
      case SPOD_C64: return launch_pipe_in<float, true, N>(p, xmap, width, d_X, m0, mcount, s, nlaunch);
      case SPOD_C128: return launch_pipe_in<double, true, N>(p, xmap, width, d_X, m0, mcount, s, nlaunch);
      default: return launch_pipe_in<__nv_bfloat16, false, N>(p, xmap, width, d_X, m0, mcount, s, nlaunch);
    }
  };
  return e;
}

}  // namespace
}  // namespace spod
