// Expansion coefficients and reconstruction ("SPOD for data compression",
// Eqs. coeffs and SPODrec):
//   A = (Phi_r^* W Phi_r)^{-1} Phi_r^* W Q,   Q~ = Phi_r A_r,
// Q = X^T - mu, over the leading nmodes_r modes of the selected one-sided bins
// and, for the bins other than DC and Nyquist, their complex conjugates (the
// modes of the negative frequencies, so that the set is closed under
// conjugation and the reconstruction of real data is real).
//
// The computation runs in the equivalent real basis: the complex span of
// {phi, conj phi} meets the real vectors in the real span of {Re phi, Im phi}
// (DC and Nyquist modes are real), so with the K real basis rows b_r
//   B = P_w X^T - P_w mu 1^T   (P_w rows W b_r; a plain GEMM over the M points),
//   G = P_w P_b^T               (P_b rows b_r; FP64 sums),
//   C = G^{-1} B,
// and a = c_re / 2 - i c_im / 2 for a conjugate pair (a = c_re at DC and
// Nyquist) recovers the complex coefficient of the mode at the positive bin
// (its conjugate bin carries conj(a)).  The reconstruction is
//   X~ = mu + P_b^T C  (real rows [nt][M]).
// The two large products run on k_gemm_f32 (FP32 plans) or k_gemm_simt (FP64), this
// file's SIMT GEMMs; the product over the M points is split over CTAs and the
// parts summed in FP64 in a fixed order.  C = G^{-1} B runs on k_gemm_simt.
#include <algorithm>
#include <vector>

#include "spod_internal.cuh"

namespace spod {
namespace {

struct BasisRow {
  int f, k, part;   // bin, mode, 0: Re phi, 1: Im phi
};

// P_w[r][m] = W_m b_r[m] (Pw may be NULL), P_b[r][m] = b_r[m]; phi is the interleaved complex
// mode array [nf][nmodes][M].
template <typename R>
__global__ void k_coeff_basis(const R* __restrict__ phi, int nmodes, int64_t M, const BasisRow* __restrict__ rows,
                              const R* __restrict__ sqrtW, R* __restrict__ Pw, R* __restrict__ Pb) {
  const int r = blockIdx.y;
  const BasisRow br = rows[r];
  const R* src = phi + ((int64_t)br.f * nmodes + br.k) * M * 2 + br.part;
  for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < M; m += (int64_t)gridDim.x * blockDim.x) {
    const R b = src[2 * m];
    const R sw = sqrtW[m];
    Pb[(int64_t)r * M + m] = b;
    if (Pw) Pw[(int64_t)r * M + m] = b * sw * sw;
  }
}

// G[i][j] = G[j][i] = sum_m P_w[i][m] P_b[j][m] for the 4 x 4 tiles (bi, bj), bi <= bj,
// and, for bj one past the last tile, v[i] = sum_m P_w[i][m] mu[m]; FP64 sums in a
// fixed order (thread t takes m = t, t + 256, ..).  What bounds it: the FP64 pipe.  K = 64,
// M = 65 536: 0.86 ms, against 0.80 with one pair per CTA; but those 4160 CTAs kept the
// product that runs beside it (Fork) off the SMs, and these 152 leave it most of each.
// Fewer rows make fewer tiles than SMs, whose CTAs would then walk all the points one
// FP64 FMA after another while the rest of the chip idles: split z takes the points
// [z mper, (z + 1) mper) and writes part z of G [gridDim.z][K][K] and v [gridDim.z][K],
// which k_spd_inverse adds up in order (coeff_gram_splits says how many).
template <typename R>
__global__ void __launch_bounds__(256) k_coeff_gram(const R* __restrict__ Pw, const R* __restrict__ Pb,
                                                    const double* __restrict__ mu, int64_t M, int64_t mper, int K,
                                                    double* __restrict__ G, double* __restrict__ v) {
  __shared__ double red[16][8];
  const int i0 = 4 * blockIdx.x, j0 = 4 * blockIdx.y;
  if (j0 < i0) return;
  const int64_t m0 = (int64_t)blockIdx.z * mper, m1 = min(M, m0 + mper);
  G += (int64_t)blockIdx.z * K * K;
  v += (int64_t)blockIdx.z * K;
  const bool isv = j0 >= K;
  const R *a[4], *b[4];
  for (int q = 0; q < 4; ++q) {                       // rows past K repeat the last one
    a[q] = Pw + (int64_t)min(i0 + q, K - 1) * M;
    b[q] = Pb + (int64_t)min(j0 + q, K - 1) * M;
  }
  double acc[4][4];
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = 0.0;
  if (!isv) {
    for (int64_t m = m0 + threadIdx.x; m < m1; m += 256) {
      double av[4], bv[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) { av[q] = (double)a[q][m]; bv[q] = (double)b[q][m]; }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = fma(av[x], bv[y], acc[x][y]);
    }
  } else {
    for (int64_t m = m0 + threadIdx.x; m < m1; m += 256) {
      const double c = mu[m];
#pragma unroll
      for (int x = 0; x < 4; ++x) acc[x][0] = fma((double)a[x][m], c, acc[x][0]);
    }
  }
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      double t = acc[x][y];
      for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
      if (lane == 0) red[4 * x + y][w] = t;
    }
  __syncthreads();
  if (threadIdx.x >= 16) return;
  const int i = i0 + (int)threadIdx.x / 4, j = j0 + (int)threadIdx.x % 4;
  double t = 0.0;
  for (int q = 0; q < 8; ++q) t += red[threadIdx.x][q];
  if (isv) {
    if (j == j0 && i < K) v[i] = t;
  } else if (i < K && j < K && i <= j) {
    G[(int64_t)i * K + j] = t;
    G[(int64_t)j * K + i] = t;
  }
}

// Ginv = G^{-1} for the symmetric positive definite G (K x K, FP64) by
// Gauss-Jordan elimination without pivoting (one CTA; G is overwritten).  A
// pivot that is not positive (a basis that is not linearly independent)
// raises FLAG_NOTCONV and leaves Ginv unusable.  G and v come as nparts parts
// (k_coeff_gram), added up first; v's total goes to its first part.  At step c the columns of G up to c
// are those of I already and the columns of Ginv past c still are, so a row is K
// entries: Ginv's up to c and G's past it.  With smem the two matrices are held in
// shared memory (K <= kInvSmemK: the elimination is a chain of K short steps, and
// through L2 each one waited for its loads; K = 64: 0.31 -> 0.16 ms).
constexpr int kInvSmemK = 96;
__global__ void __launch_bounds__(1024) k_spd_inverse(double* __restrict__ Gg, double* __restrict__ v,
                                                      double* __restrict__ Ginv_g, int K, int nparts, int smem,
                                                      unsigned* __restrict__ flags) {
  extern __shared__ double sh[];    // fac [K], then (smem) G and Ginv, rows of K + 1
  double* const fac = sh;
  double* const G = smem ? sh + K : Gg;
  double* const Ginv = smem ? G + (size_t)K * (K + 1) : Ginv_g;
  const int64_t ld = smem ? K + 1 : K;
  const int tid = threadIdx.x, nth = blockDim.x;
  for (int idx = tid; idx < K * K; idx += nth) {
    const int i = idx / K, j = idx - i * K;
    double g = Gg[idx];
    for (int z = 1; z < nparts; ++z) g += Gg[(size_t)z * K * K + idx];
    G[i * ld + j] = g;
    Ginv[i * ld + j] = i == j ? 1.0 : 0.0;
  }
  if (nparts > 1)
    for (int i = tid; i < K; i += nth) {
      double t = v[i];
      for (int z = 1; z < nparts; ++z) t += v[(size_t)z * K + i];
      v[i] = t;
    }
  __syncthreads();
  for (int c = 0; c < K; ++c) {
    const double piv = G[c * ld + c];
    if (!(piv > 0.0)) {
      if (tid == 0) atomicOr(flags, FLAG_NOTCONV);
      return;
    }
    for (int i = tid; i < K; i += nth) fac[i] = G[i * ld + c];
    __syncthreads();
    for (int j = tid; j < K; j += nth) {
      double* const e = (j > c ? G : Ginv) + c * ld + j;
      *e /= piv;
    }
    __syncthreads();
    for (int idx = tid; idx < K * K; idx += nth) {
      const int i = idx / K, j = idx - i * K;
      if (i == c) continue;
      double* const X = j > c ? G : Ginv;
      X[i * ld + j] -= fac[i] * X[c * ld + j];
    }
    __syncthreads();
  }
  if (smem)
    for (int idx = tid; idx < K * K; idx += nth) Ginv_g[idx] = Ginv[(idx / K) * ld + idx % K];
}

// d_A[q][t] (q = j * nmodes_r + k) from the real coefficients C (column-major
// K x nt): a = c[re] (DC, Nyquist) or c[re] / 2 - i c[im] / 2.
__global__ void k_coeff_pack(const double* __restrict__ C, const int2* __restrict__ qrows, int nq, int K,
                             int64_t nt, double2* __restrict__ A) {
  const int q = blockIdx.y;
  const int2 rr = qrows[q];
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nt; t += (int64_t)gridDim.x * blockDim.x) {
    const double cre = C[t * K + rr.x];
    A[(int64_t)q * nt + t] = rr.y < 0 ? make_double2(cre, 0.0) : make_double2(0.5 * cre, -0.5 * C[t * K + rr.y]);
  }
}

// The real coefficients C (column-major K x nt, type R) from d_A.
template <typename R>
__global__ void k_coeff_unpack(const double2* __restrict__ A, const int2* __restrict__ qrows, int K, int64_t nt,
                               R* __restrict__ C) {
  const int q = blockIdx.y;
  const int2 rr = qrows[q];
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nt; t += (int64_t)gridDim.x * blockDim.x) {
    const double2 a = A[(int64_t)q * nt + t];
    if (rr.y < 0) {
      C[t * K + rr.x] = (R)a.x;
    } else {
      C[t * K + rr.x] = (R)(2.0 * a.x);
      C[t * K + rr.y] = (R)(-2.0 * a.y);
    }
  }
}

// Xrec[t][m] = mu[m].
template <typename R>
__global__ void k_fill_mean(const double* __restrict__ mu, int64_t M, int64_t n, R* __restrict__ X) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    X[e] = (R)mu[e % M];
}

// D(i, j) = beta D(i, j) + sum_k A(i, k) B(k, j) over the split's range of k,
// every operand given by element strides: A(i, k) = A[i sai + k sak],
// B(k, j) = B[k sbk + j sbj], D(i, j) = D[i sdi + j sdj].  64 x 64 tiles of D,
// 256 threads with 4 x 4 results each, k in steps of 16 staged in shared
// memory (loads along whichever index is contiguous).  Split z covers
// k in [z kper, (z + 1) kper) and writes D + z dsplit.
template <typename R>
__global__ void __launch_bounds__(256) k_gemm_simt(int ni, int nj, int64_t nk, const R* __restrict__ A, int64_t sai,
                                                   int64_t sak, const R* __restrict__ B, int64_t sbk, int64_t sbj,
                                                   R* __restrict__ D, int64_t sdi, int64_t sdj, int64_t dsplit,
                                                   R beta, int64_t kper) {
  constexpr int TI = 64, TJ = 64, TK = 16;
  __shared__ R As[TK][TI + 4];
  __shared__ R Bs[TK][TJ + 4];
  const int i0 = blockIdx.x * TI, j0 = blockIdx.y * TJ;
  const int64_t k0 = (int64_t)blockIdx.z * kper;
  const int64_t k1 = k0 + kper < nk ? k0 + kper : nk;
  R* Dz = D + (int64_t)blockIdx.z * dsplit;
  const int tid = threadIdx.x;
  // the output index that is contiguous in D varies fastest across threads
  const bool jfast = sdj == 1;
  const int ti = (jfast ? tid / 16 : tid % 16) * 4, tj = (jfast ? tid % 16 : tid / 16) * 4;
  R acc[4][4];
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = (R)0;
  for (int64_t kb = k0; kb < k1; kb += TK) {
    for (int e = tid; e < TI * TK; e += 256) {
      const int kk = sak == 1 ? e % TK : e / TI, ii = sak == 1 ? e / TK : e % TI;
      const int gi = i0 + ii;
      const int64_t gk = kb + kk;
      As[kk][ii] = (gi < ni && gk < k1) ? A[(int64_t)gi * sai + gk * sak] : (R)0;
    }
    for (int e = tid; e < TK * TJ; e += 256) {
      const int kk = sbk == 1 ? e % TK : e / TJ, jj = sbk == 1 ? e / TK : e % TJ;
      const int gj = j0 + jj;
      const int64_t gk = kb + kk;
      Bs[kk][jj] = (gj < nj && gk < k1) ? B[gk * sbk + (int64_t)gj * sbj] : (R)0;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      R a[4], b[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) { a[q] = As[kk][ti + q]; b[q] = Bs[kk][tj + q]; }
#pragma unroll
      for (int x = 0; x < 4; ++x)
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = fma(a[x], b[y], acc[x][y]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int x = 0; x < 4; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) {
      const int gi = i0 + ti + x, gj = j0 + tj + y;
      if (gi < ni && gj < nj) {
        R* d = Dz + (int64_t)gi * sdi + (int64_t)gj * sdj;
        *d = beta == (R)0 ? acc[x][y] : beta * *d + acc[x][y];
      }
    }
}

// The FP32 products: D(i, j) = c(j) + sum_k A(i, k) B(k, j) over the split's range of
// k in ascending order, A(i, k) = A[i sai + k], B(k, j) = B[j ldb + k] (BK) or
// B[k ldb + j], D(i, j) = D[i sdi + j sdj], c(j) = mean[j] rounded (or 0).  64 x 128
// tiles of D, 128 threads with 8 x 8 results each (rows 4 a .. and 32 + 4 a .., columns
// 4 b .. and 64 + 4 b ..: conflict-free 16-byte shared loads), packed FMAs on pairs of
// columns, k in steps of 16 through two shared buffers, the next step's loads in
// registers meanwhile.  VEC: 16-byte loads (strides and bases multiples of 16 bytes).
// What bounds it: FP32 issue (four shared loads and eight duplications for 32 packed
// FMAs).  Same order of the same FMAs as k_gemm_simt, so the same results: K = 64,
// nt = 4096, M = 65 536: 1.87 -> 0.97 ms over
// the points, 1.50 (and 0.46 to fill in the mean) -> 0.66 for the reconstruction.
template <bool BK, bool VEC>
__global__ void __launch_bounds__(128, 3) k_gemm_f32(int ni, int nj, int64_t nk, const float* __restrict__ A,
                                                     int64_t sai, const float* __restrict__ B, int64_t ldb,
                                                     float* __restrict__ D, int64_t sdi, int64_t sdj, int64_t dsplit,
                                                     const double* __restrict__ mean, int64_t kper) {
  constexpr int TI = 64, TJ = 128, TK = 16;
  __shared__ __align__(16) float As[2][TK][TI + 4];
  __shared__ __align__(16) float Bs[2][TK][TJ + 4];
  const int i0 = blockIdx.y * TI, j0 = blockIdx.x * TJ;
  const int64_t k0 = (int64_t)blockIdx.z * kper;
  const int64_t k1 = k0 + kper < nk ? k0 + kper : nk;
  D += (int64_t)blockIdx.z * dsplit;
  const int tid = threadIdx.x;
  const int ta = tid / 16, tb = tid % 16;
  // four consecutive elements p[0 .. 3], those past n (and all of a row not in) as zeros
  auto load4 = [](const float* p, bool in, int64_t n) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (VEC) {
      if (in && n > 0) v = *reinterpret_cast<const float4*>(p);   // n is a multiple of 4
    } else if (in) {
      if (n > 0) v.x = p[0];
      if (n > 1) v.y = p[1];
      if (n > 2) v.z = p[2];
      if (n > 3) v.w = p[3];
    }
    return v;
  };
  float4 pa[2], pb[4];
  auto fetch = [&](int64_t kb) {
    const int q = tid % 4;
    const int64_t k = kb + 4 * q;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int i = i0 + tid / 4 + 32 * r;
      pa[r] = load4(A + (int64_t)i * sai + k, i < ni, k1 - k);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (BK) {
        const int j = j0 + tid / 4 + 32 * r;
        pb[r] = load4(B + (int64_t)j * ldb + k, j < nj, k1 - k);
      } else {
        const int64_t kk = kb + tid / 32 + 4 * r;
        const int j = j0 + 4 * (tid % 32);
        pb[r] = load4(B + kk * ldb + j, kk < k1, nj - j);
      }
    }
  };
  auto put = [&](int s) {
    const int q = 4 * (tid % 4);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int i = tid / 4 + 32 * r;
      As[s][q][i] = pa[r].x; As[s][q + 1][i] = pa[r].y; As[s][q + 2][i] = pa[r].z; As[s][q + 3][i] = pa[r].w;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      if (BK) {
        const int j = tid / 4 + 32 * r;
        Bs[s][q][j] = pb[r].x; Bs[s][q + 1][j] = pb[r].y; Bs[s][q + 2][j] = pb[r].z; Bs[s][q + 3][j] = pb[r].w;
      } else {
        *reinterpret_cast<float4*>(&Bs[s][tid / 32 + 4 * r][4 * (tid % 32)]) = pb[r];
      }
    }
  };
  float2 acc[8][4];
#pragma unroll
  for (int x = 0; x < 8; ++x)
#pragma unroll
    for (int y = 0; y < 4; ++y) acc[x][y] = make_float2(0.f, 0.f);
  int s = 0;
  if (k0 < k1) {
    fetch(k0);
    put(0);
  }
  __syncthreads();
  for (int64_t kb = k0; kb < k1; kb += TK, s ^= 1) {
    const bool more = kb + TK < k1;
    if (more) fetch(kb + TK);
#pragma unroll
    for (int kk = 0; kk < TK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[s][kk][4 * ta]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[s][kk][32 + 4 * ta]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[s][kk][4 * tb]);
      const float4 b1 = *reinterpret_cast<const float4*>(&Bs[s][kk][64 + 4 * tb]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y),
                            make_float2(b1.z, b1.w)};
#pragma unroll
      for (int x = 0; x < 8; ++x) {
        const float2 a2 = make_float2(av[x], av[x]);
#pragma unroll
        for (int y = 0; y < 4; ++y) acc[x][y] = __ffma2_rn(a2, bv[y], acc[x][y]);
      }
    }
    if (more) put(s ^ 1);          // last read a step ago, before the barrier below
    __syncthreads();
  }
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int j = j0 + 64 * h + 4 * tb;
    float c[4];
#pragma unroll
    for (int y = 0; y < 4; ++y) c[y] = mean && j + y < nj ? (float)mean[j + y] : 0.f;
#pragma unroll
    for (int x = 0; x < 8; ++x) {
      const int i = i0 + (x < 4 ? 0 : 28) + 4 * ta + x;
      if (i >= ni) continue;
      const float2 u = acc[x][2 * h], w = acc[x][2 * h + 1];
      const float r[4] = {c[0] + u.x, c[1] + u.y, c[2] + w.x, c[3] + w.y};
      float* const d = D + (int64_t)i * sdi + (int64_t)j * sdj;
      if (VEC && !BK) {            // rows of D (sdj = 1): whole quads, aligned
        if (j < nj) *reinterpret_cast<float4*>(d) = make_float4(r[0], r[1], r[2], r[3]);
      } else {
#pragma unroll
        for (int y = 0; y < 4; ++y)
          if (j + y < nj) d[y * sdj] = r[y];
      }
    }
  }
}

// out[e] = sum_z parts[z][e] (FP64, z in order) - v[e % K]  (B - v 1^T, column-major K x nt)
template <typename R>
__global__ void k_coeff_center_parts(const R* __restrict__ parts, int nsplit, const double* __restrict__ v, int K,
                                     int64_t n, double* __restrict__ out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    double acc = 0.0;
    for (int z = 0; z < nsplit; ++z) acc += (double)parts[(int64_t)z * n + e];
    out[e] = acc - v[e % K];
  }
}

template <typename R>
cudaError_t gemm(int ni, int nj, int64_t nk, const R* A, int64_t sai, int64_t sak, const R* B, int64_t sbk,
                 int64_t sbj, R* D, int64_t sdi, int64_t sdj, R beta, int nsplit, int64_t dsplit, cudaStream_t s) {
  const int64_t kper = ((nk + nsplit - 1) / nsplit + 15) / 16 * 16;
  dim3 grid((unsigned)((ni + 63) / 64), (unsigned)((nj + 63) / 64), (unsigned)nsplit);
  k_gemm_simt<R><<<grid, 256, 0, s>>>(ni, nj, nk, A, sai, sak, B, sbk, sbj, D, sdi, sdj, dsplit, beta, kper);
  return cudaGetLastError();
}

// FP32 form of the products (k_gemm_f32), with 16-byte loads where the sizes, strides
// and bases allow them.
template <bool BK>
cudaError_t gemm_f32(int ni, int nj, int64_t nk, const float* A, int64_t sai, const float* B, int64_t ldb, float* D,
                     int64_t sdi, int64_t sdj, const double* mean, int nsplit, int64_t dsplit, cudaStream_t s) {
  const int64_t kper = ((nk + nsplit - 1) / nsplit + 15) / 16 * 16;
  const dim3 grid((unsigned)((nj + 127) / 128), (unsigned)((ni + 63) / 64), (unsigned)nsplit);
  const uintptr_t bases = reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B) | reinterpret_cast<uintptr_t>(D);
  // rows of A (and of B, or of B and D) in whole quads
  const bool vec = bases % 16 == 0 && sai % 4 == 0 && ldb % 4 == 0 && nk % 4 == 0 && (BK || (nj % 4 == 0 && sdi % 4 == 0));
  if (vec) k_gemm_f32<BK, true><<<grid, 128, 0, s>>>(ni, nj, nk, A, sai, B, ldb, D, sdi, sdj, dsplit, mean, kper);
  else k_gemm_f32<BK, false><<<grid, 128, 0, s>>>(ni, nj, nk, A, sai, B, ldb, D, sdi, sdj, dsplit, mean, kper);
  return cudaGetLastError();
}

bool self_conjugate(int f, int nfft) { return f == 0 || (nfft % 2 == 0 && f == nfft / 2); }

// Basis rows and, per (selected bin, mode), the rows of its real and
// imaginary parts (-1: none).
void basis_rows(const spod_plan_s& p, int nmodes_r, int nsel, const int* h_freqs, std::vector<BasisRow>* rows,
                std::vector<int2>* qrows) {
  for (int j = 0; j < nsel; ++j) {
    for (int k = 0; k < nmodes_r; ++k) {
      const int f = h_freqs[j];
      int2 q;
      q.x = (int)rows->size();
      rows->push_back({f, k, 0});
      q.y = -1;
      if (!self_conjugate(f, p.nfft)) {
        q.y = (int)rows->size();
        rows->push_back({f, k, 1});
      }
      qrows->push_back(q);
    }
  }
}

struct Scratch {
  std::vector<void*> ptrs;
  cudaStream_t s;
  cudaError_t err = cudaSuccess;
  void* get(size_t bytes) {
    void* q = nullptr;
    if (err == cudaSuccess) err = cudaMallocAsync(&q, bytes, s);
    if (err == cudaSuccess) ptrs.push_back(q);
    return q;
  }
  ~Scratch() {
    for (void* q : ptrs) cudaFreeAsync(q, s);
  }
};

// The Gram and its inverse beside the product over the points: they keep the FP64
// pipe and one SM busy, the product the FP32 pipe, and neither needs the other
// (K = 64, nt = 4096, M = 65 536: 0.86 + 0.16 ms beside 0.97).  The side stream is the
// plan's copy stream, joined again whatever happens, before the scratch is given
// back; a call under stream capture stays on its own stream.
struct Fork {
  cudaStream_t s = nullptr, side = nullptr;
  cudaEvent_t ev = nullptr;
  bool open = false;
  // the stream to run beside s on (s itself when there is none to fork to)
  cudaStream_t begin(spod_plan_s& p, cudaStream_t s_) {
    s = s_;
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone) {
      cudaGetLastError();
      return s;
    }
    if (!p.h2d_stream && cudaStreamCreateWithFlags(&p.h2d_stream, cudaStreamNonBlocking) != cudaSuccess) {
      cudaGetLastError();
      p.h2d_stream = nullptr;
      return s;
    }
    if (p.host_ev.empty()) {
      if (cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) != cudaSuccess) {
        cudaGetLastError();
        return s;
      }
      p.host_ev.push_back(ev);
    }
    ev = p.host_ev[0];
    side = p.h2d_stream;
    if (cudaEventRecord(ev, s) != cudaSuccess || cudaStreamWaitEvent(side, ev, 0) != cudaSuccess) {
      cudaGetLastError();
      return s;
    }
    open = true;
    return side;
  }
  cudaError_t join() {
    if (!open) return cudaSuccess;
    open = false;
    cudaError_t e = cudaEventRecord(ev, side);
    return e == cudaSuccess ? cudaStreamWaitEvent(s, ev, 0) : e;
  }
  ~Fork() { join(); }
};

// P_w (unless Pw is NULL) and P_b (K x M, type R) of the selected modes.
template <typename R>
cudaError_t build_basis(const spod_plan_s& p, const void* d_Phi, int nmodes, const std::vector<BasisRow>& rows,
                        Scratch& sc, R** Pw, R** Pb, cudaStream_t s) {
  const int K = (int)rows.size();
  const int64_t M = p.M;
  BasisRow* d_rows = static_cast<BasisRow*>(sc.get(sizeof(BasisRow) * K));
  if (Pw) *Pw = static_cast<R*>(sc.get(sizeof(R) * (size_t)K * M));
  *Pb = static_cast<R*>(sc.get(sizeof(R) * (size_t)K * M));
  if (sc.err != cudaSuccess) return sc.err;
  cudaError_t e = cudaMemcpyAsync(d_rows, rows.data(), sizeof(BasisRow) * K, cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)std::min<int64_t>((M + 255) / 256, 1024), (unsigned)K);
  k_coeff_basis<R><<<grid, 256, 0, s>>>(static_cast<const R*>(d_Phi), nmodes, M, d_rows,
                                        static_cast<const R*>(p.d_sqrtW), Pw ? *Pw : nullptr, *Pb);
  return cudaGetLastError();
}

// Parts of the basis Gram's sums over the points: as many as fill the SMs with the
// tiles' CTAs, of at least 1024 points each (four a thread).  One from K = 41 on (152
// SMs), where the tiles alone do.  spod_coeffs, M = 262 144, nt = 300: K = 4 1.77 ms with
// one part, 0.52 so; K = 16 1.81 and 0.53; K = 32 1.88 and 1.08.
int coeff_gram_splits(int K, int64_t M, int sms) {
  const int kt = (K + 3) / 4, tiles = kt * (kt + 1) / 2 + kt;
  return (int)std::max<int64_t>(1, std::min<int64_t>(sms / tiles, M / 1024));
}

template <typename R>
cudaError_t coeffs_t(spod_plan_s& p, const void* d_X, const void* d_Phi, int nmodes, int nmodes_r, int nsel,
                     const int* h_freqs, double* d_A, cudaStream_t s) {
  std::vector<BasisRow> rows;
  std::vector<int2> qrows;
  basis_rows(p, nmodes_r, nsel, h_freqs, &rows, &qrows);
  const int K = (int)rows.size();
  const int64_t M = p.M, nt = p.nt;
  Scratch sc;
  sc.s = s;
  R *Pw = nullptr, *Pb = nullptr;
  cudaError_t e = build_basis<R>(p, d_Phi, nmodes, rows, sc, &Pw, &Pb, s);
  if (e != cudaSuccess) return e;
  // the product over the M points, split so that 64 x 64 tiles cover the GPU four times.
  // (k_gemm_f32's are 64 x 128, half as many: K = 64, nt = 4096 320 CTAs where 456 fit.
  // The count is kept because the parts are FP32 sums: another one rounds otherwise.)
  const int tiles = ((K + 63) / 64) * (int)((nt + 63) / 64);
  const int nsplit = (int)std::max<int64_t>(1, std::min<int64_t>({64, (4 * p.num_sms + tiles - 1) / tiles, M / 1024}));
  R* B = static_cast<R*>(sc.get(sizeof(R) * (size_t)K * nt * nsplit));
  double* B64 = static_cast<double*>(sc.get(sizeof(double) * (size_t)K * nt));
  double* C = static_cast<double*>(sc.get(sizeof(double) * (size_t)K * nt));
  const int nz = coeff_gram_splits(K, M, p.num_sms);
  double* G = static_cast<double*>(sc.get(sizeof(double) * (size_t)nz * K * K));
  double* Ginv = static_cast<double*>(sc.get(sizeof(double) * (size_t)K * K));
  double* v = static_cast<double*>(sc.get(sizeof(double) * (size_t)nz * K));
  int2* d_q = static_cast<int2*>(sc.get(sizeof(int2) * qrows.size()));
  if (sc.err != cudaSuccess) return sc.err;
  e = cudaMemcpyAsync(d_q, qrows.data(), sizeof(int2) * qrows.size(), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  // B = P_w X^T (column-major K x nt; X[t][m]), per split of the points, then B - v 1^T in FP64
  auto product = [&]() {
    if constexpr (sizeof(R) == 4)
      return gemm_f32<true>(K, (int)nt, M, Pw, M, static_cast<const float*>(d_X), M, B, 1, K, nullptr, nsplit,
                            (int64_t)K * nt, s);
    else
      return gemm<R>(K, (int)nt, M, Pw, M, 1, static_cast<const R*>(d_X), 1, M, B, 1, K, (R)0, nsplit,
                     (int64_t)K * nt, s);
  };
  // G and v, and G^{-1}, beside the product.  In FP64 the product goes first: both take
  // the FP64 pipe, and the Gram's CTAs, placed before it, leave the product's unevenly
  // spread (K = 16, nt = 768, M = 16 384: 2.46 ms, 2.26 so; K = 64, nt = 256: 2.00 and 1.69).
  Fork fork;
  cudaStream_t sg = fork.begin(p, s);
  if (sizeof(R) == 8 && (e = product()) != cudaSuccess) return e;
  const unsigned kt = (unsigned)((K + 3) / 4);
  k_coeff_gram<R><<<dim3(kt, kt + 1, (unsigned)nz), 256, 0, sg>>>(Pw, Pb, p.d_mu, M, (M + nz - 1) / nz, K, G, v);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  const int inv_smem = K <= kInvSmemK;
  const size_t inv_bytes = sizeof(double) * ((size_t)K + (inv_smem ? 2 * (size_t)K * (K + 1) : 0));
  e = allow_smem(k_spd_inverse, inv_bytes);
  if (e != cudaSuccess) return e;
  k_spd_inverse<<<1, 1024, inv_bytes, sg>>>(G, v, Ginv, K, nz, inv_smem, p.d_flags);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (sizeof(R) == 4 && (e = product()) != cudaSuccess) return e;
  if ((e = fork.join()) != cudaSuccess) return e;
  k_coeff_center_parts<R><<<1024, 256, 0, s>>>(B, nsplit, v, K, (int64_t)K * nt, B64);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  // C = G^{-1} (B - v 1^T)  (FP64, column-major K x nt)
  e = gemm<double>(K, (int)nt, K, Ginv, K, 1, B64, 1, K, C, 1, K, 0.0, 1, 0, s);
  if (e != cudaSuccess) return e;
  dim3 pg((unsigned)std::min<int64_t>((nt + 255) / 256, 1024), (unsigned)qrows.size());
  k_coeff_pack<<<pg, 256, 0, s>>>(C, d_q, (int)qrows.size(), K, nt, reinterpret_cast<double2*>(d_A));
  return cudaGetLastError();
}

template <typename R>
cudaError_t reconstruct_t(spod_plan_s& p, const void* d_Phi, int nmodes, int nmodes_r, int nsel, const int* h_freqs,
                          const double* d_A, void* d_Xrec, cudaStream_t s) {
  std::vector<BasisRow> rows;
  std::vector<int2> qrows;
  basis_rows(p, nmodes_r, nsel, h_freqs, &rows, &qrows);
  const int K = (int)rows.size();
  const int64_t M = p.M, nt = p.nt;
  Scratch sc;
  sc.s = s;
  R* Pb = nullptr;
  cudaError_t e = build_basis<R>(p, d_Phi, nmodes, rows, sc, nullptr, &Pb, s);
  if (e != cudaSuccess) return e;
  R* C = static_cast<R*>(sc.get(sizeof(R) * (size_t)K * nt));
  int2* d_q = static_cast<int2*>(sc.get(sizeof(int2) * qrows.size()));
  if (sc.err != cudaSuccess) return sc.err;
  e = cudaMemcpyAsync(d_q, qrows.data(), sizeof(int2) * qrows.size(), cudaMemcpyHostToDevice, s);
  if (e != cudaSuccess) return e;
  dim3 pg((unsigned)std::min<int64_t>((nt + 255) / 256, 1024), (unsigned)qrows.size());
  k_coeff_unpack<R><<<pg, 256, 0, s>>>(reinterpret_cast<const double2*>(d_A), d_q, K, nt, C);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  R* X = static_cast<R*>(d_Xrec);
  // X[t][m] = mu[m] + sum_r C[t][r] P_b[r][m]  (C column-major K x nt, P_b rows of M)
  if constexpr (sizeof(R) == 4) {
    return gemm_f32<false>((int)nt, (int)M, K, C, K, Pb, M, X, M, 1, p.d_mu, 1, 0, s);
  } else {
    k_fill_mean<R><<<2048, 256, 0, s>>>(p.d_mu, M, M * nt, X);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    return gemm<R>((int)nt, (int)M, K, C, K, 1, Pb, M, 1, X, M, 1, (R)1, 1, 0, s);
  }
}

}  // namespace

int coeff_basis_size(const spod_plan_s& p, int nmodes_r, int nsel, const int* h_freqs) {
  int K = 0;
  for (int j = 0; j < nsel; ++j) K += nmodes_r * (self_conjugate(h_freqs[j], p.nfft) ? 1 : 2);
  return K;
}

cudaError_t launch_coeffs(spod_plan_s& p, const void* d_X, const void* d_Phi, int nmodes, int nmodes_r, int nsel,
                          const int* h_freqs, double* d_A, cudaStream_t s) {
  return p.f64 ? coeffs_t<double>(p, d_X, d_Phi, nmodes, nmodes_r, nsel, h_freqs, d_A, s)
               : coeffs_t<float>(p, d_X, d_Phi, nmodes, nmodes_r, nsel, h_freqs, d_A, s);
}

cudaError_t launch_reconstruct(spod_plan_s& p, const void* d_Phi, int nmodes, int nmodes_r, int nsel,
                               const int* h_freqs, const double* d_A, void* d_Xrec, cudaStream_t s) {
  return p.f64 ? reconstruct_t<double>(p, d_Phi, nmodes, nmodes_r, nsel, h_freqs, d_A, d_Xrec, s)
               : reconstruct_t<float>(p, d_Phi, nmodes, nmodes_r, nsel, h_freqs, d_A, d_Xrec, s);
}

}  // namespace spod
