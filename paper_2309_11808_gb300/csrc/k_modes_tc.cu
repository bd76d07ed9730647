// SPOD modes on the tensor cores (Eq. spod-discrete-snapshots):
// Phi_f[:, k] = Qhat_f psi_k / sqrt(lambda_k / kappa), divided by sqrt(W_m)
// because Qhat carries sqrt(W_m).
//
// Real embedding, per frequency f and tile of 128 points (two 64-point blocks
// of the blocked Qhat layout):
//   D[128 points x NN] = A[128 x K] * B[NN x K]^T,  K = 2 nb (padded to 16)
// A is MN-major: the two TMA boxes of Qhat (K rows x 64 points each) side by
// side.  B (K-major, 128-byte swizzle) is a per-frequency image built once per
// call in global memory (k_mode_image) and copied into shared memory by one
// bulk copy whenever a CTA moves to the next frequency: row 2k holds
// [Re B_f[:, k] ; -Im B_f[:, k]], row 2k+1 holds [Im B_f[:, k] ; Re B_f[:, k]],
// B_f = Psi_f Lambda_f^{-1/2} sqrt(kappa), so D[p][2k] = Re Phi[p][k] and
// D[p][2k+1] = Im Phi[p][k]: each TMEM lane (one point) holds interleaved
// complex outputs, stored straight from registers as 8-byte values, 256
// contiguous bytes per warp and mode.  BF16X3 adds A_hi B_lo + A_lo B_hi.
// With B = G_f and scale sqrt(W) the same kernel computes W Qhat G_f for the
// adjoint.
//
// Persistent CTAs (one per SM) walk a contiguous range of the f-major list of
// (frequency, group of 128-point tiles) items.  Warp roles (576 threads): warp 16
// issues TMA (and the B image copy at each frequency change), warp 17 issues the
// MMAs into four TMEM accumulators, four groups of four warps (one warp per
// lane quadrant) drain the items in turn.  Every wait is bounded.
//
// What bounds it: HBM (Qhat read, Phi written), as long as enough bytes are in
// flight and no tile waits for a hand-over.  Hence items of about 32 KB whatever
// nb is, one hand-over per item, sixteen draining warps, and issuing warps that run
// as whole warps (elect_one): 361 x 720 x 2 points, 361 bins, nb = 7, three modes
// 10.7 -> 2.4 ms (6.4 TB/s); nb = 21, 193 bins, five modes 6.1 -> 3.3 ms; BF16, nb = 33,
// 129 bins, five modes 4.2 -> 1.7 ms; 512 x 256 x 3 points, nb = 38, five modes
// 6.5 -> 5.1 ms (6.9 TB/s).
#include <algorithm>

#include "tc_common.cuh"

namespace spod {
namespace {

constexpr int kMaxStages = 8;            // pipeline depth (fewer when shared memory is short)
constexpr int kStageTarget = 32 * 1024;  // bytes of an item's stage: as many 128-point tiles as fit (at least one)
constexpr int kMaxTiles = 8;             // 128-point tiles per item at most
constexpr int kMaxImageModes = 128;      // modes of one image (nmodes <= nb; the tensor path keeps 2 nb <= 128)
constexpr int kAcc = 4;                   // TMEM accumulators, 128 columns apart (all tiles of an item)
constexpr uint32_t kTmemCols = kAcc * 128;
constexpr int kEpiWarps = 16;
constexpr int kEpiGroups = kEpiWarps / 4;
constexpr int kEpiThreads = 4 * 32;                // one group of four warps drains an item
constexpr int kTmaWarp = kEpiWarps, kMmaWarp = kEpiWarps + 1;
constexpr int kThreadsModes = (kEpiWarps + 2) * 32;

struct ModesTcArgs {
  int nb, nmodes, np, nn, nf;             // np = K (2 nb padded to 16), nn = N (2 nmodes padded to 16)
  int64_t mcount, m0, M;                  // M: row stride of Phi in points
  int64_t phioff;                          // point of Phi's first column (tiled output)
  int64_t ntp;                             // 128-point tiles per frequency
  int64_t nit;                             // items (of `tiles` tiles) per frequency
  int tiles;                               // 128-point tiles per item
  int64_t qtile0;                          // first 128-point tile of the call inside the Qhat chunk
  int64_t nitems;                          // (f1 - f0) * nit
  int f0;                                  // first frequency of the call's range
  uint32_t box_bytes;                      // one Qhat TMA box: np rows x 128 bytes
  uint32_t img_bytes;                      // one B image (hi or lo)
  int nst;                                 // pipeline stages (2 .. kMaxStages)
};

struct ModesHdr {
  uint64_t full[kMaxStages], empty[kMaxStages], accfull[kAcc], accempty[kAcc], bfull, bempty, drain;
  uint32_t tmem_base;
  int abort;
};

__device__ __forceinline__ uint32_t sw128_offset(int r, int kk) {
  // byte offset of BF16 element (row r, k index kk < 64) in a K-major 128-byte-swizzled atom stack
  return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((((kk * 2) >> 4) ^ (r & 7)) << 4) + ((kk * 2) & 15));
}

// 1-D bulk copy global -> shared with mbarrier completion (16-byte aligned, size a multiple of 16).
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(bar)
               : "memory");
}

// 8 consecutive TMEM columns of this thread's lane (no wait).
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// B image of frequency f: rows n < nn (2k: real part of mode k, 2k+1: imaginary
// part), K index kk < np (l: Re Qhat row l, nb + l: Im Qhat row l), BF16 hi
// (and lo = bf16(v - hi)), K-major 128-byte-swizzled atoms of 64 K values.
__global__ void k_mode_image(const float* __restrict__ bmat, int nb, int nm, int np, int nn, int x3,
                             const double* __restrict__ what, uint32_t img_bytes, uint8_t* __restrict__ img) {
  const int f = blockIdx.x;
  const float* Bf = bmat + (size_t)f * nb * nm * 2;
  // folded mean: the correction row's entries -What_f c_k, c_k = sum_l B_f[l][k],
  // one thread per mode (FP64 sums of the FP32 coefficients), before the image loop
  __shared__ float2 corr[kMaxImageModes];
  if (what) {
    const double wr = what[2 * f], wi = what[2 * f + 1];
    for (int k = threadIdx.x; k < nm; k += blockDim.x) {
      double cr = 0.0, ci = 0.0;
      for (int l = 0; l < nb; ++l) {
        cr += (double)Bf[(l * nm + k) * 2];
        ci += (double)Bf[(l * nm + k) * 2 + 1];
      }
      corr[k] = make_float2((float)-(wr * cr - wi * ci), (float)-(wr * ci + wi * cr));
    }
    __syncthreads();
  }
  uint8_t* hi = img + (size_t)f * img_bytes * (x3 ? 2 : 1);
  uint8_t* lo = hi + img_bytes;
  const int katoms = (np + 63) / 64;
  for (int e = threadIdx.x; e < nn * katoms * 64; e += blockDim.x) {
    const int n = e / (katoms * 64);
    const int kk = e - n * (katoms * 64);
    const int k = n >> 1;
    float v = 0.f;
    if (kk < 2 * nb && k < nm) {
      const int l = kk < nb ? kk : kk - nb;
      const float br = Bf[(l * nm + k) * 2], bi = Bf[(l * nm + k) * 2 + 1];
      if ((n & 1) == 0) v = kk < nb ? br : -bi;
      else v = kk < nb ? bi : br;
    } else if (what && kk == 2 * nb && k < nm) {
      // folded mean: Qhat rows are the spectra Z of x - c, row 2 nb is rho; the
      // spectra of x - mu are Z - rho What_f, so column k gains -rho What_f c_k
      v = (n & 1) == 0 ? corr[k].x : corr[k].y;
    }
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    const uint32_t off = (uint32_t)(kk >> 6) * (uint32_t)(nn * 128) + sw128_offset(n, kk & 63);
    *reinterpret_cast<__nv_bfloat16*>(hi + off) = h;
    if (x3) *reinterpret_cast<__nv_bfloat16*>(lo + off) = __float2bfloat16_rn(v - __bfloat162float(h));
  }
}

// Position of a CTA's item in the (frequency, tile) list and in the stage
// ring, advanced without divisions (the issuing threads are on the critical
// path of every item).
struct Cursor {
  int f, tp;          // frequency, item (group of tiles) within it
  int s, ph;          // stage, parity of the ring pass (i / nst) & 1
  __device__ __forceinline__ void init(int64_t item0, int ntp, int f0) {
    const int fr = (int)(item0 / ntp);
    tp = (int)(item0 - (int64_t)fr * ntp);
    f = f0 + fr;
    s = 0;
    ph = 0;
  }
  __device__ __forceinline__ void next(int ntp, int nst) {
    if (++tp == ntp) { tp = 0; ++f; }
    if (++s == nst) { s = 0; ph ^= 1; }
  }
};

template <bool X3>
__global__ void __launch_bounds__(kThreadsModes, 1) k_modes_tc(const __grid_constant__ CUtensorMap map_hi,
                                                    const __grid_constant__ CUtensorMap map_lo, ModesTcArgs a,
                                                    const uint8_t* __restrict__ img, const float* __restrict__ scale,
                                                    float2* __restrict__ phi, unsigned* __restrict__ gflags) {
  using namespace tc;
  constexpr int NOPS = X3 ? 2 : 1;
  extern __shared__ unsigned char smem_raw[];
  uint8_t* sm = smem_align1024(smem_raw);
  ModesHdr* hdr = reinterpret_cast<ModesHdr*>(sm);
  uint8_t* Bhi = sm + 1024;
  uint8_t* Blo = Bhi + a.img_bytes;
  const uint32_t tile_bytes = 2u * a.box_bytes;           // a tile's two 64-point boxes of one operand
  const uint32_t op_bytes = tile_bytes * a.tiles;
  const uint32_t stage_bytes = op_bytes * NOPS;           // [hi tiles][lo tiles]
  uint8_t* stages = Bhi + NOPS * a.img_bytes;
  const uint32_t stage0 = smem_u32(stages);

  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;
  const int64_t i0 = a.nitems * blockIdx.x / gridDim.x;
  const int64_t i1 = a.nitems * (blockIdx.x + 1) / gridDim.x;
  const int nit = (int)(i1 - i0);
  const int ntp = (int)a.ntp, nitf = (int)a.nit, T = a.tiles;

  if (tid == 0) {
    for (int i = 0; i < a.nst; ++i) {
      mbar_init(smem_u32(&hdr->full[i]), 1);
      mbar_init(smem_u32(&hdr->empty[i]), 1);
    }
    for (int i = 0; i < kAcc; ++i) {
      mbar_init(smem_u32(&hdr->accfull[i]), 1);
      mbar_init(smem_u32(&hdr->accempty[i]), kEpiThreads);
    }
    mbar_init(smem_u32(&hdr->bfull), 1);
    mbar_init(smem_u32(&hdr->bempty), 1);
    mbar_init(smem_u32(&hdr->drain), 1);
    hdr->abort = 0;
    fence_mbar_init();
  }
  if (warp == kMmaWarp) {
    tmem_alloc(smem_u32(&hdr->tmem_base), kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, hdr->tmem_base, 0);
  volatile int* abort_flag = &hdr->abort;

  if (warp == kTmaWarp && nit > 0) {
    // ---------------- TMA producer (+ B image at each frequency change)
    const bool leader = elect_one();
    if (leader) {
      prefetch_tmap(&map_hi);
      if (X3) prefetch_tmap(&map_lo);
    }
    int issued = 0, seg = 0, segs_loaded = 0;
    int fcur = -1;
    Cursor cu;
    cu.init(i0, nitf, a.f0);
    for (int i = 0; i < nit; ++i, cu.next(nitf, a.nst)) {
      const int f = cu.f, tp = cu.tp;
      if (f != fcur) {
        // the MMAs of the previous frequency must be done with B before it is replaced
        if (seg >= 1 && !mbar_wait_warp(smem_u32(&hdr->bempty), (seg - 1) & 1, abort_flag, gflags)) break;
        const uint32_t bb = smem_u32(&hdr->bfull);
        const uint8_t* src = img + (size_t)f * a.img_bytes * NOPS;
        if (leader) {
          mbar_arrive_expect_tx(bb, a.img_bytes * NOPS);
          bulk_load(smem_u32(Bhi), src, a.img_bytes, bb);
          if (X3) bulk_load(smem_u32(Blo), src + a.img_bytes, a.img_bytes, bb);
        }
        __syncwarp();
        segs_loaded = seg + 1;
        fcur = f;
        ++seg;
      }
      const int s = cu.s;
      if (i >= a.nst && !mbar_wait_warp(smem_u32(&hdr->empty[s]), cu.ph ^ 1, abort_flag, gflags)) break;
      const uint32_t fb = smem_u32(&hdr->full[s]);
      const uint32_t st = stage0 + (uint32_t)s * stage_bytes;
      const int kb = 2 * (tp * T + (int)a.qtile0);
      // one copy per operand: the item's 64-point blocks side by side
      if (leader) {
        mbar_arrive_expect_tx(fb, stage_bytes);
        tma_load_4d(st, &map_hi, 0, 0, f, kb, fb);
        if (X3) tma_load_4d(st + op_bytes, &map_lo, 0, 0, f, kb, fb);
      }
      __syncwarp();
      issued = i + 1;
    }
    // copies still in flight must land before the CTA can exit
    for (int i = max(0, issued - a.nst); i < issued; ++i)
      mbar_drain(smem_u32(&hdr->full[i % a.nst]), (i / a.nst) & 1, gflags);
    if (segs_loaded > 0) mbar_drain(smem_u32(&hdr->bfull), (segs_loaded - 1) & 1, gflags);
  } else if (warp == kMmaWarp && nit > 0) {
    // ---------------- MMA issuer
    const uint32_t idesc = idesc_bf16(128, a.nn, 1, 0);      // A MN-major (points), B K-major
    const uint32_t bhi = smem_u32(Bhi), blo = smem_u32(Blo);
    const bool leader = elect_one();
    const uint32_t katom_bytes = (uint32_t)a.nn * 128u;
    const int nk16 = a.np / 16;
    int seg = 0;
    int fcur = -1;
    Cursor cu;
    cu.init(i0, nitf, a.f0);
    for (int i = 0; i < nit; ++i, cu.next(nitf, a.nst)) {
      const int f = cu.f;
      if (f != fcur) {
        if (seg >= 1 && leader) mma_commit(smem_u32(&hdr->bempty));   // B of the previous frequency is released
        if (!mbar_wait_warp(smem_u32(&hdr->bfull), seg & 1, abort_flag, gflags)) break;
        fcur = f;
        ++seg;
      }
      const int s = cu.s;
      if (!mbar_wait_warp(smem_u32(&hdr->full[s]), cu.ph, abort_flag, gflags)) break;
      tc_fence_after();
      const uint32_t st = stage0 + (uint32_t)s * stage_bytes;
      const int acc = i % kAcc;
      if (i >= kAcc && !mbar_wait_warp(smem_u32(&hdr->accempty[acc]), (i / kAcc - 1) & 1, abort_flag, gflags)) break;
      tc_fence_after();
      const int nv = min(T, ntp - cu.tp * T);
      if (leader) {
        for (int t = 0; t < nv; ++t) {
          const uint32_t d = tmem + (uint32_t)(acc * 128 + t * a.nn);
          // A: 16 K rows of both point boxes (MN atoms box_bytes apart); B: 16 K columns
          const uint64_t da0 = sdesc_sw128(st + (uint32_t)t * tile_bytes, a.box_bytes, 1024);
          const uint64_t dl0 = sdesc_sw128(st + (uint32_t)t * tile_bytes + op_bytes, a.box_bytes, 1024);
          for (int j = 0; j < nk16; ++j) {
            const uint64_t da = da0 + (uint64_t)(j * 128), dal = dl0 + (uint64_t)(j * 128);      // 2048 bytes
            const uint32_t boff = (uint32_t)(j >> 2) * katom_bytes + (uint32_t)(j & 3) * 32u;
            const uint64_t db = sdesc_sw128(bhi + boff, 16, 1024);
            mma_bf16(d, da, db, idesc, j > 0 ? 1u : 0u);
            if (X3) {
              const uint64_t dbl = sdesc_sw128(blo + boff, 16, 1024);
              mma_bf16(d, da, dbl, idesc, 1u);
              mma_bf16(d, dal, db, idesc, 1u);
            }
          }
        }
        mma_commit(smem_u32(&hdr->empty[s]));
        mma_commit(smem_u32(&hdr->accfull[acc]));
      }
      __syncwarp();
    }
    if (leader) {
      mma_commit(smem_u32(&hdr->drain));
      mbar_drain(smem_u32(&hdr->drain), 0, gflags);
    }
    __syncwarp();
  } else if (warp < kEpiWarps) {
    // ---------------- epilogue: TMEM -> registers -> scaled complex stores.
    // Groups of four warps (one per lane quadrant) take the CTA's items in turn;
    // a warp takes all columns of its 32 points of every tile of the item.
    const int quad = warp & 3, grp = warp >> 2;
    const int nm = a.nmodes;
    const int plane = quad * 32 + lane;                // point of the tile
    auto load_scale = [&](int tile) {
      const int64_t lm = (int64_t)tile * 128 + plane;
      return lm < a.mcount ? scale[a.m0 + lm] : 0.f;
    };
    int f = a.f0 + (int)(i0 / a.nit), tp = (int)(i0 % a.nit);
    auto advance = [&](int n) {
      tp += n;
      while (tp >= nitf) { tp -= nitf; ++f; }
    };
    advance(grp);
    float rw = grp < nit ? load_scale(tp * T) : 0.f;
    for (int i = grp; i < nit; i += kEpiGroups) {
      const int acc = i % kAcc;
      const int tile0 = tp * T, nv = min(T, ntp - tile0);
      float2* const of = phi + (int64_t)f * nm * a.M + (a.m0 - a.phioff);
      advance(kEpiGroups);
      // one decision per warp: the tcgen05.ld below must be executed by the whole warp
      const bool got = mbar_wait(smem_u32(&hdr->accfull[acc]), (i / kAcc) & 1, abort_flag, gflags);
      if (!__all_sync(0xffffffffu, got)) break;
      tc_fence_after();
      for (int t = 0; t < nv; ++t) {
        const int64_t lm = (int64_t)(tile0 + t) * 128 + plane;
        const bool inrange = lm < a.mcount;
        const bool last = t + 1 == nv;
        // the next tile's output scale: its latency overlaps this tile's work
        const float rw_next = !last ? load_scale(tile0 + t + 1)
                              : i + kEpiGroups < nit ? load_scale(tp * T) : 0.f;
        uint32_t taddr = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)(acc * 128 + t * a.nn);
        float2* out = of + lm;
        for (int c0 = 0; c0 < 2 * nm; c0 += 32) {      // 16 modes at a time
          float v[32];
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (c0 + c * 8 < 2 * nm) tmem_ld8(taddr + (uint32_t)(c0 + c * 8), v + c * 8);
          tmem_wait_ld();
          if (last && c0 + 32 >= 2 * nm) {
            tc_fence_before();
            mbar_arrive(smem_u32(&hdr->accempty[acc]));
          }
#pragma unroll
          for (int c = 0; c < 4; ++c)
            if (c0 + c * 8 < 2 * nm) {                 // four modes
              tmem_loaded<8>(v + c * 8);
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                if (inrange && c0 / 2 + c * 4 + j < nm) *out = make_float2(v[8 * c + 2 * j] * rw, v[8 * c + 2 * j + 1] * rw);
                out += a.M;
              }
            }
        }
        rw = rw_next;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

int modes_np(const spod_plan_s& p) { return (2 * p.nb + 15) / 16 * 16; }
int modes_nn(int nmodes) { return (2 * nmodes + 15) / 16 * 16; }
uint32_t modes_img_bytes(int np, int nn) { return (uint32_t)((np + 63) / 64) * (uint32_t)nn * 128u; }

// 128-point tiles per item: a stage of about kStageTarget bytes.  One tile of
// 16 rows (nb = 7) is 8 KB of hi and lo; with one tile per item and four
// stages 32 KB were in flight per SM and every tile cost a hand-over.
// An item's tiles share one accumulator buffer of 128 columns and one hand-over.
// No more tiles an item than leave every CTA one (ntiles tiles in all): BF16, nb = 1,
// 1001 points, 33 bins took 16.4 us a call as 33 items of eight tiles, 14.4 as 264 of one.
int modes_tiles(const spod_plan_s& p, int nn, int64_t ntiles, int64_t ctas) {
  const int nops = p.desc.precision == SPOD_PREC_BF16X3 ? 2 : 1;
  const int fit = std::min({kMaxTiles, kStageTarget / (2 * modes_np(p) * 128 * nops), 128 / nn});
  return (int)std::max<int64_t>(1, std::min<int64_t>(fit, ntiles / ctas));
}

size_t modes_tc_smem_stages(const spod_plan_s& p, int nst, int tiles) {
  const int nops = p.desc.precision == SPOD_PREC_BF16X3 ? 2 : 1;
  const int np = modes_np(p);
  const size_t img = modes_img_bytes(np, modes_nn(std::max(p.nb, p.adj_cols)));   // the adjoint's extra column
  const size_t box = (size_t)np * 128;
  return 1024 + 1024 + nops * img + (size_t)nst * tiles * 2 * box * nops;
}

}  // namespace

// Shared memory of the smallest (2-stage) configuration; launches use up to kMaxStages.
size_t modes_tc_smem_bytes(const spod_plan_s& p) { return modes_tc_smem_stages(p, 2, 1); }

// Per-frequency B images (hi [, lo]) for nmodes columns, in the plan's image buffer.
size_t modes_image_bytes(const spod_plan_s& p) {
  const int nops = p.desc.precision == SPOD_PREC_BF16X3 ? 2 : 1;
  return (size_t)p.nf * nops * modes_img_bytes(modes_np(p), modes_nn(std::max(p.nb, p.adj_cols)));
}

cudaError_t launch_mode_image(const spod_plan_s& p, int nmodes, cudaStream_t s) {
  const int np = modes_np(p), nn = modes_nn(nmodes);
  if (nmodes > kMaxImageModes) return cudaErrorInvalidValue;
  k_mode_image<<<p.nf, 256, 0, s>>>(static_cast<const float*>(p.d_bmat), p.nb, nmodes, np, nn,
                                    p.desc.precision == SPOD_PREC_BF16X3 ? 1 : 0,
                                    p.mean_fold ? p.d_what : nullptr, modes_img_bytes(np, nn),
                                    static_cast<uint8_t*>(p.d_bimg));
  return cudaGetLastError();
}

cudaError_t launch_modes_tc_chunk(const spod_plan_s& p, int64_t m0, int64_t mcount, int nmodes, void* d_Phi,
                                  cudaStream_t s, bool adjoint, int f0, int f1, int64_t qoff, int64_t out_ld,
                                  int64_t out_off) {
  if (qoff % 128 != 0) return cudaErrorInvalidValue;
  if (f1 < 0) f1 = p.nf;
  if (f0 < 0 || f1 > p.nf || f0 >= f1) return cudaErrorInvalidValue;
  const float* scale = static_cast<const float*>(adjoint ? p.d_sqrtW : p.d_rsqrtW);
  ModesTcArgs a;
  a.nb = p.nb;
  a.nmodes = nmodes;
  a.np = modes_np(p);
  a.nn = modes_nn(nmodes);
  a.nf = p.nf;
  a.mcount = mcount;
  a.m0 = m0;
  a.M = out_ld ? out_ld : (p.phi_ld && !adjoint) ? p.phi_ld : p.M;
  a.phioff = out_ld ? out_off : adjoint ? 0 : p.phi_off;
  a.ntp = (mcount + 127) / 128;
  a.qtile0 = qoff / 128;
  const int sms = p.num_sms > 0 ? p.num_sms : 148;
  int64_t grid = sms;
  if (p.modes_ctas > 0) grid = (int64_t)p.modes_ctas;   // tuning override: total CTAs
  a.tiles = modes_tiles(p, a.nn, a.ntp * (f1 - f0), grid);
  a.nit = (a.ntp + a.tiles - 1) / a.tiles;
  a.nitems = a.nit * (f1 - f0);
  a.f0 = f0;
  a.box_bytes = (uint32_t)a.np * 128u;
  a.img_bytes = modes_img_bytes(a.np, a.nn);
  grid = std::max<int64_t>(1, std::min<int64_t>(grid, a.nitems));
  int optin = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, p.device);
  a.nst = kMaxStages;
  while (a.nst > 2 && modes_tc_smem_stages(p, a.nst, a.tiles) > (size_t)optin) --a.nst;
  const size_t smem = modes_tc_smem_stages(p, a.nst, a.tiles);
  CUtensorMap mh, ml;
  const int64_t nblk = p.chunk_points / kQBlock;
  if (!make_qhat_map(p, p.d_qhat, 2 * a.tiles, nblk, &mh) ||
      !make_qhat_map(p, p.d_qlo ? p.d_qlo : p.d_qhat, 2 * a.tiles, nblk, &ml))
    return cudaErrorUnknown;
  if (p.desc.precision == SPOD_PREC_BF16X3) {
    cudaError_t e = allow_smem(k_modes_tc<true>, smem);
    if (e != cudaSuccess) return e;
    k_modes_tc<true><<<(unsigned)grid, kThreadsModes, smem, s>>>(mh, ml, a,
                                                                 static_cast<const uint8_t*>(p.d_bimg), scale,
                                                                 static_cast<float2*>(d_Phi), p.d_flags);
  } else {
    cudaError_t e = allow_smem(k_modes_tc<false>, smem);
    if (e != cudaSuccess) return e;
    k_modes_tc<false><<<(unsigned)grid, kThreadsModes, smem, s>>>(mh, mh, a,
                                                                  static_cast<const uint8_t*>(p.d_bimg), scale,
                                                                  static_cast<float2*>(d_Phi), p.d_flags);
  }
  return cudaGetLastError();
}

}  // namespace spod
