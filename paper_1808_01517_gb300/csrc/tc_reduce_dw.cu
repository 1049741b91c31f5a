// The weight gradient's last step on the tensor cores (Sec. 2.3, adjoint of the collapse):
//   dw[co,s,ci,s',k] = sum_{a,b} M_{s,s'}[k][a][b] G[(s,co,a)][(s',ci,b)],  G = sum_split P
// per shell pair a GEMM [channel pairs] x [(b,a) entries] x [kernel points k < K <= 64],
// from the FP32 partials P that the weight-gradient GEMM stored transposed (a column
// (s',ci,b) holds its rows (s,co,a) contiguously).  FP32 operands as three-part BF16
// splits, six part products.  A tensor-core accumulator cuts every addition off toward zero, so
// the products x0 M0, which carry the sum, meet few others there: two k-steps of 16 coefficients,
// the second added to the first, then the accumulator is read and added up in FP32 registers.  The
// products 2^-8 and 2^-16 of them have accumulators of their own, read once per part of the b range.
// Relative error of dw against FP64 (64 -> 64 channels): 16 voxels 1.1e-7 against 1.7e-7 for the FP32
// sum on the CUDA cores, 300 voxels 3.2e-7 against 3.2e-7, 8,192 voxels (the voxel sums') 4.4e-6
// against 4.4e-6; all products of a part in one accumulator gave 1.9e-6, 2.1e-6 and 6.0e-6.
//
// What bounds it: the thread that issues the MMAs, about 100 cycles each at these widths and 450 for
// a group's wait and commit, then reading P (58 MB per split at 16 -> 64 channels, 232 MB at
// 64 -> 64).  M's parts side by side in N make four MMAs of the six products of a k-step: 0.092 ms in the
// main kernel (64 -> 64, one split; six MMAs, small ones first, in groups of four k-steps 0.096).
// On the CUDA cores the step was bound by issue (64 FMAs per (b,a) entry and pair).  Measured, with
// the sum of the parts and db: 64 -> 64 channels, one split 0.110 ms against 0.342 on the CUDA
// cores, four splits 0.121 against 0.346; 16 -> 64 channels 0.035 and 0.047 against 0.095 and 0.100.
//
// A persistent CTA walks units (shell s, part of the b range, input shell s', tile of up to
// 128 channel pairs), consecutive units sharing the part's M images in shared memory:
//   - warp 0 copies, per b and split, the tile's runs of P (one per input channel, c_out n_out
//     consecutive floats) into a ring with untiled bulk copies;
//   - 16 converter warps sum the splits (lane = channel pair, so a lane reads its own n_out
//     floats: an odd stride, no bank conflicts for odd n_out), split the sum into BF16 parts and
//     store them to TMEM as the MMA's A operand (no shared-memory round trip);
//   - one thread issues the MMAs (A from TMEM, M images MN-major from shared memory);
//   - eight warps read the accumulators, add them up and store the partial sums, lanes along the pairs.
#include <algorithm>
#include <type_traits>
#include <vector>

#include "tc_gemm.h"
#include "tc_ptx.cuh"

namespace delimit {

namespace {

constexpr int kRdN = 64;          // kernel points (MMA N), zero-padded
constexpr int kRdConvWarps = 16;  // four per TMEM lane quarter
constexpr int kRdEpiWarps = 8;    // two per TMEM lane quarter, 32 kernel points each
constexpr int kRdConv0 = 2 + kRdEpiWarps;  // first converter warp
constexpr int kRdThreads = 32 * (kRdConv0 + kRdConvWarps);
constexpr int kRdMaxKs = 8;       // k-steps of 16 output coefficients per b
constexpr int kRdRing = 6;        // most ring slots
constexpr uint32_t kRdACols = 24; // a k-step of A: three parts of 16 coefficients, two to a column
constexpr size_t kRdSmemLimit = 226 * 1024;
// TMEM: an accumulator of x0 M0 for every other group of two k-steps; one of x0 M1 + x1 M0 and one of
// x0 M2 + x1 M1 + x2 M0 for every other unit; the A buffers of two groups
constexpr uint32_t kRdSmall = 2 * kRdN, kRdA = kRdSmall + 4 * kRdN, kRdABuf = 2 * kRdACols;
static_assert(kRdA + 2 * kRdABuf <= 512, "TMEM columns");

enum : int {
  kErrRdRing = 0x5100,
  kErrRdRingEmpty = 0x5200,
  kErrRdA = 0x5300,
  kErrRdAEmpty = 0x5400,
  kErrRdD = 0x5500,
  kErrRdB = 0x5700,
  kErrRdDrain = 0x5800
};

// M_{s,s'} -> three BF16 parts, per (pg, b) an image [part][16 ks rows a][64 kernel points] in
// the MN-major 128-byte-swizzled operand layout, zero past n_out and K
__global__ void dw_images_kernel(const __grid_constant__ LscDims d, const float* __restrict__ M,
                                 uint8_t* __restrict__ img, int npg, int ks) {
  const int rows = 16 * ks;
  const int64_t n = (int64_t)npg * d.n_in * rows * kRdN;
  const int s_of = d.m_stride_sp ? d.s_in : 1;  // resampling-free tables hold one block per shell pair
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)(i % kRdN);
    int64_t r = i / kRdN;
    const int a = (int)(r % rows);
    r /= rows;
    const int b = (int)(r % d.n_in), pg = (int)(r / d.n_in);
    const int s = pg / s_of, sp = pg - s * s_of;
    const float x = (k < d.K && a < d.n_out)
                        ? M[s * d.m_stride_s + sp * d.m_stride_sp + ((int64_t)k * d.n_out + a) * d.n_in + b]
                        : 0.f;
    const __nv_bfloat16 x0 = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(x0);
    const __nv_bfloat16 x1 = __float2bfloat16_rn(r1);
    const __nv_bfloat16 x2 = __float2bfloat16_rn(r1 - __bfloat162float(x1));
    uint8_t* base = img + ((int64_t)pg * d.n_in + b) * (3 * rows * 128);
    const int off = a * 128 + (((k >> 3) ^ (a & 7)) << 4) + (k & 7) * 2;
    *reinterpret_cast<__nv_bfloat16*>(base + off) = x0;
    *reinterpret_cast<__nv_bfloat16*>(base + rows * 128 + off) = x1;
    *reinterpret_cast<__nv_bfloat16*>(base + 2 * rows * 128 + off) = x2;
  }
}

}  // namespace

struct RdParams {
  LscDims d;
  const float* P;
  const uint8_t* img;
  float* dwp;  // [part][k][row of pairs], row = ((s s_in + s') c_in + ci) c_out + co
  int64_t ldpt, split_stride, part_stride, rows_total;
  int splits, ks, bpp, nparts;
  int nseg, co_chunks, ntiles;  // a tile: nseg input channels x all c_out, or one channel x 128 outputs
  int ring;
  uint32_t seg_stride, ring_bytes, img_bytes;  // img_bytes: one b's image
  int64_t units;
  int pg_per_pair;
  int* err;
};

// split3x2 for any FP32 value: the first two parts keep within the largest BF16 value, so that what a
// sum has beyond it, infinity or NaN included, is left to the last part.  That one meets M0 alone: the
// products have the sign (or the NaN) that the FP32 product has, and no infinity meets M1 and M2,
// whose signs differ from M's.  One instruction per pair and part: 92.7 us against 92.3 in the main kernel
// at 64 -> 64 channels (with fminf and fmaxf 97).
__device__ __forceinline__ void split3x2_any(float x, float y, uint32_t (&p)[3]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    // at most the largest BF16 value in magnitude (for NaN, the largest value)
    asm("min.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(p[q]) : "r"(ptx::pack_bf16x2f(x, y)), "r"(0x7F7F7F7Fu));
    x -= __uint_as_float(p[q] << 16);
    y -= __uint_as_float(p[q] & 0xFFFF0000u);
  }
  p[2] = ptx::pack_bf16x2f(x, y);
}

// one unit of work and its walk: (s, part, s', tile), tile fastest
struct RdUnit {
  int s, part, sp, tile;
  __device__ __forceinline__ void init(const RdParams& p, int64_t u) {
    s = 0;
    while (true) {
      const int64_t n = (int64_t)p.nparts * (p.d.win_hi[s] - p.d.win_lo[s]) * p.ntiles;
      if (u < n) break;
      u -= n;
      ++s;
    }
    const int nw = p.d.win_hi[s] - p.d.win_lo[s];
    tile = (int)(u % p.ntiles);
    u /= p.ntiles;
    sp = p.d.win_lo[s] + (int)(u % nw);
    part = (int)(u / nw);
  }
  __device__ __forceinline__ void next(const RdParams& p) {
    if (++tile < p.ntiles) return;
    tile = 0;
    if (++sp < p.d.win_hi[s]) return;
    if (++part >= p.nparts) {
      part = 0;
      do {
        ++s;
      } while (s < p.d.s_out && p.d.win_hi[s] <= p.d.win_lo[s]);
    }
    if (s < p.d.s_out) sp = p.d.win_lo[s];
  }
  // images of this unit's part: equal keys share them
  __device__ __forceinline__ int key(const RdParams& p) const {
    const int pg = p.pg_per_pair ? s * p.d.s_in + sp : s;
    return pg * p.nparts + part;
  }
};

// PER_B: most k-steps of an input coefficient that one warp converts
template <int PER_B>
__global__ void __launch_bounds__(kRdThreads, 1) reduce_dw_tc_kernel(const __grid_constant__ RdParams p) {
  using namespace ptx;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const LscDims& d = p.d;
  const uint32_t sbase = smem_u32(smem);
  const uint32_t ring_off = (uint32_t)p.bpp * p.img_bytes;  // [images of a part][ring slots][barriers]
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + ring_off + (uint32_t)p.ring * p.ring_bytes);
  // bars: ring_full[6], ring_empty[6], full[2], done[2], b_full, b_empty, drain
  uint64_t* bars2 = bars + 2 * kRdRing;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars2 + 7);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto ring_full = [&](int i) { return smem_u32(bars + i); };
  auto ring_empty = [&](int i) { return smem_u32(bars + kRdRing + i); };
  auto full = [&](int i) { return smem_u32(bars2 + i); };      // a group's A is there, its accumulators are free
  auto done = [&](int i) { return smem_u32(bars2 + 2 + i); };  // a group's MMAs: its A is free, its sums are there
  const uint32_t b_full = smem_u32(bars2 + 4), b_empty = smem_u32(bars2 + 5), drain_bar = smem_u32(bars2 + 6);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kRdRing; ++i) {
      mbar_init(ring_full(i), 1);
      mbar_init(ring_empty(i), kRdConvWarps);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(full(i), kRdConvWarps / 2 + kRdEpiWarps);
      mbar_init(done(i), 1);
    }
    mbar_init(b_full, 1);
    mbar_init(b_empty, 1);
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // this CTA's consecutive units
  const int64_t u0 = p.units * blockIdx.x / gridDim.x, u1 = p.units * (blockIdx.x + 1) / gridDim.x;
  const int cw = d.c_out < 128 ? d.c_out : 128;  // output channels of a full tile row of segments

  if (warp == 0) {
    // ---- producer: M images when the part changes, then P's runs per (b, split) ----
    RdUnit un;
    un.init(p, u0);
    int key = -1, slot = 0;
    uint32_t ph = 0, b_ph = 0;
    uint32_t used = 0;  // ring slots that have been filled
    int b_loads = 0;
    bool ok = true;
    for (int64_t u = u0; u < u1 && ok && !warp_aborted(abort_flag); ++u, un.next(p)) {
      const int b0 = un.part * p.bpp, nb = min(p.bpp, d.n_in - b0);
      if (un.key(p) != key) {
        // the images of the units before are read by MMAs that have completed
        ok = key < 0 || wait_bounded(b_empty, b_ph, abort_flag, p.err, kErrRdB);
        if (key >= 0) b_ph ^= 1u;
        if (!__all_sync(0xffffffffu, ok)) break;
        key = un.key(p);
        ++b_loads;
        if (lane == 0) {
          const int pg = key / p.nparts;
          mbar_arrive_expect_tx(b_full, (uint32_t)nb * p.img_bytes);
          bulk_load(sbase, p.img + ((int64_t)pg * d.n_in + b0) * p.img_bytes, (uint32_t)nb * p.img_bytes, b_full);
        }
      }
      const int co0 = d.c_out < 128 ? 0 : (un.tile % p.co_chunks) * 128;
      const int ci0 = d.c_out < 128 ? un.tile * p.nseg : un.tile / p.co_chunks;
      const int len = min(cw, d.c_out - co0) * d.n_out;  // floats of a run
      const int nsg = min(p.nseg, d.c_in - ci0);
      const int64_t row = ((int64_t)un.s * d.c_out + co0) * d.n_out;
      const int mis = (int)(row & 3);  // runs start on 16-byte boundaries; ldpt and split_stride are multiples of 4
      const uint32_t bytes = (uint32_t)((mis + len + 3) / 4 * 16);
      for (int b = b0; b < b0 + nb && ok; ++b) {
        for (int z = 0; z < p.splits; ++z) {
          ok = wait_bounded(ring_empty(slot), ph ^ 1u, abort_flag, p.err, kErrRdRingEmpty);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (lane == 0) mbar_arrive_expect_tx(ring_full(slot), (uint32_t)nsg * bytes);
          __syncwarp();
          const uint32_t dst = sbase + ring_off + (uint32_t)slot * p.ring_bytes;
          for (int g = lane; g < nsg; g += 32)
            bulk_load(dst + (uint32_t)g * p.seg_stride,
                      p.P + z * p.split_stride + (((int64_t)un.sp * d.c_in + ci0 + g) * d.n_in + b) * p.ldpt + row - mis,
                      bytes, ring_full(slot));
          used |= 1u << slot;
          if (++slot == p.ring) {
            slot = 0;
            ph ^= 1u;
          }
        }
      }
    }
    // copies still in flight complete before the CTA may exit: the last fill of every slot used
    // (slots before `slot` were filled in this pass of the ring, the others in the one before)
    if (b_loads) wait_drain(b_full, (uint32_t)(b_loads - 1) & 1u, p.err, kErrRdDrain);
    for (int i = 0; i < p.ring; ++i)
      if (used >> i & 1u) wait_drain(ring_full(i), i < slot ? ph : ph ^ 1u, p.err, kErrRdDrain);
  } else if (warp == 1) {
    if (lane == 0) {
      RdUnit un;
      un.init(p, u0);
      const uint32_t idesc1 = idesc_bf16(128, kRdN, false, true), idesc2 = idesc_bf16(128, 2 * kRdN, false, true);
      const uint32_t part_bytes = (uint32_t)p.ks * 2048u;
      const uint64_t part = part_bytes >> 4, img = p.img_bytes >> 4;
      const uint64_t bd0 = umma_desc(sbase, part_bytes, 1024, kSwizzle128B);
      int key = -1;
      uint32_t grp = 0, b_ph = 0;  // groups so far
      bool ok = true;
      for (int64_t u = u0; u < u1 && ok && !*abort_flag; ++u) {
        const int steps = min(p.bpp, d.n_in - un.part * p.bpp) * p.ks;
        if (un.key(p) != key) {
          key = un.key(p);
          if (!wait_bounded(b_full, b_ph, abort_flag, p.err, kErrRdB)) break;
          b_ph ^= 1u;
        }
        const uint32_t small = tmem_base + kRdSmall + (uint32_t)((u - u0) & 1) * (2 * kRdN);
        uint64_t bd = bd0;  // the k-step's image, by additions (a descriptor built per MMA took longer than the MMA)
        int kk = 0;
        for (int t = 0; t < steps; t += 2, ++grp) {
          const uint32_t set = grp & 1, lead = tmem_base + set * kRdN, x = tmem_base + kRdA + set * kRdABuf;
          if (!(ok = wait_bounded(full(set), (grp >> 1) & 1u, abort_flag, p.err, kErrRdA))) break;
          tc_fence_after();
          // four MMAs for the six part products of a k-step
          auto step = [&](uint32_t xi, uint32_t acc_lead, uint32_t acc_small) {
            mma_bf16_ts(lead, xi, bd, idesc1, acc_lead);                               // x0 M0
            mma_bf16_ts(small, xi, bd + part, idesc2, acc_small);                      // x0 [M1 M2]
            mma_bf16_ts(small, xi + kRdACols / 3, bd, idesc2, 1);                      // x1 [M0 M1]
            mma_bf16_ts(small + kRdN, xi + 2 * kRdACols / 3, bd, idesc1, 1);           // x2 M0
            bd += 128;
            if (++kk == p.ks) {  // the next input coefficient's image
              kk = 0;
              bd += img - part;
            }
          };
          step(x, 0, t > 0);
          if (t + 1 < steps) step(x + kRdACols, 1, 1);
          mma_commit(done(set));
        }
        if (!ok) break;
        un.next(p);
        if (u + 1 < u1 && un.key(p) != key) mma_commit(b_empty);
      }
      mma_commit(drain_bar);
      wait_drain(drain_bar, 0, p.err, kErrRdDrain);
    }
  } else if (warp < kRdConv0) {
    // ---- epilogue: lane = channel pair of the tile, columns = kernel points, 32 per warp of a quarter;
    // the groups' accumulators, then the small products', added up in FP32 registers ----
    const int q = warp & 3, h0 = 32 * ((warp - 2) >> 2), r = q * 32 + lane;
    const uint32_t tl = tmem_base + ((uint32_t)(q * 32) << 16) + h0;
    if (lane == 0) {  // both accumulators are free
      mbar_arrive(full(0));
      mbar_arrive(full(1));
    }
    uint32_t grp = 0;
    bool ok = true;
    RdUnit un;
    un.init(p, u0);
    for (int64_t u = u0; u < u1 && ok; ++u, un.next(p)) {
      const int steps = min(p.bpp, d.n_in - un.part * p.bpp) * p.ks;
      float sum[32];
#pragma unroll
      for (int k = 0; k < 32; ++k) sum[k] = 0.f;
      for (int t = 0; t < steps; t += 2, ++grp) {
        const uint32_t set = grp & 1;
        ok = wait_bounded_sleep(done(set), (grp >> 1) & 1u, abort_flag, p.err, kErrRdD);
        if (!(ok = __all_sync(0xffffffffu, ok))) break;
        tc_fence_after();
        if (h0 < d.K) {
          uint32_t x[16];
#pragma unroll
          for (int h = 0; h < 32; h += 16) {
            tmem_ld16_nowait(tl + set * kRdN + h, x);
            tmem_wait_ld();
#pragma unroll
            for (int k = 0; k < 16; ++k) sum[h + k] += __uint_as_float(x[k]);
          }
          if (t + 2 >= steps) {  // the unit's last group: read before its accumulator is given back, so that a
                                 // unit's first group finds the small products of the unit before last read
            const uint32_t small = kRdSmall + (uint32_t)((u - u0) & 1) * (2 * kRdN);
#pragma unroll
            for (int h = 0; h < 32; h += 8) {
              uint32_t y[8], z[8];
              tmem_ld8_nowait(tl + small + kRdN + h, y);
              tmem_ld8_nowait(tl + small + h, z);
              tmem_wait_ld();
#pragma unroll
              for (int k = 0; k < 8; ++k) sum[h + k] += __uint_as_float(y[k]) + __uint_as_float(z[k]);
            }
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(full(set));
      }
      if (!ok) break;
      const int co0 = d.c_out < 128 ? 0 : (un.tile % p.co_chunks) * 128;
      const int ci0 = d.c_out < 128 ? un.tile * p.nseg : un.tile / p.co_chunks;
      const int g = r / cw, co = co0 + r - g * cw;
      if (g < p.nseg && ci0 + g < d.c_in && co < d.c_out) {
        float* out = p.dwp + un.part * p.part_stride + h0 * p.rows_total +
                     (((int64_t)un.s * d.s_in + un.sp) * d.c_in + ci0 + g) * d.c_out + co;
#pragma unroll
        for (int k = 0; k < 32; ++k)
          if (h0 + k < d.K) out[k * p.rows_total] = sum[k];
      }
    }
  } else {
    // ---- converters: lane = channel pair; of the four warps of a quarter two take every other group, a
    // k-step each ----
    const int q = warp & 3, sub = (warp - kRdConv0) >> 2, r = q * 32 + lane;
    const int g = r / cw, cl = r - g * cw;
    const uint32_t set = (uint32_t)sub >> 1, at = tmem_base + ((uint32_t)(q * 32) << 16) + kRdA + set * kRdABuf + (sub & 1) * kRdACols;
    uint32_t fills = 0;  // groups this warp has converted
    auto wait_done = [&]() {  // the group before it in this set is done
      const bool w = wait_bounded_sleep(done(set), (fills & 1u) ^ 1u, abort_flag, p.err, kErrRdAEmpty);
      return (bool)__all_sync(0xffffffffu, w);
    };
    auto give = [&]() {
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(full(set));
      ++fills;
    };
    RdUnit un;
    un.init(p, u0);
    int slot = 0;
    uint32_t ph = 0, grp = 0;  // grp: the unit's first group
    bool ok = true;
    for (int64_t u = u0; u < u1 && ok; ++u, un.next(p)) {
      const int nb = min(p.bpp, d.n_in - un.part * p.bpp);
      const int co0 = d.c_out < 128 ? 0 : (un.tile % p.co_chunks) * 128;
      const int ci0 = d.c_out < 128 ? un.tile * p.nseg : un.tile / p.co_chunks;
      const bool valid = g < p.nseg && ci0 + g < d.c_in && co0 + cl < d.c_out;
      const int mis = (int)((((int64_t)un.s * d.c_out + co0) * d.n_out) & 3);
      const uint32_t lane_off = valid ? (uint32_t)g * p.seg_stride + (uint32_t)(mis + cl * d.n_out) * 4u : 0u;
      // this warp's k-steps of the unit: place sub & 1 of every group with the parity of `set`
      const int first = (sub & 1) + 2 * (int)((set ^ grp) & 1u);
      for (int b = 0; b < nb && ok; ++b) {
        const int kk0 = (first - b * p.ks) & 3;  // of this b: kk0, kk0 + 4
        float v[PER_B][16];
#pragma unroll
        for (int j = 0; j < PER_B; ++j)
#pragma unroll
          for (int e = 0; e < 16; ++e) v[j][e] = 0.f;
        for (int z = 0; z < p.splits; ++z) {
          ok = wait_bounded_sleep(ring_full(slot), ph, abort_flag, p.err, kErrRdRing);
          ok = __all_sync(0xffffffffu, ok);
          if (!ok) break;
          if (valid) {
            const float* src = reinterpret_cast<const float*>(smem + ring_off + (uint32_t)slot * p.ring_bytes + lane_off);
#pragma unroll
            for (int j = 0; j < PER_B; ++j) {
              const int a0 = 16 * (kk0 + 4 * j);
              if (a0 + 16 <= d.n_out) {
#pragma unroll
                for (int e = 0; e < 16; ++e) v[j][e] += src[a0 + e];
              } else if (a0 < d.n_out) {
#pragma unroll
                for (int e = 0; e < 16; ++e)
                  if (a0 + e < d.n_out) v[j][e] += src[a0 + e];
              }
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(ring_empty(slot));
          if (++slot == p.ring) {
            slot = 0;
            ph ^= 1u;
          }
        }
        if (!ok) break;
#pragma unroll
        for (int j = 0; j < PER_B; ++j) {
          if (kk0 + 4 * j >= p.ks) break;
          uint32_t part[3][8];
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            uint32_t t3[3];
            split3x2_any(v[j][2 * e], v[j][2 * e + 1], t3);
#pragma unroll
            for (int t = 0; t < 3; ++t) part[t][e] = t3[t];
          }
          if (!(ok = wait_done())) break;
          tc_fence_after();
#pragma unroll
          for (int t = 0; t < 3; ++t) tmem_st8(at + (uint32_t)(t * 8), part[t]);
          tmem_wait_st();
          give();
        }
      }
      // an odd number of k-steps: the last group has one, and its other warp has nothing to convert
      const int steps = nb * p.ks, groups = (steps + 1) / 2;
      if (ok && (steps & 1) && (sub & 1) && ((grp + groups - 1) & 1u) == set) {
        if ((ok = wait_done())) give();
      }
      grp += groups;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// dw = sum of the parts in order (zero outside the window), 32 pairs x K points per block through
// shared memory ([k][pair] in, [pair][k] out), and db in the blocks after them, one warp per
// (co, s): db[co,s] = sum_a q[s][a] (row sum of dY's row (s,co,a) over the splits)
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS) finish_dw_kernel(const __grid_constant__ RdParams p, float* __restrict__ dw,
                                                        float* __restrict__ db, const float* __restrict__ qv,
                                                        int64_t dw_blocks) {
  __shared__ float t[kRdN][33];
  const LscDims& d = p.d;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if ((int64_t)blockIdx.x < dw_blocks) {
    const uint32_t r0 = blockIdx.x * 32, row = r0 + lane;  // rows_total < 2^31 (tc_reduce_dw_supported)
    auto decode = [&](uint32_t r, uint32_t& s, uint32_t& sp, uint32_t& ci, uint32_t& co) {
      co = r % d.c_out;
      r /= d.c_out;
      ci = r % d.c_in;
      r /= d.c_in;
      sp = r % d.s_in;
      s = r / d.s_in;
    };
    uint32_t s, sp, ci, co;
    decode(row < p.rows_total ? row : 0, s, sp, ci, co);
    const bool in = row < p.rows_total && (int)sp >= d.win_lo[s] && (int)sp < d.win_hi[s];
    for (int k = warp; k < d.K; k += WARPS) {
      float a = 0.f;
      if (in) {  // eight parts' loads in flight, summed in order
        const float* src = p.dwp + k * p.rows_total + row;
        for (int z0 = 0; z0 < p.nparts; z0 += 8) {
          float v[8];
#pragma unroll
          for (int z = 0; z < 8; ++z) v[z] = z0 + z < p.nparts ? __ldg(src + (z0 + z) * p.part_stride) : 0.f;
#pragma unroll
          for (int z = 0; z < 8; ++z) a += v[z];
        }
      }
      t[k][lane] = a;
    }
    __syncthreads();
    for (int i = warp; i < 32; i += WARPS) {
      if (r0 + i >= p.rows_total) break;
      decode(r0 + i, s, sp, ci, co);
      float* out = dw + ((((int64_t)co * d.s_out + s) * d.c_in + ci) * d.s_in + sp) * d.K;
      for (int k = lane; k < d.K; k += 32) out[k] = t[k][i];
    }
  } else {
    const int64_t i = ((int64_t)blockIdx.x - dw_blocks) * WARPS + warp;
    if (i >= (int64_t)d.c_out * d.s_out) return;
    const int co = (int)(i / d.s_out), s = (int)(i % d.s_out);
    const int64_t row0 = ((int64_t)s * d.c_out + co) * d.n_out;
    float acc = 0.f;
    for (int aa = lane; aa < d.n_out; aa += 32) {
      float r = 0.f;
      for (int z = 0; z < p.splits; ++z) r += p.P[z * p.split_stride + d.rows_in * p.ldpt + row0 + aa];
      acc = fmaf(qv[s * d.n_out + aa], r, acc);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) db[co * d.s_out + s] = acc;
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

int rd_bpp(int n_in, int n_out) {
  // as many parts of the b range as the CUDA-core reduction has parts of 256 (a,b) entries
  const int parts = (n_in * n_out + 255) / 256;
  return (n_in + parts - 1) / parts;
}

// shared memory beside the ring: the part's images, alignment and barriers
size_t rd_fixed(int n_in, int n_out) {
  const int ks = (n_out + 15) / 16;
  return 1024 + (size_t)rd_bpp(n_in, n_out) * 3 * ks * 2048 + (2 * kRdRing + 7) * 8 + 64;
}

}  // namespace

cudaError_t reduce_dw_tables_create(const LscDims& dt, const float* d_M, ReduceDwTables& t, std::string& err) {
  t = ReduceDwTables();
  const int ks = (dt.n_out + 15) / 16;
  // more kernel points, coefficients or images than the kernel holds: the CUDA-core reduction
  if (dt.K > kRdN || ks > kRdMaxKs || rd_fixed(dt.n_in, dt.n_out) + 2 * 128 * (size_t)(4 * dt.n_out + 32) > kRdSmemLimit)
    return cudaSuccess;
  t.npg = dt.m_stride_sp ? dt.s_out * dt.s_in : dt.s_out;
  const size_t bytes = (size_t)t.npg * dt.n_in * 3 * ks * 2048;
  cudaError_t e = cudaMalloc(&t.d_img, bytes);
  if (e == cudaSuccess) {
    dw_images_kernel<<<152 * 4, 256>>>(dt, d_M, static_cast<uint8_t*>(t.d_img), t.npg, ks);
    count_launch();
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
  }
  if (e != cudaSuccess) {
    err = cudaGetErrorString(e);
    if (t.d_img) cudaFree(t.d_img);
    t = ReduceDwTables();
    return e;
  }
  t.ok = true;
  return cudaSuccess;
}

void reduce_dw_tables_destroy(ReduceDwTables& t) {
  if (t.d_img) cudaFree(t.d_img);
  t = ReduceDwTables();
}

bool tc_reduce_dw_supported(const LscDims& d, const ReduceDwTables& t) {
  if (!t.ok || !tc_enabled() || (int64_t)d.s_out * d.s_in * d.c_in * d.c_out > INT32_MAX) return false;
  // A tile copies a run of P per input channel, and more than 32 short ones a step take longer than
  // the CUDA cores' loads.  us, here and there, 64 -> 1 channels 26 / 24 at 2,048 voxels and 64 / 58 at
  // 16,384 (64 runs of 180 bytes), 64 -> 2 27 / 24 and 65 / 59; 64 -> 4 20 / 34 and 42 / 67 (32 runs),
  // 16 -> 1 17 / 23 and 27 / 24.
  if (std::min(128 / std::min(d.c_out, 128), d.c_in) > 32) return false;
  int dev = 0, major = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  return major == 10;
}

cudaError_t tc_reduce_dw(const LscDims& d, const ReduceDwTables& t, const float* P, int64_t ldpt, int64_t split_stride,
                         int splits, const float* q, float* dw, float* db, float* scratch, int* err, cudaStream_t st) {
  TraceScope trace("lsc_reduce_dw_tc", st);
  RdParams p;
  memset(&p, 0, sizeof p);
  p.d = d;
  p.P = P;
  p.img = static_cast<const uint8_t*>(t.d_img);
  p.dwp = scratch;
  p.ldpt = ldpt;
  p.split_stride = split_stride;
  p.splits = splits;
  p.ks = (d.n_out + 15) / 16;
  p.bpp = rd_bpp(d.n_in, d.n_out);
  p.nparts = (d.n_in + p.bpp - 1) / p.bpp;
  p.rows_total = (int64_t)d.s_out * d.s_in * d.c_in * d.c_out;
  p.part_stride = p.rows_total * d.K;
  p.nseg = d.c_out < 128 ? 128 / d.c_out : 1;
  p.co_chunks = d.c_out < 128 ? 1 : (d.c_out + 127) / 128;
  p.ntiles = d.c_out < 128 ? (d.c_in + p.nseg - 1) / p.nseg : d.c_in * p.co_chunks;
  p.seg_stride = (uint32_t)((std::min(d.c_out, 128) * d.n_out + 3 + 3) / 4 * 16);
  p.ring_bytes = (uint32_t)(p.nseg * p.seg_stride);
  p.img_bytes = (uint32_t)(3 * p.ks * 2048);
  p.pg_per_pair = d.m_stride_sp ? 1 : 0;
  p.err = err;
  for (int s = 0; s < d.s_out; ++s) p.units += (int64_t)p.nparts * std::max(0, d.win_hi[s] - d.win_lo[s]) * p.ntiles;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaError_t e;
  if (dw && p.units > 0) {
    const size_t fixed = rd_fixed(d.n_in, d.n_out);
    p.ring = (int)std::min<size_t>(kRdRing, (kRdSmemLimit - fixed) / p.ring_bytes);
    if (p.ring < 2) return cudaErrorInvalidValue;
    // at least 120 KiB so that two CTAs never share an SM (each holds 512 TMEM columns)
    const size_t smem = std::max<size_t>(120 * 1024, fixed + (size_t)p.ring * p.ring_bytes);
    auto kern = p.ks > 4 ? reduce_dw_tc_kernel<2> : reduce_dw_tc_kernel<1>;
    e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    const unsigned grid = (unsigned)std::min<int64_t>(p.units, std::max(1, sms));
    kern<<<grid, kRdThreads, smem, st>>>(p);
    count_launch();
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  const int64_t dw_blocks = dw ? (p.rows_total + 31) / 32 : 0;
  // 32 warps a block (a warp per kernel point or two, so that the parts' loads are all in flight) where
  // two such blocks per SM hold them all, else eight.  us with 32 and with eight: 1 -> 64 channels
  // 4.0 / 6.0, 16 -> 64 6.4 / 9.5, 16 -> 16 of order 10 (18 parts) 6.2 / 11.5, 64 -> 64 20.9 / 18.0
  auto finish = [&](auto kern, int warps) {
    const int64_t db_blocks = db ? ((int64_t)d.c_out * d.s_out + warps - 1) / warps : 0;
    if (dw_blocks + db_blocks == 0) return;
    kern<<<(unsigned)(dw_blocks + db_blocks), 32 * warps, 0, st>>>(p, dw, db, q, dw_blocks);
    count_launch();
  };
  if (dw_blocks <= 2 * sms)
    finish(finish_dw_kernel<32>, 32);
  else
    finish(finish_dw_kernel<8>, 8);
  return cudaGetLastError();
}

}  // namespace delimit
