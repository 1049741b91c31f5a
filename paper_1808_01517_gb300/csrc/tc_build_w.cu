// The collapsed LSC operator on the tensor cores (Sec. 2.3, the exact collapse of the
// resample / product / projection steps into one matrix per shell pair):
//   W[(s,co,a)][(s',ci,b)] = sum_k w[co,s,ci,s',k] M_{s,s'}[k][a][b]
// per shell pair a GEMM [channel pairs (co, ci)] x [kernel points k < K <= 64] x [(a,b)
// entries].  FP32 operands on the BF16 tensor cores as three-part splits (x = x0 + x1 + x2
// to 2^-27 |x|, the six part products down to 2^-18 of the leading one, FP32 accumulation in
// TMEM): FP32-level accuracy before the result is rounded to BF16 (the same rounding point as
// the CUDA-core build).  The parts of M are made once per geometry (M is fixed).
//
// What bounds it: the thread that issues the MMAs (order 8, K = 49: 48 per tile of 128 pairs, four rows
// and one input shell, about 100 cycles each whatever their width), close behind it writing
// W (149 MB at 64 -> 64 channels, 29 MB at 16 -> 64).  One tile per CTA took 20 us, its loads,
// MMAs, TMEM reads and stores one after the other; a persistent CTA that overlaps them, with
// tiles of whole rows a so that every run of W leaves in one copy, measured 0.304 -> 0.083 ms
// (64 -> 64 channels) and 0.058 -> 0.030 (16 -> 64).
//
// A tile is (output shell s, two halves of 128 / n_in rows a with all their b entries, input
// shell s', 128 / c_in output channels with all their input channels).  A CTA walks consecutive
// tiles that share the M image of (s, rows) in shared memory:
//   - four loader warps copy the tile's w (4-byte cp.async: w needs no alignment) into a ring,
//     and the M image when it changes;
//   - 8 converter warps split w into BF16 parts and store them to TMEM as the MMA's A operand;
//   - one thread issues the MMAs (6 part products, A from TMEM, M = 128 pairs, N = a half's
//     entries), a half's while the other's accumulator is read;
//   - 8 epilogue warps read the accumulator, round to BF16 and write a staging tile in W's own
//     order [co][a][ci][b];
//   - one warp copies the staging tile's rows, contiguous in W, out with bulk copies, and at the
//     end writes zeros outside the shell window.
// Every wait is bounded.
#include <algorithm>

#include "tc_gemm.h"
#include "tc_ptx.cuh"

namespace delimit {

namespace {

constexpr int kBwK = 64;                        // kernel points, zero-padded
constexpr int kBwMaxN = 256;                    // TMEM columns of the accumulators
constexpr int kBwAtomBytes = kBwK * 128;        // one 64-entry atom of an M part: [64 k][64 entries]
constexpr int kBwLoadWarps = 4, kBwEpiWarps = 8, kBwConvWarps = 8;
constexpr int kBwEpi0 = kBwLoadWarps + 2, kBwConv0 = kBwEpi0 + kBwEpiWarps;  // first warp of a role
constexpr int kBwThreads = 32 * (kBwConv0 + kBwConvWarps);
constexpr size_t kBwSmemLimit = 226 * 1024;
constexpr uint32_t kBwACols = 96;               // TMEM columns of an A buffer: 3 parts x 32

enum : int {
  kErrBwW = 0x4100,
  kErrBwWEmpty = 0x4200,
  kErrBwA = 0x4300,
  kErrBwAEmpty = 0x4400,
  kErrBwD = 0x4500,
  kErrBwDEmpty = 0x4600,
  kErrBwStg = 0x4700,
  kErrBwStgFree = 0x4800,
  kErrBwM = 0x4900,
  kErrBwDrain = 0x4A00
};

// halves of a tile (an accumulator and a staging buffer each), rows a of a half and of a tile,
// tiles of a shell's n_out rows, 64-entry atoms of a half's M image
__host__ __device__ constexpr int bw_halves(int n_in) { return n_in <= 128 ? 2 : 1; }
__host__ __device__ constexpr int bw_hrows(int n_in) { return n_in <= 128 ? 128 / n_in : 1; }
__host__ __device__ constexpr int bw_rows(int n_in) { return bw_halves(n_in) * bw_hrows(n_in); }
__host__ __device__ constexpr int bw_tiles(int n_in, int n_out) { return (n_out + bw_rows(n_in) - 1) / bw_rows(n_in); }
__host__ __device__ constexpr int bw_atoms(int n_in) { return (bw_hrows(n_in) * n_in + 63) / 64; }

// M_{s,s'} -> its three BF16 parts, per (shell or shell pair, tile of rows) an operand image
// [part][half][atom][64 k][64 entries], MN-major with the 128-byte swizzle, entry
// e = (a - a0) n_in + b of a half, zero past its rows and K
__global__ void split_m_kernel(const __grid_constant__ LscDims d, const float* __restrict__ M,
                               uint8_t* __restrict__ img, int npg) {
  const int hr = bw_hrows(d.n_in), nh = bw_halves(d.n_in), nt = bw_tiles(d.n_in, d.n_out), ha = bw_atoms(d.n_in);
  const int atoms = nh * ha;
  const int64_t n = (int64_t)npg * nt * atoms * kBwK * 64;
  const int s_of = d.m_stride_sp ? d.s_in : 1;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(i % 64), k = (int)(i / 64 % kBwK);
    int64_t r = i / (64 * kBwK);
    const int at = (int)(r % atoms);
    r /= atoms;
    const int t = (int)(r % nt), pg = (int)(r / nt), s = pg / s_of, sp = pg - s * s_of;
    const int hf = at / ha, e = (at - hf * ha) * 64 + c, al = e / d.n_in, b = e - al * d.n_in, a = (t * nh + hf) * hr + al;
    const float x = (k < d.K && al < hr && a < d.n_out)
                        ? M[s * d.m_stride_s + sp * d.m_stride_sp + ((int64_t)k * d.n_out + a) * d.n_in + b]
                        : 0.f;
    const __nv_bfloat16 x0 = __float2bfloat16_rn(x);
    const float r1 = x - __bfloat162float(x0);
    const __nv_bfloat16 x1 = __float2bfloat16_rn(r1);
    uint8_t* base = img + ((int64_t)pg * nt + t) * (3 * atoms * kBwAtomBytes) + at * kBwAtomBytes + k * 128 +
                    (((c >> 3) ^ (k & 7)) << 4) + (c & 7) * 2;
    *reinterpret_cast<__nv_bfloat16*>(base) = x0;
    *reinterpret_cast<__nv_bfloat16*>(base + atoms * kBwAtomBytes) = x1;
    *reinterpret_cast<__nv_bfloat16*>(base + 2 * atoms * kBwAtomBytes) = __float2bfloat16_rn(r1 - __bfloat162float(x1));
  }
}

}  // namespace

struct BwParams {
  LscDims d;
  const float* w;
  const uint8_t* img;
  const float* b;    // bias and q: the bias vector is made here too (bias null: not wanted)
  const float* q;
  float* bias;
  __nv_bfloat16* W;
  int64_t units;
  int nh, hr, nt, atoms, cpt, nptiles, ring, wld;  // cpt: output channels per tile; wld: odd row length of w in the ring
  int pg_per_pair;
  uint32_t img_bytes, w_bytes, stg_bytes;  // stg_bytes: one half's staging buffer, rows of in_blk elements
  int* err;
};

// one tile and its walk: (s, t, s', ptile), ptile fastest
struct BwUnit {
  int s, t, sp, pt;
  __device__ __forceinline__ void init(const BwParams& p, int64_t u) {
    s = 0;
    while (true) {
      const int64_t n = (int64_t)p.nt * (p.d.win_hi[s] - p.d.win_lo[s]) * p.nptiles;
      if (u < n) break;
      u -= n;
      ++s;
    }
    const int nw = p.d.win_hi[s] - p.d.win_lo[s];
    pt = (int)(u % p.nptiles);
    u /= p.nptiles;
    sp = p.d.win_lo[s] + (int)(u % nw);
    t = (int)(u / nw);
  }
  __device__ __forceinline__ void next(const BwParams& p) {
    if (++pt < p.nptiles) return;
    pt = 0;
    if (++sp < p.d.win_hi[s]) return;
    if (++t >= p.nt) {
      t = 0;
      do {
        ++s;
      } while (s < p.d.s_out && p.d.win_hi[s] <= p.d.win_lo[s]);
    }
    if (s < p.d.s_out) sp = p.d.win_lo[s];
  }
  __device__ __forceinline__ int key(const BwParams& p) const {
    return (p.pg_per_pair ? s * p.d.s_in + sp : s) * p.nt + t;
  }
};

__global__ void __launch_bounds__(kBwThreads, 1) build_w_tc_kernel(const __grid_constant__ BwParams p) {
  using namespace ptx;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const LscDims& d = p.d;
  const uint32_t sbase = smem_u32(smem);
  // [M image][staging buffers][w ring][barriers]
  const uint32_t stg_off = p.img_bytes, w_off = stg_off + (uint32_t)p.nh * p.stg_bytes;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + w_off + (uint32_t)p.ring * p.w_bytes);
  // bars, two of each: w_full, w_empty, a_full, a_empty, d_full, d_empty, stg_full, stg_free; m_full, m_empty, drain
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 19);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  auto w_full = [&](int i) { return smem_u32(bars + i); };
  auto w_empty = [&](int i) { return smem_u32(bars + 2 + i); };
  auto a_full = [&](int i) { return smem_u32(bars + 4 + i); };
  auto a_empty = [&](int i) { return smem_u32(bars + 6 + i); };
  auto d_full = [&](int i) { return smem_u32(bars + 8 + i); };
  auto d_empty = [&](int i) { return smem_u32(bars + 10 + i); };
  auto stg_full = [&](int i) { return smem_u32(bars + 12 + i); };
  auto stg_free = [&](int i) { return smem_u32(bars + 14 + i); };
  const uint32_t m_full = smem_u32(bars + 16), m_empty = smem_u32(bars + 17), drain_bar = smem_u32(bars + 18);
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(w_full(i), 32 * kBwLoadWarps);
      mbar_init(w_empty(i), kBwConvWarps);
      mbar_init(a_full(i), kBwConvWarps);
      mbar_init(a_empty(i), 1);
      mbar_init(d_full(i), 1);
      mbar_init(d_empty(i), kBwEpiWarps);
      mbar_init(stg_full(i), kBwEpiWarps);
      mbar_init(stg_free(i), 1);
    }
    mbar_init(m_full, 1);
    mbar_init(m_empty, 1);
    mbar_init(drain_bar, 1);
    *abort_flag = 0;
    fence_mbar_init();
  }
  if (warp == kBwLoadWarps) {
    tmem_alloc(smem_u32(tmem_slot), 512);
    tmem_relinquish();
  }
  if (p.bias) {  // bias_vec[(s,co,a)] = b[co,s] q[s][a]
    for (int64_t r = (int64_t)blockIdx.x * kBwThreads + threadIdx.x; r < d.rows_out; r += (int64_t)gridDim.x * kBwThreads) {
      const int per_out = d.c_out * d.n_out;
      const int s = (int)(r / per_out), co = (int)((r / d.n_out) % d.c_out), aa = (int)(r % d.n_out);
      p.bias[r] = p.b ? p.b[co * d.s_out + s] * p.q[s * d.n_out + aa] : 0.f;
    }
  }
  const int rowlen = (int)d.in_blk;  // a row run of W
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int64_t u0 = p.units * blockIdx.x / gridDim.x, u1 = p.units * (blockIdx.x + 1) / gridDim.x;
  const int ksteps = (d.K + 15) / 16;

  if (warp < kBwLoadWarps) {
    // ---- loaders: 32 of the tile's 128 pairs each; the first loads the M image too ----
    BwUnit un;
    un.init(p, u0);
    int key = -1, slot = 0, m_loads = 0;
    uint32_t ph = 0;
    for (int64_t u = u0; u < u1 && !warp_aborted(abort_flag); ++u, un.next(p)) {
      bool ok = wait_bounded(w_empty(slot), ph ^ 1u, abort_flag, p.err, kErrBwWEmpty);
      if (!__all_sync(0xffffffffu, ok)) break;
      if (warp == 0 && un.key(p) != key) {
        // the M image of the tiles before is read by MMAs that have completed
        ok = m_loads == 0 || wait_bounded(m_empty, (uint32_t)(m_loads - 1) & 1u, abort_flag, p.err, kErrBwM);
        if (!__all_sync(0xffffffffu, ok)) break;
        key = un.key(p);
        ++m_loads;
        if (lane == 0) {
          mbar_arrive_expect_tx(m_full, p.img_bytes);
          bulk_load(sbase, p.img + (int64_t)key * p.img_bytes, p.img_bytes, m_full);
        }
      }
      // w rows of the tile's pairs r = (co - co0) c_in + ci, K floats each, at an odd stride
      const int co0 = un.pt * p.cpt, np = min(p.cpt, d.c_out - co0) * d.c_in;
      const uint32_t dst0 = sbase + w_off + (uint32_t)slot * p.w_bytes;
      const int64_t ci_stride = (int64_t)d.s_in * d.K, co_jump = (int64_t)d.s_out * d.c_in * ci_stride;
      const int r0 = 32 * warp;
      int ci = r0 % d.c_in;
      const float* src = p.w + ((((int64_t)(co0 + r0 / d.c_in) * d.s_out + un.s) * d.c_in) * d.s_in + un.sp) * d.K;
      const float* row = src + ci * ci_stride;
      for (int r = r0; r < min(np, r0 + 32); ++r) {
        const uint32_t dst = dst0 + (uint32_t)(r * p.wld + lane) * 4u;
        if (lane < d.K) cp_async4(dst, row + lane);
        if (lane + 32 < d.K) cp_async4(dst + 128, row + lane + 32);
        row += ci_stride;
        if (++ci == d.c_in) {
          ci = 0;
          src += co_jump;
          row = src;
        }
      }
      cp_async_mbar_arrive(w_full(slot));
      if (++slot == p.ring) {
        slot = 0;
        ph ^= 1u;
      }
    }
    // copies still in flight complete before the CTA may exit
    asm volatile("cp.async.wait_all;" ::: "memory");
    if (m_loads) wait_drain(m_full, (uint32_t)(m_loads - 1) & 1u, p.err, kErrBwDrain);
  } else if (warp == kBwLoadWarps) {
    if (lane == 0) {
      BwUnit un;
      un.init(p, u0);
      int key = -1, m_loads = 0, i = 0;
      for (int64_t u = u0; u < u1 && !*abort_flag; ++u, ++i) {
        const int buf = i & 1;
        if (un.key(p) != key) {
          key = un.key(p);
          if (!wait_bounded(m_full, (uint32_t)m_loads & 1u, abort_flag, p.err, kErrBwM)) break;
          ++m_loads;
        }
        if (!wait_bounded(a_full(buf), (uint32_t)(i >> 1) & 1u, abort_flag, p.err, kErrBwA)) break;
        tc_fence_after();
        const uint32_t a_tmem = tmem_base + kBwMaxN + (uint32_t)buf * kBwACols;
        const uint32_t half_bytes = (uint32_t)(p.atoms * kBwAtomBytes), part_bytes = (uint32_t)p.nh * half_bytes;
        bool ok = true;
        for (int hf = 0; hf < p.nh; ++hf) {
          if (!(ok = wait_bounded(d_empty(hf), (uint32_t)(i & 1) ^ 1u, abort_flag, p.err, kErrBwDEmpty))) break;
          tc_fence_after();
          const int na = max(1, min(p.hr, d.n_out - (un.t * p.nh + hf) * p.hr));  // a half without rows: its zeros
          const uint32_t idesc = idesc_bf16(128, (na * d.n_in + 15) / 16 * 16, false, true);
          const uint32_t d_tmem = tmem_base + (uint32_t)(hf * 128);
          // operand addresses by one addition each: a descriptor built per MMA took longer than the MMA
          const uint64_t bd0 = umma_desc(sbase + (uint32_t)hf * half_bytes, kBwAtomBytes, 1024, kSwizzle128B);
#pragma unroll
          for (int pr = 0; pr < 6; ++pr) {  // part products, smallest first
            constexpr int pa[6] = {2, 0, 1, 1, 0, 0}, pb[6] = {0, 2, 1, 0, 1, 0};
            const uint64_t bd = bd0 + pb[pr] * (part_bytes >> 4);
#pragma unroll
            for (int k = 0; k < kBwK / 16; ++k)
              if (k < ksteps) mma_bf16_ts(d_tmem, a_tmem + (uint32_t)(pa[pr] * 32 + k * 8), bd + k * 128, idesc, (pr | k) != 0);
          }
          mma_commit(d_full(hf));
        }
        if (!ok) break;
        mma_commit(a_empty(buf));
        un.next(p);
        if (u + 1 < u1 && un.key(p) != key) mma_commit(m_empty);
      }
      mma_commit(drain_bar);
      wait_drain(drain_bar, 0, p.err, kErrBwDrain);
    }
  } else if (warp == kBwLoadWarps + 1) {
    // ---- copy-out: row (co, a) of the tile is one contiguous run of W ----
    BwUnit un;
    un.init(p, u0);
    const uint32_t run = (uint32_t)rowlen * 2u;
    int i = 0;
    bool ok = true;
    for (int64_t u = u0; u < u1 && ok; ++u, ++i, un.next(p)) {
      const int co0 = un.pt * p.cpt, nco = min(p.cpt, d.c_out - co0);
      for (int hf = 0; hf < p.nh && ok; ++hf) {
        ok = wait_bounded_sleep(stg_full(hf), (uint32_t)i & 1u, abort_flag, p.err, kErrBwStg);
        if (!(ok = __all_sync(0xffffffffu, ok))) break;
        const int a0 = (un.t * p.nh + hf) * p.hr, na = max(0, min(p.hr, d.n_out - a0));
        // consecutive rows a are contiguous in W too when it holds one shell block: one copy per channel
        const int rows = d.ldW == rowlen ? na : 1, runs = na / max(rows, 1);
        for (int r = lane; r < nco * runs; r += 32) {
          const int col = r / runs, al = r - col * runs;
          __nv_bfloat16* dst =
              p.W + (((int64_t)un.s * d.c_out + co0 + col) * d.n_out + a0 + al) * d.ldW + (int64_t)un.sp * d.in_blk;
          bulk_store(dst, sbase + stg_off + (uint32_t)hf * p.stg_bytes + (uint32_t)(col * p.hr + al) * run,
                     (uint32_t)rows * run);
        }
        bulk_commit();
        bulk_wait_read<0>();
        __syncwarp();
        if (lane == 0) mbar_arrive(stg_free(hf));
      }
    }
    // zeros outside the window: a staging buffer cleared once, then copied to every such run
    const int out_cols = (int)min((int64_t)p.stg_bytes / 2, (int64_t)d.s_in * d.in_blk);  // elements of zeros kept
    bool any = false;
    for (int s = 0; s < d.s_out; ++s) any = any || d.win_hi[s] - d.win_lo[s] < d.s_in;
    if (any && ok) {
      for (int o = lane * 16; o < out_cols * 2; o += 512) *reinterpret_cast<uint4*>(smem + stg_off + o) = make_uint4(0, 0, 0, 0);
      fence_proxy_async_smem();
      __syncwarp();
      const int per_out = d.c_out * d.n_out;
      for (int64_t r = (int64_t)blockIdx.x * 32 + lane; r < d.rows_out; r += (int64_t)gridDim.x * 32) {
        const int s = (int)(r / per_out);
        for (int side = 0; side < 2; ++side) {
          const int64_t c0 = side ? (int64_t)max(d.win_hi[s], 0) * d.in_blk : 0;
          const int64_t c1 = side ? (int64_t)d.s_in * d.in_blk : (int64_t)max(d.win_lo[s], 0) * d.in_blk;
          for (int64_t c = c0; c < c1; c += out_cols)
            bulk_store(p.W + r * d.ldW + c, sbase + stg_off, (uint32_t)min((int64_t)out_cols, c1 - c) * 2u);
        }
      }
      bulk_commit();
    }
    bulk_wait<0>();
  } else if (warp < kBwConv0) {
    // ---- epilogue: lane = channel pair; the two warps of a quarter take alternate rows a ----
    const int q = warp & 3, h = (warp - kBwEpi0) >> 2, r = q * 32 + lane;
    const int col = r / d.c_in, ci = r - col * d.c_in;
    BwUnit un;
    un.init(p, u0);
    int i = 0;
    for (int64_t u = u0; u < u1; ++u, ++i, un.next(p)) {
      const bool valid = un.pt * p.cpt + col < d.c_out;
      bool ok = true;
      for (int hf = 0; hf < p.nh; ++hf) {
        ok = wait_bounded_sleep(stg_free(hf), (uint32_t)(i & 1) ^ 1u, abort_flag, p.err, kErrBwStgFree);
        ok = ok && wait_bounded_sleep(d_full(hf), (uint32_t)i & 1u, abort_flag, p.err, kErrBwD);
        if (!(ok = __all_sync(0xffffffffu, ok))) break;
        tc_fence_after();
        const int na = min(p.hr, d.n_out - (un.t * p.nh + hf) * p.hr);
        const uint32_t tl = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(hf * 128);
        for (int al = h; al < na; al += 2) {
          __nv_bfloat16* dst = reinterpret_cast<__nv_bfloat16*>(smem + stg_off + (uint32_t)hf * p.stg_bytes) +
                               (col * p.hr + al) * rowlen + ci * d.n_in;
          for (int c = 0; c < d.n_in; c += 48) {
            uint32_t rv[3][16];
#pragma unroll
            for (int j = 0; j < 3; ++j)
              if (c + 16 * j < d.n_in) tmem_ld16_nowait(tl + (uint32_t)(al * d.n_in + c + 16 * j), rv[j]);
            tmem_wait_ld();
            if (valid) {
#pragma unroll
              for (int j = 0; j < 48; j += 2) {
                const uint32_t v = pack_bf16x2(rv[j >> 4][j & 15], rv[j >> 4][(j & 15) + 1]);
                if (c + j < d.n_in) dst[c + j] = __ushort_as_bfloat16((unsigned short)(v & 0xFFFFu));
                if (c + j + 1 < d.n_in) dst[c + j + 1] = __ushort_as_bfloat16((unsigned short)(v >> 16));
              }
            }
          }
        }
        tc_fence_before();
        fence_proxy_async_smem();  // the staging buffer is read by the copy engine
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(d_empty(hf));
          mbar_arrive(stg_full(hf));
        }
      }
      if (!ok) break;
    }
  } else {
    // ---- converters: lane = channel pair, kernel points 32 h .. 32 h + 31 ----
    const int q = warp & 3, h = (warp - kBwConv0) >> 2, r = q * 32 + lane;
    int slot = 0, i = 0;
    uint32_t ph = 0;
    BwUnit un;
    un.init(p, u0);
    for (int64_t u = u0; u < u1; ++u, ++i, un.next(p)) {
      const int buf = i & 1;
      bool ok = wait_bounded_sleep(w_full(slot), ph, abort_flag, p.err, kErrBwW);
      ok = ok && wait_bounded_sleep(a_empty(buf), ((uint32_t)(i >> 1) & 1u) ^ 1u, abort_flag, p.err, kErrBwAEmpty);
      if (!__all_sync(0xffffffffu, ok)) break;
      tc_fence_after();
      const bool valid = r < min(p.cpt, d.c_out - un.pt * p.cpt) * d.c_in;
      if (32 * h < 16 * ksteps) {
        const float* src = reinterpret_cast<const float*>(smem + w_off + (uint32_t)slot * p.w_bytes) + r * p.wld + 32 * h;
        const int kn = valid ? d.K - 32 * h : 0;
        uint32_t part[3][16];
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float x = 2 * j < kn ? src[2 * j] : 0.f, y = 2 * j + 1 < kn ? src[2 * j + 1] : 0.f;
          uint32_t t3[3];
          split3x2(x, y, t3);
#pragma unroll
          for (int t = 0; t < 3; ++t) part[t][j] = t3[t];
        }
        const uint32_t at = tmem_base + ((uint32_t)(q * 32) << 16) + kBwMaxN + (uint32_t)buf * kBwACols + 16u * h;
#pragma unroll
        for (int t = 0; t < 3; ++t) tmem_st16(at + 32u * t, part[t]);
        tmem_wait_st();
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(w_empty(slot));
        mbar_arrive(a_full(buf));
      }
      if (++slot == p.ring) {
        slot = 0;
        ph ^= 1u;
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == kBwLoadWarps) {
    tc_fence_after();
    tmem_dealloc(tmem_base, 512);
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
namespace {

int bw_wld(int K) { return K | 1; }  // odd: the converters' lanes read conflict-free

// a half's staging buffer: 128 / c_in channels x its rows, in_blk elements each
size_t bw_stg_bytes(int n_in, int c_in, int64_t in_blk) {
  return ((size_t)(128 / c_in) * bw_hrows(n_in) * in_blk * 2 + 1023) / 1024 * 1024;
}

size_t bw_smem(int n_in, int c_in, int64_t in_blk, int K, int ring) {
  const size_t img = 3 * (size_t)(bw_halves(n_in) * bw_atoms(n_in)) * kBwAtomBytes;
  return 1024 + img + bw_halves(n_in) * bw_stg_bytes(n_in, c_in, in_blk) + ring * ((128 * (size_t)bw_wld(K) * 4 + 15) / 16 * 16) +
         19 * 8 + 64;
}

}  // namespace

cudaError_t build_w_tables_create(const LscDims& dt, const float* d_M, BuildWTables& t, std::string& err) {
  t = BuildWTables();
  if (dt.K > kBwK || dt.n_in < 1 || dt.n_in > kBwMaxN) return cudaSuccess;  // the CUDA-core build takes these
  t.npg = dt.m_stride_sp ? dt.s_out * dt.s_in : dt.s_out;
  const size_t bytes =
      (size_t)t.npg * bw_tiles(dt.n_in, dt.n_out) * 3 * bw_halves(dt.n_in) * bw_atoms(dt.n_in) * kBwAtomBytes;
  void* mp = nullptr;
  cudaError_t e = cudaMalloc(&mp, bytes);
  if (e == cudaSuccess) {
    const unsigned blocks = (unsigned)std::min<size_t>((bytes / 6 + 255) / 256, 152 * 8);
    split_m_kernel<<<blocks, 256>>>(dt, d_M, static_cast<uint8_t*>(mp), t.npg);
    count_launch();
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaDeviceSynchronize();
  }
  if (e != cudaSuccess) {
    err = cudaGetErrorString(e);
    if (mp) cudaFree(mp);
    t = BuildWTables();
    return e;
  }
  t.d_mp = mp;
  t.ok = true;
  return cudaSuccess;
}

void build_w_tables_destroy(BuildWTables& t) {
  if (t.d_mp) cudaFree(t.d_mp);
  t = BuildWTables();
}

bool tc_build_w_supported(const LscDims& d, const BuildWTables& t) {
  // Other channel counts keep the CUDA-core build's sums: a network's FP32 gradients would show the
  // other rounding (1e-4 of W's entries a BF16 step away)
  if (!tc_enabled() || !t.ok || d.c_in < 1 || 128 % d.c_in != 0 || d.in_blk != (int64_t)d.c_in * d.n_in) return false;
  if (bw_smem(d.n_in, d.c_in, d.in_blk, d.K, 1) > kBwSmemLimit) return false;
  int dev = 0, major = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, dev);
  return major == 10;
}

cudaError_t tc_build_w(const LscDims& d, const BuildWTables& t, const float* w, const float* b, const float* q, void* W,
                       float* bias_vec, int* err, cudaStream_t st) {
  TraceScope trace("lsc_build_w_tc", st);
  BwParams p;
  memset(&p, 0, sizeof p);
  p.d = d;
  p.w = w;
  p.img = static_cast<const uint8_t*>(t.d_mp);
  p.b = b;
  p.q = q;
  p.bias = bias_vec;
  p.W = static_cast<__nv_bfloat16*>(W);
  p.nh = bw_halves(d.n_in);
  p.hr = bw_hrows(d.n_in);
  p.nt = bw_tiles(d.n_in, d.n_out);
  p.atoms = bw_atoms(d.n_in);
  p.cpt = 128 / d.c_in;
  p.nptiles = (d.c_out + p.cpt - 1) / p.cpt;
  p.wld = bw_wld(d.K);
  p.pg_per_pair = d.m_stride_sp ? 1 : 0;
  p.img_bytes = (uint32_t)(3 * p.nh * p.atoms * kBwAtomBytes);
  p.w_bytes = (uint32_t)((128 * p.wld * 4 + 15) / 16 * 16);
  p.stg_bytes = (uint32_t)bw_stg_bytes(d.n_in, d.c_in, d.in_blk);
  p.ring = bw_smem(d.n_in, d.c_in, d.in_blk, d.K, 2) <= kBwSmemLimit ? 2 : 1;
  p.err = err;
  for (int s = 0; s < d.s_out; ++s) p.units += (int64_t)p.nt * std::max(0, d.win_hi[s] - d.win_lo[s]) * p.nptiles;
  if (p.units == 0) return cudaErrorInvalidValue;
  // at least 120 KiB so that two CTAs never share an SM (each holds 512 TMEM columns)
  const size_t smem = std::max<size_t>(120 * 1024, bw_smem(d.n_in, d.c_in, d.in_blk, d.K, p.ring));
  cudaError_t e = cudaFuncSetAttribute(build_w_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  build_w_tc_kernel<<<(unsigned)std::min<int64_t>(p.units, std::max(1, sms)), kBwThreads, smem, st>>>(p);
  count_launch();
  return cudaGetLastError();
}

}  // namespace delimit
