// ssd_bwd.cu -- backward of the SSD form (Mamba-2: one scalar decay per head,
// B and C shared by the channels) of the block-restricted bidirectional scan,
// on the tcgen05 tensor cores of sm_103a (Sec. 4.1, eq. prefix-cache-gradient;
// Appendix C for the Mamba-2 mixers).
//
// Per block of Bs tokens, head h and direction (forward: lower-triangular,
// seeded with the state before the block; reverse: upper-triangular), with
// c the in-block cumulative dt (prefix sums forward, suffix sums reverse),
// decay[t, s] = exp(A (c_t - c_s)) on the direction's triangle, G = C B^T,
// Q = dy x^T, R' = Q o G o decay and R = R' diag(dt):
//   dx  = (G o decay diag(dt))^T dy          dC = (Q o decay diag(dt)) B
//   dB  = (Q o decay diag(dt))^T C           seed term y += diag(E) C S^T,
//   E_t = exp(A c_t): dC += diag(E) dy S, dS = (diag(E) dy)^T C,
//   dc_t = A (rowsum_t R - colsum_t R + E_t dy_t . (C S^T)_t),
//   ddt_r = colsum_r R' + sum of dc over the tokens whose c includes dt_r,
//   dA = sum_t c_t dc_t / A.
// The clean stream adds the reverse pass over block-end states
// (S_k = exp(A sumdt_k) S_{k-1} + T_k, T_k = sum_s w_s x_s B_s^T,
// w_s = exp(A sum_{r>s} dt_r) dt_s) and the transpose of T_k.
//
// Kernels: k_ssd_bwd_tile (tcgen05: the products of one 128-token tile of a
// block against every s-tile its direction reaches, one head per CTA),
// k_ssd_bwd_vec (dt, A gradients from the row and column sums), k_ssd_bwd_pass
// (reverse state pass), k_ssd_bwd_state (tcgen05: the block-state transpose),
// and fixed-order combines in ssd_api.cu's launch sequence.
#include <cstring>

#include "device.cuh"
#include "params.h"
#include "ssd.cuh"
#include "ssd_common.cuh"
#include "umma.cuh"

namespace bds {
namespace {

using umma::sw128;

constexpr int kStateBwdThreads = 256;  // k_ssd_bwd_state
constexpr int kTileThreads = 256;  // k_ssd_bwd_tile: two threads per token row

// Copies `rows` rows of `ncols` (64 or 128) bf16 into 128-byte-swizzled atom
// columns of rows * 128 bytes each, by NT threads; a null source stages zeros.
template <int NT>
__device__ __forceinline__ void stage_bf16(unsigned char* dst, const __nv_bfloat16* src, int64_t ld, int rows,
                                           int ncols) {
  const int cpr = ncols / 8;
  for (int c = threadIdx.x; c < rows * cpr; c += NT) {
    const int r = c / cpr, ch = c % cpr;
    unsigned char* d = dst + (uint32_t)(ch >> 3) * (uint32_t)rows * 128u + sw128((uint32_t)r, (uint32_t)(ch & 7));
    if (src == nullptr)
      *reinterpret_cast<uint4*>(d) = make_uint4(0u, 0u, 0u, 0u);
    else
      cp_async16(d, src + (int64_t)r * ld + ch * 8, 16);
  }
}

// An fp32 [ROWS][NC] matrix (row stride NC) as bf16 high parts bf16(v) at
// `dhi` and low parts bf16(v - bf16(v)) at `dlo` (atom columns of ROWS * 128
// bytes each), by NT threads; every load is issued before the first store.
template <int NT, int ROWS, int NC>
__device__ __forceinline__ void stage_f32_hilo(unsigned char* dhi, unsigned char* dlo, const float* src) {
  constexpr int cpr = NC / 8, per = ROWS * cpr / NT;
  static_assert(ROWS * cpr % NT == 0, "whole chunks per thread");
  float4 a[per], b[per];
#pragma unroll
  for (int q = 0; q < per; ++q) {
    const int c = (int)threadIdx.x + q * NT, r = c / cpr, ch = c % cpr;
    a[q] = *reinterpret_cast<const float4*>(src + (int64_t)r * NC + ch * 8);
    b[q] = *reinterpret_cast<const float4*>(src + (int64_t)r * NC + ch * 8 + 4);
  }
#pragma unroll
  for (int q = 0; q < per; ++q) {
    const int c = (int)threadIdx.x + q * NT, r = c / cpr, ch = c % cpr;
    const float v[8] = {a[q].x, a[q].y, a[q].z, a[q].w, b[q].x, b[q].y, b[q].z, b[q].w};
    uint32_t hi[4], lo[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const __nv_bfloat162 hv = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
      hi[e] = *reinterpret_cast<const uint32_t*>(&hv);
      lo[e] = pack_bf16(__fsub_rn(v[2 * e], __low2float(hv)), __fsub_rn(v[2 * e + 1], __high2float(hv)));
    }
    const uint32_t off = (uint32_t)(ch >> 3) * (uint32_t)ROWS * 128u + sw128((uint32_t)r, (uint32_t)(ch & 7));
    *reinterpret_cast<uint4*>(dhi + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
    *reinterpret_cast<uint4*>(dlo + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
  }
}

// Stores a warp's 32 x 32 fp32 block (lane r holds row r in v) to rows
// dst + r * ld (16-byte aligned, ld a multiple of 4), through a warp-private
// buffer tb of 1024 floats (16-byte chunks XOR-swizzled by row), so that each
// store instruction writes four 128-byte row segments.
__device__ __forceinline__ void store_block32(float* dst, int64_t ld, const float (&v)[32], float* tb) {
  const int r = threadIdx.x & 31;
#pragma unroll
  for (int c4 = 0; c4 < 8; ++c4)
    *reinterpret_cast<float4*>(tb + r * 32 + 4 * (c4 ^ (r & 7))) =
        make_float4(v[4 * c4], v[4 * c4 + 1], v[4 * c4 + 2], v[4 * c4 + 3]);
  __syncwarp();
  const int c4 = r & 7;
#pragma unroll
  for (int rr = 0; rr < 32; rr += 4) {
    const int row = rr + (r >> 3);
    *reinterpret_cast<float4*>(dst + row * ld + 4 * c4) =
        *reinterpret_cast<const float4*>(tb + row * 32 + 4 * (c4 ^ (row & 7)));
  }
  __syncwarp();
}
// 32 consecutive fp32 columns of this thread's TMEM lane, written (the
// counterpart of umma::tmem_ld32); tmem_wait_st() orders them before later loads.
__device__ __forceinline__ void tmem_st32(uint32_t ta, const float (&v)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
      "%15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};\n" ::"r"(ta),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])), "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])), "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])), "r"(__float_as_uint(v[15])), "r"(__float_as_uint(v[16])), "r"(__float_as_uint(v[17])), "r"(__float_as_uint(v[18])), "r"(__float_as_uint(v[19])), "r"(__float_as_uint(v[20])), "r"(__float_as_uint(v[21])), "r"(__float_as_uint(v[22])), "r"(__float_as_uint(v[23])), "r"(__float_as_uint(v[24])), "r"(__float_as_uint(v[25])), "r"(__float_as_uint(v[26])), "r"(__float_as_uint(v[27])), "r"(__float_as_uint(v[28])), "r"(__float_as_uint(v[29])), "r"(__float_as_uint(v[30])), "r"(__float_as_uint(v[31])));
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Barrier of the warp pair q, q + 4 of a k_ssd_bwd_tile CTA (the two column
// halves of the same 32 token rows): named barrier 1 + q over 64 threads.
__device__ __forceinline__ void pair_sync(int q) {
  asm volatile("bar.sync %0, 64;\n" ::"r"(1 + q) : "memory");
}

// bf16 high parts bf16(v) and low parts bf16(v - bf16(v)) of a pair
__device__ __forceinline__ void split_pair(float a, float b, uint32_t& hi, uint32_t& lo) {
  const __nv_bfloat162 hv = __floats2bfloat162_rn(a, b);
  hi = *reinterpret_cast<const uint32_t*>(&hv);
  lo = pack_bf16(__fsub_rn(a, __low2float(hv)), __fsub_rn(b, __high2float(hv)));
}

// Shared memory of k_ssd_bwd_tile (offsets from a 1024-aligned base).
//   C    C of tile i, [128 t][128 n] (n >= N zero)    BT  B of s-tile j, [128 s][N]
//   X    x of s-tile j, one head, [128 s][64 p]       DY  dy of tile i, one head, [128 t][64 p]
//   M    one head's M' = G o decay, bf16 high part, [128 t][128 s]
//   COL  its low part (same layout); after the head's D product, per-warp
//        32 x 32 fp32 transposition blocks of the dx stores
//   VEC  c and dt of the block for every head of the group, [2][16][256] fp32
//   CP   the second column half's partial of the column sums, [128] fp32
//   ROWS row sums per head of the group [16][128], row dots per column half [2][16][128]
//   CF   the current head's column factors exp(A (c_ref - c_s)) and their products with dt_s
// After a s-tile's heads, the head-summed dG goes to M (bf16 high part) and
// X + DY (low part). The seed phase uses DY, BT for E o dy, M for the seed's
// bf16 high and low parts.
struct TileSmem {
  static constexpr uint32_t C = 0, BT = 32768, X = 65536, DY = 81920, M = 98304, COL = 131072;
  static constexpr uint32_t VEC = COL + 128u * 65u * 4u;
  static constexpr uint32_t CP = VEC + 2u * 16u * 256u * 4u;
  static constexpr uint32_t ROWS = CP + 4u * 64u * 4u;
  static constexpr uint32_t CF = ROWS + 3u * 16u * 128u * 4u;  // one head's column factors, and times dt [2][256]
  static constexpr uint32_t total = CF + 2u * 256u * 4u + 1024u;
};
constexpr int kMaxBwdHeads = 16;  // heads per tile CTA

// One CTA of 8 warps per (batch row, block, tile i) and group of heads. Token
// row t of tile i (TMEM lane t) has two threads, t and t + 128: the first
// takes columns 0..63 of every 128-column product, the second 64..127 (a
// warp reaches the TMEM lanes 32 (warp mod 4) onward). Row s = t of s-tile j
// is the column-side row. Per s-tile j the Gram tile G = C_i B_j^T is shared
// by the group's heads; per head, Q = dy x^T, the masked decays M' = G o
// decay (bf16 high and low parts), D = M'^T dy (then dx_j = diag(dt) D and
// the column sums of R' as x_s . D_s, since R'[t, s] = (dy_t . x_s)
// M'[t, s]), and dG = Q o decay o dt summed over the heads in fp32 in TMEM. dC and dB_j then take the head-summed dG once (B and C are
// shared by the heads), split into bf16 high and low parts. TMEM: G, then
// dB_j (and the seed products) at 0; Q, then D at 128; the head sum of dG
// at 256; dC at 384.
template <int N, bool UPPER, bool SEED>
__global__ void __launch_bounds__(kTileThreads, 1) k_ssd_bwd_tile(const SsdBwdTileParams p,
                                                                  const __grid_constant__ CUtensorMap xmap,
                                                                  const __grid_constant__ CUtensorMap dymap) {
  pdl_sync();
  extern __shared__ unsigned char smraw[];
  unsigned char* sm = align1024(smraw);
  __shared__ uint64_t bar, bar_ld;  // MMAs; a head's x and dy tiles (TMA)
  __shared__ uint32_t tslot;
  using S = TileSmem;
  constexpr int NT = kTileThreads;
  const SsdGeo& g = p.g;
  const int Bs = (int)g.Bs, H = g.H, m = g.m, tid = threadIdx.x, w = tid >> 5;
  const int t = tid & 127, half = tid >> 7;  // token row, column half
  const int64_t idx = blockIdx.x;
  const int i = (int)(idx % m);
  const int64_t bk = idx / m, b = bk / g.nb;
  const int k = (int)(bk % g.nb);
  const int grp = blockIdx.y, ngrp = gridDim.y;
  const int h0 = grp * p.hg, h1 = min(H, h0 + p.hg), hg = h1 - h0;
  // debug build: the tile, the head group and its last dx partial lie inside the sizes
  if (!(dguard(kSiteSsdBwdTile, idx, g.Bt * g.nb * m) && dguard(kSiteSsdBwdTile, h0, H) &&
        dguard(kSiteSsdBwdTile, (((bk * H + h1 - 1) * m + i) * Bs + Bs - 1) * kSsdP + kSsdP - 1,
               g.Bt * g.nb * H * m * g.Bs * kSsdP)))
    return;
  const int64_t tok0 = b * g.L + (int64_t)k * Bs;  // the block's first token
  const int64_t HP = (int64_t)H * kSsdP;
  float* s_cv = reinterpret_cast<float*>(sm + S::VEC);  // [hh][256]: c of every head of the group
  float* s_dtv = s_cv + kMaxBwdHeads * 256;              // [hh][256]: dt
  float* s_col = reinterpret_cast<float*>(sm + S::COL);
  float* s_cp = reinterpret_cast<float*>(sm + S::CP);
  float* s_cf = reinterpret_cast<float*>(sm + S::CF);  // [256]
  float* s_cfd = s_cf + 256;                           // [256]
  float* s_rows = reinterpret_cast<float*>(sm + S::ROWS);                              // [hh][128]
  float* s_dots = s_rows + kMaxBwdHeads * 128 + half * kMaxBwdHeads * 128;             // [hh][128] of this half

  stage_bf16<NT>(sm + S::C, p.C + (tok0 + i * kSsdT) * N, N, 128, N);
  if (N == 64)
    for (int c = tid; c < 128 * 8; c += NT) *reinterpret_cast<uint4*>(sm + S::C + kTile16 + c * 16) = make_uint4(0u, 0u, 0u, 0u);
  cp_async_commit();
  for (int hh = 0; hh < kMaxBwdHeads; ++hh) {
    if (half == 0) s_rows[hh * 128 + t] = 0.f;
    s_dots[hh * 128 + t] = 0.f;
  }
  // dt and its in-block cumulative sums of every head of the group, once per
  // CTA: warp w takes heads w, w + 8
  for (int hh = w; hh < hg; hh += NT / 32) {
    const int h = h0 + hh;
    warp_scan_dt<UPPER>(p.dt + tok0 * H + h, H, Bs, s_cv + hh * 256, s_dtv + hh * 256);
  }
  if (tid == 0) {
    umma::bar_init(&bar, 1);
    umma::bar_init(&bar_ld, 1);
  }
  if (w == 0) tmem_alloc(&tslot, 512);
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tm = tslot, lane_base = tm + ((uint32_t)(32 * (w & 3)) << 16);
  const int tt = i * kSsdT + t;
  uint32_t phase = 0, ldphase = 0;
  bool alive = true, ld_pending = false;  // a TMA phase issued and not yet waited for
  const uint32_t y0 = umma::smem_u32(sm + S::DY), c0 = umma::smem_u32(sm + S::C), x0 = umma::smem_u32(sm + S::X),
                 b0 = umma::smem_u32(sm + S::BT), m0 = umma::smem_u32(sm + S::M);
  constexpr uint32_t id_gq = umma::idesc_bf16(128, 128, false, false);
  constexpr uint32_t id_dc = umma::idesc_bf16(128, N, false, true);
  constexpr uint32_t id_dx = umma::idesc_bf16(128, 64, true, true);
  constexpr uint32_t id_db = umma::idesc_bf16(128, N, true, true);
  auto wait_mma = [&]() {
    if (!cta_wait(&bar, phase, p.flag)) return false;
    phase ^= 1u;
    umma::fence_after_sync();
    return true;
  };
  const int j0 = UPPER ? i : 0, j1 = UPPER ? m - 1 : i;
  for (int j = j0; j <= j1 && alive; ++j) {
    const int64_t sr0 = tok0 + (int64_t)j * kSsdT;
    // x and dy of head hh are staged after head hh-1's dx products (head 0's
    // with B_j): the copies run during the previous head's epilogue
    // (by TMA, thread 0, when the launcher set up the maps; a missing dy is
    // zero-filled by the threads)
    auto stage_head = [&](int hh) {
      const int h = h0 + hh;
      if (p.tma) {
        if (tid == 0) {
          umma::fence_async_smem();  // earlier generic accesses of X and DY before the async writes
          bar_expect_tx(&bar_ld, p.dy != nullptr ? 32768u : 16384u);
          tma_load_3d(sm + S::X, &xmap, 0, h, (int)sr0, &bar_ld);
          if (p.dy != nullptr) tma_load_3d(sm + S::DY, &dymap, 0, h, (int)(tok0 + i * kSsdT), &bar_ld);
        }
        ld_pending = true;
        if (p.dy == nullptr) stage_bf16<NT>(sm + S::DY, nullptr, HP, 128, 64);
      } else {
        stage_bf16<NT>(sm + S::X, p.x + (sr0 * H + h) * kSsdP, HP, 128, 64);
        stage_bf16<NT>(sm + S::DY, p.dy != nullptr ? p.dy + ((tok0 + i * kSsdT) * H + h) * kSsdP : nullptr, HP, 128,
                       64);
      }
    };
    stage_bf16<NT>(sm + S::BT, p.B + sr0 * N, N, 128, N);
    stage_head(0);
    cp_async_commit();
    cp_async_wait_all();
    umma::fence_async_smem();
    umma::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      umma::fence_after_sync();
      const uint64_t dc = umma::sdesc(c0, 16, 1024), db = umma::sdesc(b0, 16, 1024);
#pragma unroll
      for (int kk = 0; kk < N / 16; ++kk) {  // G = C_i B_j^T, shared by the heads
        const uint32_t off = (uint32_t)(kk >> 2) * kTile16 + (uint32_t)(kk & 3) * 32u;
        umma::mma_bf16(tm, umma::sdesc_adv(dc, off), umma::sdesc_adv(db, off), id_gq, kk > 0);
      }
      umma::mma_commit(&bar);
    }
    if (!(alive = wait_mma())) break;
    for (int hh = 0; hh < hg; ++hh) {
      const int h = h0 + hh;
      // column factors of this head: exp(A (c_ref - c_s)), with c_ref the
      // cumulative dt at the last (forward) or first (reverse) token of s's
      // 32-token group, and their products with dt_s (the previous head's
      // element-wise phase is past the barrier before its dx products)
      if (tid < Bs) {
        const float* c = s_cv + hh * 256;
        const float cf = ex2(__fmul_rn(__fmul_rn(p.A[h], kLog2e), __fsub_rn(c[UPPER ? (tid & ~31) : (tid | 31)], c[tid])));
        s_cf[tid] = cf;
        s_cfd[tid] = __fmul_rn(cf, s_dtv[hh * 256 + tid]);
      }
      if (p.tma) {  // every staged head completes one phase of the load barrier
        if (!cta_wait(&bar_ld, ldphase, p.flag)) {
          alive = false;
          break;
        }
        ldphase ^= 1u;
        ld_pending = false;
      } else {
        cp_async_wait_all();
      }
      umma::fence_async_smem();
      umma::fence_before_sync();
      __syncthreads();
      if (tid == 0) {
        umma::fence_after_sync();
        const uint64_t dy = umma::sdesc(y0, 16, 1024), dx = umma::sdesc(x0, 16, 1024);
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)  // Q = dy_i x_j^T
          umma::mma_bf16(tm + 128u, umma::sdesc_adv(dy, kk * 32u), umma::sdesc_adv(dx, kk * 32u), id_gq, kk > 0);
        umma::mma_commit(&bar);
      }
      if (!(alive = wait_mma())) break;
      const float* s_c = s_cv + hh * 256;
      const float* s_dt = s_dtv + hh * 256;
      const float A2 = __fmul_rn(p.A[h], kLog2e), ct = s_c[tt];
      float rowsum = 0.f;
      // two rounds: round r takes 32-column chunk r (first half) and 2 + r
      // (second half), then the column sums of those 64 columns
#pragma unroll 1
      for (int r = 0; r < 2; ++r) {
        const int c = 2 * half + r;
        float gv[32], qv[32], dgs[32];
        umma::tmem_ld32(lane_base + 32u * (uint32_t)c, gv);
        umma::tmem_ld32(lane_base + 128u + 32u * (uint32_t)c, qv);
        if (hh > 0) umma::tmem_ld32(lane_base + 256u + 32u * (uint32_t)c, dgs);
        uint32_t mp[16], ml[16];  // M' as bf16 high and low parts, column pairs
        // the chunk's 32 columns against this warp's 32 rows: entirely inside
        // the direction's triangle (the decay factors into a row factor times
        // the column factors, both at most 1), the diagonal 32 x 32 block
        // (one ex2 per element, masked), or entirely outside (zero)
        const int rq = w & 3;  // the warp's row group in the tile
        const int mode = UPPER ? (j > i || c > rq ? 1 : (c == rq ? 2 : 0)) : (j < i || c < rq ? 1 : (c == rq ? 2 : 0));
        const int s0 = j * kSsdT + 32 * c;
        if (mode == 1) {
          const float rf = ex2(__fmul_rn(A2, __fsub_rn(ct, s_c[UPPER ? s0 : s0 + 31])));
          const float2 rf2 = f2(rf);
          float2 rs2 = f2(0.f);
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            const float2 cf = *reinterpret_cast<const float2*>(s_cf + s0 + e);
            const float2 cfd = *reinterpret_cast<const float2*>(s_cfd + s0 + e);
            const float2 g2 = make_float2(gv[e], gv[e + 1]), q2 = make_float2(qv[e], qv[e + 1]);
            const float2 L = mul2(rf2, cf), Ld = mul2(rf2, cfd);
            const float2 dg = mul2(q2, Ld);
            rs2 = fma2(g2, dg, rs2);
            const float2 old2 = make_float2(dgs[e], dgs[e + 1]);
            const float2 nd = hh > 0 ? add2(old2, dg) : dg;
            dgs[e] = nd.x;
            dgs[e + 1] = nd.y;
            const float2 mv = mul2(g2, L);
            split_pair(mv.x, mv.y, mp[e >> 1], ml[e >> 1]);
          }
          rowsum = __fadd_rn(rowsum, __fadd_rn(rs2.x, rs2.y));
        } else if (mode == 2) {
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            float mv[2];
#pragma unroll
            for (int q = 0; q < 2; ++q) {
              const int s = s0 + e + q;
              const bool valid = UPPER ? (s >= tt) : (s <= tt);
              const float L = valid ? ex2(__fmul_rn(A2, __fsub_rn(ct, s_c[s]))) : 0.f;
              const float ds = s_dt[s];
              const float gl = __fmul_rn(gv[e + q], L);
              rowsum = __fmaf_rn(__fmul_rn(qv[e + q], gl), ds, rowsum);
              const float dg = __fmul_rn(__fmul_rn(qv[e + q], L), ds);
              dgs[e + q] = hh > 0 ? __fadd_rn(dgs[e + q], dg) : dg;
              mv[q] = gl;
            }
            split_pair(mv[0], mv[1], mp[e >> 1], ml[e >> 1]);
          }
        } else {
#pragma unroll
          for (int e = 0; e < 32; e += 2) {
            if (hh == 0) dgs[e] = dgs[e + 1] = 0.f;
            mp[e >> 1] = ml[e >> 1] = 0u;
          }
        }
        tmem_st32(lane_base + 256u + 32u * (uint32_t)c, dgs);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int chunk = 4 * c + u;
          const uint32_t off = (uint32_t)(chunk >> 3) * kTile16 + sw128((uint32_t)t, (uint32_t)(chunk & 7));
          *reinterpret_cast<uint4*>(sm + S::M + off) = make_uint4(mp[4 * u], mp[4 * u + 1], mp[4 * u + 2], mp[4 * u + 3]);
          *reinterpret_cast<uint4*>(sm + S::COL + off) = make_uint4(ml[4 * u], ml[4 * u + 1], ml[4 * u + 2], ml[4 * u + 3]);
        }
      }
      if (half == 0) s_rows[hh * 128 + t] = __fadd_rn(s_rows[hh * 128 + t], rowsum);  // the second half after the barrier
      tmem_wait_st();
      umma::fence_async_smem();
      umma::fence_before_sync();
      __syncthreads();
      if (tid == 0) {
        umma::fence_after_sync();
        const uint64_t dy = umma::sdesc(y0, kTile16, 1024);
#pragma unroll
        for (int part = 0; part < 2; ++part) {  // D = M'^T dy_i: M' read as an MN-major operand (M = s, K = t)
          const uint64_t dm = umma::sdesc(part ? umma::smem_u32(sm + S::COL) : m0, kTile16, 1024);
#pragma unroll
          for (int kk = 0; kk < 8; ++kk)
            umma::mma_bf16(tm + 128u, umma::sdesc_adv(dm, kk * 2048u), umma::sdesc_adv(dy, kk * 2048u), id_dx,
                           part > 0 || kk > 0);
        }
        umma::mma_commit(&bar);
      }
      if (half == 1) s_rows[hh * 128 + t] = __fadd_rn(s_rows[hh * 128 + t], rowsum);
      if (!(alive = wait_mma())) break;
      {  // row s = j*128 + t of D, channels 32 half ..: the column sum of R'
         // is x_s . D_s, this half's 32 channels in order and then the two
         // halves; head h's dx contribution from tile i is dt_s D_s
        float v[32];
        umma::tmem_ld32(lane_base + 128u + 32u * (uint32_t)half, v);
        float cs = 0.f;
#pragma unroll
        for (int cq = 0; cq < 4; ++cq) {
          const uint4 u = *reinterpret_cast<const uint4*>(sm + S::X + sw128((uint32_t)t, (uint32_t)(4 * half + cq)));
          const __nv_bfloat162* x2 = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const float2 f = __bfloat1622float2(x2[e]);
            cs = __fmaf_rn(f.x, v[8 * cq + 2 * e], cs);
            cs = __fmaf_rn(f.y, v[8 * cq + 2 * e + 1], cs);
          }
        }
        if (p.dd_part != nullptr && j == i) {  // x and dy tiles of the same tokens: the skip term's dy . x
          float dd = 0.f;
#pragma unroll
          for (int cq = 0; cq < 4; ++cq) {
            const uint32_t off = sw128((uint32_t)t, (uint32_t)(4 * half + cq));
            const uint4 ux = *reinterpret_cast<const uint4*>(sm + S::X + off);
            const uint4 uy = *reinterpret_cast<const uint4*>(sm + S::DY + off);
            const __nv_bfloat162* x2 = reinterpret_cast<const __nv_bfloat162*>(&ux);
            const __nv_bfloat162* y2 = reinterpret_cast<const __nv_bfloat162*>(&uy);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const float2 fx = __bfloat1622float2(x2[e]), fy = __bfloat1622float2(y2[e]);
              dd = __fmaf_rn(fy.x, fx.x, dd);
              dd = __fmaf_rn(fy.y, fx.y, dd);
            }
          }
          dd = warp_sum(dd);
          if ((tid & 31) == 0) p.dd_part[((bk * H + h) * m + i) * 8 + w] = dd;
        }
        if (half == 1) s_cp[t] = cs;
        pair_sync(w & 3);  // warps w and w + 4 hold the two halves of the same rows
        if (half == 0) p.col_part[((bk * H + h) * m + i) * Bs + j * kSsdT + t] = __fadd_rn(cs, s_cp[t]);
        if (hh + 1 < hg) {  // X and DY are free: the next head's copies start now
          stage_head(hh + 1);
          cp_async_commit();
        }
        const float ds = s_dtv[hh * 256 + j * kSsdT + t];
#pragma unroll
        for (int e = 0; e < 32; ++e) v[e] = __fmul_rn(ds, v[e]);
        // the warp's 32 x 32 block goes out through COL (free after the D product)
        store_block32(p.dx_part + (((bk * H + h) * m + i) * Bs + j * kSsdT + 32 * (w & 3)) * kSsdP + 32 * half, kSsdP,
                      v, s_col + w * 1024);
      }
      umma::fence_before_sync();
    }
    if (!alive) break;
    // the head-summed dG as bf16 high (M) and low (X + DY) parts
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {
      const int c = 2 * half + r;
      float dgs[32];
      umma::tmem_ld32(lane_base + 256u + 32u * (uint32_t)c, dgs);
      uint32_t hi[16], lo[16];
#pragma unroll
      for (int e = 0; e < 32; e += 2) {
        const __nv_bfloat162 hv = __floats2bfloat162_rn(dgs[e], dgs[e + 1]);
        hi[e >> 1] = *reinterpret_cast<const uint32_t*>(&hv);
        lo[e >> 1] = pack_bf16(__fsub_rn(dgs[e], __low2float(hv)), __fsub_rn(dgs[e + 1], __high2float(hv)));
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int chunk = 4 * c + u;
        const uint32_t off = (uint32_t)(chunk >> 3) * kTile16 + sw128((uint32_t)t, (uint32_t)(chunk & 7));
        *reinterpret_cast<uint4*>(sm + S::M + off) = make_uint4(hi[4 * u], hi[4 * u + 1], hi[4 * u + 2], hi[4 * u + 3]);
        *reinterpret_cast<uint4*>(sm + S::X + off) = make_uint4(lo[4 * u], lo[4 * u + 1], lo[4 * u + 2], lo[4 * u + 3]);
      }
    }
    umma::fence_async_smem();
    umma::fence_before_sync();
    __syncthreads();
    if (tid == 0) {
      umma::fence_after_sync();
      const uint64_t db = umma::sdesc(b0, kTile16, 1024), dc = umma::sdesc(c0, kTile16, 1024);
#pragma unroll
      for (int part = 0; part < 2; ++part) {
        const uint32_t dg0 = part ? x0 : m0;
        const uint64_t dgk = umma::sdesc(dg0, 16, 1024), dgm = umma::sdesc(dg0, kTile16, 1024);
#pragma unroll
        for (int kk = 0; kk < 8; ++kk) {
          const uint32_t koff = (uint32_t)(kk >> 2) * kTile16 + (uint32_t)(kk & 3) * 32u, mn = (uint32_t)kk * 2048u;
          // dC += dG B_j: dG K-major [t][s], B_j MN-major [s][n]
          umma::mma_bf16(tm + 384u, umma::sdesc_adv(dgk, koff), umma::sdesc_adv(db, mn), id_dc,
                         j != j0 || part > 0 || kk > 0);
          // dB_j = dG^T C_i: dG read as MN-major (M = s)
          umma::mma_bf16(tm, umma::sdesc_adv(dgm, mn), umma::sdesc_adv(dc, mn), id_db, part > 0 || kk > 0);
        }
      }
      umma::mma_commit(&bar);
    }
    if (!(alive = wait_mma())) break;
    {  // rows s = j*128 + 32 (w mod 4) .. of the group's dB contribution from
       // tile i, N/2 columns per half, through the warp's block of COL
      float v[32];
      float* dbo = p.dB_part + (((bk * ngrp + grp) * m + i) * Bs + j * kSsdT + 32 * (w & 3)) * N;
#pragma unroll
      for (int q = half * (N / 64); q < (half + 1) * (N / 64); ++q) {
        umma::tmem_ld32(lane_base + 32u * (uint32_t)q, v);
        store_block32(dbo + 32 * q, N, v, s_col + w * 1024);
      }
    }
    umma::fence_before_sync();
  }

  if (alive && SEED && k > 0) {
    // seed products per head: dC += (E o dy) S, the row dot dy_t . E_t (C_t S^T)
    // and the seed gradient (E o dy)^T C; the seed as bf16 high and low parts.
    // With TMA the next head's dy tile (DY and X alternate) and raw seed (into
    // COL, free here) arrive under the current head's MMAs and epilogue.
    constexpr uint32_t id_cs = umma::idesc_bf16(128, 64, false, false);
    const float* seeds = p.states + (b * g.nb + k - 1) * H * (int64_t)kSsdP * N;  // head h at h * 64 N
    auto seed_loads = [&](int hh) {
      if (tid == 0) {
        umma::fence_async_smem();  // earlier generic accesses of the buffers before the async writes
        bar_expect_tx(&bar_ld, (p.dy != nullptr ? 16384u : 0u) + (uint32_t)(kSsdP * N * 4));
        if (p.dy != nullptr)
          tma_load_3d(sm + ((hh & 1) ? S::X : S::DY), &dymap, 0, h0 + hh, (int)(tok0 + i * kSsdT), &bar_ld);
        bulk_load(sm + S::COL, seeds + (int64_t)(h0 + hh) * kSsdP * N, (uint32_t)(kSsdP * N * 4), &bar_ld);
      }
      ld_pending = true;
    };
    __syncthreads();  // the last dB stores went through COL
    if (p.tma) seed_loads(0);
    for (int hh = 0; hh < hg && alive; ++hh) {
      const int h = h0 + hh;
      const uint32_t dyo = (p.tma && (hh & 1)) ? S::X : S::DY;  // this head's dy tile
      if (p.tma) {
        if (p.dy == nullptr) stage_bf16<NT>(sm + dyo, nullptr, HP, 128, 64);
        if (!cta_wait(&bar_ld, ldphase, p.flag)) {
          alive = false;
          break;
        }
        ldphase ^= 1u;
        ld_pending = false;
        stage_f32_hilo<NT, 64, N>(sm + S::M, sm + S::M + 16384u, reinterpret_cast<const float*>(sm + S::COL));
      } else {
        stage_bf16<NT>(sm + S::DY, p.dy != nullptr ? p.dy + ((tok0 + i * kSsdT) * H + h) * kSsdP : nullptr, HP, 128, 64);
        cp_async_commit();
        stage_f32_hilo<NT, 64, N>(sm + S::M, sm + S::M + 16384u, seeds + (int64_t)h * kSsdP * N);
        cp_async_wait_all();
      }
      __syncthreads();
      // the seeded direction is the forward one: s_cv holds prefix sums
      const float E = ex2(__fmul_rn(__fmul_rn(p.A[h], kLog2e), s_cv[hh * 256 + tt]));
#pragma unroll
      for (int cq = 0; cq < 4; ++cq) {  // 16-byte chunks 4 half .. 4 half + 3 of row t
        const int ch = 4 * half + cq;
        const uint4 u = *reinterpret_cast<const uint4*>(sm + dyo + sw128((uint32_t)t, (uint32_t)ch));
        const __nv_bfloat162* v2 = reinterpret_cast<const __nv_bfloat162*>(&u);
        uint32_t o[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = __bfloat1622float2(v2[e]);
          o[e] = pack_bf16(__fmul_rn(E, f.x), __fmul_rn(E, f.y));
        }
        *reinterpret_cast<uint4*>(sm + S::BT + sw128((uint32_t)t, (uint32_t)ch)) = make_uint4(o[0], o[1], o[2], o[3]);
      }
      umma::fence_async_smem();
      umma::fence_before_sync();
      __syncthreads();
      if (tid == 0) {
        umma::fence_after_sync();
        const uint64_t dbk = umma::sdesc(b0, 16, 1024), dck = umma::sdesc(c0, 16, 1024);
        const uint64_t dbm = umma::sdesc(b0, kTile16, 1024), dcm = umma::sdesc(c0, kTile16, 1024);
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          const uint32_t s0 = m0 + (part ? 16384u : 0u);
          const uint64_t dsm = umma::sdesc(s0, 8192, 1024), dsk = umma::sdesc(s0, 16, 1024);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)  // dC += (E o dy) S: S MN-major [p][n], atom columns of 8 KB
            umma::mma_bf16(tm + 384u, umma::sdesc_adv(dbk, kk * 32u), umma::sdesc_adv(dsm, kk * 2048u), id_dc, true);
#pragma unroll
          for (int kk = 0; kk < N / 16; ++kk)  // C S^T: S K-major [p][n]
            umma::mma_bf16(tm, umma::sdesc_adv(dck, (kk >> 2) * kTile16 + (kk & 3) * 32u),
                           umma::sdesc_adv(dsk, (kk >> 2) * 8192u + (kk & 3) * 32u), id_cs, part > 0 || kk > 0);
        }
#pragma unroll
        for (int kk = 0; kk < 8; ++kk)  // dS^T = C_i^T (E o dy): C read as MN-major (M = n)
          umma::mma_bf16(tm + 64u, umma::sdesc_adv(dcm, kk * 2048u), umma::sdesc_adv(dbm, kk * 2048u), id_dx, kk > 0);
        umma::mma_commit(&bar);
      }
      if (p.tma && hh + 1 < hg) seed_loads(hh + 1);  // COL and the other dy buffer are free
      if (!(alive = wait_mma())) break;
      float v[32], rowdot = 0.f;  // channels 32 half .. 32 half + 31 of the row dot, in order
      umma::tmem_ld32(lane_base + 32u * (uint32_t)half, v);
#pragma unroll
      for (int cq = 0; cq < 4; ++cq) {
        const uint4 u = *reinterpret_cast<const uint4*>(sm + dyo + sw128((uint32_t)t, (uint32_t)(4 * half + cq)));
        const __nv_bfloat162* v2 = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = __bfloat1622float2(v2[e]);
          rowdot = __fmaf_rn(f.x, v[8 * cq + 2 * e], rowdot);
          rowdot = __fmaf_rn(f.y, v[8 * cq + 2 * e + 1], rowdot);
        }
      }
      s_dots[hh * 128 + t] = __fmul_rn(E, rowdot);
      if (32 * (w & 3) < N) {  // row n = t of dS^T, channels 32 half ..: the seed gradient partial [p][n]
        float* dso = p.dS_part + ((bk * H + h) * m + i) * (int64_t)kSsdP * N + t;
        umma::tmem_ld32(lane_base + 64u + 32u * (uint32_t)half, v);
#pragma unroll
        for (int e = 0; e < 32; ++e) dso[(int64_t)(32 * half + e) * N] = v[e];
      }
      umma::fence_before_sync();
      __syncthreads();  // BT, M and this head's dy buffer are restaged for the next heads
    }
  }
  if (alive) {  // dC of rows 32 (w mod 4) .. of tile i, summed over the group's heads, N/2 columns per half
    float v[32];
    float* dco = p.dC_part + ((bk * ngrp + grp) * Bs + i * kSsdT + 32 * (w & 3)) * N;
#pragma unroll
    for (int q = half * (N / 64); q < (half + 1) * (N / 64); ++q) {
      umma::tmem_ld32(lane_base + 384u + 32u * (uint32_t)q, v);
      store_block32(dco + 32 * q, N, v, s_col + w * 1024);
    }
  }
  __syncthreads();  // both halves' row sums and dots are in shared memory
  if (alive) {
    const float* dots = s_rows + kMaxBwdHeads * 128;  // [half][hh][128]
    for (int hh = half; hh < hg; hh += 2) {
      const int h = h0 + hh;
      p.rowsum[(bk * H + h) * Bs + tt] = s_rows[hh * 128 + t];
      if (SEED) p.rowdot[(bk * H + h) * Bs + tt] = __fadd_rn(dots[hh * 128 + t], dots[(kMaxBwdHeads + hh) * 128 + t]);
    }
  }
  cp_async_wait_all();
  if (ld_pending) umma::bar_wait(&bar_ld, ldphase);  // after a give-up: the copies in flight, bounded
  umma::fence_before_sync();
  __syncthreads();
  if (w == 0) tmem_dealloc(tm, 512);
}

// In-place inclusive scan of n fp32 values (n a multiple of 32, at most 256)
// by one warp; REV scans from the end (suffix sums).
template <bool REV>
__device__ __forceinline__ void warp_scan_f32(float* a, int n) {
  const int lane = threadIdx.x & 31, per = n / 32;
  float loc[8];
  float s = 0.f;
  for (int q = 0; q < per; ++q) {
    const int pos = REV ? n - 1 - (lane * per + q) : lane * per + q;
    s = __fadd_rn(s, a[pos]);
    loc[q] = s;
  }
  float inc = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const float v = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc = __fadd_rn(inc, v);
  }
  float base = __shfl_up_sync(0xffffffffu, inc, 1);
  if (lane == 0) base = 0.f;
  __syncwarp();
  for (int q = 0; q < per; ++q) {
    const int pos = REV ? n - 1 - (lane * per + q) : lane * per + q;
    a[pos] = __fadd_rn(base, loc[q]);
  }
  __syncwarp();
}


// One warp per (batch row, block, head) and stream (blockIdx.y): dc_t = A (rowsum_t - dt_t colsum'_t +
// rowdot_t), ddt_r = colsum'_r + sum of dc over the tokens whose cumulative dt
// includes dt_r (t >= r forward, t <= r reverse), dA = sum_t c_t (dc_t / A).
__global__ void __launch_bounds__(128) k_ssd_bwd_vec(const __grid_constant__ SsdBwdVecParams prm) {
  pdl_sync();
  __shared__ float s_c[4][256], s_q[4][256], s_col[4][256];
  const SsdGeo& g = prm.g;
  const SsdBwdVecStream& p = prm.s[blockIdx.y];
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, Bs = (int)g.Bs, m = g.m, H = g.H;
  const int64_t u = (int64_t)blockIdx.x * 4 + w;
  if (u >= g.Bt * g.nb * H) return;  // whole warps
  const int h = (int)(u % H);
  const int64_t bk = u / H, b = bk / g.nb, k = bk % g.nb;
  const int64_t tok0 = b * g.L + k * Bs;
  const float total = p.upper ? warp_scan_dt<true>(p.dt + tok0 * H + h, H, Bs, s_c[w])
                              : warp_scan_dt<false>(p.dt + tok0 * H + h, H, Bs, s_c[w]);
  if (p.sumdt != nullptr && lane == 0) p.sumdt[bk * H + h] = total;
  __syncwarp();
  const float A = p.A[h];
  float dA = 0.f;
  const float* colp = p.col_part + (bk * H + h) * (int64_t)m * Bs;
  for (int s = lane; s < Bs; s += 32) {
    const int js = s / kSsdT;
    float col = 0.f;
    for (int i = p.upper ? 0 : js; i <= (p.upper ? js : m - 1); ++i) col = __fadd_rn(col, colp[(int64_t)i * Bs + s]);
    const float dt = __bfloat162float(p.dt[(tok0 + s) * H + h]);
    float q = __fsub_rn(p.rowsum[(bk * H + h) * Bs + s], __fmul_rn(dt, col));
    if (p.rowdot != nullptr) q = __fadd_rn(q, p.rowdot[(bk * H + h) * Bs + s]);
    dA = __fmaf_rn(s_c[w][s], q, dA);
    s_q[w][s] = __fmul_rn(A, q);
    s_col[w][s] = col;
  }
  __syncwarp();
  if (p.upper)
    warp_scan_f32<false>(s_q[w], Bs);  // reverse: c_t sums dt over r >= t, so dt_r feeds every t <= r
  else
    warp_scan_f32<true>(s_q[w], Bs);   // forward: dt_r feeds every t >= r
  for (int s = lane; s < Bs; s += 32) {
    const float v = __fadd_rn(s_col[w][s], s_q[w][s]);
    if (p.ddt_out != nullptr)
      p.ddt_out[(tok0 + s) * H + h] = __float2bfloat16_rn(v);
    else
      p.ddt[(tok0 + s) * H + h] = v;
  }
  dA = warp_sum(dA);
  if (lane == 0) p.dA[bk * H + h] = dA;
}

// One thread per (batch row, head, channel, state index), blocks last to first.
__global__ void __launch_bounds__(256) k_ssd_bwd_pass(const SsdBwdPassParams p) {
  pdl_sync();
  const SsdGeo& g = p.g;
  const int64_t PN = (int64_t)kSsdP * g.N, per_b = (int64_t)g.H * PN;
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (idx >= g.Bt * per_b) return;
  const int64_t b = idx / per_b, r = idx - b * per_b;
  const int h = (int)(r / PN);
  const int64_t pn = r - (int64_t)h * PN;
  const float A2 = __fmul_rn(p.A[h], kLog2e);
  float gS = 0.f;
  // m is 1 or 2 (blocks of 128 or 256 tokens). The loads of U blocks are
  // issued before the reverse recurrence uses them: they do not depend on gS.
  const bool two = g.m > 1;
  constexpr int U = 8;
  for (int k0 = g.nb - 1; k0 >= 0; k0 -= U) {
    float f0[U], f1[U], c0[U], c1[U], ext[U], sdt[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 - u;
      f0[u] = f1[u] = c0[u] = c1[u] = ext[u] = sdt[u] = 0.f;
      if (k < 0) continue;
      if (k + 1 < g.nb) {  // the seed gradients of block k+1 (forward noisy direction, then clean)
        const int64_t base = ((b * g.nb + k + 1) * g.H + h) * (int64_t)g.m * PN + pn;
        f0[u] = p.dS_f[base];
        c0[u] = p.dS_c[base];
        if (two) {
          f1[u] = p.dS_f[base + PN];
          c1[u] = p.dS_c[base + PN];
        }
      }
      if (p.dstates != nullptr) ext[u] = p.dstates[((b * g.nb + k) * g.H + h) * PN + pn];
      sdt[u] = p.sumdt[(b * g.nb + k) * g.H + h];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = k0 - u;
      if (k < 0) break;
      if (k + 1 < g.nb) {
        float inj = f0[u];
        if (two) inj = __fadd_rn(inj, f1[u]);
        inj = __fadd_rn(inj, c0[u]);
        if (two) inj = __fadd_rn(inj, c1[u]);
        gS = __fadd_rn(gS, inj);
      }
      if (p.dstates != nullptr) gS = __fadd_rn(gS, ext[u]);
      p.gS[((b * g.nb + k) * g.H + h) * PN + pn] = gS;
      gS = __fmul_rn(ex2(__fmul_rn(A2, sdt[u])), gS);
    }
  }
}

// Shared memory of k_ssd_bwd_state (from a 1024-aligned base):
//   G     the state gradient's bf16 high and low parts ([64 p][N] each, atom
//         columns of 8 KB); after the products per-warp 32 x 32 fp32
//         transposition blocks of the stores
//   RAW   the next state gradient as loaded (fp32)
//   X     two buffers of a head's x tiles; BT the block's B tiles
//   SUF   per head of the CTA the dt after each token, DT its dt (bf16), DW
//         x . U (one tile per block: of each half of the channels)
struct StateBwdSmem {
  uint32_t g, raw, x, bt, suf, dt, dw, total;
  __host__ __device__ StateBwdSmem(int N, int m, int hg) {
    g = 0;
    raw = 32768u;
    x = raw + 256u * (uint32_t)N;
    bt = x + 2u * (uint32_t)m * 16384u;
    suf = bt + (uint32_t)(m * (N / 64)) * kTile16;
    dw = suf + (uint32_t)hg * (uint32_t)m * 512u;
    dt = dw + (uint32_t)hg * 1024u;
    total = dt + (uint32_t)hg * (uint32_t)m * 256u + 1024u;
  }
};

// One CTA of 8 warps per (batch row, block) of the clean stream and group of
// heads, with gS = the gradient of the state after the block. Per head and
// 128-token tile U = B gS^T and V = x gS on the tensor core (gS split into
// bf16 high and low parts), then dx = w U, dw = x . U, and the dt and A
// gradients of w and of the block decay. dB is shared by the heads: w V is
// summed over the group's heads in registers, one row (two tiles) or half a
// row (one tile) per thread, and leaves once per group. The next head's gS, x
// and previous state arrive under the current head's products and epilogue.
// Bound by memory and the chain of a head's steps: 8 x 8192 x 26 heads x 128
// moves 1.1 GB in 342 us. A CTA per head, with 0.87 GB of per-head dB written
// here and read back by k_ssd_bwd_dbc, took 518 us (and the combine 241 for 109).
template <int N, bool TWO>
__global__ void __launch_bounds__(kStateBwdThreads, 1) k_ssd_bwd_state(const SsdBwdStateParams p) {
  pdl_sync();
  extern __shared__ unsigned char smraw[];
  unsigned char* sm = align1024(smraw);
  __shared__ uint64_t bar;
  __shared__ uint32_t tslot;
  __shared__ float red[kMaxStateBwdHeads][kStateBwdThreads / 32];
  constexpr int NT = kStateBwdThreads, m = TWO ? 2 : 1, Bs = 128 * m;
  constexpr int UC = TWO ? 64 : 32, VC = TWO ? N : N / 2;  // columns of U and V per thread
  const SsdGeo& g = p.g;
  const int H = g.H, tid = threadIdx.x, w = tid >> 5, lane = tid & 31, t = tid & 127, half = tid >> 7;
  const int64_t bk = blockIdx.x, b = bk / g.nb;
  const int k = (int)(bk % g.nb);
  const int grp = blockIdx.y, h0 = grp * p.hg, hg = min(H, h0 + p.hg) - h0;
  // debug build: the block and the heads lie inside the sizes
  if (!(dguard(kSiteSsdBwdState, bk, g.Bt * g.nb) && dguard(kSiteSsdBwdState, h0 + hg - 1, H))) return;
  const StateBwdSmem S(N, m, p.hg);
  const int64_t tok0 = b * g.L + (int64_t)k * Bs, HP = (int64_t)H * kSsdP, PN = (int64_t)kSsdP * N;
  float* s_suf = reinterpret_cast<float*>(sm + S.suf);                  // [hh][Bs]
  float* s_dw = reinterpret_cast<float*>(sm + S.dw);                    // [hh][256]
  __nv_bfloat16* s_dt = reinterpret_cast<__nv_bfloat16*>(sm + S.dt);    // [hh][Bs]
  const float* gS = p.gS + (bk * H + h0) * PN;                          // head h0 + hh at hh PN
  const float* prev = k > 0 ? p.states + ((bk - 1) * H + h0) * PN : nullptr;

  auto load_head = [&](int hh) {  // gS and x of head h0 + hh
    for (int c = tid; c < kSsdP * N / 4; c += NT) cp_async16(sm + S.raw + c * 16, gS + hh * PN + c * 4, 16);
#pragma unroll
    for (int j = 0; j < m; ++j)
      stage_bf16<NT>(sm + S.x + (uint32_t)((hh & 1) * m + j) * 16384u, p.x + ((tok0 + j * kSsdT) * H + h0 + hh) * kSsdP,
                     HP, 128, 64);
    cp_async_commit();
  };
  constexpr int cpr = N / 8, per = kSsdP * cpr / NT;  // 8-element pieces of a state matrix per thread
  float4 pa[per], pb[per];                            // the previous state's, for the block decay's gradient
  auto load_prev = [&](int hh) {
#pragma unroll
    for (int q = 0; q < per; ++q) {
      const float* src = prev + hh * PN + (tid + q * NT) * 8;
      pa[q] = prev != nullptr ? *reinterpret_cast<const float4*>(src) : make_float4(0.f, 0.f, 0.f, 0.f);
      pb[q] = prev != nullptr ? *reinterpret_cast<const float4*>(src + 4) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
#pragma unroll
  for (int j = 0; j < m; ++j)
    stage_bf16<NT>(sm + S.bt + (uint32_t)(j * (N / 64)) * kTile16, p.B + (tok0 + j * kSsdT) * N, N, 128, N);
  load_head(0);
  load_prev(0);
  for (int hh = w; hh < hg; hh += NT / 32) {  // dt and the dt after each token
    const __nv_bfloat16* dth = p.dt + tok0 * H + h0 + hh;
    float* suf = s_suf + hh * Bs;
    warp_scan_dt<true>(dth, H, Bs, suf);
    __syncwarp();
    for (int s = lane; s < Bs; s += 32) {
      const __nv_bfloat16 d = dth[(int64_t)s * H];
      s_dt[hh * Bs + s] = d;
      suf[s] = __fsub_rn(suf[s], __bfloat162float(d));
    }
  }
  if (tid == 0) umma::bar_init(&bar, 1);
  constexpr uint32_t kCols = m * (N + 64) <= 128 ? 128 : m * (N + 64) <= 256 ? 256 : 512;
  if (w == 0) tmem_alloc(&tslot, kCols);
  umma::fence_before_sync();
  __syncthreads();
  umma::fence_after_sync();
  const uint32_t tm = tslot, lane_base = tm + ((uint32_t)(32 * (w & 3)) << 16);
  const uint32_t gh = umma::smem_u32(sm + S.g), x0 = umma::smem_u32(sm + S.x), b0 = umma::smem_u32(sm + S.bt);
  constexpr uint32_t kGLow = 64u * (uint32_t)N * 2u;                        // low parts after the high ones
  constexpr uint32_t kU = m * N;                                            // TMEM: V_j at N j, U_j at kU + 64 j
  constexpr uint32_t id_u = umma::idesc_bf16(128, 64, false, false);
  constexpr uint32_t id_v = umma::idesc_bf16(128, N, false, true);
  const int tile = TWO ? half : 0, row = tile * kSsdT + t;                  // this thread's token
  const uint32_t ucol = kU + (TWO ? 64u * (uint32_t)half : 32u * (uint32_t)half);
  const uint32_t vcol = TWO ? (uint32_t)(N * half) : (uint32_t)(VC * half);
  const int u0 = TWO ? 0 : 32 * half;                                       // first channel of the thread's U columns
  const int64_t row0 = tile * kSsdT + 32 * (w & 3);                         // the warp's first token
  float* tb = reinterpret_cast<float*>(sm + S.g) + w * 1024;
  float acc[VC];
#pragma unroll
  for (int e = 0; e < VC; ++e) acc[e] = 0.f;
  bool alive = true;
  for (int hh = 0; hh < hg; ++hh) {
    cp_async_wait_all();
    __syncthreads();  // the head's gS and x have landed; the transposition blocks are no longer read
    float da = 0.f;   // the block decay's: sum over (p, n) of gS o S_{k-1}
#pragma unroll
    for (int q = 0; q < per; ++q) {
      const int c = tid + q * NT, r = c / cpr, ch = c % cpr;
      const float4 ga = *reinterpret_cast<const float4*>(sm + S.raw + c * 32);
      const float4 gb = *reinterpret_cast<const float4*>(sm + S.raw + c * 32 + 16);
      const float v[8] = {ga.x, ga.y, ga.z, ga.w, gb.x, gb.y, gb.z, gb.w};
      const float u[8] = {pa[q].x, pa[q].y, pa[q].z, pa[q].w, pb[q].x, pb[q].y, pb[q].z, pb[q].w};
      uint32_t hi[4], lo[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) split_pair(v[2 * e], v[2 * e + 1], hi[e], lo[e]);
#pragma unroll
      for (int e = 0; e < 8; ++e) da = __fmaf_rn(v[e], u[e], da);
      const uint32_t off = (uint32_t)(ch >> 3) * 64u * 128u + sw128((uint32_t)r, (uint32_t)(ch & 7));
      *reinterpret_cast<uint4*>(sm + S.g + off) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
      *reinterpret_cast<uint4*>(sm + S.g + kGLow + off) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
    }
    umma::fence_async_smem();
    umma::fence_before_sync();
    __syncthreads();
    const uint32_t xo = (uint32_t)((hh & 1) * m) * 16384u;
    if (tid == 0) {
      umma::fence_after_sync();
#pragma unroll
      for (int j = 0; j < m; ++j) {
        const uint64_t db = umma::sdesc(b0 + (uint32_t)(j * (N / 64)) * kTile16, 16, 1024),
                       dx = umma::sdesc(x0 + xo + (uint32_t)j * 16384u, 16, 1024);
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          const uint32_t gs0 = gh + (part ? kGLow : 0u);
          const uint64_t dgk = umma::sdesc(gs0, 16, 1024), dgm = umma::sdesc(gs0, 8192, 1024);
#pragma unroll
          for (int kk = 0; kk < N / 16; ++kk)  // U = B_j gS^T: gS K-major [p][n]
            umma::mma_bf16(tm + kU + 64u * j, umma::sdesc_adv(db, (kk >> 2) * kTile16 + (kk & 3) * 32u),
                           umma::sdesc_adv(dgk, (kk >> 2) * 8192u + (kk & 3) * 32u), id_u, part > 0 || kk > 0);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)  // V = x_j gS: gS MN-major [p][n]
            umma::mma_bf16(tm + (uint32_t)(N * j), umma::sdesc_adv(dx, kk * 32u), umma::sdesc_adv(dgm, kk * 2048u), id_v,
                           part > 0 || kk > 0);
        }
      }
      umma::mma_commit(&bar);
    }
    if (hh + 1 < hg) {
      load_head(hh + 1);
      load_prev(hh + 1);
    }
    da = warp_sum(da);
    if (lane == 0) red[hh][w] = da;
    if (!cta_wait(&bar, (uint32_t)(hh & 1), p.flag)) {
      alive = false;
      break;
    }
    umma::fence_after_sync();
    const float A2 = __fmul_rn(p.A[h0 + hh], kLog2e);
    const float ws = __fmul_rn(ex2(__fmul_rn(A2, s_suf[hh * Bs + row])), __bfloat162float(s_dt[hh * Bs + row]));
    float v[32], dw = 0.f;
    float* dxo = p.dx_state + ((bk * H + h0 + hh) * Bs + row0) * kSsdP + u0;
#pragma unroll
    for (int q = 0; q < UC / 32; ++q) {
      umma::tmem_ld32(lane_base + ucol + 32u * (uint32_t)q, v);
      const unsigned char* xr = sm + S.x + xo + (uint32_t)tile * 16384u;
#pragma unroll
      for (int cq = 0; cq < 4; ++cq) {
        const uint4 xv = *reinterpret_cast<const uint4*>(xr + sw128((uint32_t)t, (uint32_t)(u0 / 8 + 4 * q + cq)));
        const __nv_bfloat162* x2 = reinterpret_cast<const __nv_bfloat162*>(&xv);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = __bfloat1622float2(x2[e]);
          dw = __fmaf_rn(f.x, v[8 * cq + 2 * e], dw);
          dw = __fmaf_rn(f.y, v[8 * cq + 2 * e + 1], dw);
        }
      }
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = __fmul_rn(ws, v[e]);
      store_block32(dxo + 32 * q, kSsdP, v, tb);
    }
#pragma unroll
    for (int q = 0; q < VC / 32; ++q) {
      umma::tmem_ld32(lane_base + vcol + 32u * (uint32_t)q, v);
#pragma unroll
      for (int e = 0; e < 32; ++e) acc[32 * q + e] = __fmaf_rn(ws, v[e], acc[32 * q + e]);
    }
    s_dw[hh * 256 + half * 128 + t] = dw;
    umma::fence_before_sync();
  }
  cp_async_wait_all();
  __syncthreads();
  if (alive) {
    float* dbo = p.dB_state + ((bk * gridDim.y + grp) * Bs + row0) * N + (TWO ? 0 : VC * half);
    float v[32];
#pragma unroll
    for (int q = 0; q < VC / 32; ++q) {
#pragma unroll
      for (int e = 0; e < 32; ++e) v[e] = acc[32 * q + e];
      store_block32(dbo + 32 * q, N, v, tb);
    }
    // the exponent of w_s is A times the dt after s: dt_r feeds every s < r
    for (int hh = w; hh < hg; hh += NT / 32) {
      const int h = h0 + hh;
      float* suf = s_suf + hh * Bs;
      const float* dwv = s_dw + hh * 256;
      const float A = p.A[h], A2 = __fmul_rn(A, kLog2e);
      float da = red[hh][0], dA = 0.f, ev[Bs / 32], dv[Bs / 32];
#pragma unroll
      for (int q = 1; q < NT / 32; ++q) da = __fadd_rn(da, red[hh][q]);
#pragma unroll
      for (int q = 0; q < Bs / 32; ++q) {
        const int s = lane + 32 * q;
        const float dw = TWO ? dwv[s] : __fadd_rn(dwv[s], dwv[128 + s]);
        ev[q] = ex2(__fmul_rn(A2, suf[s]));
        dv[q] = dw;
        const float wdw = __fmul_rn(__fmul_rn(ev[q], __bfloat162float(s_dt[hh * Bs + s])), dw);
        dA = __fmaf_rn(suf[s], wdw, dA);
        suf[s] = __fmul_rn(A, wdw);
      }
      __syncwarp();
      warp_scan_f32<false>(suf, Bs);  // inclusive prefix sums of A w dw
      const float sd = p.sumdt[bk * H + h], ak = ex2(__fmul_rn(A2, sd));
      const float blk = __fmul_rn(__fmul_rn(A, ak), da);  // block decay exp(A sumdt) of S_{k-1}
#pragma unroll
      for (int q = 0; q < Bs / 32; ++q) {
        const int r = lane + 32 * q;
        const float before = r > 0 ? suf[r - 1] : 0.f;  // exclusive: s < r
        const float vs = __fadd_rn(__fadd_rn(__fmul_rn(ev[q], dv[q]), before), blk);
        const int64_t o = (tok0 + r) * H + h;
        p.ddt[o] = __float2bfloat16_rn(__fadd_rn(p.ddt_tile[o], vs));
      }
      dA = warp_sum(dA);
      if (lane == 0) p.dA[bk * H + h] = __fadd_rn(dA, __fmul_rn(__fmul_rn(sd, ak), da));
    }
  }
  umma::fence_before_sync();
  __syncthreads();
  if (w == 0) tmem_dealloc(tm, kCols);
}

}  // namespace

namespace {

__device__ __forceinline__ float4 add4(float4 a, float4 b) {
  return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z), __fadd_rn(a.w, b.w));
}
__device__ __forceinline__ float4 ld4(const float* p) { return *reinterpret_cast<const float4*>(p); }
__device__ __forceinline__ float4 bf4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  const float2 a = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.x));
  const float2 b = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&u.y));
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ void st_bf4(__nv_bfloat16* p, float4 v) {
  const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
  *reinterpret_cast<uint2*>(p) = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
}

// dx of both streams: the tile partials of every tile that reaches s (tiles
// i >= j(s) forward, i <= j(s) reverse), the clean state term and the skip
// terms. One thread per (token, head, 4 channels).
__global__ void __launch_bounds__(256) k_ssd_bwd_dx(const SsdGeo g, const float* dxp_c, const float* dxs,
                                                    const float* dxp_f, const float* dxp_r, const __nv_bfloat16* dyc,
                                                    const __nv_bfloat16* dyn, const float* Df, const float* Dr,
                                                    __nv_bfloat16* dxc, __nv_bfloat16* dxn) {
  pdl_sync();
  constexpr int Q = kSsdP / 4;  // 4-channel groups per head
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= g.Bt * g.L * g.H * Q) return;
  const int64_t bt = i / (g.H * Q);
  const int hq = (int)(i - bt * g.H * Q), h = hq / Q, pp = (hq - h * Q) * 4;
  const int64_t b = bt / g.L;
  const int tl = (int)(bt - b * g.L), k = tl / (int)g.Bs, s = tl - k * (int)g.Bs, j = s / kSsdT, m = g.m;
  const int64_t hb = (b * g.nb + k) * g.H + h, idx = (bt * g.H + h) * kSsdP + pp;
  const int64_t stride_i = (int64_t)g.Bs * kSsdP;  // between the tile partials of one head
  const int64_t po = (hb * m * g.Bs + s) * kSsdP + pp;
  // m is 1 or 2: only the tiles that reach s are read (j is the same for a
  // warp's threads but at the ends of 128-token tiles), every load before
  // the sums (in the order i = j..m-1 forward, 0..j reverse)
  const bool two = m > 1;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  const float4 c0 = j == 0 ? ld4(dxp_c + po) : z, f0 = j == 0 ? ld4(dxp_f + po) : z, r0 = ld4(dxp_r + po);
  const float4 c1 = two ? ld4(dxp_c + po + stride_i) : z, f1 = two ? ld4(dxp_f + po + stride_i) : z,
               r1 = j == 1 ? ld4(dxp_r + po + stride_i) : z;
  const float4 st = ld4(dxs + (hb * g.Bs + s) * kSsdP + pp);
  const float4 yc = dyc != nullptr ? bf4(dyc + idx) : z, yn = bf4(dyn + idx);
  float4 c = j == 0 ? c0 : z, n = j == 0 ? f0 : z;
  if (two) {
    c = j == 0 ? add4(c, c1) : c1;
    n = j == 0 ? add4(n, f1) : f1;
  }
  c = add4(c, st);
  const float dc = Df[h], dn = __fadd_rn(Df[h], Dr[h]);
  if (dyc != nullptr)
    c = make_float4(__fmaf_rn(dc, yc.x, c.x), __fmaf_rn(dc, yc.y, c.y), __fmaf_rn(dc, yc.z, c.z), __fmaf_rn(dc, yc.w, c.w));
  n = add4(n, r0);
  if (j == 1) n = add4(n, r1);
  n = make_float4(__fmaf_rn(dn, yn.x, n.x), __fmaf_rn(dn, yn.y, n.y), __fmaf_rn(dn, yn.z, n.z), __fmaf_rn(dn, yn.w, n.w));
  st_bf4(dxc + idx, c);
  st_bf4(dxn + idx, n);
}

// dB and dC of the three streams: the tile partials of every head group (and
// the clean state term of its own head groups), summed in order. One thread per
// (token, 4 state indices); the tile index j of a token is the same across
// a warp but at the ends of 128-token tiles, and only the tile partials that
// reach the token are read.
__global__ void __launch_bounds__(256) k_ssd_bwd_dbc(const SsdGeo g, int ngrp, int ngrp_state, const float* dBp_c,
                                                     const float* dBs,
                                                     const float* dCp_c, const float* dBp_f, const float* dCp_f,
                                                     const float* dBp_r, const float* dCp_r, __nv_bfloat16* dBc,
                                                     __nv_bfloat16* dCc, __nv_bfloat16* dBf, __nv_bfloat16* dCf,
                                                     __nv_bfloat16* dBr, __nv_bfloat16* dCr) {
  pdl_sync();
  const int N = g.N, m = g.m, Q = N / 4;
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= g.Bt * g.L * Q) return;
  const int64_t bt = i / Q, b = bt / g.L;
  const int n = (int)(i - bt * Q) * 4;
  const int tl = (int)(bt - b * g.L), k = tl / (int)g.Bs, s = tl - k * (int)g.Bs, j = s / kSsdT;
  const int64_t bk = b * g.nb + k, idx = bt * N + n;
  const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 bc = z, cc = z, bf = z, cf = z, br = z, cr = z;
  const bool two = m > 1;
  for (int q = 0; q < ngrp; ++q) {
    const int64_t gb = bk * ngrp + q;
    const int64_t tp = (gb * m * g.Bs + s) * N + n, ti = (int64_t)g.Bs * N, c1 = (gb * g.Bs + s) * N + n;
    // m is 1 or 2: the loads first, then the sums in the order i = j..m-1
    // (forward), 0..j (reverse)
    const float4 bc0 = j == 0 ? ld4(dBp_c + tp) : z, bf0 = j == 0 ? ld4(dBp_f + tp) : z, br0 = ld4(dBp_r + tp);
    const float4 bc1 = two ? ld4(dBp_c + tp + ti) : z, bf1 = two ? ld4(dBp_f + tp + ti) : z,
                 br1 = j == 1 ? ld4(dBp_r + tp + ti) : z;
    const float4 cc0 = ld4(dCp_c + c1), cf0 = ld4(dCp_f + c1), cr0 = ld4(dCp_r + c1);
    if (j == 0) {
      bc = add4(bc, bc0);
      bf = add4(bf, bf0);
    }
    if (two) {
      bc = add4(bc, bc1);
      bf = add4(bf, bf1);
    }
    br = add4(br, br0);
    if (j == 1) br = add4(br, br1);
    cc = add4(cc, cc0);
    cf = add4(cf, cf0);
    cr = add4(cr, cr0);
  }
  const float* st = dBs + (bk * ngrp_state * g.Bs + s) * N + n;
  for (int q = 0; q < ngrp_state; ++q) bc = add4(bc, ld4(st + (int64_t)q * g.Bs * N));
  st_bf4(dBc + idx, bc);
  st_bf4(dCc + idx, cc);
  st_bf4(dBf + idx, bf);
  st_bf4(dCf + idx, cf);
  st_bf4(dBr + idx, br);
  st_bf4(dCr + idx, cr);
}

// Parameter gradients per head: one CTA per head; thread t sums the (batch
// row, block) partials t, t + 256, ... in order (the dy . x partials of a
// block in tile and warp order), then a fixed tree over the threads, so the
// result does not depend on scheduling.
__global__ void __launch_bounds__(256) k_ssd_bwd_par(const SsdGeo g, const float* dd_c, const float* dd_n,
                                                     const float* dA_c, const float* dA_f, const float* dA_s,
                                                     const float* dA_r, float* dAf, float* dDf, float* dAr,
                                                     float* dDr) {
  pdl_sync();
  __shared__ float4 red[256];
  const int h = blockIdx.x, t = threadIdx.x, nd = g.m * 8;
  float af = 0.f, ar = 0.f, df = 0.f, dr = 0.f;
  for (int64_t bk = t; bk < g.Bt * g.nb; bk += 256) {
    const int64_t o = bk * g.H + h;
    af = __fadd_rn(af, __fadd_rn(__fadd_rn(dA_c[o], dA_f[o]), dA_s[o]));
    ar = __fadd_rn(ar, dA_r[o]);
    float sc = 0.f, sn = 0.f;
    for (int q = 0; q < nd; ++q) {
      sc = __fadd_rn(sc, dd_c[o * nd + q]);
      sn = __fadd_rn(sn, dd_n[o * nd + q]);
    }
    df = __fadd_rn(df, __fadd_rn(sc, sn));
    dr = __fadd_rn(dr, sn);
  }
  red[t] = make_float4(af, ar, df, dr);
  __syncthreads();
  for (int w = 128; w > 0; w >>= 1) {
    if (t < w) {
      const float4 u = red[t], v = red[t + w];
      red[t] = make_float4(__fadd_rn(u.x, v.x), __fadd_rn(u.y, v.y), __fadd_rn(u.z, v.z), __fadd_rn(u.w, v.w));
    }
    __syncthreads();
  }
  if (t == 0) {
    const float4 r = red[0];
    dAf[h] = r.x;
    dAr[h] = r.y;
    dDf[h] = r.z;
    dDr[h] = r.w;
  }
}

template <int N, bool UPPER, bool SEED>
cudaError_t bwd_tile_t(const SsdBwdTileParams& p_in, cudaStream_t s) {
  const int smem = (int)TileSmem::total;
  cudaError_t e = set_smem_cached((const void*)k_ssd_bwd_tile<N, UPPER, SEED>, smem, -1);
  if (e != cudaSuccess) return e;
  SsdBwdTileParams p = p_in;
  CUtensorMap xmap, dymap;
  memset(&xmap, 0, sizeof(xmap));
  memset(&dymap, 0, sizeof(dymap));
  const int64_t rows = p.g.Bt * p.g.L;
  p.tma = encode_head_map(&xmap, p.x, rows, p.g.H) && (p.dy == nullptr || encode_head_map(&dymap, p.dy, rows, p.g.H))
              ? 1
              : 0;
  dim3 grid((unsigned)(p.g.Bt * p.g.nb * p.g.m), (unsigned)((p.g.H + p.hg - 1) / p.hg));
  launch_pdl(k_ssd_bwd_tile<N, UPPER, SEED>, grid, kTileThreads, smem, s, p, xmap, dymap);
  return cudaGetLastError();
}

template <int N, bool TWO>
cudaError_t bwd_state_t(const SsdBwdStateParams& p, cudaStream_t s) {
  const int smem = (int)StateBwdSmem(N, p.g.m, p.hg).total;
  cudaError_t e = set_smem_cached((const void*)k_ssd_bwd_state<N, TWO>, smem, -1);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)(p.g.Bt * p.g.nb), (unsigned)((p.g.H + p.hg - 1) / p.hg));
  launch_pdl(k_ssd_bwd_state<N, TWO>, grid, kStateBwdThreads, smem, s, p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_ssd_bwd_tile(bool upper, bool seeded, const SsdBwdTileParams& p, cudaStream_t s) {
  if (p.g.N == 64) {
    if (upper) return bwd_tile_t<64, true, false>(p, s);
    return seeded ? bwd_tile_t<64, false, true>(p, s) : bwd_tile_t<64, false, false>(p, s);
  }
  if (upper) return bwd_tile_t<128, true, false>(p, s);
  return seeded ? bwd_tile_t<128, false, true>(p, s) : bwd_tile_t<128, false, false>(p, s);
}

cudaError_t launch_ssd_bwd_vec(const SsdBwdVecParams& p, cudaStream_t s) {
  const int64_t warps = p.g.Bt * p.g.nb * p.g.H;
  launch_pdl(k_ssd_bwd_vec, dim3((unsigned)((warps + 3) / 4), 3), 128, 0, s, p);
  return cudaGetLastError();
}

cudaError_t launch_ssd_bwd_pass(const SsdBwdPassParams& p, cudaStream_t s) {
  const int64_t n = p.g.Bt * p.g.H * kSsdP * p.g.N;
  launch_pdl(k_ssd_bwd_pass, (unsigned)((n + 255) / 256), 256, 0, s, p);
  return cudaGetLastError();
}

cudaError_t launch_ssd_bwd_state(const SsdBwdStateParams& p, cudaStream_t s) {
  if (p.g.N == 64) return p.g.m == 2 ? bwd_state_t<64, true>(p, s) : bwd_state_t<64, false>(p, s);
  return p.g.m == 2 ? bwd_state_t<128, true>(p, s) : bwd_state_t<128, false>(p, s);
}

cudaError_t launch_ssd_bwd_dx(const SsdGeo& g, const float* dxp_c, const float* dxs, const float* dxp_f,
                              const float* dxp_r, const __nv_bfloat16* dyc, const __nv_bfloat16* dyn, const float* Df,
                              const float* Dr, __nv_bfloat16* dxc, __nv_bfloat16* dxn, cudaStream_t s) {
  const int64_t n = g.Bt * g.L * g.H * (kSsdP / 4);
  if (n == 0) return cudaSuccess;
  launch_pdl(k_ssd_bwd_dx, (unsigned)((n + 255) / 256), 256, 0, s, g, dxp_c, dxs, dxp_f, dxp_r, dyc, dyn, Df, Dr, dxc, dxn);
  return cudaGetLastError();
}

cudaError_t launch_ssd_bwd_dbc(const SsdGeo& g, int ngrp, int ngrp_state, const float* dBp_c, const float* dBs,
                               const float* dCp_c,
                               const float* dBp_f, const float* dCp_f, const float* dBp_r, const float* dCp_r,
                               __nv_bfloat16* dBc, __nv_bfloat16* dCc, __nv_bfloat16* dBf, __nv_bfloat16* dCf,
                               __nv_bfloat16* dBr, __nv_bfloat16* dCr, cudaStream_t s) {
  const int64_t n = g.Bt * g.L * (g.N / 4);
  if (n == 0) return cudaSuccess;
  launch_pdl(k_ssd_bwd_dbc, (unsigned)((n + 255) / 256), 256, 0, s, g, ngrp, ngrp_state, dBp_c, dBs,
             dCp_c, dBp_f, dCp_f, dBp_r, dCp_r, dBc, dCc, dBf, dCf, dBr, dCr);
  return cudaGetLastError();
}

cudaError_t launch_ssd_bwd_params(const SsdGeo& g, const float* dd_c, const float* dd_n, const float* dA_c,
                                  const float* dA_f, const float* dA_s, const float* dA_r, float* dAf, float* dDf,
                                  float* dAr, float* dDr, cudaStream_t s) {
  launch_pdl(k_ssd_bwd_par, (unsigned)g.H, 256, 0, s, g, dd_c, dd_n, dA_c, dA_f, dA_s, dA_r, dAf, dDf, dAr, dDr);
  return cudaGetLastError();
}

}  // namespace bds
