// fwd.cu -- forward-side kernels of libbdscan (sm_103a).
//
// The clean prefix scan (eq. boundary-state) is split into time chunks of
// m blocks (m = max(1, 128 / Bs)) so that Bt * D channels are not the only
// source of parallelism:
//   k_chunk_local  each (batch, chunk, 128 channels): scan the chunk from a
//                  zero state; keep the end state and the sum of dt.
//   k_chunk_carry  each (batch, channel, state): walk the chunks in order,
//                  H_{c+1} = exp(A * sum_c dt) * H_c + local_c, giving the
//                  exact state at every chunk start.
//   k_block_scan   each (batch, chunk, 128 channels): rescan the chunk from
//                  its start state, emitting y_c and the state at every
//                  block end; for every noisy block of the chunk, continue
//                  the state at its start through the noisy tokens (forward
//                  direction, eq. partial-reverse first line) and run the
//                  block-local reverse scan from zero (second line), and
//                  write their sum (third line).
//   k_active_block each (batch, 32 channels): one noisy block from a cached
//                  seed (the inference step), forward and reverse scans in
//                  two warps at once.
// The state at the end of a chunk's last block is taken from the carry
// kernel (the same value the next chunk starts from), so every consumer of
// a boundary state sees one value, and boundary states of a prefix equal
// those of any longer stream: chunking depends on Bs only.
#include "device.cuh"
#include "params.h"

namespace bds {

static_assert(kCta == kCtaHost, "host and device CTA widths differ");

constexpr int kLocalSpan = 32;  // tokens staged per step of the chunk-local scan
// Tokens the block scan stages at once: longer blocks are staged in segments
// of this many tokens (shared memory, and so residency, stays that of a
// 16-token block).
constexpr int kScanSeg = 16;

// REV: the scan runs right to left in time (logical token t is row L-1-t).
// Bound by the exponentials (one ex2 per token, channel and state) together
// with the packed FP32 operations around them: 262,144 x 2048 x 16 takes
// 1182 us, of which the ex2 alone need 853. The staged spans have a
// compile-time stride, so a token's addresses are immediates (1273 us with a
// run-time stride and half the unroll).
// A thread scans NS of the N states of its channel: N / NS CTAs share a channel
// group, and each stages the group's tokens for itself. All of them in one
// thread is the least work. With few CTAs the chunk's serial walk is what takes
// the time, and it is shorter over fewer states: four of them up to one CTA on
// each of the part's 152 SMs, eight up to two (128 tokens per chunk, N = 16; 16 / 8 / 4 states each:
// 4 CTAs 20.4 / 17.2 / 13.2 us, 128 CTAs 21.5 / 19.4 / 17.6, 304 CTAs
// 23.9 / 22.8 / 26.9, 608 CTAs 32.4 / 38.2 / 45.2; N = 8, 8 / 4 states: 15.0 /
// 14.0, 15.1 / 14.8, 17.3 / 17.2, 21.5 / 25.6). Each state is the same sequence
// of operations either way.
constexpr int kLocalQuarter = 152, kLocalHalf = 304;
template <typename T, int N, int NS, bool REV>
__global__ void __launch_bounds__(kCta) k_chunk_local(const FwdParams p) {
  pdl_sync();
  extern __shared__ __align__(16) unsigned char smem[];
  const Geo& g = p.g;
  const int64_t b = blockIdx.z;
  const int c = blockIdx.y;
  constexpr int Q = N / NS;
  const int n0 = (int)(blockIdx.x % Q) * NS;
  const int64_t d0 = (int64_t)(blockIdx.x / Q) * kCta, d = d0 + threadIdx.x;
  const bool act = d < g.D;
  {  // debug build: the chunk's tokens, channels and state slot lie inside the sizes
    const int64_t tc = (int64_t)g.m * g.Bs, dl = (d0 + kCta < g.D ? d0 + kCta : g.D) - 1;
    if (!(dguard(kSiteChunkLocal, b, g.Bt) && dguard(kSiteChunkLocal, (c + 1) * tc - 1, g.L) &&
          dguard(kSiteChunkLocal, d0, g.D) &&
          dguard(kSiteChunkLocal, ((b * (g.nc + 1) + c) * g.D + dl) * N + N - 1, g.Bt * (g.nc + 1) * g.D * N)))
      return;
  }
  Stage<T, N, 2, 1, 2, kLocalSpan, REV> st;
  st.carve(smem, kLocalSpan);
  auto prow = [&](int64_t t) { return b * g.L + (REV ? g.L - 1 - t : t); };  // row of logical token t
  st.td_src[0] = (const T*)p.xc;
  st.td_src[1] = (const T*)p.dtc;
  st.row_src[0] = (const T*)p.Bc;

  float2 A2[NS / 2], h[NS / 2];
  vzero2<NS>(A2);
  vzero2<NS>(h);
  if (act) {
    vload2<NS>(A2, p.Af + d * N + n0, 0);
#pragma unroll
    for (int j = 0; j < NS / 2; ++j) A2[j] = mul2(A2[j], f2(kLog2e));
  }
  float sdt = 0.f;
  const int64_t tc = (int64_t)g.m * g.Bs;
  const int64_t tbeg = (int64_t)c * tc;
  const int nspan = (int)((tc + kLocalSpan - 1) / kLocalSpan);
  st.issue(0, prow(tbeg), (int)(tc < kLocalSpan ? tc : kLocalSpan), g.D, d0);
  for (int sp = 0; sp < nspan; ++sp) {
    const int64_t t = (int64_t)sp * kLocalSpan;
    const int ns = (int)((tc - t) < kLocalSpan ? (tc - t) : kLocalSpan);
    __syncthreads();  // the other buffer is no longer read
    if (sp + 1 < nspan) {
      const int64_t tn = t + kLocalSpan;
      st.issue((sp + 1) & 1, prow(tbeg + tn), (int)((tc - tn) < kLocalSpan ? (tc - tn) : kLocalSpan), g.D, d0);
    }
    st.complete(sp & 1, ns, sp + 1 < nspan ? 1 : 0);
#pragma unroll 8
    for (int i = 0; i < ns; ++i) {
      const float dt = st.at(1, i);
      scan_state<NS>(h, A2, dt, st.at(0, i), st.row(0, i) + n0);
      sdt = __fadd_rn(sdt, dt);
    }
  }
  if (act) {
    vstore2<NS>(p.hst + ((b * (g.nc + 1) + c) * g.D + d) * N + n0, h, 0);
    if (n0 == 0) p.sdt[(b * g.nc + c) * g.D + d] = sdt;
  }
}

// The carry over a few chunks: one thread per (batch row, channel, state).
template <int N>
__global__ void __launch_bounds__(256) k_chunk_carry(const FwdParams p) {
  pdl_sync();
  const Geo& g = p.g;
  const int64_t idx = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (idx >= g.Bt * g.D * N) return;
  const int n = (int)(idx % N);
  const int64_t d = (idx / N) % g.D, b = idx / ((int64_t)N * g.D);
  // debug build: the last state slot this thread writes (no barrier follows)
  if (!dguard(kSiteChunkCarry, ((b * (g.nc + 1) + g.nc_full) * g.D + d) * N + n, g.Bt * (g.nc + 1) * g.D * N)) return;
  const float A2 = __fmul_rn(p.Af[d * N + n], kLog2e);
  float H = p.init ? p.init[(b * g.D + d) * N + n] : 0.f;
  const int64_t hstride = g.D * N;
  float* hs = p.hst + b * (g.nc + 1) * hstride + d * N + n;
  const float* sd = p.sdt + b * g.nc * g.D + d;
  constexpr int U = 8;
  int c = 0;
  for (; c + U <= g.nc_full; c += U) {
    float hl[U], s[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      hl[j] = hs[(int64_t)(c + j) * hstride];
      s[j] = sd[(int64_t)(c + j) * g.D];
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      hs[(int64_t)(c + j) * hstride] = H;
      H = __fmaf_rn(ex2(__fmul_rn(A2, s[j])), H, hl[j]);
    }
  }
  for (; c < g.nc_full; ++c) {
    const float hl = hs[(int64_t)c * hstride], s = sd[(int64_t)c * g.D];
    hs[(int64_t)c * hstride] = H;
    H = __fmaf_rn(ex2(__fmul_rn(A2, s)), H, hl);
  }
  hs[(int64_t)g.nc_full * hstride] = H;
  dfinite(kSiteChunkCarry, H, idx);  // debug build: a non-finite cached state
}

// The carry over chunks is one fused multiply-add per chunk and state, so the
// kernel is bound by how many bytes it keeps in flight. A CTA of 64 threads
// owns 64 consecutive (channel, state) elements of one batch row, one per
// thread, and streams the chunk rows (256 bytes of local end states plus the
// sums of dt) through a ring of kCarryStages cp.async groups of kCarryRows
// rows: 12 KB ahead of the chain per CTA: 2048 chunks x 32768 elements 102 us,
// 291 (1.8 TB/s) in k_chunk_carry, which has eight loads per thread in flight.
// Up to kCarryFew chunks that one is taken: with few rounds of loads the ring's
// fill is not made up for (16 chunks x 196608 elements: 7.8 us, 10.0 through
// the ring; 32 x 16384: 7.7 us either way).
constexpr int kCarryW = 64, kCarryRows = 16, kCarryStages = 4, kCarryFew = 32;
template <int N>
__global__ void __launch_bounds__(kCarryW) k_chunk_carry_ring(const FwdParams p) {
  pdl_sync();
  constexpr int CH = kCarryW / N;        // channels of the CTA's elements
  constexpr int HQ = kCarryW / 4, SQ = CH / 4;  // 16-byte pieces of one row of states, of dt sums
  __shared__ __align__(16) float hbuf[kCarryStages][kCarryRows][kCarryW];
  __shared__ __align__(16) float sbuf[kCarryStages][kCarryRows][CH];
  const Geo& g = p.g;
  const int64_t DN = g.D * N, b = blockIdx.y, e0 = (int64_t)blockIdx.x * kCarryW, e = e0 + threadIdx.x;
  const bool act = e < DN;
  // debug build: the last state slot the CTA writes
  if (!dguard(kSiteChunkCarry, (b * (g.nc + 1) + g.nc_full) * DN + (e0 + kCarryW < DN ? e0 + kCarryW : DN) - 1,
              g.Bt * (g.nc + 1) * DN))
    return;
  const float A2 = act ? __fmul_rn(p.Af[e], kLog2e) : 0.f;
  float H = act && p.init ? p.init[b * DN + e] : 0.f;
  float* hrow = p.hst + b * (g.nc + 1) * DN + e0;
  const float* srow = p.sdt + b * g.nc * g.D + e0 / N;
  const int nst = (g.nc_full + kCarryRows - 1) / kCarryRows;
  auto issue = [&](int st) {  // rows of stage st; pieces past the row's end or the last chunk are left out
    if (st < nst) {
      const int c0 = st * kCarryRows, slot = st % kCarryStages;
      for (int q = threadIdx.x; q < kCarryRows * HQ; q += kCarryW) {
        const int r = q / HQ, j = (q - r * HQ) * 4;
        if (c0 + r < g.nc_full && e0 + j < DN) cp_async16(&hbuf[slot][r][j], hrow + (int64_t)(c0 + r) * DN + j, 16);
      }
      for (int q = threadIdx.x; q < kCarryRows * SQ; q += kCarryW) {
        const int r = q / SQ, j = (q - r * SQ) * 4;
        if (c0 + r < g.nc_full && e0 / N + j < g.D)
          cp_async16(&sbuf[slot][r][j], srow + (int64_t)(c0 + r) * g.D + j, 16);
      }
    }
    cp_async_commit();
  };
  for (int st = 0; st < kCarryStages - 1; ++st) issue(st);
  for (int st = 0; st < nst; ++st) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kCarryStages - 2) : "memory");
    __syncthreads();  // stage st is complete, and stage st - 1 is no longer read
    issue(st + kCarryStages - 1);
    const int c0 = st * kCarryRows, slot = st % kCarryStages;
    const int nr = g.nc_full - c0 < kCarryRows ? g.nc_full - c0 : kCarryRows;
#pragma unroll
    for (int r = 0; r < kCarryRows; ++r) {
      if (r >= nr) break;
      const float hl = hbuf[slot][r][threadIdx.x], sd = sbuf[slot][r][threadIdx.x / N];
      if (act && !p.carry_last_only) hrow[(int64_t)(c0 + r) * DN + threadIdx.x] = H;
      H = __fmaf_rn(ex2(__fmul_rn(A2, sd)), H, hl);
    }
  }
  if (act) {
    hrow[(int64_t)g.nc_full * DN + threadIdx.x] = H;
    dfinite(kSiteChunkCarry, H, b * DN + e);  // debug build: a non-finite cached state
  }
}

// MODE 0: all-block forward (clean + noisy). MODE 1: clean scan only (cache
// build). MODE 2: clean scan only, right to left in time (logical token t is
// row L-1-t; the reverse direction of a full-sequence bidirectional layer).
// The active block has its own kernel (k_active_block).
template <int MODE>
struct ScanLayout {
  static_assert(MODE >= 0 && MODE <= 2, "block scan modes");
  static constexpr bool kClean = true;
  static constexpr bool kNoisy = MODE == 0;
  static constexpr int NTD = MODE == 0 ? 5 : 2;
  static constexpr int NROW = MODE == 0 ? 6 : 2;
  // token-by-channel slots
  static constexpr int XC = 0, DTC = 1;
  static constexpr int XN = 2, DTF = XN + 1, DTR = XN + 2;
  // token-by-state slots
  static constexpr int BC = 0, CC = 1;
  static constexpr int BF = 2, CF = BF + 1, BR = BF + 2, CR = BF + 3;
};

// KIND: how the chunk is walked (params.h). The clean scans copy the next block,
// tile or segment while the current one is scanned; in mode 0 a second buffer
// would cost a resident CTA per SM, which measured slower than the overlap it
// buys. There the forward pass over a segment stages the clean and forward
// tensors, the reverse pass its own.
// The stride of the staged tiles is fixed at kScanSeg tokens, so a token's
// addresses are immediates (16 tokens, 8 x 2048 x 1536 x 16, mode 0: 336 ->
// 321 us). The clean scans alone fit six CTAs per SM (65,536 x 2048 x 16,
// mode 1: 545 us with four, 528 with five, 520 with six, 610 with seven).
template <typename T, typename TO, int N, int MODE, int KIND>
__global__ void __launch_bounds__(kCta, MODE == 0 ? 4 : 6) k_block_scan(const FwdParams p) {
  pdl_sync();
  using Ly = ScanLayout<MODE>;
  extern __shared__ __align__(16) unsigned char smem[];
  const Geo& g = p.g;
  const int64_t b = blockIdx.z;
  const int c = p.c_begin + blockIdx.y;
  const int64_t d0 = (int64_t)blockIdx.x * kCta, d = d0 + threadIdx.x;
  const bool act = d < g.D;
  // debug build: the chunk's first token and the channel group lie inside the sizes
  if (!(dguard(kSiteBlockScan, b, g.Bt) && dguard(kSiteBlockScan, (int64_t)c * g.m * g.Bs, g.L) &&
        dguard(kSiteBlockScan, d0, g.D)))
    return;
  constexpr bool SEGS = KIND == kSegs, TILED = KIND == kTiles;
  const int Bs = KIND == kOneSeg ? kScanSeg : (int)g.Bs;
  const int SEG = TILED ? Bs : kScanSeg, NSEG = SEGS ? (Bs + SEG - 1) / SEG : 1;
  // blocks shorter than kScanSeg are staged TB at a time (one tile of at most
  // kScanSeg tokens), so the staging and its barriers are paid per tile
  const int TB = TILED ? kScanSeg / Bs : 1;
  constexpr bool kRev = MODE == 2;
  Stage<T, N, Ly::NTD, Ly::NROW, 2, kScanSeg, kRev> st;
  st.carve(smem, kScanSeg);
  // the row holding logical row x = b L + t (t reversed in time for MODE 2)
  auto prow = [&](int64_t x) { return kRev ? 2 * b * g.L + g.L - 1 - x : x; };
  constexpr bool dbuf = !Ly::kNoisy;
  float* yfbuf = reinterpret_cast<float*>(smem + decltype(st)::buf_bytes(kScanSeg));  // mode 0
  if (Ly::kClean) {
    st.td_src[Ly::XC] = (const T*)p.xc;
    st.td_src[Ly::DTC] = (const T*)p.dtc;
    st.row_src[Ly::BC] = (const T*)p.Bc;
    st.row_src[Ly::CC] = (const T*)p.Cc;
  }
  if (Ly::kNoisy) {
    st.td_src[Ly::XN] = (const T*)p.xn;
    st.td_src[Ly::DTF] = (const T*)p.dtf;
    st.td_src[Ly::DTR] = (const T*)p.dtr;
    st.row_src[Ly::BF] = (const T*)p.Bf;
    st.row_src[Ly::CF] = (const T*)p.Cf;
    st.row_src[Ly::BR] = (const T*)p.Br;
    st.row_src[Ly::CR] = (const T*)p.Cr;
  }

  float2 A2f[N / 2], A2r[N / 2];
  float Df = 0.f, Dr = 0.f;
  vzero2<N>(A2f);
  vzero2<N>(A2r);
  if (act) {
    vload2<N>(A2f, p.Af + d * N, 0);
    Df = p.Df[d];
    if (Ly::kNoisy) {
      vload2<N>(A2r, p.Ar + d * N, 0);
      Dr = p.Dr[d];
    }
#pragma unroll
    for (int j = 0; j < N / 2; ++j) {
      A2f[j] = mul2(A2f[j], f2(kLog2e));
      A2r[j] = mul2(A2r[j], f2(kLog2e));
    }
  }

  const int k_lo = c * g.m, k_hi = min(k_lo + g.m, g.nb) - 1;
  const bool full = c < g.nc_full;
  float2 hc[N / 2];
  vzero2<N>(hc);
  if (act) vload2<N>(hc, p.hst + ((b * (g.nc + 1) + c) * g.D + d) * N, 0);

  auto tile_blocks = [&](int k0) { return k_hi - k0 + 1 < TB ? k_hi - k0 + 1 : TB; };
  // SEGS, clean scans: the chunk's segments in order, one copied ahead
  int nk = k_lo, ns0 = 0, fill = 0, cur = 0;  // next segment to copy (block, first token), buffers
  auto copy_seg = [&]() {
    if (nk > k_hi) return false;
    st.issue(fill, prow(b * g.L + (int64_t)nk * Bs + ns0), Bs - ns0 < SEG ? Bs - ns0 : SEG, g.D, d0);
    fill ^= 1;
    ns0 += SEG;
    if (ns0 >= Bs) {
      ns0 = 0;
      ++nk;
    }
    return true;
  };
  if (dbuf && SEGS) copy_seg();
  if (dbuf && !SEGS) st.issue(0, prow(b * g.L + (int64_t)k_lo * Bs), tile_blocks(k_lo) * Bs, g.D, d0);
  for (int k0 = k_lo; k0 <= k_hi; k0 += TB) {
    const int nbk = tile_blocks(k0), tile = (k0 - k_lo) / TB;
    const int64_t trow = b * g.L + (int64_t)k0 * Bs;
    if (dbuf && !SEGS) {
      __syncthreads();  // the other buffer is no longer read
      const int k1 = k0 + TB;
      if (k1 <= k_hi) st.issue((tile + 1) & 1, prow(trow + (int64_t)nbk * Bs), tile_blocks(k1) * Bs, g.D, d0);
      st.complete(tile & 1, nbk * Bs, k1 <= k_hi ? 1 : 0);
    } else if (!SEGS) {
      st.load(prow(trow), nbk * Bs, g.D, d0);
    }
    for (int kk = 0; kk < nbk; ++kk) {
      const int k = k0 + kk;
      const int64_t row0 = trow + (int64_t)kk * Bs;
      const int toff = kk * Bs;  // the block's first token in the staged tile (0 for long blocks)
      float2 hs[N / 2];
#pragma unroll
      for (int j = 0; j < N / 2; ++j) hs[j] = hc[j];  // the block's seed: state before its first token
      for (int sg = 0; sg < NSEG; ++sg) {  // segments left to right
        const int i0 = sg * SEG, ns = Bs - i0 < SEG ? Bs - i0 : SEG;
        if (SEGS && dbuf) {
          __syncthreads();  // the other buffer is no longer read
          const bool ahead = copy_seg();
          st.complete(cur, ns, ahead ? 1 : 0);
          cur ^= 1;
        } else if (SEGS) {
          st.td_src[0] = (const T*)p.xc;
          st.td_src[1] = (const T*)p.dtc;
          st.row_src[0] = (const T*)p.Bc;
          st.row_src[1] = (const T*)p.Cc;
          st.load_first(row0 + i0, ns, g.D, d0, 4, 4);  // x_c, dt_c, x_n, dt_f; B_c, C_c, B_f, C_f
        }
        int64_t o = prow(row0 + i0) * g.D + d;  // the token's element, stepped
#pragma unroll 2
        for (int ii = 0; ii < ns; ++ii, o += kRev ? -g.D : g.D) {
          const int i = i0 + ii;
          if (Ly::kClean) {
            const float x = st.at(Ly::XC, toff + ii), dt = st.at(Ly::DTC, toff + ii);
            const float y = scan_step<N>(hc, A2f, dt, x, st.row(Ly::BC, toff + ii), st.row(Ly::CC, toff + ii));
            if (p.yc != nullptr && act) reinterpret_cast<TO*>(p.yc)[o] = to_out<TO>(with_skip(y, Df, x));
          }
          if (Ly::kNoisy) {
            const float x = st.at(Ly::XN, toff + ii), dt = st.at(Ly::DTF, toff + ii);
            const float y = scan_step<N>(hs, A2f, dt, x, st.row(Ly::BF, toff + ii), st.row(Ly::CF, toff + ii));
            yfbuf[i * kCta + threadIdx.x] = with_skip(y, Df, x);
          }
        }
      }
      if (Ly::kClean && p.emit_all && act) {
        float* dst = p.states + ((b * g.nb + k) * g.D + d) * N;
        if (k == k_hi && full) {
          float2 e[N / 2];
          vload2<N>(e, p.hst + ((b * (g.nc + 1) + c + 1) * g.D + d) * N, 0);
          vstore2<N>(dst, e, 0);
        } else {
          vstore2<N>(dst, hc, 0);
        }
      }
      if (Ly::kNoisy) {
        float2 hr[N / 2];
        vzero2<N>(hr);
        // SEGS: the reverse pass stages its tensors in the first slots
        constexpr int XR = SEGS ? 0 : Ly::XN, DTR = SEGS ? 1 : Ly::DTR, BR = SEGS ? 0 : Ly::BR, CR = SEGS ? 1 : Ly::CR;
        for (int sg = NSEG - 1; sg >= 0; --sg) {  // segments right to left
          const int i0 = sg * SEG, ns = Bs - i0 < SEG ? Bs - i0 : SEG;
          if (SEGS) {
            st.td_src[0] = (const T*)p.xn;
            st.td_src[1] = (const T*)p.dtr;
            st.row_src[0] = (const T*)p.Br;
            st.row_src[1] = (const T*)p.Cr;
            st.load_first(row0 + i0, ns, g.D, d0, 2, 2);
          }
          int64_t o = prow(row0 + i0 + ns - 1) * g.D + d;
#pragma unroll 2
          for (int ii = ns - 1; ii >= 0; --ii, o -= g.D) {  // noisy streams are never reversed
            const int i = i0 + ii;
            const float x = st.at(XR, toff + ii), dt = st.at(DTR, toff + ii);
            const float y = scan_step<N>(hr, A2r, dt, x, st.row(BR, toff + ii), st.row(CR, toff + ii));
            if (act)
              reinterpret_cast<TO*>(p.yn)[o] =
                  to_out<TO>(combine_dirs(yfbuf[i * kCta + threadIdx.x], with_skip(y, Dr, x)));
          }
        }
      }
    }
  }
  if (Ly::kClean && p.final_state != nullptr && c == g.nc - 1 && act) {
    float* dst = p.final_state + (b * g.D + d) * N;
    if (full) {
      float2 e[N / 2];
      vload2<N>(e, p.hst + ((b * (g.nc + 1) + c + 1) * g.D + d) * N, 0);
      vstore2<N>(dst, e, 0);
    } else {
      vstore2<N>(dst, hc, 0);
    }
  }
}

// ---------------------------------------------------------------------------
// Active block (the inference step): one noisy block per batch row from a
// read-only cached seed; in the all-block forward of small problems (see
// noisy_apart) every noisy block, seeded with the clean state before it. A CTA
// covers 32 channels of one block; warp 0 runs the
// seeded forward scan and warp 1 the block-local reverse scan at the same
// time, each with the per-channel arithmetic of k_block_scan (scan_step,
// with_skip, combine_dirs), so the outputs equal those of the all-block
// forward bit for bit. The step is bound by the latency of the serial scan,
// so small CTAs spread it over many SMs.
// ---------------------------------------------------------------------------
constexpr int kActW = 32;  // channels per active-block CTA

template <typename T, int N>
struct ActiveLayout {
  // [3][Bs][32] x, dt_f, dt_r as stored; [4][Bs][N] B_f, C_f, B_r, C_r as
  // loaded and widened to fp32; [2][Bs][32] forward and reverse outputs
  static __host__ __device__ size_t td_bytes(int Bs) {
    return ((size_t)3 * Bs * kActW * sizeof(T) + 15) & ~(size_t)15;
  }
  static __host__ __device__ size_t raw_bytes(int Bs) {
    return is_f32<T>::value ? 0 : (((size_t)4 * Bs * N * sizeof(T) + 15) & ~(size_t)15);
  }
  static __host__ __device__ size_t rows_bytes(int Bs) { return (size_t)4 * Bs * N * 4; }
  static __host__ __device__ size_t bytes(int Bs) {
    return td_bytes(Bs) + raw_bytes(Bs) + rows_bytes(Bs) + (size_t)2 * Bs * kActW * 4;
  }
  // with adaptive layer norm: the modulated input [Bs][32] fp32 after the outputs
  static __host__ __device__ size_t bytes_ada(int Bs) { return bytes(Bs) + (size_t)Bs * kActW * 4; }
};

// ADA: adaptive layer norm on the block (Appendix E, eq. cacheable-adaln):
// the scans read u = (1 + scale) (x - mean) rstd + shift instead of x, and
// the output is x + gate * y_n. The seed, the cache, is never modulated.
template <typename T, typename TO, int N, bool ADA = false>
__global__ void __launch_bounds__(2 * kActW, 1) k_active_block(const FwdParams p) {
  pdl_sync();
  using Ly = ActiveLayout<T, N>;
  extern __shared__ __align__(16) unsigned char smem[];
  const Geo& g = p.g;
  const int Bs = (int)g.Bs;
  const unsigned groups = (unsigned)((g.D + kActW - 1) / kActW), k = blockIdx.x / groups;  // the block of the row
  const int64_t b = blockIdx.y, d0 = (int64_t)(blockIdx.x - k * groups) * kActW;
  const int lane = threadIdx.x & 31, dir = threadIdx.x >> 5;  // dir 0: forward, 1: reverse
  const int64_t d = d0 + lane;
  const bool act = d < g.D;
  // debug build: the batch row, its block and the channel group lie inside the sizes
  if (!(dguard(kSiteActiveBlock, b, g.Bt) && dguard(kSiteActiveBlock, k, g.nb) && dguard(kSiteActiveBlock, d0, g.D)))
    return;
  T* td = reinterpret_cast<T*>(smem);
  float* rows = reinterpret_cast<float*>(smem + Ly::td_bytes(Bs) + Ly::raw_bytes(Bs));
  T* raw = is_f32<T>::value ? reinterpret_cast<T*>(rows) : reinterpret_cast<T*>(smem + Ly::td_bytes(Bs));
  float* ybuf = rows + (size_t)4 * Bs * N;

  // copies (16-byte chunks; channels past D read as zero)
  constexpr int E = 16 / (int)sizeof(T);
  constexpr int CPR = kActW / E;
  const int64_t row0 = b * g.L + (int64_t)k * Bs;
  for (int q = threadIdx.x; q < 3 * Bs * CPR; q += 2 * kActW) {
    const int j = q / (Bs * CPR), r = q - j * (Bs * CPR), t = r / CPR, cc = (r - t * CPR) * E;
    const T* src = (const T*)(j == 0 ? p.xn : (j == 1 ? p.dtf : p.dtr));
    const bool ok = d0 + cc < g.D;
    cp_async16(td + ((size_t)j * Bs + t) * kActW + cc,
               ok ? (const void*)(src + (row0 + t) * g.D + d0 + cc) : (const void*)src, ok ? 16 : 0);
  }
  const int rch = Bs * N / E;
  for (int q = threadIdx.x; q < 4 * rch; q += 2 * kActW) {
    const int j = q / rch, r = q - j * rch;
    const T* src = (const T*)(j == 0 ? p.Bf : (j == 1 ? p.Cf : (j == 2 ? p.Br : p.Cr)));
    cp_async16(raw + (size_t)j * Bs * N + r * E, src + row0 * N + (int64_t)r * E, 16);
  }
  cp_async_commit();

  // parameters and the seed while the copies are in flight
  float2 A2[N / 2], h[N / 2];
  vzero2<N>(A2);
  vzero2<N>(h);
  float Dd = 0.f;
  if (act) {
    vload2<N>(A2, (dir == 0 ? p.Af : p.Ar) + d * N, 0);
#pragma unroll
    for (int j = 0; j < N / 2; ++j) A2[j] = mul2(A2[j], f2(kLog2e));
    Dd = dir == 0 ? p.Df[d] : p.Dr[d];
    const float* seed = p.seed != nullptr ? p.seed + (b * g.D + d) * N
                        : k > 0           ? p.states + ((b * g.nb + k - 1) * g.D + d) * N
                                          : nullptr;
    if (dir == 0 && seed != nullptr) vload2<N>(h, seed, 0);
  }
  cp_async_wait_all();
  __syncthreads();
  if (!is_f32<T>::value) {
    for (int q = threadIdx.x; q < 2 * Bs * N; q += 2 * kActW)
      reinterpret_cast<float2*>(rows)[q] = make_float2(cvt(raw[2 * q]), cvt(raw[2 * q + 1]));
    __syncthreads();
  }
  float* xmod = ybuf + (size_t)2 * Bs * kActW;  // [Bs][32], ADA only
  if (ADA) {
    for (int q = threadIdx.x; q < Bs * kActW; q += 2 * kActW) {
      const int i = q / kActW, c = q - i * kActW;
      const int64_t dc = d0 + c;
      float u = 0.f;
      if (dc < g.D) {
        const float2 st = p.ln_stats[b * Bs + i];
        const float z = __fmul_rn(__fsub_rn(cvt(td[q]), st.x), st.y);
        u = __fmaf_rn(__fadd_rn(1.f, p.scale[b * g.D + dc]), z, p.shift[b * g.D + dc]);
      }
      xmod[q] = u;
    }
    __syncthreads();
  }
  // this lane's input at token i: x as stored, or the modulated input
  auto xin = [&](int i) { return ADA ? xmod[i * kActW + lane] : cvt(td[i * kActW + lane]); };

  const T* xs = td;
  const T* dts = td + (size_t)(1 + dir) * Bs * kActW;
  const float* Brow = rows + (size_t)(2 * dir) * Bs * N;
  const float* Crow = Brow + (size_t)Bs * N;
  float* yb = ybuf + (size_t)dir * Bs * kActW;
  (void)xs;
  if (dir == 0) {
#pragma unroll 4
    for (int i = 0; i < Bs; ++i) {
      const float x = xin(i), dt = cvt(dts[i * kActW + lane]);
      const float y = scan_step<N>(h, A2, dt, x, Brow + i * N, Crow + i * N);
      yb[i * kActW + lane] = with_skip(y, Dd, x);
    }
  } else {
#pragma unroll 4
    for (int i = Bs - 1; i >= 0; --i) {
      const float x = xin(i), dt = cvt(dts[i * kActW + lane]);
      const float y = scan_step<N>(h, A2, dt, x, Brow + i * N, Crow + i * N);
      yb[i * kActW + lane] = with_skip(y, Dd, x);
    }
  }
  __syncthreads();
  for (int q = threadIdx.x; q < Bs * kActW; q += 2 * kActW) {
    const int i = q / kActW, c = q - i * kActW;
    if (d0 + c < g.D) {
      const float yv = combine_dirs(ybuf[q], ybuf[(size_t)Bs * kActW + q]);
      // gated residual of the modulated step: x + gate * y_n
      const float o = ADA ? __fmaf_rn(p.gate[b * g.D + d0 + c], yv, cvt(td[q])) : yv;
      reinterpret_cast<TO*>(p.yn)[(row0 + i) * g.D + d0 + c] = to_out<TO>(o);
    }
  }
}

// Layer-norm statistics of each token (one warp per row of D elements): the
// mean, then 1/sqrt(var + eps) from the centred second moment, in fp32.
template <typename T>
__global__ void __launch_bounds__(256) k_ln_stats(const T* h, int64_t rows, int64_t D, float eps, float2* stats) {
  pdl_sync();
  const int64_t row = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= rows) return;
  const T* r = h + row * D;
  float s = 0.f;
  for (int64_t i = lane; i < D; i += 32) s = __fadd_rn(s, cvt(r[i]));
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
  const float mu = __fdiv_rn(s, (float)D);
  float v = 0.f;
  for (int64_t i = lane; i < D; i += 32) {
    const float e = __fsub_rn(cvt(r[i]), mu);
    v = __fmaf_rn(e, e, v);
  }
#pragma unroll
  for (int o = 16; o >= 1; o >>= 1) v = __fadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (lane == 0) stats[row] = make_float2(mu, __fdiv_rn(1.f, __fsqrt_rn(__fadd_rn(__fdiv_rn(v, (float)D), eps))));
}

// ---------------------------------------------------------------------------
// Sum of the two directions of a full-sequence bidirectional layer: each fp32
// input already holds its direction's output with its own skip term.
// ---------------------------------------------------------------------------
template <typename TO>
__global__ void __launch_bounds__(256) k_combine(const float* yf, const float* yr, TO* y, int64_t n4) {
  pdl_sync();
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;  // four elements each
  if (i >= n4) return;
  const float4 a = reinterpret_cast<const float4*>(yf)[i], r = reinterpret_cast<const float4*>(yr)[i];
  TO* o = y + 4 * i;
  o[0] = to_out<TO>(combine_dirs(a.x, r.x));
  o[1] = to_out<TO>(combine_dirs(a.y, r.y));
  o[2] = to_out<TO>(combine_dirs(a.z, r.z));
  o[3] = to_out<TO>(combine_dirs(a.w, r.w));
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
namespace {

template <typename T, int N, int NS, bool REV>
cudaError_t chunk_local_k(const FwdParams& p, cudaStream_t s) {
  const size_t smem = Stage<T, N, 2, 1, 2>::bytes(kLocalSpan);
  cudaError_t e = set_smem_cached((const void*)k_chunk_local<T, N, NS, REV>, (int)smem, -1);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)(p.g.G * (N / NS)), (unsigned)p.g.nc_full, (unsigned)p.g.Bt);
  launch_pdl(k_chunk_local<T, N, NS, REV>, grid, kCta, smem, s, p);
  return cudaGetLastError();
}
template <typename T, int N, bool REV>
cudaError_t chunk_local_rt(const FwdParams& p, cudaStream_t s) {
  const int64_t ctas = (int64_t)p.g.G * p.g.nc_full * p.g.Bt;
  if (ctas <= kLocalQuarter) return chunk_local_k<T, N, 4, REV>(p, s);
  if (N == 16 && ctas <= kLocalHalf) return chunk_local_k<T, N, 8, REV>(p, s);
  return chunk_local_k<T, N, N, REV>(p, s);
}
template <typename T, int N>
cudaError_t chunk_local_t(const FwdParams& p, cudaStream_t s) {
  return p.rev ? chunk_local_rt<T, N, true>(p, s) : chunk_local_rt<T, N, false>(p, s);
}

template <typename T, typename TO, int N, int MODE, int KIND>
cudaError_t block_scan_k(int nchunks, const FwdParams& p, cudaStream_t s) {
  using Ly = ScanLayout<MODE>;
  const size_t buf = Stage<T, N, Ly::NTD, Ly::NROW, 2>::buf_bytes(kScanSeg);
  const size_t smem = Ly::kNoisy ? buf + (size_t)p.g.Bs * kCta * sizeof(float) : 2 * buf;
  cudaError_t e = set_smem_cached((const void*)k_block_scan<T, TO, N, MODE, KIND>, (int)smem, -1);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)p.g.G, (unsigned)nchunks, (unsigned)p.g.Bt);
  launch_pdl(k_block_scan<T, TO, N, MODE, KIND>, grid, kCta, smem, s, p);
  return cudaGetLastError();
}
template <typename T, typename TO, int N, int MODE>
cudaError_t block_scan_t(int nchunks, const FwdParams& p, cudaStream_t s) {
  switch (block_kind(p.g.Bs)) {
    case kTiles: return block_scan_k<T, TO, N, MODE, kTiles>(nchunks, p, s);
    case kSegs: return block_scan_k<T, TO, N, MODE, kSegs>(nchunks, p, s);
    default: return block_scan_k<T, TO, N, MODE, kOneSeg>(nchunks, p, s);
  }
}

template <typename T, typename TO, int N>
cudaError_t block_scan_mode(int mode, int nchunks, const FwdParams& p, cudaStream_t s) {
  switch (mode) {
    case 0: return block_scan_t<T, TO, N, 0>(nchunks, p, s);
    case 1: return block_scan_t<T, TO, N, 1>(nchunks, p, s);
    case 2: return block_scan_t<T, TO, N, 2>(nchunks, p, s);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T, typename TO, int N, bool ADA = false>
cudaError_t active_block_t(const FwdParams& p, cudaStream_t s) {
  using Ly = ActiveLayout<T, N>;
  const size_t smem = ADA ? Ly::bytes_ada((int)p.g.Bs) : Ly::bytes((int)p.g.Bs);
  if (smem > 48 * 1024) {
    cudaError_t e = set_smem_cached((const void*)k_active_block<T, TO, N, ADA>, (int)smem, -1);
    if (e != cudaSuccess) return e;
  }
  dim3 grid((unsigned)((p.g.D + kActW - 1) / kActW * p.g.nb), (unsigned)p.g.Bt);
  launch_pdl(k_active_block<T, TO, N, ADA>, grid, 2 * kActW, smem, s, p);
  return cudaGetLastError();
}

}  // namespace

#define BDS_DISPATCH_N(N, ...)                      \
  switch (N) {                                      \
    case 8: { constexpr int NN = 8; __VA_ARGS__ }   \
    case 16: { constexpr int NN = 16; __VA_ARGS__ } \
    default: return cudaErrorInvalidValue;          \
  }

cudaError_t launch_chunk_local(int dt, int N, const FwdParams& p, cudaStream_t s) {
  if (p.g.nc_full == 0 || p.g.Bt == 0) return cudaSuccess;
  if (dt == 0) {
    BDS_DISPATCH_N(N, return chunk_local_t<float, NN>(p, s);)
  }
  BDS_DISPATCH_N(N, return chunk_local_t<bf16, NN>(p, s);)
}

cudaError_t launch_chunk_carry(int N, const FwdParams& p, cudaStream_t s) {
  if (p.g.Bt * p.g.D * N == 0) return cudaSuccess;
  if (p.g.nc_full <= kCarryFew) {
    const unsigned blocks = (unsigned)((p.g.Bt * p.g.D * N + 255) / 256);
    BDS_DISPATCH_N(N, launch_pdl(k_chunk_carry<NN>, blocks, 256, 0, s, p); return cudaGetLastError();)
  }
  const dim3 grid((unsigned)((p.g.D * N + kCarryW - 1) / kCarryW), (unsigned)p.g.Bt);
  BDS_DISPATCH_N(N, launch_pdl(k_chunk_carry_ring<NN>, grid, kCarryW, 0, s, p); return cudaGetLastError();)
}

cudaError_t launch_block_scan(int dt, int N, int mode, int nchunks, const FwdParams& p, cudaStream_t s) {
  if (nchunks == 0 || p.g.Bt == 0) return cudaSuccess;
  switch (dt) {
    case 0: BDS_DISPATCH_N(N, return block_scan_mode<float, float, NN>(mode, nchunks, p, s);)
    case 1: BDS_DISPATCH_N(N, return block_scan_mode<bf16, bf16, NN>(mode, nchunks, p, s);)
    default: BDS_DISPATCH_N(N, return block_scan_mode<bf16, float, NN>(mode, nchunks, p, s);)
  }
}

cudaError_t launch_active_block(int dt, int N, const FwdParams& p, cudaStream_t s) {
  if (p.g.Bt == 0 || p.g.D == 0) return cudaSuccess;
  switch (dt) {
    case 0: BDS_DISPATCH_N(N, return active_block_t<float, float, NN>(p, s);)
    case 1: BDS_DISPATCH_N(N, return active_block_t<bf16, bf16, NN>(p, s);)
    default: BDS_DISPATCH_N(N, return active_block_t<bf16, float, NN>(p, s);)
  }
}

cudaError_t launch_active_block_adaln(int dt, int N, const FwdParams& p, cudaStream_t s) {
  if (p.g.Bt == 0 || p.g.D == 0) return cudaSuccess;
  switch (dt) {
    case 0: BDS_DISPATCH_N(N, return active_block_t<float, float, NN, true>(p, s);)
    case 1: BDS_DISPATCH_N(N, return active_block_t<bf16, bf16, NN, true>(p, s);)
    default: BDS_DISPATCH_N(N, return active_block_t<bf16, float, NN, true>(p, s);)
  }
}

cudaError_t launch_ln_stats(int dt, const void* h, int64_t rows, int64_t D, float eps, float2* stats, cudaStream_t s) {
  if (rows == 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((rows + 7) / 8);
  if (dt == 0)
    launch_pdl(k_ln_stats<float>, blocks, 256, 0, s, reinterpret_cast<const float*>(h), rows, D, eps, stats);
  else
    launch_pdl(k_ln_stats<bf16>, blocks, 256, 0, s, reinterpret_cast<const bf16*>(h), rows, D, eps, stats);
  return cudaGetLastError();
}

cudaError_t launch_combine(int out_f32, const float* yf, const float* yr, void* y, int64_t n, cudaStream_t s) {
  const int64_t n4 = n / 4;  // D is a multiple of 4
  if (n4 == 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((n4 + 255) / 256);
  if (out_f32)
    launch_pdl(k_combine<float>, blocks, 256, 0, s, yf, yr, reinterpret_cast<float*>(y), n4);
  else
    launch_pdl(k_combine<bf16>, blocks, 256, 0, s, yf, yr, reinterpret_cast<bf16*>(y), n4);
  return cudaGetLastError();
}

}  // namespace bds
