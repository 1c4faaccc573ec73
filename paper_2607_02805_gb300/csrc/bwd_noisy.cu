// bwd_noisy.cu -- the noisy-block backward of libbdscan (sm_103a); see
// bwd_common.cuh for the derivative and the kernel sequence.
#include "bwd_common.cuh"

namespace bds {

// ---------------------------------------------------------------------------
// Noisy blocks (both directions) + the clean stream's chunk-local adjoint
// ---------------------------------------------------------------------------
template <typename T, int N, int KIND>
struct NoisyBwdSmem {
  // token-by-channel: x_n, dt_f, dt_r, dy_n, dt_c, dy_c; token-by-state: B_f, C_f, B_r, C_r, C_c.
  // Blocks of several segments stage what one pass over a segment reads: at
  // most three of the first (x_n, dt, dy_n; or dt_c, dy_c) and two of the
  // second (B, C; or C_c)
  using St = Stage<T, N, KIND == kSegs ? 3 : 6, KIND == kSegs ? 2 : 5, 2, kBwdTS>;
  // `bufs` staging buffers: 2 (the next block, tile or segment is copied while
  // the current one is used) or, where that leaves more CTAs on an SM, 1
  static __host__ __device__ size_t dx_off(int bufs) { return align16(St::buf_bytes(kBwdTS) * bufs); }
  // dx partials of a tile (several short blocks) or of one long block
  static __host__ __device__ size_t red_off(int bufs, int Bs) { return dx_off(bufs) + (size_t)(Bs < kBwdTS ? kBwdTS : Bs) * kCta * 4; }
  // red slots: both directions of a tile at once for short blocks, one
  // direction's segment at a time otherwise
  static __host__ __device__ int red_slots(int Bs) { return Bs < kBwdTS ? 4 : 2; }
  static __host__ __device__ size_t ck_off(int bufs, int Bs) { return red_off(bufs, Bs) + (size_t)red_slots(Bs) * kBwdTS * kRedRow * 4; }
  // checkpoints in shared memory up to kCkSmemMaxBs tokens, else in global memory
  static __host__ __device__ size_t slot_off(int bufs, int TS, int Bs) {
    return ck_off(bufs, Bs) + (Bs > kCkSmemMaxBs ? 0 : (size_t)(Bs / TS - 1) * N * kCta * 4);
  }
  static __host__ __device__ size_t bytes(int bufs, int TS, int Bs) { return slot_off(bufs, TS, Bs) + 16; }
};

// KIND: how the chunk is walked (params.h). Blocks of several segments
// make five passes over each: the clean local adjoint, and per direction the
// checkpoints and the segments themselves. Each pass stages what it reads, and
// the next pass's or segment's copies run under the current one's work (8 x
// 2048 x 2048, blocks of 64: 1419 -> 1199 us against staging every tensor for
// each pass). Blocks of one segment have their sizes at compile time (8 x 2048
// x 1536, blocks of 16: 801 -> 738 us).
// SPLIT (small problems, split_parts): the chunk is one block, and a CTA does
// one of the three parts of its work, none of which reads what another makes.
template <typename T, typename TO, int N, int KIND, bool SPLIT>
__global__ void __launch_bounds__(kCta, 1) k_bwd_noisy(const BwdParams p) {
  pdl_sync();
  static_assert(!(KIND == kTiles && SPLIT), "a split launch has one block per CTA");
  constexpr bool TILED = KIND == kTiles, SEGS = KIND == kSegs;
  extern __shared__ __align__(16) unsigned char smem[];
  using L = NoisyBwdSmem<T, N, KIND>;
  const Geo& g = p.g;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int sw = swz_of_lane<N>();
  const unsigned part = SPLIT ? blockIdx.z % 3 : 0;
  const bool do_clean = !SPLIT || part == 0, do_rev = !SPLIT || part == 1, do_fwd = !SPLIT || part == 2;
  const int64_t b = SPLIT ? blockIdx.z / 3 : blockIdx.z;
  const int c = blockIdx.y;
  const int64_t d0 = (int64_t)blockIdx.x * kCta, d = d0 + tid;
  const bool act = d < g.D;
  const int Bs = KIND == kOneSeg && !SPLIT ? 16 : (int)g.Bs;
  const int TS = SEGS || (KIND == kOneSeg && !SPLIT) ? 16 : Bs, NSEG = SEGS ? Bs / 16 : 1;
  const int k_lo = chunk_lo(g, c), k_hi = chunk_lo(g, c + 1) - 1;
  // debug build: the chunk's last token and the channel group lie inside the sizes
  if (!(dguard(kSiteBwdNoisy, b, g.Bt) && dguard(kSiteBwdNoisy, (int64_t)(k_hi + 1) * Bs - 1, g.L) &&
        dguard(kSiteBwdNoisy, d0, g.D)))
    return;

  constexpr int XN = 0, DTF = 1, DTR = SEGS ? 1 : 2, DYN = SEGS ? 2 : 3, DTC = SEGS ? 0 : 4, DYC = SEGS ? 1 : 5;
  constexpr int BF = 0, CF = 1, BR = SEGS ? 0 : 2, CR = SEGS ? 1 : 3, CC = SEGS ? 0 : 4;
  typename L::St st;
  st.carve(smem, TS);
  if constexpr (!SEGS) {
    st.td_src[XN] = (const T*)p.xn;
    st.td_src[DTF] = (const T*)p.dtf;
    st.td_src[DTR] = (const T*)p.dtr;
    st.td_src[DYN] = (const T*)p.dyn;
    st.td_src[DTC] = (const T*)p.dtc;
    st.td_src[DYC] = (const T*)p.dyc;
    st.row_src[BF] = (const T*)p.Bf;
    st.row_src[CF] = (const T*)p.Cf;
    st.row_src[BR] = (const T*)p.Br;
    st.row_src[CR] = (const T*)p.Cr;
    st.row_src[CC] = (const T*)p.Cc;
  }
  const int bufs = is_f32<T>::value ? p.stage_bufs : 2;
  float* dxr_part = p.dx_part;  // SPLIT: where the two directions leave their share of dx
  float* dxf_part = SPLIT ? p.dx_part + g.Bt * g.L * g.D : nullptr;
  float* dxbuf = reinterpret_cast<float*>(smem + L::dx_off(bufs));
  float* red = reinterpret_cast<float*>(smem + L::red_off(bufs, Bs));
  float* mine = red_slot<N>(red);
  float* ck = Bs > kCkSmemMaxBs
                  ? p.ck_noisy + (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) *
                                     (size_t)(NSEG - 1) * N * kCta
                  : reinterpret_cast<float*>(smem + L::ck_off(bufs, Bs));
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + L::slot_off(bufs, TS, Bs));

  const uint32_t tcols = full_cols(TS, N);
  if (warp == 0) tmem_alloc(tslot, tcols);
  tmem_sync();
  const uint32_t tbase = *tslot;
  const uint32_t tb = tbase + ((uint32_t)(warp * 32) << 16);

  float2 A2f[N / 2], A2r[N / 2];
  vzero2<N>(A2f);
  vzero2<N>(A2r);
  float Dsum = 0.f;
  if (act) {
    vload2<N>(A2f, p.Af + d * N, sw);
    vload2<N>(A2r, p.Ar + d * N, sw);
#pragma unroll
    for (int j = 0; j < N / 2; ++j) {
      A2f[j] = mul2(A2f[j], f2(kLog2e));
      A2r[j] = mul2(A2r[j], f2(kLog2e));
    }
    Dsum = __fadd_rn(p.Df[d], p.Dr[d]);
  }
  float2 dAf[N / 2], dAr[N / 2];
  vzero2<N>(dAf);
  vzero2<N>(dAr);
  float dDn = 0.f, sdt = 0.f;
  float2 carry[N / 2];  // clean stream: a_{t+1} gbar_{t+1} (+ injections) entering token t from the right
  vzero2<N>(carry);
  float2 dSn[N / 2];  // seed gradient of the block to the right of the current one
  vzero2<N>(dSn);

  // SEGS: the steps (pass, segment) of a block in the order they are used, one
  // step staged ahead. Passes 0: clean, 1 / 2: reverse checkpoints / segments,
  // 3 / 4: forward checkpoints / segments.
  int nk = k_hi, np = 0, ns = NSEG - 1, fill = 0, cur = 0;  // next step to copy, buffers
  auto enter = [&](int pass) {
    for (;; ++pass) {
      if (pass > 4) {
        pass = 0;
        --nk;
      }
      if (pass == 0 ? do_clean : pass <= 2 ? do_rev : do_fwd) break;
    }
    np = pass;
    ns = pass == 2 || pass == 3 ? 0 : NSEG - 1;
  };
  auto copy_step = [&]() {
    if (nk < k_lo) return false;
    const bool fwd = np >= 3, adj = np == 2 || np == 4;
    st.td_src[0] = (const T*)(np == 0 ? p.dtc : p.xn);
    st.td_src[1] = (const T*)(np == 0 ? p.dyc : fwd ? p.dtf : p.dtr);
    st.row_src[0] = (const T*)(np == 0 ? p.Cc : fwd ? p.Bf : p.Br);
    if constexpr (SEGS) {
      st.td_src[2] = (const T*)p.dyn;
      st.row_src[1] = (const T*)(fwd ? p.Cf : p.Cr);
    }
    st.issue_first(fill, b * g.L + (int64_t)nk * Bs + ns * TS, TS, g.D, d0, adj ? 3 : 2, adj ? 2 : 1);
    fill ^= bufs - 1;
    if (np == 2 || np == 3) {
      if (++ns > (np == 2 ? NSEG - 1 : NSEG - 2)) enter(np + 1);
    } else {
      if (--ns < (np == 1 ? 1 : 0)) enter(np + 1);
    }
    return true;
  };
  auto next_step = [&](int nrow) {  // the next step's tiles become current
    __syncthreads();                // the buffer to fill is no longer read
    const bool ahead = copy_step() && bufs == 2;
    st.complete(cur, TS, ahead ? 1 : 0, nrow);
    cur ^= bufs - 1;
  };
  if (SEGS) {
    enter(0);
    if (bufs == 2) copy_step();
  }

  // everything for block k, whose tokens start at `off` in the staged tile
  auto block = [&](int k, int off) {
    const int64_t t0 = (int64_t)k * Bs;
    const int64_t row0 = b * g.L + t0;

    // ---- clean stream: chunk-local adjoint over block k ----
    if (k < k_hi) {
#pragma unroll
      for (int j = 0; j < N / 2; ++j) carry[j] = add2(carry[j], dSn[j]);
      if (p.dstates != nullptr && act) {
        float2 e[N / 2];
        vload2<N>(e, p.dstates + ((b * g.nb + k) * g.D + d) * N, sw);
#pragma unroll
        for (int j = 0; j < N / 2; ++j) carry[j] = add2(carry[j], e[j]);
      }
    }
    if (do_clean) for (int s = NSEG - 1; s >= 0; --s) {
      if (SEGS) next_step(1);
#pragma unroll 4
      for (int i = TS - 1; i >= 0; --i) {
        const float dt = st.at(DTC, off + i), dy = st.at(DYC, off + i);
        const float2 dt2 = f2(dt), dy2 = f2(dy);
        float2 C[N / 2];
        vload2<N>(C, st.row(CC, off + i), sw);
#pragma unroll
        for (int j = 0; j < N / 2; ++j) carry[j] = mul2(ex2x2(mul2(dt2, A2f[j])), fma2(C[j], dy2, carry[j]));
        sdt = __fadd_rn(sdt, dt);
      }
    }

    // ---- noisy block k, reverse direction (zero state at the block end) ----
    if (do_rev) {
      if (SEGS) {
        float2 h[N / 2];
        vzero2<N>(h);
        for (int s = NSEG - 1; s >= 1; --s) {
          next_step(1);
#pragma unroll 4
          for (int i = TS - 1; i >= 0; --i) scan_state_swz<N>(h, A2r, st.at(DTR, i), st.at(XN, i), st.row(BR, i), sw);
          ck_store<N>(ck, s - 1, h);
        }
      }
      float2 gr[N / 2];  // a_{t-1} gbar_{t-1}, entering token t from the left
      vzero2<N>(gr);
      for (int s = 0; s < NSEG; ++s) {
        if (SEGS) next_step(2);
        float2 h[N / 2];
        if (s == NSEG - 1)
          vzero2<N>(h);
        else
          ck_load<N>(h, ck, s);
        int64_t o = (row0 + (int64_t)s * TS) * g.D + d;  // the token's element, stepped
        seg_bwd<N, false>(st, TS, XN, DTR, DYN, BR, CR, A2r, sw, h, gr, dAr, tb, mine, off, 0,
                          [&](int i, float dt, float x, float dy, float sgB, float sAq) {
                            const int ib = s * TS + i;
                            if (act)
                              reinterpret_cast<TO*>(p.ddtr)[o] =
                                  to_out<TO>(__fmaf_rn(x, sgB, __fmul_rn(kLn2, sAq)));
                            if (!SPLIT)
                              dxbuf[(off + ib) * kCta + tid] = __fmul_rn(dt, sgB);
                            else if (act)
                              dxr_part[o] = __fmul_rn(dt, sgB);
                            o += g.D;
                          });
        if (!TILED) red_flush<N>(p, red, 0, 1, 4, 5, b, t0 + (int64_t)s * TS, TS);
      }
    }

    // ---- noisy block k, forward direction (seeded with states[k-1]) ----
    if (do_fwd) {
      float2 seed[N / 2];
      vzero2<N>(seed);
      if (k > 0 && act) vload2<N>(seed, p.states + ((b * g.nb + (k - 1)) * g.D + d) * N, sw);
      if (SEGS) {
        float2 h[N / 2];
#pragma unroll
        for (int j = 0; j < N / 2; ++j) h[j] = seed[j];
        for (int s = 0; s < NSEG - 1; ++s) {
          next_step(1);
#pragma unroll 4
          for (int i = 0; i < TS; ++i) scan_state_swz<N>(h, A2f, st.at(DTF, i), st.at(XN, i), st.row(BF, i), sw);
          ck_store<N>(ck, s, h);
        }
      }
      float2 gf[N / 2];  // a_{t+1} gbar_{t+1}, entering token t from the right
      vzero2<N>(gf);
      for (int s = NSEG - 1; s >= 0; --s) {
        if (SEGS) next_step(2);
        float2 h[N / 2];
        if (s == 0) {
#pragma unroll
          for (int j = 0; j < N / 2; ++j) h[j] = seed[j];
        } else {
          ck_load<N>(h, ck, s - 1);
        }
        int64_t o = (row0 + (int64_t)(s + 1) * TS - 1) * g.D + d;
        seg_bwd<N, true>(st, TS, XN, DTF, DYN, BF, CF, A2f, sw, h, gf, dAf, tb, mine, off, TILED ? 2 : 0,
                         [&](int i, float dt, float x, float dy, float sgB, float sAq) {
                           const int ib = s * TS + i;
                           if (act) {
                             reinterpret_cast<TO*>(p.ddtf)[o] = to_out<TO>(__fmaf_rn(x, sgB, __fmul_rn(kLn2, sAq)));
                             const float dxf = __fmul_rn(dt, sgB);
                             if (SPLIT)
                               dxf_part[o] = dxf;
                             else
                               reinterpret_cast<TO*>(p.dxn)[o] = to_out<TO>(
                                   __fmaf_rn(Dsum, dy, __fadd_rn(dxbuf[(off + ib) * kCta + tid], dxf)));
                           }
                           dDn = __fmaf_rn(dy, x, dDn);
                           o -= g.D;
                         });
        if (!TILED) red_flush<N>(p, red, 0, 1, 2, 3, b, t0 + (int64_t)s * TS, TS);
      }
      // gradient of this block's seed, states[k-1]: a_{t0} gbar_{t0}
#pragma unroll
      for (int j = 0; j < N / 2; ++j) dSn[j] = gf[j];
      if (k > 0 && act) vstore2<N>(p.dS + ((b * g.nb + (k - 1)) * g.D + d) * N, gf, sw);
    }
  };

  if (TILED) {
    // Short blocks are staged in tiles of TB blocks (at most kBwdTS tokens),
    // the next tile copied while the current one is used, and the dB/dC
    // partials of a tile are flushed once for both directions.
    const int TB = kBwdTS / Bs;
    auto tile_lo = [&](int hi) { return hi - TB + 1 > k_lo ? hi - TB + 1 : k_lo; };
    auto issue_tile = [&](int buf, int lo, int hi) { st.issue(buf, b * g.L + (int64_t)lo * Bs, (hi - lo + 1) * Bs, g.D, d0); };
    if (bufs == 2) issue_tile(0, tile_lo(k_hi), k_hi);
    int tile = 0;
    for (int kt_hi = k_hi; kt_hi >= k_lo; ++tile) {
      const int kt_lo = tile_lo(kt_hi), nbk = kt_hi - kt_lo + 1;
      const int buf = bufs == 2 ? tile & 1 : 0;
      const bool ahead = bufs == 2 && kt_lo > k_lo;
      __syncthreads();  // the buffer to fill is no longer read
      if (bufs == 1) issue_tile(0, kt_lo, kt_hi);
      if (ahead) issue_tile(buf ^ 1, tile_lo(kt_lo - 1), kt_lo - 1);
      st.complete(buf, nbk * Bs, ahead ? 1 : 0);
      for (int k = kt_hi; k >= kt_lo; --k) block(k, (k - kt_lo) * Bs);
      const int64_t ts0 = (int64_t)kt_lo * Bs;  // the tile's dB/dC partials, both directions
      if (do_rev) red_flush<N>(p, red, 0, 1, 4, 5, b, ts0, nbk * Bs);
      if (do_fwd) red_flush<N>(p, red, 2, 3, 2, 3, b, ts0, nbk * Bs);
      kt_hi = kt_lo - 1;
    }
  } else if (SEGS) {
    for (int k = k_hi; k >= k_lo; --k) block(k, 0);
  } else {
    // two buffers: block k-1 is copied while block k is processed
    if (bufs == 2) st.issue(0, b * g.L + (int64_t)k_hi * Bs, TS, g.D, d0);
    for (int k = k_hi; k >= k_lo; --k) {
      const int64_t row0 = b * g.L + (int64_t)k * Bs;
      const int buf = bufs == 2 ? (k_hi - k) & 1 : 0;
      const bool ahead = bufs == 2 && k > k_lo;
      __syncthreads();  // the buffer to fill is no longer read
      if (bufs == 1) st.issue(0, row0, TS, g.D, d0);
      if (ahead) st.issue(buf ^ 1, row0 - Bs, TS, g.D, d0);
      st.complete(buf, TS, ahead ? 1 : 0);
      block(k, 0);
    }
  }

  if (act) {
    const int64_t u = b * g.nc + c, U = g.Bt * g.nc;
    if (do_clean) {
      vstore2<N>(p.Lc + (u * g.D + d) * N, carry, sw);
      p.sdtc[u * g.D + d] = sdt;
    }
    if (do_fwd) {
      vstore2<N>(p.part_A + ((0 * U + u) * g.D + d) * N, dAf, sw);
      p.part_D[(0 * U + u) * g.D + d] = dDn;
    }
    if (do_rev) vstore2<N>(p.part_A + ((1 * U + u) * g.D + d) * N, dAr, sw);
  }
  tmem_sync();
  if (warp == 0) tmem_dealloc(tbase, tcols);
}

namespace {

template <typename T, typename TO, int N, int KIND, bool SPLIT>
BwdLaunch noisy_launch(int Bs, int dev) {
  return bwd_launch<NoisyBwdSmem<T, N, KIND>, is_f32<T>::value>(k_bwd_noisy<T, TO, N, KIND, SPLIT>, Bs,
                                                               full_cols(Bs < 16 ? Bs : 16, N), dev);
}
template <typename T, typename TO, int N, int KIND, bool SPLIT>
cudaError_t bwd_noisy_tt(const BwdParams& p_in, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const BwdLaunch l = noisy_launch<T, TO, N, KIND, SPLIT>((int)p_in.g.Bs, dev);
  BwdParams p = p_in;
  p.stage_bufs = l.bufs;
  e = set_bwd_attrs(k_bwd_noisy<T, TO, N, KIND, SPLIT>, l.smem);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)p.g.G, (unsigned)p.g.nc, (unsigned)(SPLIT ? 3 * p.g.Bt : p.g.Bt));
  launch_pdl(k_bwd_noisy<T, TO, N, KIND, SPLIT>, grid, kCta, l.smem, s, p);
  return cudaGetLastError();
}
template <typename T, typename TO, int N>
cudaError_t bwd_noisy_t(const BwdParams& p, cudaStream_t s) {
  const bool split = p.dx_part != nullptr;
  switch (split && p.g.Bs < 16 ? kOneSeg : block_kind(p.g.Bs)) {
    case kTiles: return bwd_noisy_tt<T, TO, N, kTiles, false>(p, s);
    case kSegs: return split ? bwd_noisy_tt<T, TO, N, kSegs, true>(p, s) : bwd_noisy_tt<T, TO, N, kSegs, false>(p, s);
    default: return split ? bwd_noisy_tt<T, TO, N, kOneSeg, true>(p, s) : bwd_noisy_tt<T, TO, N, kOneSeg, false>(p, s);
  }
}

template <typename T, typename TO, int N, int KIND>
int noisy_resident(int Bs, int dev) {
  return resident_ctas(k_bwd_noisy<T, TO, N, KIND, false>, noisy_launch<T, TO, N, KIND, false>(Bs, dev).smem,
                       full_cols(Bs < 16 ? Bs : 16, N), dev);
}
template <typename T, typename TO, int N>
int bwd_noisy_per_sm_t(int Bs, int dev) {
  switch (block_kind(Bs)) {
    case kTiles: return noisy_resident<T, TO, N, kTiles>(Bs, dev);
    case kSegs: return noisy_resident<T, TO, N, kSegs>(Bs, dev);
    default: return noisy_resident<T, TO, N, kOneSeg>(Bs, dev);
  }
}

}  // namespace

cudaError_t launch_bwd_noisy(int dt, int N, const BwdParams& p, cudaStream_t s) {
  switch (dt) {
    case 0: BDS_DISPATCH_N(N, return bwd_noisy_t<float, float, NN>(p, s);)
    case 1: BDS_DISPATCH_N(N, return bwd_noisy_t<bf16, bf16, NN>(p, s);)
    default: BDS_DISPATCH_N(N, return bwd_noisy_t<bf16, float, NN>(p, s);)
  }
}

int bwd_noisy_per_sm(int dt, int N, int Bs, int dev) {
  if (dt == 0) return N == 8 ? bwd_noisy_per_sm_t<float, float, 8>(Bs, dev) : bwd_noisy_per_sm_t<float, float, 16>(Bs, dev);
  if (dt == 1) return N == 8 ? bwd_noisy_per_sm_t<bf16, bf16, 8>(Bs, dev) : bwd_noisy_per_sm_t<bf16, bf16, 16>(Bs, dev);
  return N == 8 ? bwd_noisy_per_sm_t<bf16, float, 8>(Bs, dev) : bwd_noisy_per_sm_t<bf16, float, 16>(Bs, dev);
}

}  // namespace bds
