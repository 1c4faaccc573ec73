// bwd_clean.cu -- the clean-stream backward of libbdscan (sm_103a); see
// bwd_common.cuh for the derivative and the kernel sequence.
#include "bwd_common.cuh"

namespace bds {

// ---------------------------------------------------------------------------
// Clean stream backward from the exact chunk carries
// ---------------------------------------------------------------------------
template <typename T, int N>
struct CleanBwdSmem {
  using St = Stage<T, N, 3, 2, 2, kBwdTS>;  // x_c, dt_c, dy_c; B_c, C_c
  // `bufs` staging buffers, as for the noisy kernel
  static __host__ __device__ size_t red_off(int bufs) { return align16(St::buf_bytes(kBwdTS) * bufs); }
  static __host__ __device__ size_t ck_off(int bufs) { return red_off(bufs) + (size_t)2 * kBwdTS * kRedRow * 4; }
  // checkpoints in shared memory up to kCkSmemMaxBs tokens, else in global memory
  static __host__ __device__ size_t slot_off(int bufs, int TS, int Bs) {
    return ck_off(bufs) + (Bs > kCkSmemMaxBs ? 0 : (size_t)(Bs / TS - 1) * N * kCta * 4);
  }
  // one-segment blocks: the seed of each buffer's block
  static __host__ __device__ size_t seed_off(int bufs, int TS, int Bs) { return slot_off(bufs, TS, Bs) + 16; }
  static __host__ __device__ size_t bytes(int bufs, int TS, int Bs) {
    return seed_off(bufs, TS, Bs) + (Bs / TS == 1 ? (size_t)bufs * kCta * N * 4 : 0);
  }
};

// KIND: how the chunk is walked (params.h). Blocks of several segments
// make two passes, the checkpoints and the segments, each staging what it
// reads, one segment ahead.
template <typename T, typename TO, int N, int KIND>
__global__ void __launch_bounds__(kCta, 3) k_bwd_clean(const BwdParams p) {
  pdl_sync();
  extern __shared__ __align__(16) unsigned char smem[];
  using L = CleanBwdSmem<T, N>;
  constexpr bool TILED = KIND == kTiles, SEGS = KIND == kSegs;
  const Geo& g = p.g;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int sw = swz_of_lane<N>();
  const int64_t b = blockIdx.z;
  const int c = blockIdx.y;
  const int64_t d0 = (int64_t)blockIdx.x * kCta, d = d0 + tid;
  const bool act = d < g.D;
  const int Bs = KIND == kOneSeg ? 16 : (int)g.Bs, TS = TILED ? Bs : 16, NSEG = SEGS ? Bs / 16 : 1;
  const int k_lo = chunk_lo(g, c), k_hi = chunk_lo(g, c + 1) - 1;
  // debug build: the chunk's last token and the channel group lie inside the sizes
  if (!(dguard(kSiteBwdClean, b, g.Bt) && dguard(kSiteBwdClean, (int64_t)(k_hi + 1) * Bs - 1, g.L) &&
        dguard(kSiteBwdClean, d0, g.D)))
    return;

  enum { XC = 0, DTC = 1, DYC = 2 };
  enum { BC = 0, CC = 1 };
  typename L::St st;
  st.carve(smem, TS);
  st.td_src[XC] = (const T*)p.xc;
  st.td_src[DTC] = (const T*)p.dtc;
  st.td_src[DYC] = (const T*)p.dyc;
  st.row_src[BC] = (const T*)p.Bc;
  st.row_src[CC] = (const T*)p.Cc;
  const int bufs = is_f32<T>::value ? p.stage_bufs : 2;
  float* red = reinterpret_cast<float*>(smem + L::red_off(bufs));
  float* mine = red_slot<N>(red);
  float* ck = Bs > kCkSmemMaxBs
                  ? p.ck_clean + (((size_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x) *
                                     (size_t)(NSEG - 1) * N * kCta
                  : reinterpret_cast<float*>(smem + L::ck_off(bufs));
  uint32_t* tslot = reinterpret_cast<uint32_t*>(smem + L::slot_off(bufs, TS, Bs));
  float* seedb = reinterpret_cast<float*>(smem + L::seed_off(bufs, TS, Bs));  // [2][kCta][N]

  const uint32_t tcols = half_cols(TS, N);  // held states of a segment
  if (warp == 0) tmem_alloc(tslot, tcols);
  tmem_sync();
  const uint32_t tbase = *tslot;
  const uint32_t tb = tbase + ((uint32_t)(warp * 32) << 16);

  float2 A2[N / 2];
  vzero2<N>(A2);
  float Df = 0.f;
  if (act) {
    vload2<N>(A2, p.Af + d * N, sw);
#pragma unroll
    for (int j = 0; j < N / 2; ++j) A2[j] = mul2(A2[j], f2(kLog2e));
    Df = p.Df[d];
  }
  float2 dA[N / 2];
  vzero2<N>(dA);
  float dDc = 0.f;
  float2 gc[N / 2];  // a_{t+1} gbar_{t+1} (+ injections) entering token t from the right
  vzero2<N>(gc);

  // SEGS: the steps (pass, segment) of a block in the order they are used, one
  // step staged ahead: checkpoints of segments 0 .. NSEG-2, then every segment
  // from the last.
  int nk = k_hi, ns = 0, fill = 0, cur = 0;  // next step to copy, buffers
  bool nadj = false;                         // the next step is of the second pass
  auto copy_step = [&]() {
    if (nk < k_lo) return false;
    st.issue_first(fill, b * g.L + (int64_t)nk * Bs + ns * TS, TS, g.D, d0, nadj ? 3 : 2, nadj ? 2 : 1);
    fill ^= bufs - 1;
    if (!nadj) {
      nadj = ++ns > NSEG - 2;  // ns is the last segment then
    } else if (--ns < 0) {
      nadj = false;
      ns = 0;
      --nk;
    }
    return true;
  };
  auto next_step = [&](int nrow) {  // the next step's tiles become current
    __syncthreads();                // the buffer to fill is no longer read
    const bool ahead = copy_step() && bufs == 2;
    st.complete(cur, TS, ahead ? 1 : 0, nrow);
    cur ^= bufs - 1;
  };
  if (SEGS && bufs == 2) copy_step();

  // everything for block k, whose tokens start at `off` in the staged tile;
  // seed_staged: its seed is in seedb[buf]
  auto block = [&](int k, int off, int buf, bool seed_staged) {
    const int64_t t0 = (int64_t)k * Bs;
    const int64_t row0 = b * g.L + t0;
    if (k == k_hi) {
      if (act) vload2<N>(gc, p.Lc + ((b * g.nc + c) * g.D + d) * N, sw);
    } else if (act) {
      float2 e[N / 2];
      vload2<N>(e, p.dS + ((b * g.nb + k) * g.D + d) * N, sw);
#pragma unroll
      for (int j = 0; j < N / 2; ++j) gc[j] = add2(gc[j], e[j]);
      if (p.dstates != nullptr) {
        vload2<N>(e, p.dstates + ((b * g.nb + k) * g.D + d) * N, sw);
#pragma unroll
        for (int j = 0; j < N / 2; ++j) gc[j] = add2(gc[j], e[j]);
      }
    }
    float2 seed[N / 2];
    vzero2<N>(seed);
    if (seed_staged)
      vload2<N>(seed, seedb + (buf * kCta + tid) * N, sw);  // staged with the tile
    else if (k > 0 && act)
      vload2<N>(seed, p.states + ((b * g.nb + (k - 1)) * g.D + d) * N, sw);
    if (SEGS) {
      float2 h[N / 2];
#pragma unroll
      for (int j = 0; j < N / 2; ++j) h[j] = seed[j];
      for (int s = 0; s < NSEG - 1; ++s) {
        next_step(1);
#pragma unroll 4
        for (int i = 0; i < TS; ++i) scan_state_swz<N>(h, A2, st.at(DTC, i), st.at(XC, i), st.row(BC, i), sw);
        ck_store<N>(ck, s, h);
      }
    }
    for (int s = NSEG - 1; s >= 0; --s) {
      if (SEGS) next_step(2);
      float2 h[N / 2];
      if (s == 0) {
#pragma unroll
        for (int j = 0; j < N / 2; ++j) h[j] = seed[j];
      } else {
        ck_load<N>(h, ck, s - 1);
      }
      int64_t o = (row0 + (int64_t)(s + 1) * TS - 1) * g.D + d;  // the token's element, stepped
      seg_bwd_half<N, true>(st, TS, XC, DTC, DYC, BC, CC, A2, sw, h, gc, dA, tb, mine, off, 0,
                       [&](int i, float dt, float x, float dy, float sgB, float sAq) {
                         if (act) {
                           reinterpret_cast<TO*>(p.ddtc)[o] = to_out<TO>(__fmaf_rn(x, sgB, __fmul_rn(kLn2, sAq)));
                           reinterpret_cast<TO*>(p.dxc)[o] = to_out<TO>(__fmaf_rn(Df, dy, __fmul_rn(dt, sgB)));
                         }
                         dDc = __fmaf_rn(dy, x, dDc);
                         o -= g.D;
                       });
      if (!TILED) red_flush<N>(p, red, 0, 1, 0, 1, b, t0 + (int64_t)s * TS, TS);
    }
  };

  if (TILED) {
    // Short blocks are staged in tiles of TB blocks (at most kBwdTS tokens)
    // together with the seed of the tile's last block, the next tile copied
    // while the current one is used, and the dB/dC partials of a tile are
    // flushed once.
    const int TB = kBwdTS / Bs;
    auto tile_lo = [&](int hi) { return hi - TB + 1 > k_lo ? hi - TB + 1 : k_lo; };
    auto issue_tile = [&](int buf, int lo, int hi) {
      issue_seed<N>(seedb + buf * kCta * N, p.states, g, b, hi, d0);  // same cp.async group as the tile
      st.issue(buf, b * g.L + (int64_t)lo * Bs, (hi - lo + 1) * Bs, g.D, d0);
    };
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
      for (int k = kt_hi; k >= kt_lo; --k) block(k, (k - kt_lo) * Bs, buf, k == kt_hi);
      red_flush<N>(p, red, 0, 1, 0, 1, b, (int64_t)kt_lo * Bs, nbk * Bs);  // the tile's dB/dC
      kt_hi = kt_lo - 1;
    }
  } else if (SEGS) {
    for (int k = k_hi; k >= k_lo; --k) block(k, 0, 0, false);
  } else {
    // two buffers: block k-1 (and its seed) is copied while block k is processed
    auto issue_block = [&](int buf, int k) {
      issue_seed<N>(seedb + buf * kCta * N, p.states, g, b, k, d0);  // same cp.async group as the block
      st.issue(buf, b * g.L + (int64_t)k * Bs, TS, g.D, d0);
    };
    if (bufs == 2) issue_block(0, k_hi);
    for (int k = k_hi; k >= k_lo; --k) {
      const int buf = bufs == 2 ? (k_hi - k) & 1 : 0;
      const bool ahead = bufs == 2 && k > k_lo;
      __syncthreads();  // the buffer to fill is no longer read
      if (bufs == 1) issue_block(0, k);
      if (ahead) issue_block(buf ^ 1, k - 1);
      st.complete(buf, TS, ahead ? 1 : 0);
      block(k, 0, buf, true);
    }
  }
  if (act) {
    const int64_t u = b * g.nc + c, U = g.Bt * g.nc;
    vstore2<N>(p.part_A + ((2 * U + u) * g.D + d) * N, dA, sw);
    p.part_D[(1 * U + u) * g.D + d] = dDc;
  }
  tmem_sync();
  if (warp == 0) tmem_dealloc(tbase, tcols);
}

namespace {

template <typename T, typename TO, int N, int KIND>
BwdLaunch clean_launch(int Bs, int dev) {
  return bwd_launch<CleanBwdSmem<T, N>, is_f32<T>::value>(k_bwd_clean<T, TO, N, KIND>, Bs,
                                                          half_cols(Bs < 16 ? Bs : 16, N), dev);
}

template <typename T, typename TO, int N, int KIND>
cudaError_t bwd_clean_tt(const BwdParams& p_in, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const BwdLaunch l = clean_launch<T, TO, N, KIND>((int)p_in.g.Bs, dev);
  BwdParams p = p_in;
  p.stage_bufs = l.bufs;
  e = set_bwd_attrs(k_bwd_clean<T, TO, N, KIND>, l.smem);
  if (e != cudaSuccess) return e;
  dim3 grid((unsigned)p.g.G, (unsigned)p.g.nc, (unsigned)p.g.Bt);
  launch_pdl(k_bwd_clean<T, TO, N, KIND>, grid, kCta, l.smem, s, p);
  return cudaGetLastError();
}
template <typename T, typename TO, int N>
cudaError_t bwd_clean_t(const BwdParams& p, cudaStream_t s) {
  switch (block_kind(p.g.Bs)) {
    case kTiles: return bwd_clean_tt<T, TO, N, kTiles>(p, s);
    case kSegs: return bwd_clean_tt<T, TO, N, kSegs>(p, s);
    default: return bwd_clean_tt<T, TO, N, kOneSeg>(p, s);
  }
}

template <typename T, typename TO, int N, int KIND>
int clean_resident(int Bs, int dev) {
  return resident_ctas(k_bwd_clean<T, TO, N, KIND>, clean_launch<T, TO, N, KIND>(Bs, dev).smem,
                       half_cols(Bs < 16 ? Bs : 16, N), dev);
}
template <typename T, typename TO, int N>
int bwd_clean_per_sm_t(int Bs, int dev) {
  switch (block_kind(Bs)) {
    case kTiles: return clean_resident<T, TO, N, kTiles>(Bs, dev);
    case kSegs: return clean_resident<T, TO, N, kSegs>(Bs, dev);
    default: return clean_resident<T, TO, N, kOneSeg>(Bs, dev);
  }
}

}  // namespace

cudaError_t launch_bwd_clean(int dt, int N, const BwdParams& p, cudaStream_t s) {
  switch (dt) {
    case 0: BDS_DISPATCH_N(N, return bwd_clean_t<float, float, NN>(p, s);)
    case 1: BDS_DISPATCH_N(N, return bwd_clean_t<bf16, bf16, NN>(p, s);)
    default: BDS_DISPATCH_N(N, return bwd_clean_t<bf16, float, NN>(p, s);)
  }
}

int bwd_clean_per_sm(int dt, int N, int Bs, int dev) {
  if (dt == 0) return N == 8 ? bwd_clean_per_sm_t<float, float, 8>(Bs, dev) : bwd_clean_per_sm_t<float, float, 16>(Bs, dev);
  if (dt == 1) return N == 8 ? bwd_clean_per_sm_t<bf16, bf16, 8>(Bs, dev) : bwd_clean_per_sm_t<bf16, bf16, 16>(Bs, dev);
  return N == 8 ? bwd_clean_per_sm_t<bf16, float, 8>(Bs, dev) : bwd_clean_per_sm_t<bf16, float, 16>(Bs, dev);
}

}  // namespace bds
