// mixer.cu -- the steps either side of the scan in a Mamba mixer (see
// include/bdscan_mixer.h): the width-4 causal depthwise convolution with
// SiLU (its last three inputs are part of the cache, Sec. 4.1 eq. cache-c4),
// the step size softplus(dt_raw + bias), and the SiLU-gated output; forward,
// backward, cache build and cached active block.
//
// These steps are elementwise per (token, channel), against the scan's work
// per (token, channel, state), and memory-bound: each runs as one fused pass
// over the tensors (convolution, SiLU and softplus together; gate and its
// derivative together) around the scan kernels of the library, which run in
// fp32 on intermediates kept in the workspace. The channel sums of the
// parameter gradients (taps, biases) are fixed-order two-level reductions,
// so results are deterministic.
#include <cstdio>
#include <cstring>

#include "bdscan_mixer.h"
#include "device.cuh"
#include "params.h"

namespace bds {
namespace {

constexpr int kW = 4;           // convolution width
constexpr int kParSplit = 256;  // most token slices of the parameter-gradient reduction

// The logistic function and softplus on the fast hardware paths (__expf,
// __logf, __fdividef): relative errors of order 1e-6, far inside the
// tolerance of the path, and the same functions serve every entry point, so
// the cache paths stay bit-identical to the all-block ones.
__device__ __forceinline__ float sigm(float z) { return __fdividef(1.f, __fadd_rn(1.f, __expf(-z))); }
__device__ __forceinline__ float silu(float z) { return __fmul_rn(z, sigm(z)); }
// d SiLU / dz = s (1 + z (1 - s))
__device__ __forceinline__ float dsilu(float z) {
  const float s = sigm(z);
  return __fmul_rn(s, __fmaf_rn(z, __fsub_rn(1.f, s), 1.f));
}
__device__ __forceinline__ float softplus(float z) {
  return __fadd_rn(fmaxf(z, 0.f), __logf(__fadd_rn(1.f, __expf(-fabsf(z)))));
}

// Arguments of the input-side kernels. Token-by-channel tensors [Bt][L][D].
template <typename T>
struct MixIn {
  int64_t Bt, L, D, Bs;
  const T *xr_c, *dtr_c, *xr_n, *dtr_f, *dtr_r;
  const float *w, *cb, *bias_f, *bias_r;
  const float* conv_init;  // [Bt][3][D] or null
};

// Raw clean input at position u of batch row b, channel d (positions before 0
// read the initial convolution state).
template <typename T>
__device__ __forceinline__ float raw_c(const MixIn<T>& a, int64_t b, int64_t u, int64_t d) {
  if (u >= 0) return cvt(a.xr_c[(b * a.L + u) * a.D + d]);
  return a.conv_init != nullptr ? a.conv_init[(b * (kW - 1) + (kW - 1) + u) * a.D + d] : 0.f;
}
// Vector access: V = 16 / sizeof(T) consecutive channels per thread (8 for
// bf16, 4 for fp32; d_inner is a multiple of V), so every token-by-channel
// load is 16 bytes per thread.
template <typename T>
struct Vec {
  static constexpr int V = 16 / (int)sizeof(T);
};
__device__ __forceinline__ void ld16(const bf16* p, float (&v)[8]) {
  const uint4 u = *reinterpret_cast<const uint4*>(p);
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&u);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 f = __bfloat1622float2(h[e]);
    v[2 * e] = f.x;
    v[2 * e + 1] = f.y;
  }
}
__device__ __forceinline__ void ld16(const float* p, float (&v)[4]) {
  const float4 u = *reinterpret_cast<const float4*>(p);
  v[0] = u.x;
  v[1] = u.y;
  v[2] = u.z;
  v[3] = u.w;
}
template <int V>
__device__ __forceinline__ void ldf(const float* p, float (&v)[V]) {
#pragma unroll
  for (int q = 0; q < V / 4; ++q) {
    const float4 u = *reinterpret_cast<const float4*>(p + 4 * q);
    v[4 * q] = u.x;
    v[4 * q + 1] = u.y;
    v[4 * q + 2] = u.z;
    v[4 * q + 3] = u.w;
  }
}
template <int V>
__device__ __forceinline__ void stv(float* p, const float (&v)[V]) {
#pragma unroll
  for (int q = 0; q < V / 4; ++q)
    *reinterpret_cast<float4*>(p + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
}
template <int V>
__device__ __forceinline__ void stv(bf16* p, const float (&v)[V]) {
#pragma unroll
  for (int q = 0; q < V / 4; ++q) {
    const __nv_bfloat162 a = __floats2bfloat162_rn(v[4 * q], v[4 * q + 1]);
    const __nv_bfloat162 c = __floats2bfloat162_rn(v[4 * q + 2], v[4 * q + 3]);
    *reinterpret_cast<uint2*>(p + 4 * q) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&c));
  }
}

// Q = 2 or 4 consecutive channels of one row; d_inner is a multiple of 4, so
// the rows of Q channels are aligned to the access.
template <int Q>
__device__ __forceinline__ void ldq(const float* p, float (&v)[Q]) {
  if (Q == 4) {
    const float4 u = *reinterpret_cast<const float4*>(p);
    v[0] = u.x, v[1] = u.y, v[Q - 2] = u.z, v[Q - 1] = u.w;
  } else {
    const float2 u = *reinterpret_cast<const float2*>(p);
    v[0] = u.x, v[1] = u.y;
  }
}
template <int Q>
__device__ __forceinline__ void ldq(const bf16* p, float (&v)[Q]) {
  uint32_t u[Q / 2];
  if (Q == 4)
    *reinterpret_cast<uint2*>(u) = *reinterpret_cast<const uint2*>(p);
  else
    u[0] = *reinterpret_cast<const uint32_t*>(p);
#pragma unroll
  for (int e = 0; e < Q / 2; ++e) {
    v[2 * e] = __uint_as_float(u[e] << 16);
    v[2 * e + 1] = __uint_as_float(u[e] & 0xffff0000u);
  }
}
template <int Q>
__device__ __forceinline__ void stq(float* p, const float (&v)[Q]) {
  if (Q == 4)
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[Q - 2], v[Q - 1]);
  else
    *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
}
template <int Q>
__device__ __forceinline__ void stq(bf16* p, const float (&v)[Q]) {
#pragma unroll
  for (int e = 0; e < Q / 2; ++e)
    reinterpret_cast<__nv_bfloat162*>(p)[e] = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
}
template <int Q>
__device__ __forceinline__ void zeroq(float (&v)[Q]) {
#pragma unroll
  for (int e = 0; e < Q; ++e) v[e] = 0.f;
}

// Raw clean inputs at position u of batch row b for Q channels from d: the
// clean stream, the initial convolution state before token 0, zero past the
// end (or without a clean stream, where no window reads them).
template <typename T, int Q>
__device__ __forceinline__ void raw_cq(const MixIn<T>& a, int64_t b, int u, int64_t d, float (&r)[Q]) {
  if (u >= 0 && u < a.L && a.xr_c != nullptr)
    ldq<Q>(a.xr_c + (b * a.L + u) * a.D + d, r);
  else if (u < 0 && a.conv_init != nullptr)
    ldq<Q>(a.conv_init + (b * (kW - 1) + (kW - 1) + u) * a.D + d, r);
  else
    zeroq<Q>(r);
}
// The noisy stream's raw inputs at u, zero outside the stream.
template <typename T, int Q>
__device__ __forceinline__ void raw_nq(const MixIn<T>& a, int64_t b, int u, int64_t d, float (&r)[Q]) {
  if (u >= 0 && u < a.L)
    ldq<Q>(a.xr_n + (b * a.L + u) * a.D + d, r);
  else
    zeroq<Q>(r);
}
// Positions fit 32 bits (the checks on dims bound len by 65535 chunks of at
// most 256 tokens), so block offsets are 32-bit remainders.
template <typename T>
__device__ __forceinline__ int block_off(const MixIn<T>& a, int t) {
  return (int)((uint32_t)t % (uint32_t)a.Bs);
}

// The token sweeps below read their rows through a ring in shared memory: each
// thread copies (cp.async) the Q channels it will use itself, kAhead tokens
// before it uses them, so no barrier is needed and enough bytes are in flight
// without holding them in registers.
template <int BYTES>
__device__ __forceinline__ void copy_async(void* smem, const void* gmem) {
  const uint32_t s = (uint32_t)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(s), "l"(gmem), "n"(BYTES) : "memory");
}
template <int PENDING>
__device__ __forceinline__ void wait_async() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(PENDING) : "memory");
}

// Scan inputs in fp32: x = SiLU(conv), dt = softplus(dt_raw + bias), for the
// clean stream (if x_c) and the noisy stream (if x_n). A thread sweeps Ls
// consecutive tokens of 4 channels with the convolution window in registers
// (slot q holds the last row whose position is q modulo 4 of the sweep).
// Bound by memory: 8 x 2048 x 1536 bf16 moves 755 MB; one element per thread,
// each with its own window loads and two 64-bit divisions, took 391 us.
constexpr int kPrepCta = 128, kPrepRing = 8, kPrepAhead = kPrepRing - 1;
template <typename T>
constexpr size_t prep_smem() {
  return (size_t)kPrepRing * 5 * kPrepCta * 4 * sizeof(T);
}
template <typename T>
__global__ void __launch_bounds__(kPrepCta, 4) k_mix_prep(const MixIn<T> a, float* x_c, float* dt_c, float* x_n,
                                                       float* dt_f, float* dt_r, int Ls) {
  pdl_sync();
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int Q = 4, S = 4, W1 = kW - 1;
  const int64_t d = ((int64_t)blockIdx.y * blockDim.x + threadIdx.x) * Q, b = blockIdx.z;
  const int tb = (int)(blockIdx.x * blockDim.y + threadIdx.y) * Ls, L = (int)a.L, Bs = (int)a.Bs;
  if (d >= a.D || tb >= L) return;
  const int te = tb + Ls < L ? tb + Ls : L;
  T* ring = reinterpret_cast<T*>(smem) + (threadIdx.y * blockDim.x + threadIdx.x) * Q;  // [slot][tensor][thread]
  auto slot = [&](int t, int k) { return ring + ((t & (kPrepRing - 1)) * 5 + k) * (kPrepCta * Q); };
  constexpr int BYTES = Q * (int)sizeof(T);
  auto issue = [&](int t) {
    if (t < te) {
      const int64_t i = (b * a.L + t) * a.D + d;
      if (a.xr_c != nullptr) {
        copy_async<BYTES>(slot(t, 0), a.xr_c + i);
        if (x_c != nullptr) copy_async<BYTES>(slot(t, 1), a.dtr_c + i);
      }
      if (x_n != nullptr) {
        copy_async<BYTES>(slot(t, 2), a.xr_n + i);
        copy_async<BYTES>(slot(t, 3), a.dtr_f + i);
        copy_async<BYTES>(slot(t, 4), a.dtr_r + i);
      }
    }
    cp_async_commit();
  };
#pragma unroll
  for (int q = 0; q < kPrepAhead; ++q) issue(tb + q);
  float c[S][Q], n[S][Q];
#pragma unroll
  for (int q = 0; q < S; ++q) {
    zeroq<Q>(c[q]);
    zeroq<Q>(n[q]);
  }
#pragma unroll
  for (int q = 1; q < S; ++q) {
    raw_cq<T, Q>(a, b, tb - S + q, d, c[q]);
    if (x_n != nullptr) raw_nq<T, Q>(a, b, tb - S + q, d, n[q]);
  }
  float w[kW * Q], cb[Q], bf[Q], br[Q];
  ldf<kW * Q>(a.w + d * kW, w);
  ldq<Q>(a.cb + d, cb);
  ldq<Q>(a.bias_f + d, bf);
  ldq<Q>(a.bias_r + d, br);
  int off = block_off(a, tb);
  for (int t0 = tb; t0 < te; t0 += S) {
#pragma unroll
    for (int q = 0; q < S; ++q) {
      const int t = t0 + q;
      if (t >= te) break;
      issue(t + kPrepAhead);
      wait_async<kPrepAhead>();
      const int64_t i = (b * a.L + t) * a.D + d;
      float o[Q], v[Q];
      if (a.xr_c != nullptr) ldq<Q>(slot(t, 0), c[q]);
      if (x_c != nullptr) {
        ldq<Q>(slot(t, 1), v);
#pragma unroll
        for (int e = 0; e < Q; ++e) {
          float pre = cb[e];
#pragma unroll
          for (int j = 0; j < kW; ++j) pre = __fmaf_rn(w[e * kW + j], c[(q + 1 + j) % S][e], pre);
          o[e] = silu(pre);
          v[e] = softplus(__fadd_rn(v[e], bf[e]));
        }
        stq<Q>(x_c + i, o);
        stq<Q>(dt_c + i, v);
      }
      if (x_n != nullptr) {
        ldq<Q>(slot(t, 2), n[q]);
        ldq<Q>(slot(t, 3), v);
#pragma unroll
        for (int e = 0; e < Q; ++e) {
          float pre = cb[e];
#pragma unroll
          for (int j = 0; j < kW; ++j)  // tap j is at t - 3 + j: inside the block from its first token on
            pre = __fmaf_rn(w[e * kW + j], off >= W1 - j ? n[(q + 1 + j) % S][e] : c[(q + 1 + j) % S][e], pre);
          o[e] = silu(pre);
          v[e] = softplus(__fadd_rn(v[e], bf[e]));
        }
        stq<Q>(x_n + i, o);
        stq<Q>(dt_f + i, v);
        ldq<Q>(slot(t, 4), v);
#pragma unroll
        for (int e = 0; e < Q; ++e) v[e] = softplus(__fadd_rn(v[e], br[e]));
        stq<Q>(dt_r + i, v);
      }
      off = off + 1 == Bs ? 0 : off + 1;
    }
  }
}

// The backward from the scan's fp32 gradients to the raw inputs, in one pass:
// through SiLU (gp = gx SiLU'(pre)), softplus (the step-size gradients), the
// convolution's transpose (raw position u feeds tap j of token u + 3 - j; a
// noisy token's taps before its block feed the clean stream) and the partial
// sums of the parameter gradients, part[slice][v][d] for v = tap 0..3, conv
// bias, dt_bias_f, dt_bias_r. gp exists in registers only.
// A warp sweeps segments of Ls consecutive tokens (and the three after each,
// whose gp the transpose needs) for 64 channels, with windows of the last four
// raw rows and gp rows (slot q: position q modulo 4 of the sweep); the eight
// warps of a CTA share the channels and leave one slice of sums.
// Bound by memory: 8 x 2048 x 1536 bf16 moves 1.0 GB; as three kernels that
// exchanged gp through memory the same work took 795 us.
constexpr int kBwdGroups = 8, kBwdRing = 4, kBwdAhead = kBwdRing - 1;  // warps per CTA; ring of token rows
template <typename T>
constexpr size_t mix_bwd_smem() {
  return (size_t)kBwdRing * 5 * 32 * kBwdGroups * 2 * (sizeof(T) + 4);
}
template <typename T, typename TO>
__global__ void __launch_bounds__(32 * kBwdGroups, 2)
    k_mix_bwd(const MixIn<T> a, const float* gx_c, const float* gdt_c, const float* gx_n, const float* gdt_f,
              const float* gdt_r, TO* dxr_c, TO* ddtr_c, TO* dxr_n, TO* ddtr_f, TO* ddtr_r, int Ls, int nseg,
              float* part) {
  pdl_sync();
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int Q = 2, W1 = kW - 1, S = 4, TH = 32 * kBwdGroups;
  __shared__ float red[kBwdGroups][kW + 3][32 * Q];
  const int lane = threadIdx.x, grp = threadIdx.y;
  const int64_t d = ((int64_t)blockIdx.y * 32 + lane) * Q;
  const int L = (int)a.L, Bs = (int)a.Bs;
  // ring[slot][tensor][thread]: fp32 gx_c, gx_n, gdt_c, gdt_f, gdt_r, then xr_c, xr_n, dtr_c, dtr_f, dtr_r
  float* fring = reinterpret_cast<float*>(smem) + (grp * 32 + lane) * Q;
  T* tring = reinterpret_cast<T*>(smem + (size_t)kBwdRing * 5 * TH * Q * 4) + (grp * 32 + lane) * Q;
  auto fslot = [&](int t, int k) { return fring + ((t & (kBwdRing - 1)) * 5 + k) * (TH * Q); };
  auto tslot = [&](int t, int k) { return tring + ((t & (kBwdRing - 1)) * 5 + k) * (TH * Q); };
  float s[kW + 3][Q];
#pragma unroll
  for (int q = 0; q < kW + 3; ++q) zeroq<Q>(s[q]);
  if (d < a.D) {
    float w[kW * Q], cb[Q], bf[Q], br[Q];
    ldf<kW * Q>(a.w + d * kW, w);
    ldq<Q>(a.cb + d, cb);
    ldq<Q>(a.bias_f + d, bf);
    ldq<Q>(a.bias_r + d, br);
    const int64_t segs = a.Bt * nseg;
    for (int64_t seg = (int64_t)blockIdx.x * kBwdGroups + grp; seg < segs; seg += (int64_t)gridDim.x * kBwdGroups) {
      const int64_t b = seg / nseg;
      const int tb = (int)(seg - b * nseg) * Ls, te = tb + Ls < L ? tb + Ls : L;
      const int th = te + W1 < L ? te + W1 : L;  // tokens whose gp is needed
      auto issue = [&](int t) {
        if (t < th) {
          const int64_t i = (b * a.L + t) * a.D + d;
          copy_async<8>(fslot(t, 0), gx_c + i);
          copy_async<8>(fslot(t, 1), gx_n + i);
          copy_async<2 * sizeof(T)>(tslot(t, 0), a.xr_c + i);
          copy_async<2 * sizeof(T)>(tslot(t, 1), a.xr_n + i);
          if (t < te) {
            copy_async<8>(fslot(t, 2), gdt_c + i);
            copy_async<8>(fslot(t, 3), gdt_f + i);
            copy_async<8>(fslot(t, 4), gdt_r + i);
            copy_async<2 * sizeof(T)>(tslot(t, 2), a.dtr_c + i);
            copy_async<2 * sizeof(T)>(tslot(t, 3), a.dtr_f + i);
            copy_async<2 * sizeof(T)>(tslot(t, 4), a.dtr_r + i);
          }
        }
        cp_async_commit();
      };
#pragma unroll
      for (int q = 0; q < kBwdAhead; ++q) issue(tb + q);
      float c[S][Q], n[S][Q], pc[S][Q], pn[S][Q];
      int off[S];  // the token's offset in its block
#pragma unroll
      for (int q = 0; q < S; ++q) {
        zeroq<Q>(c[q]);
        zeroq<Q>(n[q]);
        zeroq<Q>(pc[q]);
        zeroq<Q>(pn[q]);
        off[q] = 0;
      }
#pragma unroll
      for (int q = 1; q < S; ++q) {
        raw_cq<T, Q>(a, b, tb - S + q, d, c[q]);
        raw_nq<T, Q>(a, b, tb - S + q, d, n[q]);
      }
      int o = block_off(a, tb);
      for (int t0 = tb; t0 < te + W1; t0 += S) {
#pragma unroll
        for (int q = 0; q < S; ++q) {
          const int t = t0 + q;
          if (t >= te + W1) break;
          issue(t + kBwdAhead);
          wait_async<kBwdAhead>();
          off[q] = o;
          o = o + 1 == Bs ? 0 : o + 1;
          if (t < L) {
            ldq<Q>(tslot(t, 0), c[q]);
            ldq<Q>(tslot(t, 1), n[q]);
            ldq<Q>(fslot(t, 0), pc[q]);
            ldq<Q>(fslot(t, 1), pn[q]);
#pragma unroll
            for (int e = 0; e < Q; ++e) {
              float rc[kW], rn[kW], prc = cb[e], prn = cb[e];
#pragma unroll
              for (int j = 0; j < kW; ++j) {
                rc[j] = c[(q + 1 + j) % S][e];
                rn[j] = off[q] >= W1 - j ? n[(q + 1 + j) % S][e] : rc[j];
                prc = __fmaf_rn(w[e * kW + j], rc[j], prc);
                prn = __fmaf_rn(w[e * kW + j], rn[j], prn);
              }
              pc[q][e] = __fmul_rn(pc[q][e], dsilu(prc));
              pn[q][e] = __fmul_rn(pn[q][e], dsilu(prn));
              if (t < te) {
#pragma unroll
                for (int j = 0; j < kW; ++j) s[j][e] = __fmaf_rn(pn[q][e], rn[j], __fmaf_rn(pc[q][e], rc[j], s[j][e]));
                s[kW][e] = __fadd_rn(s[kW][e], __fadd_rn(pc[q][e], pn[q][e]));
              }
            }
            if (t < te) {
              const int64_t i = (b * a.L + t) * a.D + d;
              float v1[Q], v2[Q], v3[Q], r1[Q], r2[Q], r3[Q];
              ldq<Q>(fslot(t, 2), v1);
              ldq<Q>(fslot(t, 3), v2);
              ldq<Q>(fslot(t, 4), v3);
              ldq<Q>(tslot(t, 2), r1);
              ldq<Q>(tslot(t, 3), r2);
              ldq<Q>(tslot(t, 4), r3);
#pragma unroll
              for (int e = 0; e < Q; ++e) {
                v1[e] = __fmul_rn(v1[e], sigm(__fadd_rn(r1[e], bf[e])));
                v2[e] = __fmul_rn(v2[e], sigm(__fadd_rn(r2[e], bf[e])));
                v3[e] = __fmul_rn(v3[e], sigm(__fadd_rn(r3[e], br[e])));
                s[kW + 1][e] = __fadd_rn(s[kW + 1][e], __fadd_rn(v1[e], v2[e]));
                s[kW + 2][e] = __fadd_rn(s[kW + 2][e], v3[e]);
              }
              stq<Q>(ddtr_c + i, v1);
              stq<Q>(ddtr_f + i, v2);
              stq<Q>(ddtr_r + i, v3);
            }
          }
          // gp of tokens u ... u + 3 is complete: the raw gradients of u = t - 3
          const int u = t - W1;
          if (u >= tb) {
            float ac[Q], an[Q];
            zeroq<Q>(ac);
            zeroq<Q>(an);
#pragma unroll
            for (int j = 0; j < kW; ++j) {
              if (t - j >= L) continue;
              const int k = (q + S - j) % S;
              const bool inside = off[k] >= W1 - j;  // the same block as the consuming noisy token
#pragma unroll
              for (int e = 0; e < Q; ++e) {
                const float wj = w[e * kW + j];
                ac[e] = __fmaf_rn(wj, pc[k][e], ac[e]);
                if (inside)
                  an[e] = __fmaf_rn(wj, pn[k][e], an[e]);
                else
                  ac[e] = __fmaf_rn(wj, pn[k][e], ac[e]);
              }
            }
            const int64_t i = (b * a.L + u) * a.D + d;
            stq<Q>(dxr_c + i, ac);
            stq<Q>(dxr_n + i, an);
          }
        }
      }
    }
  }
#pragma unroll
  for (int q = 0; q < kW + 3; ++q)
#pragma unroll
    for (int e = 0; e < Q; ++e) red[grp][q][lane * Q + e] = s[q][e];
  __syncthreads();
  for (int i = grp * 32 + lane; i < (kW + 3) * 32 * Q; i += TH) {
    const int q = i / (32 * Q), k = i - q * (32 * Q);
    const int64_t dk = (int64_t)blockIdx.y * 32 * Q + k;
    float v = red[0][q][k];
#pragma unroll
    for (int r = 1; r < kBwdGroups; ++r) v = __fadd_rn(v, red[r][q][k]);
    if (dk < a.D) part[((int64_t)blockIdx.x * (kW + 3) + q) * a.D + dk] = v;
  }
}

// The slices summed in order: dconv_w [D][4], dconv_b, ddt_bias_f, ddt_bias_r [D].
__global__ void __launch_bounds__(256) k_mix_par_red(int64_t D, int slices, const float* part, float* dw, float* db,
                                                     float* dbf, float* dbr) {
  pdl_sync();
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= D * (kW + 3)) return;
  const int v = (int)(i / D);
  const int64_t d = i % D;
  float s = 0.f;
#pragma unroll 16
  for (int sl = 0; sl < slices; ++sl) s = __fadd_rn(s, part[((int64_t)sl * (kW + 3) + v) * D + d]);
  if (v < kW)
    dw[d * kW + v] = s;
  else if (v == kW)
    db[d] = s;
  else if (v == kW + 1)
    dbf[d] = s;
  else
    dbr[d] = s;
}

// out = y * SiLU(z), V elements per thread.
template <typename T, typename TO>
__global__ void __launch_bounds__(256) k_mix_gate(int64_t n, const float* y, const T* z, TO* out) {
  pdl_sync();
  constexpr int V = Vec<T>::V;
  const int64_t i = ((int64_t)blockIdx.x * 256 + threadIdx.x) * V;
  if (i >= n) return;
  float yv[V], zv[V];
  ldf<V>(y + i, yv);
  ld16(z + i, zv);
#pragma unroll
  for (int v = 0; v < V; ++v) yv[v] = __fmul_rn(yv[v], silu(zv[v]));
  stv<V>(out + i, yv);
}

// The gate's backward: dy = dout * SiLU(z), dz = dout * y * SiLU'(z) (zero
// without dout), V elements per thread.
template <typename T, typename TO>
__global__ void __launch_bounds__(256) k_mix_gate_bwd(int64_t n, const float* y, const T* z, const T* dout, float* dy,
                                                      TO* dz) {
  pdl_sync();
  constexpr int V = Vec<T>::V;
  const int64_t i = ((int64_t)blockIdx.x * 256 + threadIdx.x) * V;
  if (i >= n) return;
  float yv[V], zv[V], gv[V], a[V], c[V];
  ldf<V>(y + i, yv);
  ld16(z + i, zv);
  if (dout != nullptr) {
    ld16(dout + i, gv);
  } else {
#pragma unroll
    for (int v = 0; v < V; ++v) gv[v] = 0.f;
  }
#pragma unroll
  for (int v = 0; v < V; ++v) {
    a[v] = __fmul_rn(gv[v], silu(zv[v]));
    c[v] = __fmul_rn(__fmul_rn(gv[v], yv[v]), dsilu(zv[v]));
  }
  stv<V>(dy + i, a);
  stv<V>(dz + i, c);
}

// Element type conversion of up to six tensors of n elements (B, C to fp32
// for the scan; their gradients back), one per blockIdx.y; four elements per
// thread (rows of d_state are multiples of 4).
struct CvtSet {
  const void* src[6];
  void* dst[6];
};
template <typename TI, typename TO>
__global__ void __launch_bounds__(256) k_mix_cvt(int64_t n, const __grid_constant__ CvtSet c) {
  pdl_sync();
  const int64_t i = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 4;
  if (i >= n) return;
  float v[4];
  ldq<4>((const TI*)c.src[blockIdx.y] + i, v);
  stq<4>((TO*)c.dst[blockIdx.y] + i, v);
}

// Convolution part of the cache: the raw clean inputs of the three tokens
// before each emitted boundary (every block end, or the end of the stream).
template <typename T>
__global__ void __launch_bounds__(256) k_mix_conv_states(const MixIn<T> a, int emit_all, float* cs) {
  pdl_sync();
  const int64_t nS = emit_all ? a.L / a.Bs : 1;
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= a.Bt * nS * (kW - 1) * a.D) return;
  const int64_t d = i % a.D, r = i / a.D;
  const int q = (int)(r % (kW - 1));
  const int64_t k = (r / (kW - 1)) % nS, b = r / ((kW - 1) * nS);
  const int64_t end = emit_all ? (k + 1) * a.Bs : a.L;
  cs[i] = raw_c(a, b, end - (kW - 1) + q, d);
}

}  // namespace

// ---------------------------------------------------------------------------
// entry points
// ---------------------------------------------------------------------------
namespace {

size_t al(size_t x) { return (x + 255) & ~(size_t)255; }

// Workspace regions (byte offsets): fp32 scan inputs x_c, dt_c, x_n, dt_f,
// dt_r; fp32 B_c, C_c, B_f, C_f, B_r, C_r; fp32 scan outputs y_c, y_n; the
// scan's workspace. The backward adds the recomputed boundary states, the
// gate's fp32 gradients dy_c, dy_n, the scan's fp32 gradients (x, dt of the
// five streams, then B, C) and its workspace, and the parameter partials.
struct MixWs {
  size_t x[5], bc[6], y[2], scan, fwd_total;
  size_t states, dy[2], gx[5], gbc[6], bws, part, bwd_total;
};
MixWs mix_ws(const Geo& g, int N) {
  MixWs w;
  const size_t td = al((size_t)g.Bt * g.L * g.D * 4), tn = al((size_t)g.Bt * g.L * N * 4);
  size_t o = 0;
  for (int i = 0; i < 5; ++i, o += td) w.x[i] = o;
  for (int i = 0; i < 6; ++i, o += tn) w.bc[i] = o;
  for (int i = 0; i < 2; ++i, o += td) w.y[i] = o;
  w.scan = o;
  o += al(api_fwd_workspace(g, N));
  w.fwd_total = o;
  w.states = o;
  o += al((size_t)g.Bt * g.nb * g.D * N * 4);
  for (int i = 0; i < 2; ++i, o += td) w.dy[i] = o;
  for (int i = 0; i < 5; ++i, o += td) w.gx[i] = o;
  for (int i = 0; i < 6; ++i, o += tn) w.gbc[i] = o;
  w.bws = o;
  o += al(api_bwd_workspace(g, N));
  w.part = o;
  o += al((size_t)kParSplit * (kW + 3) * g.D * 4);
  w.bwd_total = o;
  return w;
}

bool a16(const void* p) { return ((uintptr_t)p & 15u) == 0; }

int bad_arg(const char* fn, const char* what) {
  char m[256];
  snprintf(m, sizeof(m), "%s: %s", fn, what);
  return api_fail(BDSCAN_ERR_ARG, m);
}
int cuda_err(const char* fn, cudaError_t e) {
  char m[256];
  snprintf(m, sizeof(m), "%s: %s", fn, cudaGetErrorString(e));
  return api_fail(BDSCAN_ERR_CUDA, m);
}

#define MIX_REQ(ptr, name) \
  if ((ptr) == nullptr || !a16(ptr)) return bad_arg(fn, name " is NULL or not 16-byte aligned")
#define MIX_OPT(ptr, name) \
  if ((ptr) != nullptr && !a16(ptr)) return bad_arg(fn, name " is not 16-byte aligned")

int check_mparams(const bdscan_mixer_params* m, const char* fn) {
  if (m == nullptr) return bad_arg(fn, "mparams is NULL");
  MIX_REQ(m->conv_w, "mparams.conv_w");
  MIX_REQ(m->conv_b, "mparams.conv_b");
  MIX_REQ(m->dt_bias_f, "mparams.dt_bias_f");
  MIX_REQ(m->dt_bias_r, "mparams.dt_bias_r");
  return BDSCAN_OK;
}

unsigned blocks_of(int64_t n) { return (unsigned)((n + 255) / 256); }
template <typename T>
unsigned vec_blocks(int64_t n) {
  constexpr int64_t span = 256 * Vec<T>::V;
  return (unsigned)((n + span - 1) / span);
}

template <typename T>
MixIn<T> mix_in(const Geo& g, const bdscan_clean* c, const bdscan_noisy* n, const bdscan_mixer_params* m,
                const float* conv_init) {
  MixIn<T> a;
  memset(&a, 0, sizeof(a));
  a.Bt = g.Bt;
  a.L = g.L;
  a.D = g.D;
  a.Bs = g.Bs;
  if (c != nullptr) {
    a.xr_c = (const T*)c->x;
    a.dtr_c = (const T*)c->dt;
  }
  if (n != nullptr) {
    a.xr_n = (const T*)n->x;
    a.dtr_f = (const T*)n->dt_f;
    a.dtr_r = (const T*)n->dt_r;
  }
  a.w = m->conv_w;
  a.cb = m->conv_b;
  a.bias_f = m->dt_bias_f;
  a.bias_r = m->dt_bias_r;
  a.conv_init = conv_init;
  return a;
}

template <typename TI, typename TO>
cudaError_t cvt_all(const CvtSet& c, int count, int64_t n, cudaStream_t s) {
  launch_pdl(k_mix_cvt<TI, TO>, dim3((unsigned)((n / 4 + 255) / 256), (unsigned)count), 256, 0, s, n, c);
  return api_launched(cudaGetLastError(), s);
}
// B and C of the given streams converted to fp32 into the workspace slots.
template <typename T>
cudaError_t to_f32(const void* const* src, const size_t* slot, int count, char* ws, int64_t n, cudaStream_t s) {
  CvtSet c;
  memset(&c, 0, sizeof(c));
  for (int i = 0; i < count; ++i) {
    c.src[i] = src[i];
    c.dst[i] = ws + slot[i];
  }
  return cvt_all<T, float>(c, count, n, s);
}

// Tokens per sweep of the elementwise kernels: 32 where that still leaves two
// CTAs to every SM, else 8 (shorter serial sweeps). `ctas(Ls)` is the CTA count.
template <typename F>
int sweep_len(F ctas) {
  return ctas(32) >= 2 * (int64_t)sm_count_cached() ? 32 : 8;
}

template <typename T>
cudaError_t prep(const Geo& g, const MixIn<T>& a, float* x_c, float* dt_c, float* x_n, float* dt_f, float* dt_r,
                 cudaStream_t s) {
  const int64_t quads = (g.D + 3) / 4;
  unsigned tx = 8;  // threads along the channels, the rest along the sweeps
  while (tx < kPrepCta && tx < quads) tx <<= 1;
  const unsigned ty = kPrepCta / tx, tiles = (unsigned)((quads + tx - 1) / tx);
  auto runs = [&](int ls) { return (unsigned)(((g.L + ls - 1) / ls + ty - 1) / ty); };
  const int Ls = sweep_len([&](int ls) { return g.Bt * tiles * runs(ls); });
  cudaError_t e = set_smem_cached((const void*)k_mix_prep<T>, (int)prep_smem<T>(), -1);
  if (e != cudaSuccess) return e;
  launch_pdl(k_mix_prep<T>, dim3(runs(Ls), tiles, (unsigned)g.Bt), dim3(tx, ty), prep_smem<T>(), s, a, x_c, dt_c, x_n, dt_f,
             dt_r, Ls);
  return api_launched(cudaGetLastError(), s);
}

// The forward of both streams up to the scan outputs: prep, B/C to fp32, the
// all-block scan in fp32 (states into `states`).
template <typename T>
cudaError_t mix_forward_core(const Geo& g, int N, const bdscan_clean* cl, const bdscan_noisy* nz,
                             const bdscan_params* pr, const bdscan_mixer_params* mp, float* states, char* ws,
                             const MixWs& w, cudaStream_t s) {
  const MixIn<T> a = mix_in<T>(g, cl, nz, mp, nullptr);
  const int64_t nn = g.Bt * g.L * N;
  float* X[5];
  for (int i = 0; i < 5; ++i) X[i] = (float*)(ws + w.x[i]);
  cudaError_t e = prep<T>(g, a, X[0], X[1], X[2], X[3], X[4], s);
  const void* bc[6] = {cl->B, cl->C, nz->B_f, nz->C_f, nz->B_r, nz->C_r};
  if (e == cudaSuccess) e = to_f32<T>(bc, w.bc, 6, ws, nn, s);
  if (e != cudaSuccess) return e;
  FwdParams p;
  memset(&p, 0, sizeof(p));
  p.g = g;
  p.xc = X[0];
  p.dtc = X[1];
  p.Bc = ws + w.bc[0];
  p.Cc = ws + w.bc[1];
  p.xn = X[2];
  p.dtf = X[3];
  p.Bf = ws + w.bc[2];
  p.Cf = ws + w.bc[3];
  p.dtr = X[4];
  p.Br = ws + w.bc[4];
  p.Cr = ws + w.bc[5];
  p.Af = pr->A_f;
  p.Df = pr->D_f;
  p.Ar = pr->A_r;
  p.Dr = pr->D_r;
  p.yc = ws + w.y[0];
  p.yn = ws + w.y[1];
  p.states = states;
  return api_run_forward(0, N, p, ws + w.scan, s);
}

template <typename T, typename TO>
cudaError_t gate(int64_t n, const char* ws, size_t yslot, const void* z, void* out, cudaStream_t s) {
  launch_pdl(k_mix_gate<T, TO>, vec_blocks<T>(n), 256, 0, s, n, (const float*)(ws + yslot), (const T*)z, (TO*)out);
  return api_launched(cudaGetLastError(), s);
}

template <typename T, typename TO>
cudaError_t mix_forward_t(const Geo& g, int N, const bdscan_clean* cl, const void* z_c, const bdscan_noisy* nz,
                          const void* z_n, const bdscan_params* pr, const bdscan_mixer_params* mp, void* out_c,
                          void* out_n, float* states, char* ws, cudaStream_t s) {
  const MixWs w = mix_ws(g, N);
  cudaError_t e = mix_forward_core<T>(g, N, cl, nz, pr, mp, states, ws, w, s);
  const int64_t n = g.Bt * g.L * g.D;
  if (e == cudaSuccess) e = gate<T, TO>(n, ws, w.y[0], z_c, out_c, s);
  if (e == cudaSuccess) e = gate<T, TO>(n, ws, w.y[1], z_n, out_n, s);
  return e;
}

template <typename T, typename TO>
cudaError_t mix_backward_t(const Geo& g, int N, const bdscan_clean* cl, const void* z_c, const bdscan_noisy* nz,
                           const void* z_n, const bdscan_params* pr, const bdscan_mixer_params* mp,
                           const void* dout_c, const void* dout_n, const float* dstates,
                           const bdscan_clean_grads* gc, void* dz_c, const bdscan_noisy_grads* gn, void* dz_n,
                           const bdscan_param_grads* gp, const bdscan_mixer_grads* gm, char* ws, cudaStream_t s) {
  const MixWs w = mix_ws(g, N);
  float* states = (float*)(ws + w.states);
  // recompute the forward's scan inputs, outputs and boundary states
  cudaError_t e = mix_forward_core<T>(g, N, cl, nz, pr, mp, states, ws, w, s);
  if (e != cudaSuccess) return e;
  const int64_t n = g.Bt * g.L * g.D, nn = g.Bt * g.L * N;
  float* dy[2] = {(float*)(ws + w.dy[0]), (float*)(ws + w.dy[1])};
  launch_pdl(k_mix_gate_bwd<T, TO>, vec_blocks<T>(n), 256, 0, s, n, (const float*)(ws + w.y[0]), (const T*)z_c,
             (const T*)dout_c, dy[0], (TO*)dz_c);
  e = api_launched(cudaGetLastError(), s);
  if (e != cudaSuccess) return e;
  launch_pdl(k_mix_gate_bwd<T, TO>, vec_blocks<T>(n), 256, 0, s, n, (const float*)(ws + w.y[1]), (const T*)z_n,
             (const T*)dout_n, dy[1], (TO*)dz_n);
  e = api_launched(cudaGetLastError(), s);
  if (e != cudaSuccess) return e;
  float* G[5];
  for (int i = 0; i < 5; ++i) G[i] = (float*)(ws + w.gx[i]);
  BwdParams q;
  memset(&q, 0, sizeof(q));
  q.g = g;
  q.xc = ws + w.x[0];
  q.dtc = ws + w.x[1];
  q.Bc = ws + w.bc[0];
  q.Cc = ws + w.bc[1];
  q.xn = ws + w.x[2];
  q.dtf = ws + w.x[3];
  q.Bf = ws + w.bc[2];
  q.Cf = ws + w.bc[3];
  q.dtr = ws + w.x[4];
  q.Br = ws + w.bc[4];
  q.Cr = ws + w.bc[5];
  q.Af = pr->A_f;
  q.Df = pr->D_f;
  q.Ar = pr->A_r;
  q.Dr = pr->D_r;
  q.states = states;
  q.dyc = dy[0];
  q.dyn = dy[1];
  q.dstates = dstates;
  q.dxc = G[0];
  q.ddtc = G[1];
  q.dBc = ws + w.gbc[0];
  q.dCc = ws + w.gbc[1];
  q.dxn = G[2];
  q.ddtf = G[3];
  q.dBf = ws + w.gbc[2];
  q.dCf = ws + w.gbc[3];
  q.ddtr = G[4];
  q.dBr = ws + w.gbc[4];
  q.dCr = ws + w.gbc[5];
  q.dAf = gp->dA_f;
  q.dDf = gp->dD_f;
  q.dAr = gp->dA_r;
  q.dDr = gp->dD_r;
  e = api_run_backward(0, N, q, ws + w.bws, s);
  if (e != cudaSuccess) return e;
  // through SiLU, softplus and the convolution
  const MixIn<T> a = mix_in<T>(g, cl, nz, mp, nullptr);
  float* part = (float*)(ws + w.part);
  const int64_t tiles = (g.D + 63) / 64;
  auto ctas = [&](int ls) { return (g.Bt * ((g.L + ls - 1) / ls) + kBwdGroups - 1) / kBwdGroups; };
  const int Ls = sweep_len([&](int ls) { return ctas(ls) * tiles; });
  const int64_t want = ctas(Ls);
  const int slices = (int)(want < kParSplit ? want : kParSplit);
  if ((e = set_smem_cached((const void*)k_mix_bwd<T, TO>, (int)mix_bwd_smem<T>(), -1)) != cudaSuccess) return e;
  launch_pdl(k_mix_bwd<T, TO>, dim3((unsigned)slices, (unsigned)tiles), dim3(32, kBwdGroups), mix_bwd_smem<T>(), s,
             a, G[0], G[1], G[2], G[3], G[4], (TO*)gc->dx, (TO*)gc->ddt, (TO*)gn->dx, (TO*)gn->ddt_f, (TO*)gn->ddt_r, Ls,
             (int)((g.L + Ls - 1) / Ls), part);
  e = api_launched(cudaGetLastError(), s);
  if (e != cudaSuccess) return e;
  CvtSet cv;
  void* gbc_out[6] = {gc->dB, gc->dC, gn->dB_f, gn->dC_f, gn->dB_r, gn->dC_r};
  for (int i = 0; i < 6; ++i) {
    cv.src[i] = ws + w.gbc[i];
    cv.dst[i] = gbc_out[i];
  }
  if ((e = cvt_all<float, TO>(cv, 6, nn, s)) != cudaSuccess) return e;
  launch_pdl(k_mix_par_red, blocks_of(g.D * (kW + 3)), 256, 0, s, g.D, slices, part, gm->dconv_w, gm->dconv_b,
             gm->ddt_bias_f, gm->ddt_bias_r);
  return api_launched(cudaGetLastError(), s);
}

template <typename T, typename TO>
cudaError_t mix_boundary_t(const Geo& g, int N, const bdscan_clean* cl, const void* z_c, const float* A_f,
                           const float* D_f, const bdscan_mixer_params* mp, const float* init_state,
                           const float* conv_init, void* out_c, float* states, float* conv_states, int emit_all,
                           char* ws, cudaStream_t s) {
  const MixWs w = mix_ws(g, N);
  const MixIn<T> a = mix_in<T>(g, cl, nullptr, mp, conv_init);
  const int64_t n = g.Bt * g.L * g.D, nn = g.Bt * g.L * N;
  cudaError_t e = prep<T>(g, a, (float*)(ws + w.x[0]), (float*)(ws + w.x[1]), nullptr, nullptr, nullptr, s);
  const void* bc[2] = {cl->B, cl->C};
  if (e == cudaSuccess) e = to_f32<T>(bc, w.bc, 2, ws, nn, s);
  if (e != cudaSuccess) return e;
  FwdParams p;
  memset(&p, 0, sizeof(p));
  p.g = g;
  p.xc = ws + w.x[0];
  p.dtc = ws + w.x[1];
  p.Bc = ws + w.bc[0];
  p.Cc = ws + w.bc[1];
  p.Af = A_f;
  p.Df = D_f;
  p.init = init_state;
  p.yc = out_c != nullptr ? (void*)(ws + w.y[0]) : nullptr;
  p.hst = (float*)(ws + w.scan);
  p.sdt = (float*)(ws + w.scan + al((size_t)g.Bt * (g.nc + 1) * g.D * N * 4));
  e = api_run_boundary(0, N, p, states, emit_all, s);
  if (e == cudaSuccess && out_c != nullptr) e = gate<T, TO>(n, ws, w.y[0], z_c, out_c, s);
  if (e != cudaSuccess) return e;
  const int64_t nc = g.Bt * (emit_all ? g.nb : 1) * (kW - 1) * g.D;
  launch_pdl(k_mix_conv_states<T>, blocks_of(nc), 256, 0, s, a, emit_all, conv_states);
  return api_launched(cudaGetLastError(), s);
}

template <typename T, typename TO>
cudaError_t mix_active_t(const Geo& g, int N, const float* seed, const float* conv_seed, const bdscan_noisy* nz,
                         const void* z_n, const bdscan_params* pr, const bdscan_mixer_params* mp, void* out_n,
                         char* ws, cudaStream_t s) {
  const MixWs w = mix_ws(g, N);
  // one block: every window position before its first token reads the cached
  // convolution state
  const MixIn<T> a = mix_in<T>(g, nullptr, nz, mp, conv_seed);
  const int64_t n = g.Bt * g.L * g.D, nn = g.Bt * g.L * N;
  cudaError_t e = prep<T>(g, a, nullptr, nullptr, (float*)(ws + w.x[2]), (float*)(ws + w.x[3]),
                          (float*)(ws + w.x[4]), s);
  const void* bc[4] = {nz->B_f, nz->C_f, nz->B_r, nz->C_r};
  if (e == cudaSuccess) e = to_f32<T>(bc, w.bc + 2, 4, ws, nn, s);
  if (e != cudaSuccess) return e;
  FwdParams p;
  memset(&p, 0, sizeof(p));
  p.g = g;
  p.xn = ws + w.x[2];
  p.dtf = ws + w.x[3];
  p.Bf = ws + w.bc[2];
  p.Cf = ws + w.bc[3];
  p.dtr = ws + w.x[4];
  p.Br = ws + w.bc[4];
  p.Cr = ws + w.bc[5];
  p.Af = pr->A_f;
  p.Df = pr->D_f;
  p.Ar = pr->A_r;
  p.Dr = pr->D_r;
  p.yn = ws + w.y[1];
  p.seed = seed;
  e = api_launched(launch_active_block(0, N, p, s), s);
  if (e == cudaSuccess) e = gate<T, TO>(n, ws, w.y[1], z_n, out_n, s);
  return e;
}

// dt code: 0 f32 in and out, 1 bf16 in and out, 2 bf16 in, f32 out
#define MIX_DISPATCH(dt, CALL)                      \
  switch (dt) {                                     \
    case 0: { using T = float; using TO = float; return CALL; } \
    case 1: { using T = bf16; using TO = bf16; return CALL; }   \
    default: { using T = bf16; using TO = float; return CALL; } \
  }

}  // namespace
}  // namespace bds

using bds::Geo;
using bds::a16;
using bds::bad_arg;
using bds::bf16;

namespace {

template <typename F>
int mix_run(const char* fn, F f) {
  const cudaError_t e = f();
  if (e != cudaSuccess) return bds::cuda_err(fn, e);
  return bds::api_ok();
}

int mix_check_streams(const char* fn, const bdscan_clean* cl, const bdscan_noisy* nz) {
  if (cl != nullptr) {
    MIX_REQ(cl->x, "clean.x");
    MIX_REQ(cl->dt, "clean.dt");
    MIX_REQ(cl->B, "clean.B");
    MIX_REQ(cl->C, "clean.C");
  }
  if (nz != nullptr) {
    MIX_REQ(nz->x, "noisy.x");
    MIX_REQ(nz->dt_f, "noisy.dt_f");
    MIX_REQ(nz->B_f, "noisy.B_f");
    MIX_REQ(nz->C_f, "noisy.C_f");
    MIX_REQ(nz->dt_r, "noisy.dt_r");
    MIX_REQ(nz->B_r, "noisy.B_r");
    MIX_REQ(nz->C_r, "noisy.C_r");
  }
  return BDSCAN_OK;
}
int mix_check_params(const char* fn, const bdscan_params* pr) {
  if (pr == nullptr) return bds::bad_arg(fn, "params is NULL");
  MIX_REQ(pr->A_f, "params.A_f");
  MIX_REQ(pr->D_f, "params.D_f");
  MIX_REQ(pr->A_r, "params.A_r");
  MIX_REQ(pr->D_r, "params.D_r");
  return BDSCAN_OK;
}
int mix_check_ws(const char* fn, void* ws, size_t have, size_t need) {
  MIX_REQ(ws, "workspace");
  if (have < need) {
    char m[200];
    snprintf(m, sizeof(m), "workspace of %zu bytes, %zu needed", have, need);
    return bds::bad_arg(fn, m);
  }
  return BDSCAN_OK;
}

}  // namespace

extern "C" {

size_t bdscan_mixer_forward_workspace_size(const bdscan_dims* dims) {
  Geo g;
  int dt = 0, N = 0;
  if (bds::api_check_forward_dims(dims, &g, &dt, &N, "bdscan_mixer_forward_workspace_size")) return 0;
  return bds::mix_ws(g, N).fwd_total;
}
size_t bdscan_mixer_backward_workspace_size(const bdscan_dims* dims) {
  Geo g;
  int dt = 0, N = 0;
  if (bds::api_check_forward_dims(dims, &g, &dt, &N, "bdscan_mixer_backward_workspace_size")) return 0;
  return bds::mix_ws(g, N).bwd_total;
}
size_t bdscan_mixer_boundary_states_workspace_size(const bdscan_dims* dims) {
  return bdscan_mixer_forward_workspace_size(dims);
}
size_t bdscan_mixer_active_block_workspace_size(const bdscan_dims* dims) {
  return bdscan_mixer_forward_workspace_size(dims);
}

int bdscan_mixer_forward(const bdscan_dims* dims, const bdscan_clean* clean, const void* z_c,
                         const bdscan_noisy* noisy, const void* z_n, const bdscan_params* params,
                         const bdscan_mixer_params* mparams, void* out_c, void* out_n, float* states,
                         void* workspace, size_t workspace_bytes, void* stream) {
  const char* fn = "bdscan_mixer_forward";
  Geo g;
  int dt = 0, N = 0;
  int rc = bds::api_check_forward_dims(dims, &g, &dt, &N, fn);
  if (rc) return rc;
  if (g.Bt == 0 || g.L == 0) return bds::api_ok();
  if (clean == nullptr || noisy == nullptr) return bds::bad_arg(fn, "clean or noisy is NULL");
  if ((rc = mix_check_streams(fn, clean, noisy)) || (rc = mix_check_params(fn, params)) ||
      (rc = bds::check_mparams(mparams, fn)))
    return rc;
  MIX_REQ(z_c, "z_c");
  MIX_REQ(z_n, "z_n");
  MIX_REQ(out_c, "out_c");
  MIX_REQ(out_n, "out_n");
  MIX_REQ(states, "states");
  if ((rc = mix_check_ws(fn, workspace, workspace_bytes, bds::mix_ws(g, N).fwd_total))) return rc;
  char* ws = (char*)workspace;
  cudaStream_t s = (cudaStream_t)stream;
  return mix_run(fn, [&]() -> cudaError_t {
    MIX_DISPATCH(dt, (bds::mix_forward_t<T, TO>(g, N, clean, z_c, noisy, z_n, params, mparams, out_c, out_n, states,
                                               ws, s)))
  });
}

int bdscan_mixer_backward(const bdscan_dims* dims, const bdscan_clean* clean, const void* z_c,
                          const bdscan_noisy* noisy, const void* z_n, const bdscan_params* params,
                          const bdscan_mixer_params* mparams, const void* dout_c, const void* dout_n,
                          const float* dstates, const bdscan_clean_grads* gclean, void* dz_c,
                          const bdscan_noisy_grads* gnoisy, void* dz_n, const bdscan_param_grads* gparams,
                          const bdscan_mixer_grads* gmparams, void* workspace, size_t workspace_bytes,
                          void* stream) {
  const char* fn = "bdscan_mixer_backward";
  Geo g;
  int dt = 0, N = 0;
  int rc = bds::api_check_forward_dims(dims, &g, &dt, &N, fn);
  if (rc) return rc;
  if (g.Bs > 256)
    return bds::api_fail(BDSCAN_ERR_UNSUPPORTED, "bdscan_mixer_backward: backward block above 256");
  if (g.Bs > 16 && g.Bs % 16 != 0)
    return bds::api_fail(BDSCAN_ERR_UNSUPPORTED, "bdscan_mixer_backward: backward needs block <= 16 or a multiple of 16");
  if (gparams == nullptr || gmparams == nullptr) return bds::bad_arg(fn, "gparams or gmparams is NULL");
  MIX_REQ(gparams->dA_f, "dA_f");
  MIX_REQ(gparams->dD_f, "dD_f");
  MIX_REQ(gparams->dA_r, "dA_r");
  MIX_REQ(gparams->dD_r, "dD_r");
  MIX_REQ(gmparams->dconv_w, "dconv_w");
  MIX_REQ(gmparams->dconv_b, "dconv_b");
  MIX_REQ(gmparams->ddt_bias_f, "ddt_bias_f");
  MIX_REQ(gmparams->ddt_bias_r, "ddt_bias_r");
  if (g.Bt == 0 || g.L == 0) return bds::api_fail(BDSCAN_ERR_UNSUPPORTED, "bdscan_mixer_backward: empty problem");
  if (clean == nullptr || noisy == nullptr) return bds::bad_arg(fn, "clean or noisy is NULL");
  if ((rc = mix_check_streams(fn, clean, noisy)) || (rc = mix_check_params(fn, params)) ||
      (rc = bds::check_mparams(mparams, fn)))
    return rc;
  MIX_REQ(z_c, "z_c");
  MIX_REQ(z_n, "z_n");
  MIX_OPT(dout_c, "dout_c");
  MIX_REQ(dout_n, "dout_n");
  MIX_OPT(dstates, "dstates");
  MIX_REQ(dz_c, "dz_c");
  MIX_REQ(dz_n, "dz_n");
  if (gclean == nullptr || gnoisy == nullptr) return bds::bad_arg(fn, "gradient struct is NULL");
  MIX_REQ(gclean->dx, "gclean.dx");
  MIX_REQ(gclean->ddt, "gclean.ddt");
  MIX_REQ(gclean->dB, "gclean.dB");
  MIX_REQ(gclean->dC, "gclean.dC");
  MIX_REQ(gnoisy->dx, "gnoisy.dx");
  MIX_REQ(gnoisy->ddt_f, "gnoisy.ddt_f");
  MIX_REQ(gnoisy->dB_f, "gnoisy.dB_f");
  MIX_REQ(gnoisy->dC_f, "gnoisy.dC_f");
  MIX_REQ(gnoisy->ddt_r, "gnoisy.ddt_r");
  MIX_REQ(gnoisy->dB_r, "gnoisy.dB_r");
  MIX_REQ(gnoisy->dC_r, "gnoisy.dC_r");
  if ((rc = mix_check_ws(fn, workspace, workspace_bytes, bds::mix_ws(g, N).bwd_total))) return rc;
  char* ws = (char*)workspace;
  cudaStream_t s = (cudaStream_t)stream;
  return mix_run(fn, [&]() -> cudaError_t {
    MIX_DISPATCH(dt, (bds::mix_backward_t<T, TO>(g, N, clean, z_c, noisy, z_n, params, mparams, dout_c, dout_n,
                                                dstates, gclean, dz_c, gnoisy, dz_n, gparams, gmparams, ws, s)))
  });
}

int bdscan_mixer_boundary_states(const bdscan_dims* dims, const bdscan_clean* clean, const void* z_c,
                                 const float* A_f, const float* D_f, const bdscan_mixer_params* mparams,
                                 const float* init_state, const float* conv_init, void* out_c, float* states,
                                 float* conv_states, int emit_all, void* workspace, size_t workspace_bytes,
                                 void* stream) {
  const char* fn = "bdscan_mixer_boundary_states";
  Geo g;
  int dt = 0, N = 0;
  int rc = bds::api_check_forward_dims(dims, &g, &dt, &N, fn);
  if (rc) return rc;
  if (g.Bt == 0) return bds::api_ok();
  MIX_OPT(init_state, "init_state");
  MIX_OPT(conv_init, "conv_init");
  cudaStream_t s = (cudaStream_t)stream;
  if (g.L == 0) {  // the cache is the initial state
    if (emit_all) return bds::api_ok();
    MIX_REQ(states, "states");
    MIX_REQ(conv_states, "conv_states");
    const size_t sb = (size_t)g.Bt * g.D * N * 4, cb = (size_t)g.Bt * 3 * g.D * 4;
    cudaError_t e = init_state ? cudaMemcpyAsync(states, init_state, sb, cudaMemcpyDeviceToDevice, s)
                               : cudaMemsetAsync(states, 0, sb, s);
    if (e == cudaSuccess)
      e = conv_init ? cudaMemcpyAsync(conv_states, conv_init, cb, cudaMemcpyDeviceToDevice, s)
                    : cudaMemsetAsync(conv_states, 0, cb, s);
    return e == cudaSuccess ? bds::api_ok() : bds::cuda_err(fn, e);
  }
  if (clean == nullptr) return bds::bad_arg(fn, "clean is NULL");
  if ((rc = mix_check_streams(fn, clean, nullptr)) || (rc = bds::check_mparams(mparams, fn))) return rc;
  MIX_REQ(A_f, "A_f");
  MIX_REQ(D_f, "D_f");
  MIX_REQ(states, "states");
  MIX_REQ(conv_states, "conv_states");
  MIX_OPT(out_c, "out_c");
  MIX_OPT(z_c, "z_c");
  if ((out_c == nullptr) != (z_c == nullptr)) return bds::bad_arg(fn, "give both z_c and out_c, or neither");
  if ((rc = mix_check_ws(fn, workspace, workspace_bytes, bds::mix_ws(g, N).fwd_total))) return rc;
  char* ws = (char*)workspace;
  return mix_run(fn, [&]() -> cudaError_t {
    MIX_DISPATCH(dt, (bds::mix_boundary_t<T, TO>(g, N, clean, z_c, A_f, D_f, mparams, init_state, conv_init, out_c,
                                                states, conv_states, emit_all ? 1 : 0, ws, s)))
  });
}

int bdscan_mixer_active_block(const bdscan_dims* dims, const float* seed, const float* conv_seed,
                              const bdscan_noisy* noisy, const void* z_n, const bdscan_params* params,
                              const bdscan_mixer_params* mparams, void* out_n, void* workspace,
                              size_t workspace_bytes, void* stream) {
  const char* fn = "bdscan_mixer_active_block";
  Geo g;
  int dt = 0, N = 0;
  int rc = bds::api_check_forward_dims(dims, &g, &dt, &N, fn);
  if (rc) return rc;
  if (dims->len != dims->block && dims->len != 0) return bds::bad_arg(fn, "len must equal block");
  if (g.Bt == 0 || g.L == 0) return bds::api_ok();
  MIX_REQ(seed, "seed");
  MIX_REQ(conv_seed, "conv_seed");
  if (noisy == nullptr) return bds::bad_arg(fn, "noisy is NULL");
  if ((rc = mix_check_streams(fn, nullptr, noisy)) || (rc = mix_check_params(fn, params)) ||
      (rc = bds::check_mparams(mparams, fn)))
    return rc;
  MIX_REQ(z_n, "z_n");
  MIX_REQ(out_n, "out_n");
  if ((rc = mix_check_ws(fn, workspace, workspace_bytes, bds::mix_ws(g, N).fwd_total))) return rc;
  char* ws = (char*)workspace;
  cudaStream_t s = (cudaStream_t)stream;
  return mix_run(fn, [&]() -> cudaError_t {
    MIX_DISPATCH(dt, (bds::mix_active_t<T, TO>(g, N, seed, conv_seed, noisy, z_n, params, mparams, out_n, ws, s)))
  });
}

}  // extern "C"
