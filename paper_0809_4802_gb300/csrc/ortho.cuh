// One step of the Arnoldi process in one launch: the new vector w = V_kk is orthogonalised against
// V_0 .. V_{kk-1} by classical Gram-Schmidt with one re-orthogonalisation pass and normalised
// (Section 6: Krylov solves of the condensed system).
//
// What bounds it: on the vectors of one problem (1e4 to 1e6 entries) the four passes over the basis
// take a few microseconds of L2, and the nine launches they used to be (two dot products with their
// reductions and combinations, a norm, a scaling) about 60 us. Here one block per SM keeps a range
// of the rows through all passes, and the sums over the blocks are exchanged as polled words
// (cooperative launch, so every block is resident; grid barriers took 1.1 us each). Measured per GMRES step, launches
// and gaps included: 22^3 nodes, FP32 vectors 58 -> 25 us, 33^3 nodes 67 -> 32 us; FP64 vectors 89 ->
// 45 and 123 -> 68 us (bases up to 100 vectors; there the FP64 unit bounds the passes).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace vms {

constexpr int OG_THREADS = 512, OG_WARPS = OG_THREADS / 32;
constexpr int OG_K = 8;                  // vectors a warp takes at a time
constexpr int OG_MAX = 480;              // most basis vectors (MAX_RESTART)
constexpr int OG_BLOCKS = 256;           // most blocks
constexpr unsigned long long OG_UNSET = ~0ull;
// Exchange words of one launch (doubles): the blocks' shares of the dot products of the two passes
// and of the norm, the dot products.
constexpr int64_t OG_P = 0, OG_N = 2 * (int64_t)OG_MAX * OG_BLOCKS, OG_H = OG_N + OG_BLOCKS,
                  OG_SET = OG_H + 2 * OG_MAX;

// Words are exchanged between blocks by their values: a buffer holds an all-ones pattern (a NaN that
// arithmetic never produces but from an operand that is one) until a word is written, once, and its readers
// poll the word itself. Two buffers take turns; each launch sets the other one's used words back for the next.
__device__ __forceinline__ void og_put(double* p, double v) {
  if (__double_as_longlong(v) == (long long)OG_UNSET) v = __longlong_as_double(0x7ff8000000000000ll);  // another NaN
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(p), "d"(v) : "memory");
}
__device__ __forceinline__ unsigned long long og_peek(const double* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// The word at p once it is written; clears `ok` when it does not come within `lim` polls, or at once where
// an earlier wait of the thread has.
__device__ __forceinline__ double og_get(const double* p, uint32_t lim, bool& ok) {
  unsigned long long v = og_peek(p);
  for (uint32_t it = 0; v == OG_UNSET; ++it) {
    if (it >= lim || !ok) {
      ok = false;
      return 0.0;
    }
    v = og_peek(p);
  }
  return __longlong_as_double((long long)v);
}

template <typename VT> struct OgQuad;
template <> struct OgQuad<float> {
  using V4 = float4;
  // A lane's sum of products as an unevaluated pair hi + lo (two-sum), so that its accuracy does
  // not depend on how many rows the lane takes.
  struct Acc {
    float hi = 0.f, lo = 0.f;
    __device__ __forceinline__ void add(const float4& a, const float4& b) {
      const float s = fmaf(a.w, b.w, fmaf(a.z, b.z, fmaf(a.y, b.y, a.x * b.x)));
      const float t = __fadd_rn(hi, s);
      const float z = __fsub_rn(t, hi);
      lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(s, z)));
      hi = t;
    }
    __device__ __forceinline__ float value() const { return __fadd_rn(hi, lo); }
  };
  __device__ __forceinline__ static float4 zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ static void fma4(float4& s, float c, const float4& v) {
    s.x = fmaf(c, v.x, s.x); s.y = fmaf(c, v.y, s.y); s.z = fmaf(c, v.z, s.z); s.w = fmaf(c, v.w, s.w);
  }
  // s c rounded to FP32, c split into two FP32 parts: one rounding, as of an FP64 product
  __device__ __forceinline__ static void scale4(float4& s, double c) {
    const float h = (float)c, l = (float)(c - (double)h);
    s.x = fmaf(s.x, h, s.x * l); s.y = fmaf(s.y, h, s.y * l); s.z = fmaf(s.z, h, s.z * l); s.w = fmaf(s.w, h, s.w * l);
  }
};
struct alignas(16) OgD4 {
  double x, y, z, w;
};
template <> struct OgQuad<double> {
  using V4 = OgD4;
  struct Acc {
    double s = 0.0;
    __device__ __forceinline__ void add(const OgD4& a, const OgD4& b) {
      s = fma(a.w, b.w, fma(a.z, b.z, fma(a.y, b.y, fma(a.x, b.x, s))));
    }
    __device__ __forceinline__ double value() const { return s; }
  };
  __device__ __forceinline__ static OgD4 zero() { return OgD4{0.0, 0.0, 0.0, 0.0}; }
  __device__ __forceinline__ static void fma4(OgD4& s, double c, const OgD4& v) {
    s.x = fma(c, v.x, s.x); s.y = fma(c, v.y, s.y); s.z = fma(c, v.z, s.z); s.w = fma(c, v.w, s.w);
  }
  __device__ __forceinline__ static void scale4(OgD4& s, double c) { s.x *= c; s.y *= c; s.z *= c; s.w *= c; }
};

// 1 / sqrt(d) for a positive normal d: the approximation of the PTX instruction set and two Newton
// steps r <- r + r (1 - d r^2) / 2, each of which squares its relative error. A square root and a
// division are about a hundred FP64 instructions, 64 cycles each on one warp.
__device__ __forceinline__ double og_rsqrt(double d) {
  double r;
  asm("rsqrt.approx.f64 %0, %1;" : "=d"(r) : "d"(d));
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const double e = fma(-d * r, r, 1.0);
    r = fma(0.5 * r, e, r);
  }
  return r;
}

// V: basis, vectors of n entries (n a multiple of 4, V 16-byte aligned) at V + k n; w = V_kk. X: this
// launch's exchange words, Y: those of the launch before, which had kprev vectors and gprev blocks.
// out (host or device, kk + 2 doubles) receives the coefficients V_k . w of both passes added, the
// squared norm of what is left of w before it is scaled to unit length (to zero if that norm is zero
// or not a number), and the status: left alone, or 1 when a wait gave up after `lim` polls.
template <typename VT>
__global__ void __launch_bounds__(OG_THREADS, 1)
    ortho_kernel(VT* V, int64_t n, int kk, double* X, double* Y, int kprev, int gprev, uint32_t lim, double* out) {
  using Q = OgQuad<VT>;
  using V4 = typename Q::V4;
  __shared__ double sh[512];       // warps' sums (parts x vectors)
  __shared__ double hs[2][OG_MAX];
  __shared__ VT cs[OG_MAX];
  __shared__ V4 red[OG_THREADS];
  __shared__ double s_norm, s_scale;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int G = gridDim.x, c = blockIdx.x;
  const int64_t n4 = n >> 2;
  const int64_t q0 = n4 * c / G, q1 = n4 * (c + 1) / G;
  const int64_t len = q1 - q0;
  const V4* B = reinterpret_cast<const V4*>(V);
  V4* w = reinterpret_cast<V4*>(V + (int64_t)kk * n);
  bool ok = true;
  // ok of every thread of the block; a wait that gave up ends the kernel (the other blocks' waits
  // give up too)
  auto all_ok = [&]() {
    if (__syncthreads_and(ok)) return true;
    if (tid == 0) out[kk + 1] = 1.0;
    return false;
  };
  {
    const double unset = __longlong_as_double((long long)OG_UNSET);
    for (int64_t i = (int64_t)c * OG_THREADS + tid; i < (int64_t)kprev * gprev; i += (int64_t)G * OG_THREADS) {
      Y[OG_P + i] = unset;
      Y[OG_P + (int64_t)OG_MAX * OG_BLOCKS + i] = unset;
    }
    if (c == G - 1) {
      for (int i = tid; i < gprev; i += OG_THREADS) Y[OG_N + i] = unset;
      for (int i = tid; i < kprev; i += OG_THREADS) Y[OG_H + i] = Y[OG_H + OG_MAX + i] = unset;
    }
  }
  for (int pass = 0; pass < 2; ++pass) {
    double* P = X + OG_P + pass * (int64_t)OG_MAX * OG_BLOCKS;
    double* H = X + OG_H + pass * OG_MAX;
    // this block's shares of the dot products: a warp takes eight vectors over a part of the rows
    {
      // (whole warps of quads: every part costs an FP64 addition per vector)
      const int groups = (kk + OG_K - 1) / OG_K, units = (int)((len + 31) / 32);
      const int most = groups < OG_WARPS ? OG_WARPS / groups : 1, parts = units < 1 ? 1 : (units < most ? units : most);
      for (int t = warp; t < groups * parts; t += OG_WARPS) {
        const int k0 = OG_K * (t % groups), part = t / groups;
        const int64_t a = q0 + 32 * ((int64_t)units * part / parts);
        const int64_t b = part + 1 == parts ? q1 : q0 + 32 * ((int64_t)units * (part + 1) / parts);
        typename Q::Acc acc[OG_K];
        for (int64_t i = a + lane; i < b; i += 32) {
          const V4 wv = w[i];
          V4 vv[OG_K];
#pragma unroll
          for (int k = 0; k < OG_K; ++k)
            if (k0 + k < kk) vv[k] = B[(int64_t)(k0 + k) * n4 + i];
#pragma unroll
          for (int k = 0; k < OG_K; ++k)
            if (k0 + k < kk) acc[k].add(vv[k], wv);
        }
        VT v[OG_K];
#pragma unroll
        for (int k = 0; k < OG_K; ++k) v[k] = acc[k].value();
        // reduce-scatter: lane ends with vector 4 b16 + 2 b8 + b4 of the eight (bits of the lane)
#pragma unroll
        for (int m = OG_K / 2, o = 16; m > 0; m >>= 1, o >>= 1) {
          const bool up = lane & o;
#pragma unroll
          for (int k = 0; k < m; ++k) {
            const VT send = up ? v[k] : v[k + m];
            v[k] = (up ? v[k + m] : v[k]) + __shfl_xor_sync(0xffffffffu, send, o);
          }
        }
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
        if ((lane & 3) == 0) sh[part * groups * OG_K + k0 + (lane >> 2)] = (double)v[0];
      }
      __syncthreads();
      for (int k = tid; k < kk; k += OG_THREADS) {
        double s = 0.0;
        for (int part = 0; part < parts; ++part) s += sh[part * groups * OG_K + k];
        og_put(P + (int64_t)k * G + c, s);
      }
    }
    // vector k is summed over the blocks by block k mod G, its sum taken by all
    for (int k = c + G * warp; k < kk; k += G * OG_WARPS) {
      double s = 0.0;
      for (int b = lane; b < G; b += 32) s += og_get(P + (int64_t)k * G + b, lim, ok);
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (lane == 0) og_put(H + k, s);
    }
    for (int k = tid; k < kk; k += OG_THREADS) {
      const double x = og_get(H + k, lim, ok);
      hs[pass][k] = x;
      cs[k] = (VT)-x;
    }
    if (!all_ok()) return;
    // w -= V h on this block's rows; where the rows are fewer than the threads, several threads
    // share a quad's vectors
    typename Q::Acc nrm;
    const int ks = len >= OG_THREADS || len == 0 ? 1 : (int)(OG_THREADS / len < 16 ? OG_THREADS / len : 16);
    auto combine = [&](int64_t i, int ka, int kb, V4 s) {
      int k = ka;
      for (; k + OG_K <= kb; k += OG_K) {
        V4 vv[OG_K];
#pragma unroll
        for (int t = 0; t < OG_K; ++t) vv[t] = B[(int64_t)(k + t) * n4 + i];
#pragma unroll
        for (int t = 0; t < OG_K; ++t) Q::fma4(s, cs[k + t], vv[t]);
      }
      for (; k < kb; ++k) Q::fma4(s, cs[k], B[(int64_t)k * n4 + i]);
      return s;
    };
    if (ks == 1) {
      for (int64_t i = q0 + tid; i < q1; i += OG_THREADS) {
        const V4 s = combine(i, 0, kk, w[i]);
        w[i] = s;
        nrm.add(s, s);
      }
    } else {
      const int m = (int)len, part = tid / m, qi = tid - part * m;
      if (part < ks) red[tid] = combine(q0 + qi, kk * part / ks, kk * (part + 1) / ks, part == 0 ? w[q0 + qi] : Q::zero());
      __syncthreads();
      if (tid < m) {
        V4 s = red[tid];
        for (int p = 1; p < ks; ++p) Q::fma4(s, VT(1), red[p * m + tid]);
        w[q0 + tid] = s;
        nrm.add(s, s);
      }
    }
    __syncthreads();  // the next pass reads other threads' rows
    if (pass == 1) {  // only the warps that hold rows take part
      const int rows_t = ks == 1 ? OG_THREADS : (int)len, nw = (rows_t + 31) / 32;
      if (warp < nw) {
        VT v = nrm.value();
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) sh[warp] = (double)v;
      }
      __syncthreads();
      if (warp == 0) {
        double s = lane < nw ? sh[lane] : 0.0;
        for (int o = 8; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) og_put(X + OG_N + c, s);
      }
    }
  }
  if (warp == 0) {  // every block forms the same norm
    double s = 0.0;
    for (int b = lane; b < G; b += 32) s += og_get(X + OG_N + b, lim, ok);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      s_norm = s;
      s_scale = s > 0.0 ? og_rsqrt(s) : 0.0;
    }
  }
  if (!all_ok()) return;
  const double nn = s_norm, sc = s_scale;
  for (int64_t i = q0 + tid; i < q1; i += OG_THREADS) {
    V4 s = w[i];
    Q::scale4(s, sc);
    w[i] = s;
  }
  if (c == 0) {
    for (int k = tid; k < kk; k += OG_THREADS) out[k] = hs[0][k] + hs[1][k];
    if (tid == 0) out[kk] = nn;
  }
}

}  // namespace vms
