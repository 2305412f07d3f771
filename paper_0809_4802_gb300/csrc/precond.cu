// Block ILU(0) preconditioner of the condensed system (Section 6: Krylov solves with the solver
// library's default preconditioner, which on one process is an incomplete LU factorisation that
// keeps the sparsity pattern of the matrix).
//
// The matrix is viewed as 4x4 node blocks in natural node order. With no fill, the factorisation
// of block row i is, for each lower block k < i in increasing order,
//   L_ik = A_ik U_kk^-1,   A_ij -= L_ik U_kj   for every block j > k present in both rows,
// after which U_ii = A_ii and its inverse is kept for the backward sweep.
//
// GPU mapping of the factorisation: one CTA owns one node row at a time and claims rows from a counter in
// the order of their dependency levels, so a row only ever waits for rows claimed earlier, by CTAs that
// are already running. A row publishes itself by writing its epoch into a flag with release semantics;
// dependants poll the flag with acquire loads (bounded: after Ilu::spin_limit polls the kernel
// records a timeout and returns), and read data published in the same launch through L2
// (ld.global.cg), never through L1. The triangular sweeps read the finished factor from per-row
// records in their own layout and claim chunks of grid-line segments per CTA (ilu_sweep_kernel).
#include <algorithm>
#include <type_traits>
#include <vector>

#include "precond.h"
#include "solver.h"

namespace vms {

namespace {

constexpr int FACTOR_CTAS = 6, FACTOR_WIDE_CTAS = 24;  // of the factorisation, per SM: four warps a row; one
constexpr unsigned FULL = 0xffffffffu;

__device__ __forceinline__ uint32_t ld_acquire(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release(uint32_t* p, uint32_t v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Wait until *f == epoch. Gives up (returns false) when another warp has recorded an error or
// after `lim` polls (Ilu::spin_limit), recording a timeout.
__device__ __forceinline__ bool wait_ready(const uint32_t* f, uint32_t epoch, int* err, uint32_t lim) {
  if (ld_acquire(f) == epoch) return true;
  for (uint32_t it = 1; it <= lim; ++it) {
    __nanosleep(32);
    if (ld_acquire(f) == epoch) return true;
    if ((it & 1023u) == 0 && *(volatile int*)err != 0) return false;
  }
  atomicCAS(err, 0, ILU_ERR_TIMEOUT);
  return false;
}

// ---------------------------------------------------------------------------------------------
// factorisation: one CTA per node row; the row is eliminated in shared memory
//
// What bounds it where levels are narrow: the chain of rows (224 levels on a lattice of 33^3 nodes, about 160
// rows wide), and in a row the FP64 instructions of its block products, 64 cycles each on one warp: 34 for a lower block of 17
// pairs, and up to three lower blocks were finished only one level before. So a row's pairs are shared
// by four warps, one per FP64 unit, eight pairs a step; what is known beforehand (neighbours, row starts,
// pairs) is read before the first wait; U_kk^-1 and the blocks of row k are read as soon as row k is
// published, while the products of the block before are still under way; and a lower block costs one
// barrier: every warp forms L_ik for itself, the row keeps A_ik. Rows are claimed by level: in natural order
// the rows that can run lie planes apart, and the resident CTAs would hold half a plane (6.7 ms on 33^3 nodes).
// Where a level has more rows than the GPU has SMs (factor_wide), the rows in flight bound it instead: one warp
// per row, so that an SM holds 24 rows, not 6. Measured in ms, one warp per row in natural order; four warps; one warp
// now: lattices of 13^3 nodes (26 rows a level) 0.91, 0.46, 0.55; 25^3 (93) 1.96, 1.02, 1.19; 33^3 (160) 4.05, 1.66, 1.68;
// 45^3 (296) 11.6, 3.3, 2.8; 91^3 (1,183) 120, 24.2, 14.7; 40^3 nodes of a tetrahedral mesh 3.99, 1.34, 0.99; in random
// node order, whose levels are few, 25^3 0.45, 0.53, 0.40; 45^3 1.71, 3.06, 1.78; 91^3 15.9, 26.2, 14.8.
// ---------------------------------------------------------------------------------------------
template <typename T, int FW>
__global__ void __launch_bounds__(FW * 32, FW == 1 ? FACTOR_WIDE_CTAS : FACTOR_CTAS)
    ilu_factor_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                      const T* __restrict__ A, T* F, T* Dinv, const int32_t* __restrict__ dpos,
                      const int32_t* __restrict__ lptr, const int32_t* __restrict__ pptr,
                      const uint16_t* __restrict__ pairs, const int32_t* __restrict__ order, int64_t n_nodes, uint32_t* flags,
                      uint32_t epoch, unsigned long long* ticket, unsigned long long base, int* err,
                      uint32_t lim) {
  constexpr int PS = 2 * FW, PMAX = FW == 1 ? 4 : (ILU_MAX_DEG + PS - 1) / PS;  // pairs a step; steps read ahead
  __shared__ T row[ILU_MAX_DEG * 16];
  // FW > 1: L_ik as each warp reads it and as the row is stored (other warps may still need A_ik); 1: in A_ik's place
  __shared__ T lrows[FW == 1 ? 1 : ILU_MAX_DEG * 16], lw[FW][FW == 1 ? 1 : 16];
  T* const lrow = FW == 1 ? row : lrows;
  __shared__ int32_t s_k[ILU_MAX_DEG], s_pp[ILU_MAX_DEG + 1], s_rk[ILU_MAX_DEG][4];
  __shared__ uint16_t s_pairs[ILU_MAX_DEG * ILU_MAX_DEG];
  __shared__ int64_t s_row;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int q = (lane >> 2) & 3, c = lane & 3, half = lane >> 4;
  for (;;) {
    // the next row of this launch. A claim below the launch's base (the counter was disturbed by a launch that
    // stopped early) records an error and ends the block, so that no row outside [0, n_nodes) is ever formed.
    if (tid == 0) {
      const unsigned long long t = atomicAdd(ticket, 1ull);
      if (t < base) atomicCAS(err, 0, ILU_ERR_TIMEOUT);
      s_row = t >= base && t - base < (unsigned long long)n_nodes ? (int64_t)(t - base) : -1;
    }
    __syncthreads();
    if (s_row < 0) return;
    const int64_t i = order[s_row];
    const int32_t r0 = rowptr[4 * i];
    const int deg = (rowptr[4 * i + 1] - r0) >> 2, dp = dpos[i];
    const int32_t l0 = lptr[i], p0 = pptr[l0], np = pptr[l0 + dp] - p0;
    // row i into shared memory, block-major: row[16 kk + 4 q + c] = A(4i+q, 4 adj_kk + c)
    for (int e = tid; e < deg * 16; e += FW * 32)
      row[e] = A[rowptr[4 * i + ((e >> 2) & 3)] + 4 * (e >> 4) + (e & 3)];
    for (int kk = tid; kk <= dp; kk += FW * 32) {
      s_pp[kk] = pptr[l0 + kk] - p0;
      if (kk < dp) {
        const int32_t k = colidx[r0 + 4 * kk] >> 2;
        s_k[kk] = k;
        for (int m = 0; m < 4; ++m) s_rk[kk][m] = rowptr[4 * (int64_t)k + m];
      }
    }
    for (int p = tid; p < np; p += FW * 32) s_pairs[p] = pairs[p0 + p];
    __syncthreads();
    for (int kk = 0; kk < dp; ++kk) {
      const int64_t k = s_k[kk];
      int ok = 1;
      if (lane == 0) ok = wait_ready(flags + k, epoch, err, lim);
      ok = __shfl_sync(FULL, ok, 0);
      // U_kk^-1 (lane: column c) and the blocks U_kj of this half-warp's pairs (lane: column c)
      T d[4], u[PMAX][4];
      int jj[PMAX];
      if (ok) {
        for (int m = 0; m < 4; ++m) d[m] = __ldcg(Dinv + 16 * k + 4 * m + c);
#pragma unroll
        for (int s = 0; s < PMAX; ++s) {
          const int p = s_pp[kk] + PS * s + 2 * warp + half;
          jj[s] = -1;
          if (p < s_pp[kk + 1]) {
            const uint32_t pr = s_pairs[p];
            jj[s] = pr & 255;
            for (int m = 0; m < 4; ++m) u[s][m] = __ldcg(F + s_rk[kk][m] + 4 * (int)(pr >> 8) + c);
          }
        }
      }
      // the products of the lower blocks before are done
      if (__syncthreads_or(!ok)) return;
      // L_ik = A_ik U_kk^-1 (lane: entry (q, c), both halves alike)
      T l = T(0);
      for (int m = 0; m < 4; ++m) l += row[16 * kk + 4 * q + m] * d[m];
      if (FW == 1) __syncwarp();
      if (half == 0) {
        if (FW > 1) lw[warp][lane] = l;
        if (warp == 0) lrow[16 * kk + lane] = l;
      }
      __syncwarp();
      const T* L = FW == 1 ? row + 16 * kk : lw[warp];
      // A_ij -= L_ik U_kj (the products are subtracted one by one, so that each is a fused multiply-add)
#pragma unroll
      for (int s = 0; s < PMAX; ++s)
        if (jj[s] >= 0) {
          T v = row[16 * jj[s] + 4 * q + c];
          for (int m = 0; m < 4; ++m) v -= L[4 * q + m] * u[s][m];
          row[16 * jj[s] + 4 * q + c] = v;
        }
      if constexpr (PS * PMAX < ILU_MAX_DEG)
        for (int p = s_pp[kk] + PS * PMAX + 2 * warp + half; p < s_pp[kk + 1]; p += PS) {
          const uint32_t pr = s_pairs[p];
          const int j = pr & 255;
          T v = row[16 * j + 4 * q + c];
          for (int m = 0; m < 4; ++m) v -= L[4 * q + m] * __ldcg(F + s_rk[kk][m] + 4 * (int)(pr >> 8) + c);
          row[16 * j + 4 * q + c] = v;
        }
      __syncwarp();  // L is read before the next block's is written
    }
    __syncthreads();
    if (warp == 0) {
      // U_ii^-1 = adj(U_ii) / det on lanes 0..15 (lane 4r + c forms the cofactor of entry (r, c)); lanes 16..31
      // sum the squares of the rows in the same instructions
      const T* D = row + 16 * dp;
      const int r = q;
      double mnr[3][3];  // the minor: rows other than r, columns other than c
#pragma unroll
      for (int a2 = 0; a2 < 3; ++a2)
#pragma unroll
        for (int b2 = 0; b2 < 3; ++b2)
          mnr[a2][b2] = (double)D[4 * (a2 + (a2 >= r)) + b2 + (b2 >= c)];
      const double m3 = mnr[0][0] * (mnr[1][1] * mnr[2][2] - mnr[1][2] * mnr[2][1]) -
                        mnr[0][1] * (mnr[1][0] * mnr[2][2] - mnr[1][2] * mnr[2][0]) +
                        mnr[0][2] * (mnr[1][0] * mnr[2][1] - mnr[1][1] * mnr[2][0]);
      const double cf = ((r + c) & 1) ? -m3 : m3;
      const double dv = (double)D[lane & 15];
      double dt = dv * (half ? dv : cf);  // lanes 0..3: det by the first row; 16..31: squared row norms
      dt += __shfl_xor_sync(FULL, dt, 1);
      dt += __shfl_xor_sync(FULL, dt, 2);
      const double det = __shfl_sync(FULL, dt, 0);
      // singular unless |det| is a fair fraction of the product of the row norms (Hadamard's
      // bound; independent of the rows' scales), compared squared: det^2 > 1e-28 prod |row|^2
      const double hb2 = __shfl_sync(FULL, dt, 16) * __shfl_sync(FULL, dt, 20) *
                         __shfl_sync(FULL, dt, 24) * __shfl_sync(FULL, dt, 28);
      const bool good = isfinite(det) && hb2 > 0.0 && det * det > 1e-28 * hb2;
      if (!good && lane == 0) atomicCAS(err, 0, ILU_ERR_PIVOT);
      if (lane < 16) Dinv[16 * i + 4 * c + r] = good ? T(cf / det) : T(r == c ? 1.0 : 0.0);
    }
    if (FW == 1 || warp > 0) {
      constexpr int SW = FW == 1 ? 1 : FW - 1;  // warps that store
      for (int e = tid - (FW - SW) * 32; e < deg * 16; e += SW * 32)
        F[rowptr[4 * i + ((e >> 2) & 3)] + 4 * (e >> 4) + (e & 3)] = (e >> 4) < dp ? lrow[e] : row[e];
    }
    __threadfence();
    __syncthreads();
    if (tid == 0) st_release(flags + i, epoch);
  }
}

// ---------------------------------------------------------------------------------------------
// sweeps: y = L^-1 v (rows ascending), z = U^-1 y (rows descending)
//
// What bounds them: the dependency chain. A 27-point lattice of 33^3 nodes has 224 levels (128 steps
// along a line, 64 to the next line, 32 to the next plane on the longest path), while a sweep's
// data, 39 MB of FP32 records, would take 6 us of HBM. So everything off the chain is moved off the
// warp that solves a row: values of earlier chunks are fetched by one warp, records by another, and
// a row is one sum of block products without a test in its way. Measured on 33^3 nodes (jittered
// cavity): FP32 sweep 239 -> 127 us, FP64 524 -> 260 us; 22^3 nodes of a tetrahedral mesh 57 -> 46
// and 160 -> 65 us; in random node order, where rows in flight bound them, 33^3 nodes 61 -> 70 and 184 -> 136 us.
// What is left: a row takes about 0.2 us (FP32; FP64 11 instructions of 64 cycles each on its partition's FP64
// unit, about 0.5 us), and a value from another chunk about 0.9 us from its publication to the slot. Four segments a chunk: eight are alike in FP32 and slower in FP64
// (315 us: the SM's FP64 unit is shared), and a second fetching warp changes nothing.
// ---------------------------------------------------------------------------------------------

// A sweep publishes a node's four values with single stores into buffers that hold an all-ones bit
// pattern before the sweep (a NaN that arithmetic never produces): a global one, read through L2,
// and the chunk's slots in shared memory. Every word is written once, so a node is ready once none
// of its words holds the pattern: no flag, no fence, and the read that finds it ready has its values.
constexpr uint32_t UNSET32 = 0xffffffffu;

// One attempt to read a node's values from L2 (`p`) or from a slot (`s`, a shared-memory address).
// `m` is raised to the largest of the words (FP64: of the words' halves combined), which is all
// ones while one of them is not written.
__device__ __forceinline__ void words_max(uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t& m) {
  m = max(max(max(a, b), max(c, d)), m);
}
__device__ __forceinline__ void ld_relaxed4(const float* p, float x[4], uint32_t& m) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  const uint32_t w[4] = {(uint32_t)a, (uint32_t)(a >> 32), (uint32_t)b, (uint32_t)(b >> 32)};
  for (int k = 0; k < 4; ++k) x[k] = __uint_as_float(w[k]);
  words_max(w[0], w[1], w[2], w[3], m);
}
__device__ __forceinline__ void pairs_max(unsigned long long a, unsigned long long b, unsigned long long c,
                                          unsigned long long d, double x[4], uint32_t& m) {
  x[0] = __longlong_as_double((long long)a); x[1] = __longlong_as_double((long long)b);
  x[2] = __longlong_as_double((long long)c); x[3] = __longlong_as_double((long long)d);
  // both halves of a word are all ones only while it is not written
  words_max((uint32_t)a & (uint32_t)(a >> 32), (uint32_t)b & (uint32_t)(b >> 32), (uint32_t)c & (uint32_t)(c >> 32),
            (uint32_t)d & (uint32_t)(d >> 32), m);
}
__device__ __forceinline__ void ld_relaxed4(const double* p, double x[4], uint32_t& m) {
  unsigned long long a, b, c, d;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(c), "=l"(d) : "l"(p + 2) : "memory");
  pairs_max(a, b, c, d, x, m);
}
__device__ __forceinline__ void ld_slot(unsigned s, float x[4], uint32_t& m) {
  uint32_t a, b, c, d;
  asm volatile("ld.volatile.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "r"(s) : "memory");
  x[0] = __uint_as_float(a); x[1] = __uint_as_float(b);
  x[2] = __uint_as_float(c); x[3] = __uint_as_float(d);
  words_max(a, b, c, d, m);
}
__device__ __forceinline__ void ld_slot(unsigned s, double x[4], uint32_t& m) {
  unsigned long long a, b, c, d;
  asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(s) : "memory");
  asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];" : "=l"(c), "=l"(d) : "r"(s + 16) : "memory");
  pairs_max(a, b, c, d, x, m);
}
__device__ __forceinline__ void put_slot(unsigned s, const float x[4]) {
  asm volatile("st.volatile.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(s), "f"(x[0]), "f"(x[1]), "f"(x[2]), "f"(x[3]) : "memory");
}
__device__ __forceinline__ void put_slot(unsigned s, const double x[4]) {
  asm volatile("st.volatile.shared.v2.f64 [%0], {%1, %2};" ::"r"(s), "d"(x[0]), "d"(x[1]) : "memory");
  asm volatile("st.volatile.shared.v2.f64 [%0], {%1, %2};" ::"r"(s + 16), "d"(x[2]), "d"(x[3]) : "memory");
}
// Publish a node's four values with one 16-byte store per lane (generic addresses; `dst` is the
// lane's own): FP32 lane 0 writes the shared slot, lane 1 the global publication, lane 2 the plain
// vector; FP64 two lanes each.
__device__ __forceinline__ void publish(int lane, const float r[4], unsigned long long dst) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b64 a, b;\n\tsetp.lt.s32 p, %0, 3;\n\tmov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "@p st.relaxed.gpu.v2.b64 [%1], {a, b};\n\t}"
      ::"r"(lane), "l"(dst), "f"(r[0]), "f"(r[1]), "f"(r[2]), "f"(r[3]) : "memory");
}
__device__ __forceinline__ void publish(int lane, const double r[4], unsigned long long dst) {
  const double a = lane & 1 ? r[2] : r[0], b = lane & 1 ? r[3] : r[1];
  asm volatile("{\n\t.reg .pred p;\n\tsetp.lt.s32 p, %0, 6;\n\t@p st.relaxed.gpu.v2.f64 [%1], {%2, %3};\n\t}"
               ::"r"(lane), "l"(dst), "d"(a), "d"(b) : "memory");
}
// Whether one of four values is not a number (FP32: or two infinities cancel).
__device__ __forceinline__ bool any_nan(const float r[4]) {
  const float s = (r[0] + r[1]) + (r[2] + r[3]);
  return s != s;
}
__device__ __forceinline__ bool any_nan(const double r[4]) {
  uint32_t m = 0;
  for (int k = 0; k < 4; ++k) m = max(m, (uint32_t)__double2hiint(r[k]) & 0x7fffffffu);
  return m >= 0x7ff80000u;
}
__device__ __forceinline__ void ld_shared4(unsigned s, int, float o[4]) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(o[0]), "=f"(o[1]), "=f"(o[2]), "=f"(o[3]) : "r"(s));
}
__device__ __forceinline__ void ld_shared4(unsigned s, int half, double o[4]) {
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(o[0]), "=d"(o[1]) : "r"(s));
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(o[2]), "=d"(o[3]) : "r"(s + half));
}
__device__ __forceinline__ void ld_shared1(unsigned s, float& o) { asm volatile("ld.shared.f32 %0, [%1];" : "=f"(o) : "r"(s)); }
__device__ __forceinline__ void ld_shared1(unsigned s, double& o) { asm volatile("ld.shared.f64 %0, [%1];" : "=d"(o) : "r"(s)); }
__device__ __forceinline__ void ld_shared1(unsigned s, unsigned& o) { asm volatile("ld.shared.u32 %0, [%1];" : "=r"(o) : "r"(s)); }

// Bulk copies global -> shared, completed on an mbarrier.
__device__ __forceinline__ void mbar_init(unsigned bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_copy(unsigned dst, const void* src, unsigned bytes, unsigned bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(unsigned bar, unsigned parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_test(unsigned bar, unsigned parity) {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// A bulk copy completes by hardware; the limit only keeps the wait finite.
__device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity) {
  for (uint32_t it = 0; it < (1u << 22); ++it)
    if (mbar_try(bar, parity)) return true;
  return false;
}

// A row of the factor as a sweep reads it (Ilu::rec): 8 NP blocks (4 x 4), then the byte offsets of
// their values in shared memory (8 NP words). Row q of block 8 p + g belongs to lane 8 q + g in pass
// p: a pass holds its lanes' 16-byte pieces side by side (FP64: first halves, then second halves),
// so that a warp's loads meet no bank twice. The forward record holds -L_ik, the last
// place kept for the row before in the segment; the backward one -U_ii^-1 U_ij, the last place the
// same, the one before it U_ii^-1, whose value is the right-hand side. A row is then one sum of
// block products in either sweep (the forward one adds its right-hand side). Places without a
// block hold zeros and point to slot 0, which holds zeros.
template <typename T, int NP> constexpr int sweep_rec_bytes() { return 8 * NP * (16 * (int)sizeof(T) + 4); }
// Rows of a bulk copy and copies in flight per warp; one each where segments are SHORT (sweep_short). (8 rows: 190 us
// instead of 213 on 49^3 nodes, but 331 instead of 237 on lines of 151 nodes, and fewer blocks fit an SM.)
template <int NP, bool SHORT> constexpr int sweep_rb() { return SHORT ? 1 : (NP <= 2 ? 4 : 2); }
template <bool SHORT> constexpr int sweep_st() { return SHORT ? 1 : 3; }
// shared memory of a sweep: value slots (zeros, the chunk's rows, their far neighbours), the rings
// of row records and right-hand sides, the barriers
template <typename T, int NP, bool SHORT>
constexpr size_t sweep_smem_bytes(int warps, int slots) {
  return (size_t)slots * 4 * sizeof(T) +
         (size_t)warps * sweep_st<SHORT>() * (sweep_rb<NP, SHORT>() * (sweep_rec_bytes<T, NP>() + 4 * sizeof(T)) + 16);
}

// a chunk of one segment may have any number of far neighbours: 64 rows of at most 31
static_assert(sweep_smem_bytes<double, 5, false>(ILU_CHUNK, 1 + ILU_SEG_MAX * ILU_MAX_DEG) + 1024 <= (227 << 10) &&
                  ILU_CHUNK * ILU_SEG_MAX + ILU_FAR_MAX < ILU_SEG_MAX * ILU_MAX_DEG,
              "the largest chunk's shared memory");

// The records of one sweep from the factor (CSR layout, FP64): one thread per 16-byte piece.
template <typename T, bool LOWER, int NP>
__global__ void sweep_pack_kernel(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ dpos,
                                  const uint8_t* __restrict__ inl, const int32_t* __restrict__ at,
                                  const double* __restrict__ F, const double* __restrict__ Dinv, int64_t n_nodes,
                                  unsigned char* __restrict__ rec) {
  constexpr int PB = (int)sizeof(T);            // 16-byte pieces of a block
  constexpr int EP = 16 / (int)sizeof(T);       // values of a piece
  constexpr int PIECES = 8 * NP * PB + 2 * NP;  // pieces of a record
  for (int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; w < n_nodes * PIECES;
       w += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = w / PIECES;
    const int pc = (int)(w - i * PIECES);
    const int l = pc & 31, half = (pc >> 5) % (PB / 4), blk = 8 * ((pc >> 5) / (PB / 4)) + (l & 7);
    const int32_t rp = rowptr[4 * i];
    const int deg = (rowptr[4 * i + 1] - rp) >> 2, dp = dpos[i];
    const int has = inl[i] >> (LOWER ? 0 : 1) & 1;          // the row before in the segment is a neighbour
    const int own = (LOWER ? dp : deg - 1 - dp) - has;      // this row's other blocks
    if (pc < 8 * NP * PB) {
      int kk = -1;
      if (blk < own) kk = LOWER ? blk : deg - 1 - blk;
      else if (blk == 8 * NP - 1 && has) kk = LOWER ? dp - 1 : dp + 1;
      const int r = l >> 3, c0 = half * EP;
      T o[EP];
      for (int t = 0; t < EP; ++t) {
        const int c = c0 + t;
        double x = 0.0;
        if (!LOWER && blk == 8 * NP - 2) {
          x = Dinv[16 * i + 4 * r + c];
        } else if (kk >= 0) {
          const double* f = F + rp + 4 * kk + c;
          if (LOWER) x = -f[r * 4 * deg];
          else
            for (int m = 0; m < 4; ++m) x -= Dinv[16 * i + 4 * r + m] * f[m * 4 * deg];
        }
        o[t] = T(x);
      }
      T* dst = reinterpret_cast<T*>(rec + w * 16);
      for (int t = 0; t < EP; ++t) dst[t] = o[t];
    } else {
      int32_t* dst = reinterpret_cast<int32_t*>(rec + w * 16);
      const int k0 = (pc - 8 * NP * PB) * 4;
      for (int t = 0; t < 4; ++t) {
        const int k = k0 + t;
        dst[t] = k < own ? 4 * (int)sizeof(T) * at[(rp >> 4) + (LOWER ? k : deg - 1 - k)] : 0;
      }
    }
  }
}

// T: element type of the factor.
// Rows [n0, n0 + n_rows); `v` and `out` are compact (index i - n0), the publication buffers `pub`
// (written) and `clr` (the other sweep's, set to all ones for its next run) are indexed by node
// over the whole mesh. NP: passes of eight blocks (a record's 8 NP places).
//
// The rows are cut into segments (seg[s] .. seg[s+1]): maximal runs of consecutive nodes in which
// every node is coupled to the one before it (a grid line in a lattice numbering), at most
// ILU_SEG_MAX long, and the segments into chunks of at most W (Ilu::chunk). A CTA claims the next
// chunk in sweep order and each of its first W warps does one segment's rows in order: lane
// 8 q + g holds row q of the blocks g, g + 8, ..., and reads every neighbour's value from the
// chunk's slots in shared memory once it no longer holds the all-ones pattern. The rows of the
// chunk write theirs there, and the next FW warps fetch the neighbours in earlier chunks (the
// chunk's far list) from the L2 publication as they appear, so that the L2 round trips run beside
// the rows instead of inside them. The last warp streams the row records and right-hand sides into
// a ring per compute warp with bulk copies. Chunks are claimed in order by running CTAs, so every
// wait is for work that is already in progress. The blocks per SM of the launch bounds leave the variants their
// registers without spills (44 to 168 a thread; FP64 with 40 places and SHORT spills 84 bytes); left to itself the
// compiler spilled up to 68 bytes in the row loop.
template <typename T, bool LOWER, int NP, int W, int FW, bool SHORT>
__global__ void __launch_bounds__((W + FW + 1) * 32, sizeof(T) == 4 ? (SHORT ? 5 : NP <= 3 ? 4 : 3) : (SHORT ? 3 : 2))
    ilu_sweep_kernel(const unsigned char* __restrict__ rec, const int32_t* __restrict__ seg,
                     const int32_t* __restrict__ chunk, const int32_t* __restrict__ farptr,
                     const int32_t* __restrict__ far, int64_t c0, int64_t n_chunks, const T* __restrict__ v,
                     T* pub, uint4* __restrict__ clr, T* __restrict__ out, int n0, int n_rows, int slots,
                     unsigned long long* ticket, unsigned long long base, int* err, uint32_t lim) {
  constexpr int ST = sweep_st<SHORT>(), RB = sweep_rb<NP, SHORT>(), VB = 4 * (int)sizeof(T);  // VB: bytes of a node's values
  constexpr int RS = sweep_rec_bytes<T, NP>(), STAGE = RB * (RS + VB);
  constexpr int dir = LOWER ? 1 : -1;
  __shared__ int64_t s_chunk;
  extern __shared__ __align__(16) unsigned char smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int q = lane >> 3, g = lane & 7;
  const int n1 = n0 + n_rows;
  const unsigned sx = (unsigned)__cvta_generic_to_shared(smem);
  const unsigned rings = sx + slots * VB, bars = rings + W * ST * STAGE;
  // stage n of compute warp w: barrier `full` (its copies have landed), then `empty` (it was read)
  auto full = [&](int w, unsigned n) { return bars + (w * ST + n % ST) * 16; };
  auto empty = [&](int w, unsigned n) { return bars + (w * ST + n % ST) * 16 + 8; };
  if (threadIdx.x < W * ST * 2) mbar_init(bars + 8 * threadIdx.x);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  unsigned copies = 0;  // compute warp: copies read; producer lane w: copies started for warp w
  for (;;) {
    if (threadIdx.x == 0) {
      int64_t c = -1;
      if (*(volatile int*)err == 0) {
        const unsigned long long t = atomicAdd(ticket, 1ull);
        if (t < base) atomicCAS(err, 0, ILU_ERR_TIMEOUT);  // the counter was disturbed
        else if (t - base < (unsigned long long)n_chunks)
          c = LOWER ? c0 + (int64_t)(t - base) : c0 + n_chunks - 1 - (int64_t)(t - base);
      }
      s_chunk = c;
    }
    for (int l = threadIdx.x; l < slots * VB / 16; l += (W + FW + 1) * 32) {
      const uint32_t z = l < VB / 16 ? 0u : UNSET32;  // slot 0: zeros
      reinterpret_cast<uint4*>(smem)[l] = make_uint4(z, z, z, z);
    }
    __syncthreads();
    const int64_t c = s_chunk;
    if (c < 0) {
      // no copy may land after the block has ended: a warp that gave up has left some unread
      if (warp == W + FW && lane < W)
        for (unsigned n = copies < ST ? 0 : copies - ST; n < copies; ++n) mbar_wait(full(lane, n), (n / ST) & 1);
      return;
    }
    const int slo = chunk[c], shi = chunk[c + 1];  // its segments
    const int a = seg[slo];                        // its first node (slot 1)
    // rows r = 0 .. len - 1 of a segment in sweep order are the nodes first + r * dir
    auto segment = [&](int w, int& first) {
      const int s = LOWER ? slo + w : shi - 1 - w;
      int lo = seg[s], hi = seg[s + 1];
      lo = lo > n0 ? lo : n0;
      hi = hi < n1 ? hi : n1;
      first = LOWER ? lo : hi - 1;
      return hi > lo ? hi - lo : 0;
    };
    if (warp == W + FW) {
      // producer: lane w streams the segment of compute warp w, RB rows a copy
      int first = 0, left = lane < W && slo + lane < shi ? segment(lane, first) : 0;
      uint32_t idle = 0;
      bool stop = false;
      while (!__all_sync(FULL, left == 0)) {
        bool sent = false;
        if (left > 0 && (copies < ST || mbar_test(empty(lane, copies), (copies / ST - 1) & 1))) {
          const int n = left < RB ? left : RB;
          const int64_t i0 = LOWER ? first : first - n + 1;  // its lowest node
          const unsigned bar = full(lane, copies), dst = rings + (lane * ST + copies % ST) * STAGE;
          mbar_expect(bar, n * (RS + VB));
          bulk_copy(dst, rec + i0 * RS, n * RS, bar);
          bulk_copy(dst + RB * RS, v + 4 * (i0 - n0), n * VB, bar);
          ++copies;
          first += dir * n;
          left -= n;
          sent = true;
        }
        idle = __any_sync(FULL, sent) ? 0 : idle + 1;
        if (idle > 16u) __nanosleep(40);
        // give up after lim polls without progress or once another warp has recorded an error
        // (uniform decisions)
        if (idle > lim || ((idle & 63u) == 63u && __any_sync(FULL, *(volatile int*)err != 0))) {
          stop = true;
          break;
        }
      }
      if (stop && lane == 0) atomicCAS(err, 0, ILU_ERR_TIMEOUT);
    } else if (warp >= W) {
      // far neighbours: lane takes entries of the list in order, each until it is published
      const int b = seg[shi], fb = farptr[c], nf = farptr[c + 1] - fb;
      for (int l = (a > n0 ? a : n0) * (VB / 16) + (warp - W) * 32 + lane; l < (b < n1 ? b : n1) * (VB / 16); l += FW * 32)
        clr[l] = make_uint4(UNSET32, UNSET32, UNSET32, UNSET32);
      int e = (warp - W) * 32 + lane;
      int node = e < nf ? far[fb + e] : -1;
      int rest = 0;  // this warp's entries not delivered yet
      for (int k = (warp - W) * 32; k < nf; k += FW * 32) rest += nf - k < 32 ? nf - k : 32;
      uint32_t idle = 0;
      while (rest > 0) {
        const int en = e + FW * 32;
        const int next = en < nf ? far[fb + en] : -1;
        bool done = false;
        if (node >= 0) {
          if (node < n0 || node >= n1) {
            done = true;  // another block's node: no row here reads it
          } else {
            T x[4];
            uint32_t m = 0;
            ld_relaxed4(pub + 4 * (int64_t)node, x, m);
            if (m != UNSET32) {
              put_slot(sx + (1 + b - a + e) * VB, x);
              done = true;
            }
          }
        }
        if (done) {
          e = en;
          node = next;
        }
        const unsigned dm = __ballot_sync(FULL, done);
        rest -= __popc(dm);
        idle = dm ? 0 : idle + 1;
        // give up after lim / 8 polls (of an L2 round trip) without progress or once another warp
        // has recorded an error (uniform decisions)
        if (idle > lim >> 3 || ((idle & 255u) == 255u && __any_sync(FULL, *(volatile int*)err != 0))) {
          if (lane == 0) atomicCAS(err, 0, ILU_ERR_TIMEOUT);
          break;
        }
      }
    } else if (slo + warp < shi) {
      int first;
      const int len = segment(warp, first);
      // this lane's store address (publish); the step from row to row is dir * VB for all three
      unsigned long long dst;
      {
        const int role = lane / (VB / 16), half = 16 * (lane % (VB / 16));
        if (role == 0) dst = (unsigned long long)(smem + (1 + first - a) * VB) + half;
        else if (role == 1) dst = (unsigned long long)(pub + 4 * (int64_t)first) + half;
        else dst = (unsigned long long)(out + 4 * (int64_t)(first - n0)) + half;
      }
      T res[4] = {T(0), T(0), T(0), T(0)};  // the row before (every lane holds all four values)
      bool ok = true;
      // Rows are taken without asking whether their neighbours' values are there: one that is not
      // is a NaN and makes the row's result one, which all lanes see alike. Such a row is done again
      // with an explicit wait. Inside a batch (straight-line code for a full one) the next row's
      // record is loaded while the sums of the current row go through the shuffles, and its
      // neighbours' values right after.
      unsigned rc, rv;  // the batch's first record (this lane's pieces) and right-hand side
      unsigned from[RB][NP];
      T f[NP][4], x[NP][4], t = T(0);
      constexpr int RD = LOWER ? RS : -RS, VD = LOWER ? VB : -VB;
      auto record = [&](int rr) {
#pragma unroll
        for (int p = 0; p < NP; ++p) ld_shared4(rc + rr * RD + p * 128 * (int)sizeof(T), 512, f[p]);
        if (LOWER) ld_shared1(rv + rr * VD + q * (int)sizeof(T), t);
      };
      auto values = [&](int rr, uint32_t& um) {
#pragma unroll
        for (int p = 0; p < NP; ++p) ld_slot(from[rr][p], x[p], um);
      };
      auto products = [&]() {  // place 7 of the last pass is the row before
        T s0 = LOWER ? (g == 0 ? t : T(0)) : T(0);
        if constexpr (sizeof(T) == 4) {
          T s1 = T(0);  // two chains: the latency of one FMA chain would show
#pragma unroll
          for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int m = 0; m < 4; ++m) {
              const T xv = p == NP - 1 && g == 7 ? res[m] : x[p][m];
              if (m & 1) s1 += f[p][m] * xv;
              else s0 += f[p][m] * xv;
            }
          s0 += s1;
        } else {
#pragma unroll
          for (int p = 0; p < NP; ++p)
#pragma unroll
            for (int m = 0; m < 4; ++m) s0 += f[p][m] * (p == NP - 1 && g == 7 ? res[m] : x[p][m]);
        }
        return s0;
      };
      auto batch = [&](auto whole, int n) {
#pragma unroll
        for (int rr = 0; rr < RB; ++rr)
          if (whole || rr < n) {
#pragma unroll
            for (int p = 0; p < NP; ++p) {
              unsigned o;
              ld_shared1(rc - 16 * lane + rr * RD + 8 * NP * 16 * (int)sizeof(T) + 32 * p + 4 * g, o);
              from[rr][p] = !LOWER && p == NP - 1 && g == 6 ? rv + rr * VD : sx + o;  // U_ii^-1 times the right-hand side
            }
          }
        uint32_t um = 0;
        record(0);
        values(0, um);
#pragma unroll
        for (int rr = 0; rr < RB; ++rr) {
          if (!whole && rr >= n) break;
          const bool more = rr + 1 < RB && (whole || rr + 1 < n);
          T sum = products();
          if (more) record(rr + 1);
          sum += __shfl_xor_sync(FULL, sum, 4);
          sum += __shfl_xor_sync(FULL, sum, 2);
          sum += __shfl_xor_sync(FULL, sum, 1);
          T w[4];
#pragma unroll
          for (int m = 0; m < 4; ++m) w[m] = __shfl_sync(FULL, sum, 8 * m);
          if (more) values(rr + 1 < RB ? rr + 1 : 0, um);
          if (__builtin_expect(any_nan(w), 0)) {  // uniform: every lane holds the same values
            record(rr);
            for (uint32_t it = 0;; ++it) {
              um = 0;
              values(rr, um);
              if (__all_sync(FULL, um != UNSET32)) break;
              if (it >= 256u) __nanosleep(20);
              // give up after lim polls or once another warp has recorded an error (uniform decisions)
              if (it >= lim || ((it & 1023u) == 1023u && __any_sync(FULL, *(volatile int*)err != 0))) return false;
            }
            sum = products();
            if (more) record(rr + 1);
            sum += __shfl_xor_sync(FULL, sum, 4);
            sum += __shfl_xor_sync(FULL, sum, 2);
            sum += __shfl_xor_sync(FULL, sum, 1);
#pragma unroll
            for (int m = 0; m < 4; ++m) w[m] = __shfl_sync(FULL, sum, 8 * m);
            if (more) values(rr + 1 < RB ? rr + 1 : 0, um);
          }
#pragma unroll
          for (int m = 0; m < 4; ++m) res[m] = w[m];
          publish(lane, res, dst);
          dst += dir * VB;
        }
        return true;
      };
      // Whether the copy has landed: its producer may have stopped before starting it, which an error tells.
      auto landed = [&](unsigned bar, unsigned parity) {
        for (uint32_t it = 0; !mbar_try(bar, parity); ++it)
          if (it >= lim || ((it & 15u) == 15u && *(volatile int*)err != 0)) return false;
        return true;
      };
      for (int r0 = 0; r0 < len && ok; r0 += RB) {
        const int n = len - r0 < RB ? len - r0 : RB;
        if (!__all_sync(FULL, landed(full(warp, copies), (copies / ST) & 1))) {
          ok = false;
          break;
        }
        const unsigned st = rings + (warp * ST + copies % ST) * STAGE;
        rc = st + (LOWER ? 0 : (n - 1) * RS) + 16 * lane;
        rv = st + RB * RS + (LOWER ? 0 : (n - 1) * VB);
        ok = n == RB ? batch(std::true_type{}, RB) : batch(std::false_type{}, n);
        // every lane has read the stage
        __syncwarp();
        if (lane == 0) mbar_arrive(empty(warp, copies));
        ++copies;
      }
      if (!ok && lane == 0) atomicCAS(err, 0, ILU_ERR_TIMEOUT);
    }
    __syncthreads();
  }
}

unsigned resident_ctas(int64_t rows, int warps_per_cta, unsigned cap) {
  const int64_t b = (rows + warps_per_cta - 1) / warps_per_cta;
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(b, cap));
}

uint32_t next_epoch(Ilu& p, cudaStream_t st) {
  if (++p.epoch == 0) {  // wrapped: clear every flag so no stale epoch can match
    cudaMemsetAsync(p.flags, 0, sizeof(uint32_t) * p.n_nodes, st);
    p.epoch = 1;
  }
  return p.epoch;
}

// Host-side pattern of the factorisation from the CSR pattern: diagonal positions, lower blocks
// and, for every lower block (i, k), the pairs (j in row i, j in row k) with j > k.
int build_pattern(vms_ctx* ctx, Ilu& p, const Mesh& m) {
  const int64_t N = m.n_nodes;
  std::vector<int32_t> rowptr(4 * N + 1), colidx(m.nnz);
  cudaError_t e = cudaMemcpy(rowptr.data(), m.rowptr, sizeof(int32_t) * rowptr.size(), cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(colidx.data(), m.colidx, sizeof(int32_t) * colidx.size(), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return ctx_fail(ctx, VMS_ERR_CUDA, cudaGetErrorString(e));
  std::vector<int32_t> start(N + 1), adj, dpos(N), lptr(N + 1, 0), pptr(1, 0);
  std::vector<uint16_t> pairs;
  adj.reserve((size_t)m.nnz / 16);
  for (int64_t i = 0; i < N; ++i) {
    const int32_t r0 = rowptr[4 * i];
    const int deg = (rowptr[4 * i + 1] - r0) / 4;
    if (deg > ILU_MAX_DEG)
      return ctx_fail(ctx, VMS_ERR_UNSUPPORTED, "ILU(0): a node has more than 32 neighbours");
    start[i] = (int32_t)adj.size();
    int d = -1;
    for (int kk = 0; kk < deg; ++kk) {
      const int32_t j = colidx[r0 + 4 * kk] / 4;
      if (j == i) d = kk;
      adj.push_back(j);
    }
    if (d < 0) return ctx_fail(ctx, VMS_ERR_INVALID_ARG, "ILU(0): a node belongs to no element");
    dpos[i] = d;
  }
  start[N] = (int32_t)adj.size();
  std::vector<uint8_t> place(N, 0);  // of row i's neighbours in it, from 1; 0: no neighbour
  for (int64_t i = 0; i < N; ++i) {
    const int32_t* ai = adj.data() + start[i];
    const int degi = start[i + 1] - start[i];
    for (int jj = 0; jj < degi; ++jj) place[ai[jj]] = (uint8_t)(jj + 1);
    for (int kk = 0; kk < dpos[i]; ++kk) {
      const int32_t k = ai[kk];
      const int32_t* ak = adj.data() + start[k];
      const int degk = start[k + 1] - start[k];
      uint16_t found[ILU_MAX_DEG];
      int n = 0;
      for (int jk = dpos[k] + 1; jk < degk; ++jk) {  // without a branch: in random order none could be predicted
        const int jj = place[ak[jk]];
        found[n] = (uint16_t)((jj - 1) | (jk << 8));
        n += jj != 0;
      }
      pairs.insert(pairs.end(), found, found + n);
      pptr.push_back((int32_t)pairs.size());
    }
    for (int jj = 0; jj < degi; ++jj) place[ai[jj]] = 0;
    lptr[i + 1] = lptr[i] + dpos[i];
  }
  if (pairs.size() >= (size_t)INT32_MAX)
    return ctx_fail(ctx, VMS_ERR_UNSUPPORTED, "ILU(0): too many update pairs");
  // sweep segments: node i continues the segment of i - 1 when the two are coupled (adjacency
  // lists are sorted, so i - 1 is the entry just before the diagonal)
  std::vector<int32_t> seg;
  seg.reserve((size_t)N / 8 + 2);
  int run = 0;
  for (int64_t i = 0; i < N; ++i) {
    const bool coupled = i > 0 && dpos[i] > 0 && adj[start[i] + dpos[i] - 1] == i - 1;
    if (coupled && run < ILU_SEG_MAX) {
      ++run;
    } else {
      seg.push_back((int32_t)i);
      run = 1;
    }
  }
  seg.push_back((int32_t)N);
  // the most blocks a row has on either side, the row before in its segment not counted
  std::vector<uint8_t> inl(N, 0);  // bit 0: the node before is in the same segment, bit 1: the node after
  p.side_lo = p.side_up = 0;
  for (size_t s = 0; s + 1 < seg.size(); ++s)
    for (int32_t i = seg[s]; i < seg[s + 1]; ++i) {
      const int deg = start[i + 1] - start[i];
      inl[i] = (uint8_t)((i > seg[s] ? 1 : 0) | (i + 1 < seg[s + 1] ? 2 : 0));
      p.side_lo = std::max(p.side_lo, dpos[i] - (i > seg[s] ? 1 : 0));
      p.side_up = std::max(p.side_up, deg - 1 - dpos[i] - (i + 1 < seg[s + 1] ? 1 : 0));
    }
  // chunks of at most ILU_CHUNK segments, fewer where a chunk's distinct neighbours in other chunks
  // on one side would exceed ILU_FAR_MAX (one segment alone is a chunk whatever their number);
  // every neighbour's place in its row's chunk: the chunk's own rows first, then the far list of
  // its side
  std::vector<int32_t> chunk(1, 0), at(adj.size(), 0), farptr[2], far[2], mark(N, -1), order(N);
  p.slots = 0;
  {
    const int32_t n_segs = (int32_t)seg.size() - 1;
    // dependency levels of the two sweeps: the far lists are in the order in which their nodes appear
    std::vector<int32_t> level[2] = {std::vector<int32_t>(N, 0), std::vector<int32_t>(N, 0)};
    for (int64_t i = 0; i < N; ++i)
      for (int32_t t = start[i]; t < start[i] + dpos[i]; ++t) level[0][i] = std::max(level[0][i], level[0][adj[t]] + 1);
    for (int64_t i = N - 1; i >= 0; --i)
      for (int32_t t = start[i] + dpos[i] + 1; t < start[i + 1]; ++t) level[1][i] = std::max(level[1][i], level[1][adj[t]] + 1);
    // rows by level, for the factorisation
    std::vector<int32_t> first(N + 1, 0);
    for (int64_t i = 0; i < N; ++i) ++first[level[0][i] + 1];
    p.n_levels = 1 + *std::max_element(level[0].begin(), level[0].end());
    for (int64_t l = 0; l < N; ++l) first[l + 1] += first[l];
    for (int64_t i = 0; i < N; ++i) order[first[level[0][i]]++] = (int32_t)i;
    farptr[0].push_back(0);
    farptr[1].push_back(0);
    std::vector<uint64_t> lists[2];  // far neighbours of a chunk, level and node
    for (int32_t lo = 0; lo < n_segs;) {
      int32_t hi = std::min(lo + ILU_CHUNK, n_segs);
      for (;; --hi) {
        const int32_t a = seg[lo], b = seg[hi];
        for (int32_t t = start[a]; t < start[b]; ++t) {
          const int32_t j = adj[t];
          if (j >= a && j < b) {
            at[t] = 1 + j - a;
          } else if (mark[j] == -1) {
            const int side = j >= b;
            mark[j] = 0;
            lists[side].push_back((uint64_t)level[side][j] << 32 | (uint32_t)j);
          }
        }
        for (auto& list : lists) {
          std::sort(list.begin(), list.end());
          for (size_t k = 0; k < list.size(); ++k) mark[(uint32_t)list[k]] = (int32_t)k;
        }
        const size_t most = std::max(lists[0].size(), lists[1].size());
        const bool fits = most <= (size_t)ILU_FAR_MAX || hi == lo + 1;
        if (fits) {
          for (int32_t t = start[a]; t < start[b]; ++t)
            if (adj[t] < a || adj[t] >= b) at[t] = 1 + b - a + mark[adj[t]];
          p.slots = std::max(p.slots, 1 + (int)(b - a + (int32_t)most));
        }
        for (int side = 0; side < 2; ++side) {
          for (uint64_t e : lists[side]) {
            mark[(uint32_t)e] = -1;
            if (fits) far[side].push_back((int32_t)(uint32_t)e);
          }
          if (fits) farptr[side].push_back((int32_t)far[side].size());
          lists[side].clear();
        }
        if (fits) break;
      }
      chunk.push_back(hi);
      lo = hi;
    }
  }
  p.n_chunks = (int64_t)chunk.size() - 1;
  p.n_nodes = N;
  p.n_lower = lptr[N];
  p.n_pairs = (int64_t)pairs.size();
  p.n_segs = (int64_t)seg.size() - 1;
  e = cudaMalloc(&p.dpos, sizeof(int32_t) * N);
  if (e == cudaSuccess) e = cudaMalloc(&p.inl, N);
  if (e == cudaSuccess) e = cudaMemcpy(p.inl, inl.data(), N, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(&p.seg, sizeof(int32_t) * seg.size());
  if (e == cudaSuccess) e = cudaMemcpy(p.seg, seg.data(), sizeof(int32_t) * seg.size(), cudaMemcpyHostToDevice);
  auto up = [&](int32_t*& d, const std::vector<int32_t>& h) {
    if (e == cudaSuccess) e = cudaMalloc(&d, sizeof(int32_t) * std::max<size_t>(1, h.size()));
    if (e == cudaSuccess && !h.empty()) e = cudaMemcpy(d, h.data(), sizeof(int32_t) * h.size(), cudaMemcpyHostToDevice);
  };
  up(p.chunk, chunk);
  up(p.order, order);
  up(p.at, at);
  for (int side = 0; side < 2; ++side) {
    up(p.farptr[side], farptr[side]);
    up(p.far[side], far[side]);
  }
  p.chunk_node.resize(chunk.size());
  for (size_t c = 0; c < chunk.size(); ++c) p.chunk_node[c] = seg[chunk[c]];
  if (e == cudaSuccess) e = cudaMalloc(&p.lptr, sizeof(int32_t) * (N + 1));
  if (e == cudaSuccess) e = cudaMalloc(&p.pptr, sizeof(int32_t) * pptr.size());
  if (e == cudaSuccess) e = cudaMalloc(&p.pairs, sizeof(uint16_t) * std::max<size_t>(1, pairs.size()));
  if (e == cudaSuccess) e = cudaMemcpy(p.dpos, dpos.data(), sizeof(int32_t) * N, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(p.lptr, lptr.data(), sizeof(int32_t) * (N + 1), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(p.pptr, pptr.data(), sizeof(int32_t) * pptr.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess && !pairs.empty())
    e = cudaMemcpy(p.pairs, pairs.data(), sizeof(uint16_t) * pairs.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess)
    return ctx_fail(ctx, e == cudaErrorMemoryAllocation ? VMS_ERR_OUT_OF_MEMORY : VMS_ERR_CUDA,
                    cudaGetErrorString(e));
  return VMS_OK;
}

// passes of the sweeps: the places a record needs are a row's other blocks, the row before and
// (backward sweep) the diagonal block
int sweep_np(const Ilu& p, int side) {
  const int places = side ? p.side_up + 2 : p.side_lo + 1;
  return places <= 8 ? 1 : (places <= 16 ? 2 : (places <= 24 ? 3 : (places <= 32 ? 4 : 5)));
}
// f(std::integral_constant<int, NP>) for the sweep's number of passes
template <class F>
auto with_np(const Ilu& p, int side, const F& f) {
  switch (sweep_np(p, side)) {
    case 1: return f(std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, 2>{});
    case 3: return f(std::integral_constant<int, 3>{});
    case 4: return f(std::integral_constant<int, 4>{});
    default: return f(std::integral_constant<int, 5>{});
  }
}
template <typename T>
size_t rec_bytes(const Ilu& p, int side) {
  return with_np(p, side, [&](auto np) { return (size_t)p.n_nodes * sweep_rec_bytes<T, decltype(np)::value>(); });
}

int ensure_work(vms_ctx* ctx, Ilu& p, const Mesh& m, bool fp32) {
  cudaError_t e = cudaSuccess;
  if (!p.F) {
    e = cudaMalloc(&p.F, sizeof(double) * m.nnz);
    if (e == cudaSuccess) e = cudaMalloc(&p.Dinv, sizeof(double) * 16 * m.n_nodes);
  }
  if (e == cudaSuccess && fp32 && !p.vals64) {
    e = cudaMalloc(&p.vals64, sizeof(double) * m.nnz);
    for (float** b : {&p.y32, &p.yp32, &p.xp32})
      if (e == cudaSuccess) e = cudaMalloc(b, sizeof(float) * 4 * m.n_nodes);
    for (float* b : {p.yp32, p.xp32})
      if (e == cudaSuccess) e = cudaMemset(b, 0xff, sizeof(float) * 4 * m.n_nodes);
    for (int side = 0; side < 2; ++side)
      if (e == cudaSuccess) e = cudaMalloc(&p.rec32[side], rec_bytes<float>(p, side));
  }
  if (e == cudaSuccess && !p.flags) {
    e = cudaMalloc(&p.flags, sizeof(uint32_t) * m.n_nodes);
    if (e == cudaSuccess) e = cudaMemset(p.flags, 0, sizeof(uint32_t) * m.n_nodes);
    if (e == cudaSuccess) e = cudaMalloc(&p.tickets, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMemset(p.tickets, 0, sizeof(unsigned long long));
    if (e == cudaSuccess) e = cudaMalloc(&p.err, sizeof(int));
    if (e == cudaSuccess) e = cudaMemset(p.err, 0, sizeof(int));
    p.epoch = 0;
    p.base = 0;
  }
  if (e != cudaSuccess)
    return ctx_fail(ctx, e == cudaErrorMemoryAllocation ? VMS_ERR_OUT_OF_MEMORY : VMS_ERR_CUDA,
                    cudaGetErrorString(e));
  return VMS_OK;
}

template <typename A, typename B>
__global__ void convert_kernel(const A* __restrict__ x, B* __restrict__ y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = B(x[i]);
}

template <typename A, typename B>
int convert(const A* x, B* y, int64_t n, cudaStream_t st) {
  const int64_t b = (n + 255) / 256;
  const int64_t cap = (int64_t)sm_count() * 8;
  convert_kernel<A, B><<<(unsigned)(b > cap ? cap : (b < 1 ? 1 : b)), 256, 0, st>>>(x, y, n);
  return 1;
}

// The row records of both sweeps from the factor.
template <typename T, bool LOWER>
void pack_side(const Ilu& p, const Mesh& m, unsigned char* rec, cudaStream_t st) {
  with_np(p, LOWER ? 0 : 1, [&](auto np) {
    sweep_pack_kernel<T, LOWER, decltype(np)::value>
        <<<16 * (unsigned)sm_count(), 256, 0, st>>>(m.rowptr, p.dpos, p.inl, p.at, p.F, p.Dinv, m.n_nodes, rec);
  });
}
template <typename T>
int pack(const Ilu& p, const Mesh& m, unsigned char* const rec[2], cudaStream_t st) {
  pack_side<T, true>(p, m, rec[0], st);
  pack_side<T, false>(p, m, rec[1], st);
  return 2;
}

}  // namespace

void free_ilu(Ilu& p) {
  const uint32_t lim = p.spin_limit;  // a setting of the context, kept across meshes
  void* bufs[] = {p.dpos, p.order, p.lptr, p.pptr, p.pairs, p.F, p.Dinv, p.y, p.yp64, p.xp64,
                  p.vals64, p.flags, p.yp32, p.xp32, p.tickets, p.err, p.seg, p.inl, p.chunk, p.at,
                  p.farptr[0], p.farptr[1], p.far[0], p.far[1], p.rec[0], p.rec[1], p.rec32[0], p.rec32[1], p.y32};
  for (void* b : bufs)
    if (b) cudaFree(b);
  p = Ilu();
  p.spin_limit = lim;
}

// One warp per row where the levels hold more rows than there are SMs on average (see ilu_factor_kernel).
static bool factor_wide(const Ilu& p) { return p.n_nodes > (int64_t)sm_count() * p.n_levels; }

int ilu_sweeps64(vms_ctx* ctx, Ilu& p, const Mesh& m) {
  if (p.rec[1]) return VMS_OK;
  cudaError_t e = cudaSuccess;
  for (double** b : {&p.y, &p.yp64, &p.xp64})
    if (e == cudaSuccess) e = cudaMalloc(b, sizeof(double) * 4 * m.n_nodes);
  for (double* b : {p.yp64, p.xp64})
    if (e == cudaSuccess) e = cudaMemset(b, 0xff, sizeof(double) * 4 * m.n_nodes);
  for (int side = 0; side < 2; ++side)
    if (e == cudaSuccess) e = cudaMalloc(&p.rec[side], rec_bytes<double>(p, side));
  if (e == cudaSuccess) return VMS_OK;
  for (double** b : {&p.y, &p.yp64, &p.xp64}) {
    cudaFree(*b);
    *b = nullptr;
  }
  for (unsigned char*& r : p.rec) {
    cudaFree(r);
    r = nullptr;
  }
  return ctx_fail(ctx, e == cudaErrorMemoryAllocation ? VMS_ERR_OUT_OF_MEMORY : VMS_ERR_CUDA, cudaGetErrorString(e));
}

int ilu_factor(vms_ctx* ctx, Ilu& p, const Mesh& m, bool fp32, const void* values, cudaStream_t st,
               int* launches) {
  *launches = 0;
  if (p.dpos && p.n_nodes != m.n_nodes) free_ilu(p);
  // a part that was allocated would be taken for the whole by the next call: none is kept
  int rc = p.dpos ? VMS_OK : build_pattern(ctx, p, m);
  if (rc == VMS_OK) rc = ensure_work(ctx, p, m, fp32);
  if (rc != VMS_OK) {
    free_ilu(p);
    return rc;
  }
  // The elimination always runs in FP64 (from the FP32 values in mixed precision): FP32
  // elimination of the condensed systems of distorted meshes, whose condition numbers reach
  // 1e9-1e10, gives factors too poor for GMRES to converge. Mixed precision then rounds the
  // finished factor to FP32 for the FP32 sweeps.
  const double* A = reinterpret_cast<const double*>(values);
  if (fp32) {
    *launches += convert<float, double>((const float*)values, p.vals64, m.nnz, st);
    A = p.vals64;
  }
  const bool wide = factor_wide(p);
  const unsigned ctas = resident_ctas(m.n_nodes, 1, (wide ? FACTOR_WIDE_CTAS : FACTOR_CTAS) * sm_count());
  const uint32_t ep = next_epoch(p, st);
  auto go = [&](auto kern, int warps) {
    kern<<<ctas, warps * 32, 0, st>>>(m.rowptr, m.colidx, A, p.F, p.Dinv, p.dpos, p.lptr, p.pptr, p.pairs, p.order,
                                      m.n_nodes, p.flags, ep, p.tickets, p.base, p.err, p.spin_limit);
  };
  if (wide) go(ilu_factor_kernel<double, 1>, 1);
  else go(ilu_factor_kernel<double, 4>, 4);
  p.base += (unsigned long long)m.n_nodes + ctas;  // + each CTA's last claim
  *launches += 1;
  if (fp32) *launches += pack<float>(p, m, p.rec32, st);
  p.packed64 = false;  // the FP64 records are made on the first FP64 sweep
  p.factored = true;
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? VMS_OK : ctx_fail(ctx, VMS_ERR_CUDA, cudaGetErrorString(e));
}

// Rows without lines: one row a copy and one copy a warp, so that an SM holds more CTAs (FP32 5, FP64 3 instead of 3 and 2
// on hexahedra); rings for the rows to come stay empty there. A GMRES step's two sweeps in us, with the rings and
// without, random node order (one row a segment): 33^3 nodes FP32 180, 139, FP64 343, 272; 91^3 2,925, 1,958 and 6,357, 4,863;
// 40^3 nodes of a tetrahedral mesh 191, 144 and 421, 265. With segments of 5 rows on average (13^3 nodes in reverse
// Cuthill-McKee order) and more the rings win: a solve's sweeps 8.6 and 12.0 ms in FP32.
static bool sweep_short(const Ilu& p) { return p.n_nodes < 2 * p.n_segs; }

// One sweep over rows [n0, n1): the chunks that cover it (rows outside are clamped away in the kernel;
// a block solve has no couplings outside its rows, so n0 and n1 are segment starts).
template <typename T>
struct SweepArgs {
  const unsigned char* rec;
  int64_t n0, n1;
  const T* v;
  T *pub, *clr;
  T* out;
};
template <typename T, bool LOWER, int NP, bool SHORT>
static void launch_sweep(Ilu& p, const SweepArgs<T>& s, cudaStream_t st) {
  const std::vector<int32_t>& cn = p.chunk_node;
  const int64_t c0 = std::max<int64_t>(0, (int64_t)(std::upper_bound(cn.begin(), cn.end() - 1, (int32_t)s.n0) - cn.begin()) - 1);
  const int64_t nc = (int64_t)(std::lower_bound(cn.begin(), cn.end() - 1, (int32_t)s.n1) - cn.begin()) - c0;
  constexpr int W = ILU_CHUNK, FW = 1;
  const int side = LOWER ? 0 : 1;
  const size_t smem = sweep_smem_bytes<T, NP, SHORT>(W, p.slots);
  const int per_sm = (int)std::min<size_t>(48 / (W + FW + 1), (size_t)(227 << 10) / (smem + 2048));
  const unsigned ctas = resident_ctas(nc, 1, (unsigned)std::max(1, per_sm) * sm_count());
  auto kern = ilu_sweep_kernel<T, LOWER, NP, W, FW, SHORT>;
  // more than the default 48 KB of dynamic shared memory (set for the current device)
  cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  kern<<<ctas, (W + FW + 1) * 32, smem, st>>>(s.rec, p.seg, p.chunk, p.farptr[side], p.far[side], c0, nc, s.v,
                                          s.pub, (uint4*)s.clr, s.out, (int)s.n0, (int)(s.n1 - s.n0),
                                          p.slots, p.tickets, p.base, p.err, p.spin_limit);
  p.base += (unsigned long long)nc + ctas;  // + each CTA's last claim
}
template <typename T, bool LOWER>
static void sweep(Ilu& p, const SweepArgs<T>& s, cudaStream_t st) {
  const bool short_segs = sweep_short(p);
  with_np(p, LOWER ? 0 : 1, [&](auto np) {
    if (short_segs) launch_sweep<T, LOWER, decltype(np)::value, true>(p, s, st);
    else launch_sweep<T, LOWER, decltype(np)::value, false>(p, s, st);
  });
}

template <>
int ilu_apply<float, float>(Ilu& p, const Mesh& m, int64_t n0, int64_t n1, const float* v, float* z,
                            cudaStream_t st) {
  sweep<float, true>(p, {p.rec32[0], n0, n1, v, p.yp32, p.xp32, p.y32}, st);
  sweep<float, false>(p, {p.rec32[1], n0, n1, p.y32, p.xp32, p.yp32, z}, st);
  return 2;
}

template <>
int ilu_apply<double, double>(Ilu& p, const Mesh& m, int64_t n0, int64_t n1, const double* v,
                              double* z, cudaStream_t st) {
  int n = 2;
  if (!p.packed64) {
    n += pack<double>(p, m, p.rec, st);
    p.packed64 = true;
  }
  sweep<double, true>(p, {p.rec[0], n0, n1, v, p.yp64, p.xp64, p.y}, st);
  sweep<double, false>(p, {p.rec[1], n0, n1, p.y, p.xp64, p.yp64, z}, st);
  return n;
}

int ilu_status(vms_ctx* ctx, Ilu& p, cudaStream_t st) {
  if (!p.err) return VMS_OK;
  int h = 0;
  cudaError_t e = cudaMemcpyAsync(&h, p.err, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return ctx_fail(ctx, VMS_ERR_CUDA, cudaGetErrorString(e));
  if (h == 0) return VMS_OK;
  // a launch stopped early: its claims and flags are unknown, so start both afresh
  cudaMemsetAsync(p.err, 0, sizeof(int), st);
  cudaMemsetAsync(p.tickets, 0, sizeof(unsigned long long), st);
  cudaMemsetAsync(p.flags, 0, sizeof(uint32_t) * p.n_nodes, st);
  if (p.yp32) cudaMemsetAsync(p.yp32, 0xff, sizeof(float) * 4 * p.n_nodes, st);
  if (p.xp32) cudaMemsetAsync(p.xp32, 0xff, sizeof(float) * 4 * p.n_nodes, st);
  if (p.yp64) cudaMemsetAsync(p.yp64, 0xff, sizeof(double) * 4 * p.n_nodes, st);
  if (p.xp64) cudaMemsetAsync(p.xp64, 0xff, sizeof(double) * 4 * p.n_nodes, st);
  cudaStreamSynchronize(st);
  p.base = 0;
  p.epoch = 0;
  p.factored = false;
  return h == ILU_ERR_PIVOT
             ? ctx_fail(ctx, VMS_ERR_ZERO_PIVOT, "ILU(0): zero pivot in a diagonal block")
             : ctx_fail(ctx, VMS_ERR_TIMEOUT, "ILU(0): a row waited longer than its limit");
}

}  // namespace vms
