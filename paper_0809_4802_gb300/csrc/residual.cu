// FP64 element residual kernel (Section 4.1), one thread per element; arithmetic in
// residual_math.cuh.
#include "residual_math.cuh"
#include "residual_table.cuh"
#include "vms_internal.h"

namespace vms {

// Threads per block: 64 by default; the autotuner (vms_autotune) may choose 32.
constexpr int RES_THREADS = 64;
static_assert(FLAG_NEG_JACOBIAN == 1u && FLAG_NAN == 4u, "residual_element error bits");

template <bool TRANSIENT, bool FORCE, int THREADS>
__global__ void __launch_bounds__(THREADS) residual_kernel(
    const double4_32a* __restrict__ xyz, const double4_32a* __restrict__ u,
    const double4_32a* __restrict__ uprev, const int32_t* __restrict__ conn,
    const double* __restrict__ beta, KParams kp, const QpRow* __restrict__ qp, int64_t first,
    int64_t count,
    double* __restrict__ elemR, double* __restrict__ resid, const uint32_t* __restrict__ dir_mask,
    int64_t n_nodes, int mode, unsigned int* __restrict__ flags) {
  extern __shared__ __align__(16) unsigned char res_smem[];
  double (*sc)[THREADS] = reinterpret_cast<double (*)[THREADS]>(res_smem);
  const int tid = threadIdx.x;
  const int64_t t = (int64_t)blockIdx.x * THREADS + tid;
  if (t >= count) return;
  const int64_t e = first + t;

  int nd[8];
  SmemStore<THREADS> C{sc, tid};
  double Rcp[32], Rf[3];
  const unsigned bad = residual_element<TRANSIENT, FORCE>(e, C, GlobalTable{qp}, kp, xyz, u, uprev,
                                                          conn, beta, nd, Rcp, Rf);
  if (bad) atomicOr(flags, bad);  // bits 1 and 4: FLAG_NEG_JACOBIAN, FLAG_NAN
  if (mode == 0) {
    store_elem_residual(elemR + 36 * e, Rcp, Rf);
  } else {
    const uint32_t msk = dir_mask[e];
#pragma unroll
    for (int a = 0; a < 8; ++a)
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (!(msk >> (4 * a + c) & 1u)) atomicAdd(resid + 4 * (int64_t)nd[a] + c, Rcp[4 * a + c]);
    double* rf = resid + 4 * n_nodes + 3 * e;
    rf[0] = Rf[0]; rf[1] = Rf[1]; rf[2] = Rf[2];
  }
}

// The residual with a lane per line of the Gauss rule (residual_lines), one warp per block.
template <bool TRANSIENT, bool FORCE, int N1>
__global__ void __launch_bounds__(32) residual_lines_kernel(
    const double4_32a* __restrict__ xyz, const double4_32a* __restrict__ u,
    const double4_32a* __restrict__ uprev, const int32_t* __restrict__ conn,
    const double* __restrict__ beta, KParams kp, const QpRow* __restrict__ qp, int64_t first,
    int64_t count, double* __restrict__ elemR, double* __restrict__ resid,
    const uint32_t* __restrict__ dir_mask, int64_t n_nodes, int mode, unsigned int* __restrict__ flags) {
  constexpr int S = N1 * N1, EPW = 32 / S;
  __shared__ double sm[EPW][rl_doubles<N1>()];
  const int lane = threadIdx.x, el = lane / S, ln = lane - el * S;
  const int64_t t = (int64_t)blockIdx.x * EPW + el;
  const bool valid = el < EPW && t < count;
  const int64_t e = first + (valid ? t : 0);
  const uint32_t msk = mode ? dir_mask[e] : 0u;
  const unsigned bad = residual_lines<TRANSIENT, FORCE, N1>(
      valid, e, ln, sm[el < EPW ? el : 0], GlobalTable{qp}, kp, xyz, u, uprev, conn, beta,
      [&](int a, int c, double v) {
        if (mode == 0) elemR[36 * e + 4 * a + c] = v;
        else if (!(msk >> (4 * a + c) & 1u)) atomicAdd(resid + 4 * (int64_t)conn[8 * e + a] + c, v);
      },
      [&](int i, double v) {
        if (mode == 0) elemR[36 * e + 32 + i] = v;
        else resid[4 * n_nodes + 3 * e + i] = v;
      });
  if (bad) atomicOr(flags, bad);
}

template <int N1>
static void launch_lines(const Mesh& m, const State& s, const KParams& kp, const QpRow* qp,
                         double* elemR, double* resid, int64_t first, int64_t count, int mode,
                         unsigned int* flags, cudaStream_t st) {
  constexpr int EPW = 32 / (N1 * N1);
  const unsigned grid = (unsigned)((count + EPW - 1) / EPW);
  auto launch = [&](auto kern) {
    kern<<<grid, 32, 0, st>>>(m.xyz, s.u, s.u_prev, m.conn, s.beta, kp, qp, first, count, elemR, resid,
                              m.dir_mask, m.n_nodes, mode, flags);
  };
  if (kp.transient) {
    if (kp.has_force) launch(residual_lines_kernel<true, true, N1>);
    else launch(residual_lines_kernel<true, false, N1>);
  } else {
    if (kp.has_force) launch(residual_lines_kernel<false, true, N1>);
    else launch(residual_lines_kernel<false, false, N1>);
  }
}

template <int THREADS>
static void launch_r(const Mesh& m, const State& s, const KParams& kp, const QpRow* qp,
                     double* elemR, double* resid, int64_t first, int64_t count, int mode,
                     unsigned int* flags, cudaStream_t st) {
  const dim3 grid((unsigned)((count + THREADS - 1) / THREADS));
  const size_t smem = sizeof(double) * RC_N * THREADS;  // the coefficient store: above 48 KB at 64
  auto launch = [&](auto kern) {
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    kern<<<grid, THREADS, smem, st>>>(m.xyz, s.u, s.u_prev, m.conn, s.beta, kp, qp, first, count,
                                      elemR, resid, m.dir_mask, m.n_nodes, mode, flags);
  };
  if (kp.transient) {
    if (kp.has_force) launch(residual_kernel<true, true, THREADS>);
    else launch(residual_kernel<true, false, THREADS>);
  } else {
    if (kp.has_force) launch(residual_kernel<false, true, THREADS>);
    else launch(residual_kernel<false, false, THREADS>);
  }
}

// Elements of `count` that go to the lane-per-line kernel: those past the last whole round, a round
// being 64 elements per SM and half an SM's threads (2 U, one warp per SM partition), where the lines
// take less time than a part of a round of threads. Measured in us (27 points; 8; 64), U = 9,728
// elements on 152 SMs: threads U 184, 2 U 195, 3 U 288, 4 U 371 (75, 82, 115, 146; 396, 420, 636, 815)
// in steps of U and again from there; lines 29 up to 1,728 elements (25; 34), then 14 + 12.6 per
// thousand (10 + 3.9; 10 + 24). The bounds below are where the two meet. (Both take 5 % less since the
// lines' sums were shortened: 32,768 elements 371 -> 353, 10,648 142 -> 137.)
// Beside a tangent kernel (`beside`) the lines of up to 2 U elements fill the tangent's gaps better. An assembly in us
// with lines and with threads, FP64; FP32 tangent on a second stream; split-TF32 tangent: 512 elements 109 and 196, 53
// and 195, 57 and 198; 4,096 303 and 341, 115 and 232, 137 and 222; 6,069 415 and 566, 158 and 316, 177 and 237; 9,702
// 639 and 858, 232 and 380, 259 and 426; 12,696 822 and 982, 280 and 426, 319 and 463; 17,576 1,129 and 1,229, 386 and
// 514, 436 and 565. Past 2 U the lines' extra FP64 work (a third) costs more than it hides (32,768 in FP64, before the
// tangent took a fifth less: 2,318 and 2,253; a part of them in lines: up to 4 % more).
int64_t residual_rest(int nq, int64_t count, bool beside) {
  const int64_t U = 64 * (int64_t)sm_count(), r = count % (2 * U);
  if (beside) return count <= 2 * U ? count : 0;
  const bool half = (count / (2 * U)) & 1;  // the SMs already hold two blocks each
  const int pct = nq == 27 ? (half ? (r <= U ? 64 : 130) : 135) : (half ? (r <= U ? 75 : 150) : 160);
  return r * 100 <= U * pct ? r : 0;
}

int launch_residual(const Mesh& m, const State& s, const KParams& kp, const QpRow* qp,
                     double* elemR, double* resid, int64_t first, int64_t count, int mode,
                     unsigned int* flags, cudaStream_t st, bool beside) {
  if (count <= 0) return 0;
  // whole rounds with a thread per element, a remainder that would leave the SMs half empty (all of a
  // small mesh) with a lane per line
  const int64_t rest = residual_rest(kp.nq, count, beside), whole = count - rest;
  int n = 0;
  if (whole > 0) {
    if (kp.residual_threads == 32)
      launch_r<32>(m, s, kp, qp, elemR, resid, first, whole, mode, flags, st);
    else
      launch_r<RES_THREADS>(m, s, kp, qp, elemR, resid, first, whole, mode, flags, st);
    ++n;
  }
  if (rest > 0) {
    const int64_t f = first + whole;
    if (kp.nq == 27) launch_lines<3>(m, s, kp, qp, elemR, resid, f, rest, mode, flags, st);
    else if (kp.nq == 8) launch_lines<2>(m, s, kp, qp, elemR, resid, f, rest, mode, flags, st);
    else launch_lines<4>(m, s, kp, qp, elemR, resid, f, rest, mode, flags, st);
    ++n;
  }
  return n;
}

}  // namespace vms
