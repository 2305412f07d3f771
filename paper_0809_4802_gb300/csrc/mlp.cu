// Learned warm start of the transient Newton iteration (Remark of Section 4.1, Section 4.2): a
// 3-layer MLP (12 -> 128 -> 128 -> 4, tanh) that predicts each node's increment over the next
// backward-Euler step. Weights are stored in BF16, biases, activations and accumulation in FP32.
// Forward, backward (mean squared error) and Adam run in these kernels; Newton then converges to
// the same tolerance from the predicted start, so the network only changes the starting point.
// The forward pass runs both hidden layers on tcgen05 tensor cores (mlp_forward_kernel). In the gradient
// kernel the three 128-wide contractions of a 64-node tile (H1 W2, H1^T D and D W2^T) run on mma.sync
// m16n8k16, BF16 operands, FP32 accumulation. Either way the FP32 activations are split into sums of
// BF16 terms: three terms against the BF16 weights (exact products, FP32-level results), two times
// two terms (three products) for H1^T D. The 4-wide output layer and, in the gradient kernel, the
// 12-wide input layer and the small gradient blocks stay on the CUDA cores.
//
// Layout of the parameter vector (row-major): W1 [12][128], b1 [128], W2 [128][128], b2 [128],
// W3 [128][4], b3 [4].
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "mma_bf16.cuh"
#include "solver.h"
#include "vms_internal.h"

struct vms_mlp {
  int device = 0;
  cudaStream_t stream = nullptr;
  float* master = nullptr;  // FP32 master copy of all parameters (Adam updates it)
  float* m = nullptr;       // Adam first moments
  float* v = nullptr;       // Adam second moments
  float* grad = nullptr;    // gradient of the last vms_mlp_grad call
  __nv_bfloat16* w = nullptr;  // W1, W2, W3 in BF16 (offsets below)
  float* bias = nullptr;       // b1, b2, b3 in FP32
  double* loss = nullptr;      // device loss accumulator, behind grad
  float* host = nullptr;       // page-locked: gradient and loss on their way to the caller, the status word
  int* status = nullptr;       // behind them: 1 once a forward pass has given up (until it is reported)
  uint32_t wait_limit = 0;     // polls of one wait of the forward pass; 0: the default
  float* scratch = nullptr;    // P_N floats (parameter read-back)
  double* colsum = nullptr;    // 16 column sums of squares (vms_mlp_column_rms)
  int t = 0;                   // Adam steps taken
  std::string err;
};

namespace {

using vms::bf16x2_split2;
using vms::bf16x2_split3;
using vms::mma_bf16;

constexpr int NI = VMS_MLP_IN, NW = VMS_MLP_WIDTH, NO = VMS_MLP_OUT;
constexpr int P_W1 = 0, P_B1 = P_W1 + NI * NW, P_W2 = P_B1 + NW, P_B2 = P_W2 + NW * NW,
              P_W3 = P_B2 + NW, P_B3 = P_W3 + NW * NO, P_N = P_B3 + NO;
static_assert(P_N == VMS_MLP_PARAMS, "parameter count");
constexpr size_t GRAD_BYTES = sizeof(float) * P_N + sizeof(double);  // the gradient, then the loss
static_assert(P_N % 2 == 0, "the loss behind the gradient");
constexpr size_t HOST_BYTES = GRAD_BYTES + sizeof(int);
// BF16 weight array: W1 | W2 | W3; FP32 bias array: b1 | b2 | b3
constexpr int WB_1 = 0, WB_2 = NI * NW, WB_3 = WB_2 + NW * NW, WB_N = WB_3 + NW * NO;
constexpr int BB_1 = 0, BB_2 = NW, BB_3 = 2 * NW, BB_N = 2 * NW + NO;

constexpr int THREADS = 256;   // 8 warps
constexpr int HLD = NW + 4;    // padded FP32 activation row (conflict-free MMA fragment loads)
constexpr int WLD = NW + 8;    // padded BF16 weight row (68 words: conflict-free fragment loads)

// ROWS (16, 32 or 64) rows (nodes) per tile.
template <int ROWS>
struct SmemGrad {
  float W1[NI][NW];
  __nv_bfloat16 W2[NW][WLD];   // W2 [k][j]
  float W3[NW][NO];
  float b1[NW], b2[NW], b3[NO];
  float X[ROWS][NI];
  float H1[ROWS][HLD];
  float H2[ROWS][HLD];
  float D[ROWS][HLD];
  float dY[ROWS][NO];
};

// W2 arrives by asynchronous 16-byte copies while the first layer runs (wait_weights before its use).
template <int ROWS>
__device__ void load_weights(SmemGrad<ROWS>& s, const __nv_bfloat16* __restrict__ w, const float* __restrict__ bias) {
  for (int i = threadIdx.x; i < NW * NW / 8; i += THREADS) {
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(&s.W2[i / (NW / 8)][i % (NW / 8) * 8]);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(w + WB_2 + 8 * i) : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
#pragma unroll
  for (int i = threadIdx.x; i < NI * NW / 2; i += THREADS) {
    const float2 v = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w + WB_1)[i]);
    reinterpret_cast<float2*>(&s.W1[0][0])[i] = v;
  }
  {
    const float2 v = __bfloat1622float2(reinterpret_cast<const __nv_bfloat162*>(w + WB_3)[threadIdx.x]);
    reinterpret_cast<float2*>(&s.W3[0][0])[threadIdx.x] = v;
    static_assert(NW * NO == 2 * THREADS && 2 * NW == THREADS, "one pair, one bias per thread");
    (threadIdx.x < NW ? s.b1 : s.b2 - NW)[threadIdx.x] = bias[BB_1 + threadIdx.x];
  }
  if (threadIdx.x < NO) s.b3[threadIdx.x] = bias[BB_3 + threadIdx.x];
}
__device__ __forceinline__ void wait_weights() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// C[ROWS x 128] = A[ROWS x 128] B on the tensor cores, A FP32 split into three BF16 terms, B = W (BWD false)
// or W^T (true), W [128][128] in BF16. A warp owns 16 rows (warp w rows 16 (w % RT) ..) and NT column
// tiles of 8; acc[nt][*] is the standard m16n8 C fragment (rows g, g + 8 and columns 2t, 2t + 1 of
// tile nt, g = lane / 4, t = lane % 4), initialised by the caller.
template <int ROWS> struct WarpTile {
  static constexpr int RT = ROWS / 16, NT = 2 * RT;  // row tiles; column tiles per warp
  static __device__ __forceinline__ int row(int w) { return 16 * (w % RT); }
  static __device__ __forceinline__ int col(int w) { return 8 * NT * (w / RT); }
};
template <int ROWS, bool BWD>
__device__ __forceinline__ void mma_rows(const float (*A)[HLD], const __nv_bfloat16 (*W)[WLD], float (*acc)[4]) {
  constexpr int NT = WarpTile<ROWS>::NT;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int r0 = WarpTile<ROWS>::row(w) + g, c0 = WarpTile<ROWS>::col(w);
#pragma unroll 2
  for (int k0 = 0; k0 < NW; k0 += 16) {
    uint32_t ah[4], am[4], al[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const float2 x = *reinterpret_cast<const float2*>(&A[r0 + 8 * (f & 1)][k0 + 2 * t + 8 * (f >> 1)]);
      bf16x2_split3(x.x, x.y, ah[f], am[f], al[f]);
    }
#pragma unroll
    for (int nt = 0; nt < NT; nt += 2) {
      // two column tiles: rows k0 .. + 15 of W transposed on the way in, or K contiguous as it lies
      uint32_t b[4];
      const int q = lane >> 3, i = lane & 7;
      const __nv_bfloat16* at = BWD ? &W[c0 + 8 * (nt + (q >> 1)) + i][k0 + 8 * (q & 1)]
                                    : &W[k0 + 8 * (q & 1) + i][c0 + 8 * (nt + (q >> 1))];
      const uint32_t addr = (uint32_t)__cvta_generic_to_shared(at);
      if (BWD)
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(addr) : "memory");
      else
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                     : "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]) : "r"(addr) : "memory");
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        mma_bf16(acc[nt + h], al, b[2 * h], b[2 * h + 1]);
        mma_bf16(acc[nt + h], am, b[2 * h], b[2 * h + 1]);
        mma_bf16(acc[nt + h], ah, b[2 * h], b[2 * h + 1]);
      }
    }
  }
}

// H2 = tanh(H1 W2 + b2) on the tensor cores
template <int ROWS>
__device__ __forceinline__ void dense2_tanh(SmemGrad<ROWS>& s) {
  constexpr int NT = WarpTile<ROWS>::NT;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int r0 = WarpTile<ROWS>::row(w) + g, c0 = WarpTile<ROWS>::col(w);
  float acc[NT][4];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const int c = c0 + 8 * nt + 2 * t;
    acc[nt][0] = acc[nt][2] = s.b2[c];
    acc[nt][1] = acc[nt][3] = s.b2[c + 1];
  }
  mma_rows<ROWS, false>(s.H1, s.W2, acc);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const int c = c0 + 8 * nt + 2 * t;
    *reinterpret_cast<float2*>(&s.H2[r0][c]) = make_float2(tanhf(acc[nt][0]), tanhf(acc[nt][1]));
    *reinterpret_cast<float2*>(&s.H2[r0 + 8][c]) = make_float2(tanhf(acc[nt][2]), tanhf(acc[nt][3]));
  }
}

// rows [r0, r0 + ROWS) of X (through `rows` if given) into shared memory, zero beyond n
template <int ROWS>
__device__ void load_tile(SmemGrad<ROWS>& s, const float* __restrict__ X, const int32_t* __restrict__ rows,
                          int64_t r0, int64_t n) {
  for (int i = threadIdx.x; i < ROWS * NI; i += THREADS) {
    const int r = i / NI, c = i % NI;
    const int64_t g = r0 + r;
    float x = 0.f;
    if (g < n) x = X[(rows ? (int64_t)rows[g] : g) * NI + c];
    s.X[r][c] = x;
  }
}

// H1 = tanh(X W1 + b1) for the tile on the CUDA cores; warp w owns ROWS / 8 rows, lane l columns l + 32 j
template <int ROWS>
__device__ void dense1_tanh(SmemGrad<ROWS>& s) {
  constexpr int R = ROWS / 8;
  const int w = threadIdx.x >> 5, l = threadIdx.x & 31;
  float acc[R][4];
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[r][j] = s.b1[l + 32 * j];
#pragma unroll 4
  for (int k = 0; k < NI; ++k) {
    float wv[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) wv[j] = s.W1[k][l + 32 * j];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float a = s.X[R * w + r][k];
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[r][j] = fmaf(a, wv[j], acc[r][j]);
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r)
#pragma unroll
    for (int j = 0; j < 4; ++j) s.H1[R * w + r][l + 32 * j] = tanhf(acc[r][j]);
}

// ---------------------------------------------------------------------------------------------
// Forward pass on the fifth-generation tensor cores (tcgen05.mma, accumulators in tensor memory)
// ---------------------------------------------------------------------------------------------
// A CTA takes tiles of 128 rows, one row per TMEM lane; two CTAs share an SM, so one's matrix products
// run under the other's tanh. Both hidden layers are MMAs of 128 x 128 x 16 with BF16 operands from
// shared memory: the FP32 activations as three BF16 terms whose sum is exact (truncated, 8 bits each),
// the weights as they are stored; the low terms of a group of K are summed first. Biases ride along as
// three rows of a K step whose activations are 1. Per tile: X -> D1 (K = 16, three MMAs) -> H1 = tanh ->
// D2 (eight K steps, three MMAs each, in two halves of K so that the operand buffer holds half of H1
// and two CTAs fit) -> tanh -> the 4-wide output layer in FP32 as the values leave tensor memory. H2 and D2
// never touch shared memory, H1 only as an operand.
// Bound by instruction issue and the FP32 pipe (tanh, the split); the products alone would take 60 us of
// the 191 us for 975,583 rows. With mma.sync from FP32 tiles in shared memory, bound by the traffic there, it
// took 661 us (1,024 rows 14.5, now 10.8; 100,000 79, now 29), with errors against 64 bits of 4.7e-7 rms, now
// 3.9e-7 (the low terms are summed first).
constexpr int FT = 128;                       // rows per tile
constexpr uint32_t OP_K = FT * 16;            // bytes between core matrices along K (LBO)
constexpr uint32_t OP_R = 128;                // bytes between groups of 8 rows (SBO)
constexpr uint32_t OP_STEP = 2 * OP_K;        // a K step of 16: two core matrices
struct SmemFwd {
  // operands in the canonical K-major layout without swizzle: [k / 8][row][k % 8]
  __nv_bfloat16 W1[2 * FT * 8];               // W1 (k < 12), the bias' three terms (k = 12..14), 0
  __nv_bfloat16 W1f[2 * FT * 8];              // W1 with 0 for its infinities, 0: the partner of X's lower terms
  __nv_bfloat16 B2[2 * FT * 8];               // 0, the second bias' three terms, 0
  __nv_bfloat16 one[2 * FT * 8];              // its activations: 0 (not X's, which may be infinite), 1, 1, 1, 0
  __nv_bfloat16 X[3][2 * FT * 8];             // the terms of X; 1 in k = 12..14 of the first
  __nv_bfloat16 W2[16 * FT * 8];
  __nv_bfloat16 H[3][8 * FT * 8];             // the terms of half of H1
  float4 W3[NW];
  float4 part[FT];                            // output sums of columns 64..127
  float b3[NO];
  uint32_t tmem;
  unsigned long long bar[4];                  // D1; first half of D2 (operand buffers free); D2; all, after giving up
};
static_assert(sizeof(SmemFwd) + 1024 <= (228 << 10) / 2, "two CTAs per SM");

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
// Shared-memory matrix descriptor: start, LBO and SBO in 16-byte units, version 1, no swizzle.
__device__ __forceinline__ uint64_t op_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3ffffu) >> 4) | (uint64_t)(OP_K >> 4) << 16 | (uint64_t)(OP_R >> 4) << 32 | 1ull << 46;
}
// Instruction descriptor of kind::f16: FP32 accumulators, BF16 operands, both K-major, N = 128, M = 128.
constexpr uint32_t OP_IDESC = 1u << 4 | 1u << 7 | 1u << 10 | (NW >> 3) << 17 | (FT >> 4) << 24;
__device__ __forceinline__ void tc_mma(uint32_t d, uint32_t a, uint32_t b, bool add) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(op_desc(a)), "l"(op_desc(b)), "r"(OP_IDESC), "r"((uint32_t)add)
      : "memory");
}
__device__ __forceinline__ void tc_commit(unsigned long long* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
// Wait of a whole warp for the barrier's phase of this parity; false for all its lanes if it has not come after `lim`
// polls: a test, then waits of up to a microsecond each (counted, not timed: a process that is switched out has not
// waited).
constexpr uint32_t WAIT_DEFAULT = 1u << 20;
__device__ __forceinline__ bool bar_wait(unsigned long long* bar, uint32_t parity, uint32_t lim) {
  const uint32_t a = smem_u32(bar);
  uint32_t done;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(done) : "r"(a), "r"(parity) : "memory");
  for (uint32_t it = 1; !done && it < lim; ++it)
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(a), "r"(parity), "r"(1000u) : "memory");
  return __all_sync(0xffffffffu, done);
}
// 32 columns of the warp's 32 lanes of tensor memory; the values may be used when it returns.
__device__ __forceinline__ void tc_load32(uint32_t addr, float v[32]) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  __syncwarp();
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(addr)
      : "memory");
}
// x = h + m + l, each the leading 8 bits of what is left (bit patterns with the BF16 in the upper half):
// exact for every finite x whose low term is a BF16 number. NaN makes all of them NaN, an infinity m and l: where x
// may be one, finite_terms() keeps it in h alone.
struct Terms {
  uint32_t h, m, l;
};
__device__ __forceinline__ Terms split_exact(float x) {
  Terms t;
  t.h = __float_as_uint(x) & 0xffff0000u;
  const float r = x - __uint_as_float(t.h);
  t.m = __float_as_uint(r) & 0xffff0000u;
  t.l = __float_as_uint(r - __uint_as_float(t.m));
  return t;
}
__device__ __forceinline__ Terms finite_terms(float x) {
  Terms t = split_exact(x);
  if (fabsf(x) == INFINITY) t.m = t.l = 0u;
  return t;
}
// tanh of two values: x N(x^2) / D(x^2) with N of degree 4 and D of degree 5, the minimax quotient on [0, 9.02]
// (fitted with the Remez exchange algorithm in 40 digits), beyond which tanh rounds to +-1. Its relative error is 1.1e-8
// with the coefficients rounded to FP32 and, evaluated in FP32, 6.4e-8 rms and at most 2.8e-7 over 28,000 arguments
// (tanhf: 2.6e-8 and 1.7e-7), largest near +-8.8, where a value may also be 1 + 2^-22. The sums of products leave
// more: the output's error is 0.80 to 0.88 of the earlier kernel's rms (mma.sync, tanhf) on inputs of unit variance and
// initial weights, and over 45 settings of weights (1 to 10 times) and inputs (0.01 to 100) 0.36 to 1.10 of it (above 1
// in one) and 0.16 to 0.99 of its largest. Branch-free and two at a time: the tile is bound by instruction issue, and
// tanhf took two thirds of it (975,583 rows 214 us, now 191).
constexpr float NTH1 = 0.137853637f, NTH2 = 0.00400850875f, NTH3 = 3.15890575e-05f, NTH4 = 5.07622211e-08f;
constexpr float DTH1 = 0.471186966f, DTH2 = 0.0277375113f, DTH3 = 0.000420740689f, DTH4 = 1.61748528e-06f,
                DTH5 = 7.37443662e-10f;
__device__ __forceinline__ float2 tanh2(float2 v) {
  float2 x;
  asm("{\n\t.reg .f32 t;\n\tmax.NaN.f32 t, %2, 0fC11051EC;\n\tmin.NaN.f32 %0, t, 0f411051EC;\n\t"
      "max.NaN.f32 t, %3, 0fC11051EC;\n\tmin.NaN.f32 %1, t, 0f411051EC;\n\t}"
      : "=f"(x.x), "=f"(x.y)
      : "f"(v.x), "f"(v.y));
  auto c = [](float a) { return make_float2(a, a); };
  const float2 s = __fmul2_rn(x, x);
  float2 n = __ffma2_rn(c(NTH4), s, c(NTH3)), d = __ffma2_rn(c(DTH5), s, c(DTH4));
  n = __ffma2_rn(n, s, c(NTH2));
  d = __ffma2_rn(d, s, c(DTH3));
  n = __ffma2_rn(n, s, c(NTH1));
  d = __ffma2_rn(d, s, c(DTH2));
  n = __ffma2_rn(n, s, c(1.f));
  d = __ffma2_rn(d, s, c(DTH1));
  d = __ffma2_rn(d, s, c(1.f));
  float2 r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.x) : "f"(d.x));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r.y) : "f"(d.y));
  return __fmul2_rn(__fmul2_rn(n, x), r);
}

// Eight consecutive K of one row, as the three terms' 16-byte pieces.
__device__ __forceinline__ void store_terms(__nv_bfloat16* h, __nv_bfloat16* m, __nv_bfloat16* l, const float v[8]) {
  uint32_t H[4], M[4], L[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const Terms a = split_exact(v[2 * i]), b = split_exact(v[2 * i + 1]);
    H[i] = __byte_perm(a.h, b.h, 0x7632);
    M[i] = __byte_perm(a.m, b.m, 0x7632);
    L[i] = __byte_perm(a.l, b.l, 0x7632);
  }
  *reinterpret_cast<uint4*>(h) = make_uint4(H[0], H[1], H[2], H[3]);
  *reinterpret_cast<uint4*>(m) = make_uint4(M[0], M[1], M[2], M[3]);
  *reinterpret_cast<uint4*>(l) = make_uint4(L[0], L[1], L[2], L[3]);
}
__device__ __forceinline__ __nv_bfloat16 upper_bf16(uint32_t u) { return __ushort_as_bfloat16((unsigned short)(u >> 16)); }

// Eight of the sixteen K of a row of X (half 0: columns 0..7; half 1: columns 8..11, 1, 1, 1, 0); `vec`: X is 16-byte aligned.
__device__ __forceinline__ void load_x(const float* __restrict__ X, int64_t row, int64_t n, int half, bool vec, float v[8]) {
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = half && i >= 4 && i < 7 ? 1.f : 0.f;
  if (row >= n) return;
  const float* p = X + row * NI + 8 * half;
  if (vec) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(p));
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    if (!half) {
      const float4 b = __ldg(reinterpret_cast<const float4*>(p) + 1);
      v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = __ldg(p + i);
    if (!half)
#pragma unroll
      for (int i = 4; i < 8; ++i) v[i] = __ldg(p + i);
  }
}
__device__ __forceinline__ void store_x(SmemFwd& s, int row, int half, const float v[8]) {
  const int at = half * FT * 8 + row * 8;
  store_terms(&s.X[0][at], &s.X[1][at], &s.X[2][at], v);
#pragma unroll
  for (int i = 0; i < 8; ++i)
    if (fabsf(v[i]) == INFINITY) {  // infinity minus infinity would be NaN
      s.X[1][at + i] = __ushort_as_bfloat16(0);
      s.X[2][at + i] = __ushort_as_bfloat16(0);
    }
}

__global__ void __launch_bounds__(THREADS, 2) mlp_forward_kernel(const __nv_bfloat16* __restrict__ w,
                                                                 const float* __restrict__ bias,
                                                                 const float* __restrict__ X, int64_t n,
                                                                 float* __restrict__ Y, uint32_t lim, int* status) {
  extern __shared__ __align__(128) unsigned char raw[];
  SmemFwd& s = *reinterpret_cast<SmemFwd*>(raw);
  const int tid = threadIdx.x, wp = tid >> 5, half = wp >> 2, row = (wp & 3) * 32 + (tid & 31);
  const bool vec = (reinterpret_cast<uintptr_t>(X) & 15) == 0;
  const int64_t stride = (int64_t)gridDim.x * FT;
  int64_t r0 = (int64_t)blockIdx.x * FT;
  float x[8];
  load_x(X, r0 + row, n, half, vec, x);
  // operands of the weights, K (8 at a time) contiguous
  for (int i = tid; i < 16 * NW; i += THREADS) {
    const int c = i / NW, j = i % NW;
    alignas(16) __nv_bfloat16 v[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) v[k] = w[WB_2 + (8 * c + k) * NW + j];
    *reinterpret_cast<uint4*>(&s.W2[c * FT * 8 + j * 8]) = *reinterpret_cast<const uint4*>(v);
  }
  {
    const int c = tid / NW, j = tid % NW;  // 2 x 128
    const Terms b1 = finite_terms(bias[BB_1 + j]), b2 = finite_terms(bias[BB_2 + j]);
    const __nv_bfloat16 z = __ushort_as_bfloat16(0);
    alignas(16) __nv_bfloat16 v[8], f[8], u[8], o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      v[k] = 8 * c + k < NI ? w[WB_1 + (8 * c + k) * NW + j] : z;
      f[k] = (__bfloat16_as_ushort(v[k]) & 0x7fffu) == 0x7f80u ? z : v[k];
      u[k] = z;
      o[k] = c && k >= 4 && k < 7 ? __ushort_as_bfloat16(0x3f80) : z;
    }
    *reinterpret_cast<uint4*>(&s.one[c * FT * 8 + j * 8]) = *reinterpret_cast<const uint4*>(o);
    if (c) {
      v[4] = upper_bf16(b1.h); v[5] = upper_bf16(b1.m); v[6] = upper_bf16(b1.l);
      u[4] = upper_bf16(b2.h); u[5] = upper_bf16(b2.m); u[6] = upper_bf16(b2.l);
    }
    *reinterpret_cast<uint4*>(&s.W1[c * FT * 8 + j * 8]) = *reinterpret_cast<const uint4*>(v);
    *reinterpret_cast<uint4*>(&s.W1f[c * FT * 8 + j * 8]) = *reinterpret_cast<const uint4*>(f);
    *reinterpret_cast<uint4*>(&s.B2[c * FT * 8 + j * 8]) = *reinterpret_cast<const uint4*>(u);
  }
  for (int i = tid; i < NW * NO; i += THREADS) reinterpret_cast<float*>(s.W3)[i] = __bfloat162float(w[WB_3 + i]);
  if (tid < NO) s.b3[tid] = bias[BB_3 + tid];
  store_x(s, row, half, x);
  if (tid == 0) {
    for (int i = 0; i < 4; ++i)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&s.bar[i])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (wp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(&s.tmem)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  fence_async_shared();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t d1 = s.tmem, d2 = d1 + NW, lanes = (uint32_t)(wp & 3) << 21;  // the warp's lanes, in bits 16..31
  const uint32_t aX = smem_u32(s.X), aH = smem_u32(s.H), aW1 = smem_u32(s.W1), aW1f = smem_u32(s.W1f), aB2 = smem_u32(s.B2), aOne = smem_u32(s.one), aW2 = smem_u32(s.W2);
  constexpr uint32_t XT = sizeof(s.X[0]), HT = sizeof(s.H[0]);
  auto layer1 = [&]() {
    for (int t = 2; t >= 0; --t) tc_mma(d1, aX + t * XT, t ? aW1f : aW1, t != 2);  // (a zero term times an infinity is NaN)
    tc_commit(&s.bar[0]);
  };
  if (tid == 0) layer1();
  uint32_t par = 0;
  bool ok = true;
  for (; r0 < n; r0 += stride, par ^= 1u) {
    const bool more = r0 + stride < n;
    if (more) load_x(X, r0 + stride + row, n, half, vec, x);
    // H1, columns 0..63 (the warp's 32), then their products
    float v[32] = {};
    bool good = bar_wait(&s.bar[0], par, lim);
    tc_fence_after();
    if (good) tc_load32(d1 + lanes + 32 * half, v);
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float h[8];
#pragma unroll
      for (int i = 0; i < 8; i += 2) {
        const float2 t = tanh2(make_float2(v[8 * c + i], v[8 * c + i + 1]));
        h[i] = t.x; h[i + 1] = t.y;
      }
      const int at = (4 * half + c) * FT * 8 + row * 8;
      store_terms(&s.H[0][at], &s.H[1][at], &s.H[2][at], h);
    }
    fence_async_shared();
    tc_fence_before();
    if (__syncthreads_or(!good)) { ok = false; break; }
    if (tid == 0) {
      tc_fence_after();
      tc_mma(d2, aOne, aB2, false);
      for (int t = 2; t >= 0; --t)
        for (int k = 0; k < 4; ++k) tc_mma(d2, aH + t * HT + k * OP_STEP, aW2 + k * OP_STEP, true);
      tc_commit(&s.bar[1]);
    }
    // columns 64..127
    tc_load32(d1 + lanes + 64 + 32 * half, v);
#pragma unroll
    for (int i = 0; i < 32; i += 2) {
      const float2 t = tanh2(make_float2(v[i], v[i + 1]));
      v[i] = t.x; v[i + 1] = t.y;
    }
    good = bar_wait(&s.bar[1], par, lim);
    if (good)
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        const int at = (4 * half + c) * FT * 8 + row * 8;
        store_terms(&s.H[0][at], &s.H[1][at], &s.H[2][at], v + 8 * c);
      }
    if (more) store_x(s, row, half, x);
    fence_async_shared();
    tc_fence_before();
    if (__syncthreads_or(!good)) { ok = false; break; }
    if (tid == 0) {
      tc_fence_after();
      for (int t = 2; t >= 0; --t)
        for (int k = 0; k < 4; ++k) tc_mma(d2, aH + t * HT + k * OP_STEP, aW2 + (4 + k) * OP_STEP, true);
      tc_commit(&s.bar[2]);
      if (more) layer1();
    }
    // H2 and the output layer, columns 64 half ..
    good = bar_wait(&s.bar[2], par, lim);
    tc_fence_after();
    float2 ya = make_float2(0.f, 0.f), yb = ya;
#pragma unroll
    for (int q = 0; q < 2 && good; ++q) {
      tc_load32(d2 + lanes + 64 * half + 32 * q, v);
#pragma unroll
      for (int i = 0; i < 32; i += 2) {
        const float2 h = tanh2(make_float2(v[i], v[i + 1]));
        const float4 w0 = s.W3[64 * half + 32 * q + i], w1 = s.W3[64 * half + 32 * q + i + 1];
        ya = __ffma2_rn(make_float2(h.x, h.x), make_float2(w0.x, w0.y), ya);
        yb = __ffma2_rn(make_float2(h.x, h.x), make_float2(w0.z, w0.w), yb);
        ya = __ffma2_rn(make_float2(h.y, h.y), make_float2(w1.x, w1.y), ya);
        yb = __ffma2_rn(make_float2(h.y, h.y), make_float2(w1.z, w1.w), yb);
      }
    }
    if (half) s.part[row] = make_float4(ya.x, ya.y, yb.x, yb.y);
    tc_fence_before();
    if (__syncthreads_or(!good)) { ok = false; break; }
    if (!half && r0 + row < n) {
      const float4 p = s.part[row];
      const float y[4] = {s.b3[0] + ya.x + p.x, s.b3[1] + ya.y + p.y, s.b3[2] + yb.x + p.z, s.b3[3] + yb.y + p.w};
      float* o = Y + (r0 + row) * NO;
      if ((reinterpret_cast<uintptr_t>(Y) & 15) == 0) {
        *reinterpret_cast<float4*>(o) = make_float4(y[0], y[1], y[2], y[3]);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = y[i];
      }
    }
  }
  if (!ok) {
    // a product did not finish in time. Wait for all that are in flight (the next tile's first layer may be), which
    // write tensor memory and read shared memory; then say so in the rows and in the handle's status.
    if (tid == 0) {
      tc_commit(&s.bar[3]);
      *reinterpret_cast<volatile int*>(status) = 1;
      __threadfence_system();
    }
    __syncwarp();
    bar_wait(&s.bar[3], 0, WAIT_DEFAULT);
    for (; r0 < n; r0 += stride)
      for (int i = tid; i < FT * NO; i += THREADS)
        if (r0 + i / NO < n) Y[r0 * NO + i] = NAN;
  }
  __syncthreads();
  if (wp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(d1) : "memory");
}

// Gradient of loss = sum over the n rows and 4 outputs of (y - t)^2 / (4 n), accumulated per CTA
// in registers and added to grad (FP32) once; the loss (FP64) likewise. ROWS rows per tile: a CTA's tile is a
// chain of eight dependent stages whose length goes with ROWS, so as long as there are SMs for it a batch
// is cut finer (grad_rows).
template <int ROWS>
__global__ void __launch_bounds__(THREADS) mlp_grad_kernel(
    const __nv_bfloat16* __restrict__ w, const float* __restrict__ bias, const float* __restrict__ X,
    const float* __restrict__ T, const int32_t* __restrict__ rows, int64_t n, float scale,
    float* __restrict__ grad, double* __restrict__ loss) {
  extern __shared__ __align__(16) unsigned char raw[];
  SmemGrad<ROWS>& s = *reinterpret_cast<SmemGrad<ROWS>*>(raw);
  load_weights(s, w, bias);
  const int tid = threadIdx.x, wp = tid >> 5, l = tid & 31, g = l >> 2, t = l & 3;
  // register partials: dW2 as MMA C fragments (warp wp: rows k = 16 wp + g (+ 8) of dW2, column
  // tiles 0..15), dW1 (6 entries), dW3 (2 entries), db1/db2 (threads < 128: column tid), db3
  // (threads < 4)
  float gW2[16][4], gW1[6], gW3[2], gb1 = 0.f, gb2 = 0.f, gb3 = 0.f;
#pragma unroll
  for (int nt = 0; nt < 16; ++nt)
#pragma unroll
    for (int q = 0; q < 4; ++q) gW2[nt][q] = 0.f;
#pragma unroll
  for (int i = 0; i < 6; ++i) gW1[i] = 0.f;
  gW3[0] = gW3[1] = 0.f;
  double lsum = 0.0;
  for (int64_t r0 = (int64_t)blockIdx.x * ROWS; r0 < n; r0 += (int64_t)gridDim.x * ROWS) {
    __syncthreads();
    load_tile(s, X, rows, r0, n);
    __syncthreads();
    dense1_tanh(s);
    wait_weights();
    __syncthreads();
    dense2_tanh(s);
    __syncthreads();
    {
      // y[r][o] = b3[o] + sum_k H2[r][k] W3[k][o]: KS threads per output
      constexpr int KS = 64 / ROWS;
      const int o = tid & 3, ks = (tid >> 2) % KS, r = tid / (4 * KS);
      const int64_t gr = r0 + r;
      float y = ks ? 0.f : s.b3[o], d = 0.f;
#pragma unroll 8
      for (int k = ks; k < NW; k += KS) y = fmaf(s.H2[r][k], s.W3[k][o], y);
#pragma unroll
      for (int m = 4; m < 4 * KS; m <<= 1) y += __shfl_xor_sync(0xffffffffu, y, m);
      if (gr < n) {
        const float e = y - T[(rows ? (int64_t)rows[gr] : gr) * NO + o];
        if (ks == 0) lsum += (double)e * (double)e;
        d = 2.f * scale * e;
      }
      if (ks == 0) s.dY[r][o] = d;
      // db3: the warp's rows (lanes 0..3 of each warp keep the sums)
      float c = ks == 0 ? d : 0.f;
#pragma unroll
      for (int m = 4; m < 32; m <<= 1) c += __shfl_xor_sync(0xffffffffu, c, m);
      gb3 += c;
    }
    __syncthreads();
    // dW3
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int e = tid + THREADS * q, k = e / NO, o = e % NO;
      float a = 0.f;
      for (int r = 0; r < ROWS; ++r) a = fmaf(s.H2[r][k], s.dY[r][o], a);
      gW3[q] += a;
    }
    // D = dH2 = (dY W3^T) * (1 - H2^2)
#pragma unroll
    for (int r = 0; r < ROWS / 8; ++r)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int rr = ROWS / 8 * wp + r, c = l + 32 * j;
        float a = 0.f;
#pragma unroll
        for (int o = 0; o < NO; ++o) a = fmaf(s.dY[rr][o], s.W3[c][o], a);
        const float h = s.H2[rr][c];
        s.D[rr][c] = a * (1.f - h * h);
      }
    __syncthreads();
    // dW2[k][j] += sum_r H1[r][k] D[r][j] on the tensor cores: A = H1^T (rows k = 16 wp ..), B = D,
    // both split into two BF16 terms, products hi hi + hi lo + lo hi
#pragma unroll 1
    for (int k0 = 0; k0 < ROWS; k0 += 16) {
      uint32_t ah[4], al[4];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const int m = 16 * wp + g + 8 * (f & 1), kr = k0 + 2 * t + 8 * (f >> 1);
        bf16x2_split2(s.H1[kr][m], s.H1[kr + 1][m], ah[f], al[f]);
      }
#pragma unroll
      for (int nt = 0; nt < 16; ++nt) {
        const int c = 8 * nt + g, kr = k0 + 2 * t;
        uint32_t bh0, bl0, bh1, bl1;
        bf16x2_split2(s.D[kr][c], s.D[kr + 1][c], bh0, bl0);
        bf16x2_split2(s.D[kr + 8][c], s.D[kr + 9][c], bh1, bl1);
        mma_bf16(gW2[nt], al, bh0, bh1);
        mma_bf16(gW2[nt], ah, bl0, bl1);
        mma_bf16(gW2[nt], ah, bh0, bh1);
      }
    }
    if (tid < NW)
#pragma unroll 16
      for (int r = 0; r < ROWS; ++r) gb2 += s.D[r][tid];
    // dH1 = (D W2^T) * (1 - H1^2) on the tensor cores (B = W2 [k][j], K = j contiguous), written
    // over H2 (no longer needed)
    {
      constexpr int NT = WarpTile<ROWS>::NT;
      const int rr = WarpTile<ROWS>::row(wp) + g, c0 = WarpTile<ROWS>::col(wp);
      float acc[NT][4];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[nt][q] = 0.f;
      mma_rows<ROWS, true>(s.D, s.W2, acc);
#pragma unroll
      for (int nt = 0; nt < NT; ++nt) {
        const int c = c0 + 8 * nt + 2 * t;
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
          const int r = rr + 8 * hf;
          const float h0 = s.H1[r][c], h1 = s.H1[r][c + 1];
          *reinterpret_cast<float2*>(&s.H2[r][c]) =
              make_float2(acc[nt][2 * hf] * (1.f - h0 * h0), acc[nt][2 * hf + 1] * (1.f - h1 * h1));
        }
      }
    }
    __syncthreads();
    // dW1[k][j] += sum_r X[r][k] dH1[r][j], db1
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int e = tid + THREADS * q, k = e / NW, j = e % NW;
      float a = 0.f;
      for (int r = 0; r < ROWS; ++r) a = fmaf(s.X[r][k], s.H2[r][j], a);
      gW1[q] += a;
    }
    if (tid < NW)
#pragma unroll 16
      for (int r = 0; r < ROWS; ++r) gb1 += s.H2[r][tid];
  }
  // flush the partials
#pragma unroll
  for (int nt = 0; nt < 16; ++nt)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int k = 16 * wp + g + 8 * q, j = 8 * nt + 2 * t;
      atomicAdd(reinterpret_cast<float2*>(grad + P_W2 + k * NW + j), make_float2(gW2[nt][2 * q], gW2[nt][2 * q + 1]));
    }
#pragma unroll
  for (int q = 0; q < 6; ++q) atomicAdd(grad + P_W1 + tid + THREADS * q, gW1[q]);
#pragma unroll
  for (int q = 0; q < 2; ++q) atomicAdd(grad + P_W3 + tid + THREADS * q, gW3[q]);
  if (tid < NW) {
    atomicAdd(grad + P_B1 + tid, gb1);
    atomicAdd(grad + P_B2 + tid, gb2);
  }
  if (l < NO) atomicAdd(grad + P_B3 + l, gb3);
  for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
  if (l == 0) atomicAdd(loss, lsum * (double)scale);
}

// Adam on every parameter; the BF16 weights and FP32 biases the kernels use are refreshed from
// the master copy. c1 = 1 / (1 - beta1^t), c2 = 1 / (1 - beta2^t).
__global__ void mlp_adam_kernel(float* __restrict__ master, float* __restrict__ m,
                                float* __restrict__ v, const float* __restrict__ grad,
                                __nv_bfloat16* __restrict__ w, float* __restrict__ bias, float lr,
                                float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P_N) return;
  const float g = grad[i];
  const float mi = b1 * m[i] + (1.f - b1) * g;
  const float vi = b2 * v[i] + (1.f - b2) * g * g;
  m[i] = mi;
  v[i] = vi;
  const float x = master[i] - lr * (mi * c1) / (sqrtf(vi * c2) + eps);
  master[i] = x;
  if (i < P_B1) w[WB_1 + i] = __float2bfloat16_rn(x);
  else if (i < P_W2) bias[BB_1 + i - P_B1] = x;
  else if (i < P_B2) w[WB_2 + i - P_W2] = __float2bfloat16_rn(x);
  else if (i < P_W3) bias[BB_2 + i - P_B2] = x;
  else if (i < P_B3) w[WB_3 + i - P_W3] = __float2bfloat16_rn(x);
  else bias[BB_3 + i - P_B3] = x;
}

__global__ void mlp_store_kernel(const float* __restrict__ master, __nv_bfloat16* __restrict__ w,
                                 float* __restrict__ bias) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P_N) return;
  const float x = master[i];
  if (i < P_B1) w[WB_1 + i] = __float2bfloat16_rn(x);
  else if (i < P_W2) bias[BB_1 + i - P_B1] = x;
  else if (i < P_B2) w[WB_2 + i - P_W2] = __float2bfloat16_rn(x);
  else if (i < P_W3) bias[BB_2 + i - P_B2] = x;
  else if (i < P_B3) w[WB_3 + i - P_W3] = __float2bfloat16_rn(x);
  else bias[BB_3 + i - P_B3] = x;
}

__global__ void mlp_stored_kernel(const __nv_bfloat16* __restrict__ w, const float* __restrict__ bias,
                                  float* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= P_N) return;
  float x;
  if (i < P_B1) x = __bfloat162float(w[WB_1 + i]);
  else if (i < P_W2) x = bias[BB_1 + i - P_B1];
  else if (i < P_B2) x = __bfloat162float(w[WB_2 + i - P_W2]);
  else if (i < P_W3) x = bias[BB_2 + i - P_B2];
  else if (i < P_B3) x = __bfloat162float(w[WB_3 + i - P_W3]);
  else x = bias[BB_3 + i - P_B3];
  out[i] = x;
}

unsigned grid_rows(int64_t n, int rows) {
  const int64_t tiles = (n + rows - 1) / rows;
  const int64_t sms = vms::sm_count();
  return (unsigned)(tiles < 1 ? 1 : (tiles > sms ? sms : tiles));
}
// Rows per tile of the gradient kernel: the fewest for which a batch is one round of CTAs. Measured in us with
// 16, 32 and 64 rows: 1,024 rows 16.6, 20.7, 26.9; 2,432 20.7, 20.7, 26.8; 4,864 26.8, 22.7, 28.1; 9,728
// 39.1, 32.9, 30.9 (64 rows with W2 read and transposed two bytes at a time: 31.5, and 36.4 for 9,728).
int grad_rows(int64_t n) {
  const int64_t sms = vms::sm_count();
  return n <= 16 * sms ? 16 : (n <= 32 * sms ? 32 : 64);
}

int mfail(vms_mlp* p, int code, const char* msg) {
  if (p) p->err = msg;
  return code;
}

#define MCK(call)                                                             \
  do {                                                                        \
    cudaError_t e_ = (call);                                                  \
    if (e_ != cudaSuccess)                                                    \
      return mfail(mlp, e_ == cudaErrorMemoryAllocation ? VMS_ERR_OUT_OF_MEMORY \
                                                        : VMS_ERR_CUDA,        \
                   cudaGetErrorString(e_));                                   \
  } while (0)

// Reports, once, a forward pass that has given up by now.
int mlp_status(vms_mlp* mlp) {
  volatile int* s = mlp->status;
  if (*s == 0) return VMS_OK;
  *s = 0;
  return mfail(mlp, VMS_ERR_TIMEOUT, "a forward pass waited longer than its limit: rows of its result are NaN");
}
#define MSTATUS()                            \
  do {                                       \
    if (int s_ = mlp_status(mlp)) return s_; \
  } while (0)

// ---------------------------------------------------------------------------------------------
// node features and increments on a context's state
// ---------------------------------------------------------------------------------------------
struct Scales {
  float in[NI];
  float out[NO];
};

// X[n] = [u^n, u^{n-1}, mean of u^n over the 1-ring] / scale_in; the 1-ring is read from the CSR
// pattern (node row n lists its neighbours, the node itself included)
__global__ void node_features_kernel(const int32_t* __restrict__ rowptr,
                                     const int32_t* __restrict__ colidx,
                                     const double4_32a* __restrict__ u,
                                     const double4_32a* __restrict__ up, int64_t n_nodes,
                                     Scales sc, float* __restrict__ X) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_nodes) return;
  const int32_t r0 = rowptr[4 * i];
  const int deg = (rowptr[4 * i + 1] - r0) >> 2;
  double s[4] = {0.0, 0.0, 0.0, 0.0};
  int cnt = 0;
  for (int k = 0; k < deg; ++k) {
    const int64_t j = colidx[r0 + 4 * k] >> 2;
    if (j == i) continue;
    const double4_32a w = u[j], wp = up[j];
    s[0] += w.x - wp.x; s[1] += w.y - wp.y; s[2] += w.z - wp.z; s[3] += w.w - wp.w;
    ++cnt;
  }
  const double inv = cnt ? 1.0 / cnt : 0.0;
  const double4_32a a = u[i], b = up[i];
  // the last step's increment is given directly: a network with BF16 weights cannot form it from
  // u^n and u^(n-1), which agree in their leading digits
  const double f[NI] = {a.x, a.y, a.z, a.w, a.x - b.x, a.y - b.y, a.z - b.z, a.w - b.w,
                        s[0] * inv, s[1] * inv, s[2] * inv, s[3] * inv};
#pragma unroll
  for (int c = 0; c < NI; ++c) X[i * NI + c] = (float)(f[c] / (double)sc.in[c]);
}

__global__ void node_increment_kernel(const double4_32a* __restrict__ u,
                                      const double4_32a* __restrict__ up, int64_t n_nodes,
                                      Scales sc, float* __restrict__ D) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_nodes) return;
  const double4_32a a = u[i], b = up[i];
  D[4 * i + 0] = (float)((a.x - b.x) / sc.out[0]);
  D[4 * i + 1] = (float)((a.y - b.y) / sc.out[1]);
  D[4 * i + 2] = (float)((a.z - b.z) / sc.out[2]);
  D[4 * i + 3] = (float)((a.w - b.w) / sc.out[3]);
}

__global__ void apply_increment_kernel(double4_32a* __restrict__ u, int64_t n_nodes, Scales sc,
                                       const float* __restrict__ D) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n_nodes) return;
  double4_32a a = u[i];
  a.x += (double)sc.out[0] * D[4 * i + 0];
  a.y += (double)sc.out[1] * D[4 * i + 1];
  a.z += (double)sc.out[2] * D[4 * i + 2];
  a.w += (double)sc.out[3] * D[4 * i + 3];
  u[i] = a;
}

// per-column sums of squares (FP64): each thread accumulates the columns of a grid-stride set of
// rows, the block combines them in shared memory and adds them to sums once
constexpr int COLS_MAX = 16;
struct ColMul {
  float m[COLS_MAX];
};

__global__ void column_sumsq_kernel(const float* __restrict__ X, int64_t n, int cols,
                                    double* __restrict__ sums) {
  __shared__ double part[COLS_MAX];
  if (threadIdx.x < COLS_MAX) part[threadIdx.x] = 0.0;
  __syncthreads();
  double acc[COLS_MAX];
#pragma unroll
  for (int c = 0; c < COLS_MAX; ++c) acc[c] = 0.0;
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x)
#pragma unroll
    for (int c = 0; c < COLS_MAX; ++c)
      if (c < cols) {
        const double x = X[r * cols + c];
        acc[c] += x * x;
      }
  for (int c = 0; c < cols; ++c) {
    double v = acc[c];
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if ((threadIdx.x & 31) == 0) atomicAdd(&part[c], v);
  }
  __syncthreads();
  if (threadIdx.x < cols) atomicAdd(sums + threadIdx.x, part[threadIdx.x]);
}

__global__ void scale_columns_kernel(const float* __restrict__ X, int64_t n, int cols, ColMul mul,
                                     float* __restrict__ out) {
  const int64_t total = n * cols;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = X[i] * mul.m[i % cols];
}

}  // namespace

extern "C" {

int vms_mlp_create(vms_mlp** out, int device) {
  if (!out) return VMS_ERR_INVALID_ARG;
  *out = nullptr;
  vms_mlp* mlp = new vms_mlp();
  mlp->device = device;
  auto cleanup = [&](int rc) { vms_mlp_destroy(mlp); return rc; };
  if (cudaSetDevice(device) != cudaSuccess) return cleanup(VMS_ERR_CUDA);
  cudaError_t e = cudaMalloc(&mlp->master, sizeof(float) * P_N);
  if (e == cudaSuccess) e = cudaMalloc(&mlp->m, sizeof(float) * P_N);
  if (e == cudaSuccess) e = cudaMalloc(&mlp->v, sizeof(float) * P_N);
  if (e == cudaSuccess) e = cudaMalloc(&mlp->grad, GRAD_BYTES);
  if (e == cudaSuccess) e = cudaMallocHost(&mlp->host, HOST_BYTES);
  if (e == cudaSuccess) {
    mlp->status = reinterpret_cast<int*>(reinterpret_cast<char*>(mlp->host) + GRAD_BYTES);
    *mlp->status = 0;
  }
  if (e == cudaSuccess) e = cudaMalloc(&mlp->w, sizeof(__nv_bfloat16) * WB_N);
  if (e == cudaSuccess) e = cudaMalloc(&mlp->bias, sizeof(float) * BB_N);
  mlp->loss = reinterpret_cast<double*>(mlp->grad + P_N);
  if (e == cudaSuccess) e = cudaMalloc(&mlp->scratch, sizeof(float) * P_N);
  if (e == cudaSuccess) e = cudaMalloc(&mlp->colsum, sizeof(double) * 16);
  for (void* p : {(void*)mlp->master, (void*)mlp->m, (void*)mlp->v, (void*)mlp->grad, (void*)mlp->bias})
    if (e == cudaSuccess) e = cudaMemset(p, 0, sizeof(float) * (p == (void*)mlp->bias ? BB_N : P_N));
  if (e == cudaSuccess) e = cudaMemset(mlp->w, 0, sizeof(__nv_bfloat16) * WB_N);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_forward_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmemFwd));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_grad_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmemGrad<16>));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_grad_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmemGrad<32>));
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(mlp_grad_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SmemGrad<64>));
  if (e != cudaSuccess) return cleanup(e == cudaErrorMemoryAllocation ? VMS_ERR_OUT_OF_MEMORY : VMS_ERR_CUDA);
  *out = mlp;
  return VMS_OK;
}

int vms_mlp_destroy(vms_mlp* mlp) {
  if (!mlp) return VMS_OK;
  cudaSetDevice(mlp->device);
  if (mlp->stream) cudaStreamSynchronize(mlp->stream);
  for (void* p : {(void*)mlp->master, (void*)mlp->m, (void*)mlp->v, (void*)mlp->grad, (void*)mlp->w,
                  (void*)mlp->bias, (void*)mlp->scratch, (void*)mlp->colsum})
    if (p) cudaFree(p);
  if (mlp->host) cudaFreeHost(mlp->host);
  delete mlp;
  return VMS_OK;
}

const char* vms_mlp_last_error(vms_mlp* mlp) { return mlp ? mlp->err.c_str() : "null handle"; }

int vms_mlp_set_stream(vms_mlp* mlp, void* stream) {
  if (!mlp) return VMS_ERR_INVALID_ARG;
  mlp->stream = reinterpret_cast<cudaStream_t>(stream);
  return VMS_OK;
}

int vms_mlp_set_params(vms_mlp* mlp, const float* params) {
  if (!mlp || !params) return mfail(mlp, VMS_ERR_INVALID_ARG, "null argument");
  MCK(cudaSetDevice(mlp->device));
  MCK(cudaMemcpyAsync(mlp->master, params, sizeof(float) * P_N, cudaMemcpyDefault, mlp->stream));
  MCK(cudaMemsetAsync(mlp->m, 0, sizeof(float) * P_N, mlp->stream));
  MCK(cudaMemsetAsync(mlp->v, 0, sizeof(float) * P_N, mlp->stream));
  mlp_store_kernel<<<(P_N + 255) / 256, 256, 0, mlp->stream>>>(mlp->master, mlp->w, mlp->bias);
  MCK(cudaGetLastError());
  MCK(cudaStreamSynchronize(mlp->stream));
  mlp->t = 0;
  return VMS_OK;
}

int vms_mlp_get_params(vms_mlp* mlp, float* params, int stored) {
  if (!mlp || !params) return mfail(mlp, VMS_ERR_INVALID_ARG, "null argument");
  MCK(cudaSetDevice(mlp->device));
  if (stored) {
    mlp_stored_kernel<<<(P_N + 255) / 256, 256, 0, mlp->stream>>>(mlp->w, mlp->bias, mlp->scratch);
    MCK(cudaGetLastError());
    MCK(cudaMemcpyAsync(params, mlp->scratch, sizeof(float) * P_N, cudaMemcpyDefault, mlp->stream));
  } else {
    MCK(cudaMemcpyAsync(params, mlp->master, sizeof(float) * P_N, cudaMemcpyDefault, mlp->stream));
  }
  MCK(cudaStreamSynchronize(mlp->stream));
  MSTATUS();
  return VMS_OK;
}

int vms_mlp_set_wait_limit(vms_mlp* mlp, int64_t polls) {
  if (!mlp || polls < 0 || polls > ((int64_t)1 << 30)) return mfail(mlp, VMS_ERR_INVALID_ARG, "wait limit out of range");
  mlp->wait_limit = (uint32_t)polls;
  return VMS_OK;
}

int vms_mlp_forward(vms_mlp* mlp, int64_t n, const float* X, float* Y) {
  if (!mlp || n < 0 || (n > 0 && (!X || !Y))) return mfail(mlp, VMS_ERR_INVALID_ARG, "invalid arguments");
  MSTATUS();
  if (n == 0) return VMS_OK;
  MCK(cudaSetDevice(mlp->device));
  const int64_t tiles = (n + FT - 1) / FT, most = 2 * (int64_t)vms::sm_count();
  mlp_forward_kernel<<<(unsigned)(tiles < most ? tiles : most), THREADS, sizeof(SmemFwd), mlp->stream>>>(
      mlp->w, mlp->bias, X, n, Y, mlp->wait_limit ? mlp->wait_limit : WAIT_DEFAULT, mlp->status);
  MCK(cudaGetLastError());
  return VMS_OK;
}

int vms_mlp_grad(vms_mlp* mlp, int64_t n, const int32_t* rows, const float* X, const float* T,
                 double* loss, float* grads) {
  if (!mlp || n <= 0 || !X || !T) return mfail(mlp, VMS_ERR_INVALID_ARG, "invalid arguments");
  MSTATUS();
  MCK(cudaSetDevice(mlp->device));
  MCK(cudaMemsetAsync(mlp->grad, 0, GRAD_BYTES, mlp->stream));
  const float scale = (float)(1.0 / (4.0 * (double)n));
  auto launch = [&](auto kern, int r, size_t smem) {
    kern<<<grid_rows(n, r), THREADS, smem, mlp->stream>>>(mlp->w, mlp->bias, X, T, rows, n, scale, mlp->grad, mlp->loss);
  };
  const int r = grad_rows(n);
  if (r == 16) launch(mlp_grad_kernel<16>, r, sizeof(SmemGrad<16>));
  else if (r == 32) launch(mlp_grad_kernel<32>, r, sizeof(SmemGrad<32>));
  else launch(mlp_grad_kernel<64>, r, sizeof(SmemGrad<64>));
  MCK(cudaGetLastError());
  if (!loss && !grads) return VMS_OK;
  // To ordinary host memory both go in one copy through the handle's page-locked buffer; a device (or
  // managed) destination is copied to directly.
  cudaPointerAttributes at{};
  const bool host = grads && cudaPointerGetAttributes(&at, grads) == cudaSuccess &&
                    (at.type == cudaMemoryTypeUnregistered || at.type == cudaMemoryTypeHost);
  double* hl = reinterpret_cast<double*>(mlp->host + P_N);
  if (host) {
    MCK(cudaMemcpyAsync(mlp->host, mlp->grad, GRAD_BYTES, cudaMemcpyDeviceToHost, mlp->stream));
  } else {
    if (grads) MCK(cudaMemcpyAsync(grads, mlp->grad, sizeof(float) * P_N, cudaMemcpyDefault, mlp->stream));
    if (loss) MCK(cudaMemcpyAsync(hl, mlp->loss, sizeof(double), cudaMemcpyDeviceToHost, mlp->stream));
  }
  MCK(cudaStreamSynchronize(mlp->stream));
  if (host) std::memcpy(grads, mlp->host, sizeof(float) * P_N);
  if (loss) *loss = *hl;
  MSTATUS();
  return VMS_OK;
}

int vms_mlp_adam(vms_mlp* mlp, float lr) {
  if (!mlp || !(lr > 0.f)) return mfail(mlp, VMS_ERR_INVALID_ARG, "invalid arguments");
  MSTATUS();
  MCK(cudaSetDevice(mlp->device));
  mlp->t += 1;
  const double b1 = 0.9, b2 = 0.999;
  const float c1 = (float)(1.0 / (1.0 - std::pow(b1, mlp->t)));
  const float c2 = (float)(1.0 / (1.0 - std::pow(b2, mlp->t)));
  mlp_adam_kernel<<<(P_N + 255) / 256, 256, 0, mlp->stream>>>(mlp->master, mlp->m, mlp->v, mlp->grad,
                                                              mlp->w, mlp->bias, lr, (float)b1,
                                                              (float)b2, 1e-8f, c1, c2);
  MCK(cudaGetLastError());
  return VMS_OK;
}

int vms_mlp_column_rms(vms_mlp* mlp, int64_t n, int cols, const float* X, double* rms) {
  if (!mlp || n <= 0 || cols < 1 || cols > COLS_MAX || !X || !rms)
    return mfail(mlp, VMS_ERR_INVALID_ARG, "invalid arguments");
  MCK(cudaSetDevice(mlp->device));
  MCK(cudaMemsetAsync(mlp->colsum, 0, sizeof(double) * COLS_MAX, mlp->stream));
  const int64_t blocks = std::min<int64_t>((n + 255) / 256, 4 * (int64_t)vms::sm_count());
  column_sumsq_kernel<<<(unsigned)blocks, 256, 0, mlp->stream>>>(X, n, cols, mlp->colsum);
  MCK(cudaGetLastError());
  double h[COLS_MAX];
  MCK(cudaMemcpyAsync(h, mlp->colsum, sizeof(double) * cols, cudaMemcpyDeviceToHost, mlp->stream));
  MCK(cudaStreamSynchronize(mlp->stream));
  for (int c = 0; c < cols; ++c) rms[c] = std::sqrt(h[c] / (double)n);
  MSTATUS();
  return VMS_OK;
}

int vms_mlp_scale_columns(vms_mlp* mlp, int64_t n, int cols, const float* X, const float* mul,
                          float* out) {
  if (!mlp || n < 0 || cols < 1 || cols > COLS_MAX || !mul || (n > 0 && (!X || !out)))
    return mfail(mlp, VMS_ERR_INVALID_ARG, "invalid arguments");
  if (n == 0) return VMS_OK;
  MCK(cudaSetDevice(mlp->device));
  ColMul m{};
  for (int c = 0; c < cols; ++c) m.m[c] = mul[c];
  const int64_t blocks = std::min<int64_t>((n * cols + 255) / 256, 4 * (int64_t)vms::sm_count());
  scale_columns_kernel<<<(unsigned)blocks, 256, 0, mlp->stream>>>(X, n, cols, m, out);
  MCK(cudaGetLastError());
  return VMS_OK;
}

}  // extern "C"

// ---------------------------------------------------------------------------------------------
// context-side calls of the transient driver
// ---------------------------------------------------------------------------------------------
using namespace vms;

extern "C" {

int vms_node_features(vms_ctx* ctx, const float* scale_in, float* X) {
  if (!ctx || !X) return ctx_fail(ctx, VMS_ERR_INVALID_ARG, "null argument");
  const Mesh& m = ctx_mesh(ctx);
  State& s = ctx_state(ctx);
  if (!s.valid) return ctx_fail(ctx, VMS_ERR_STATE, "no state uploaded");
  Scales sc;
  for (int c = 0; c < NI; ++c) sc.in[c] = scale_in ? scale_in[c] : 1.f;
  for (int c = 0; c < NO; ++c) sc.out[c] = 1.f;
  for (int c = 0; c < NI; ++c)
    if (!(sc.in[c] != 0.f)) return ctx_fail(ctx, VMS_ERR_INVALID_ARG, "zero feature scale");
  cudaSetDevice(ctx_device(ctx));
  const unsigned blocks = (unsigned)((m.n_nodes + 255) / 256);
  node_features_kernel<<<blocks, 256, 0, ctx_stream(ctx)>>>(m.rowptr, m.colidx, s.u, s.u_prev,
                                                              m.n_nodes, sc, X);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? VMS_OK : ctx_fail(ctx, VMS_ERR_CUDA, cudaGetErrorString(e));
}

int vms_node_increment(vms_ctx* ctx, const float* scale_out, float* D) {
  if (!ctx || !D) return ctx_fail(ctx, VMS_ERR_INVALID_ARG, "null argument");
  const Mesh& m = ctx_mesh(ctx);
  State& s = ctx_state(ctx);
  if (!s.valid) return ctx_fail(ctx, VMS_ERR_STATE, "no state uploaded");
  Scales sc;
  for (int c = 0; c < NO; ++c) sc.out[c] = scale_out ? scale_out[c] : 1.f;
  for (int c = 0; c < NO; ++c)
    if (!(sc.out[c] != 0.f)) return ctx_fail(ctx, VMS_ERR_INVALID_ARG, "zero output scale");
  cudaSetDevice(ctx_device(ctx));
  const unsigned blocks = (unsigned)((m.n_nodes + 255) / 256);
  node_increment_kernel<<<blocks, 256, 0, ctx_stream(ctx)>>>(s.u, s.u_prev, m.n_nodes, sc, D);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? VMS_OK : ctx_fail(ctx, VMS_ERR_CUDA, cudaGetErrorString(e));
}

int vms_apply_increment(vms_ctx* ctx, const float* scale_out, const float* D) {
  if (!ctx || !D) return ctx_fail(ctx, VMS_ERR_INVALID_ARG, "null argument");
  const Mesh& m = ctx_mesh(ctx);
  State& s = ctx_state(ctx);
  if (!s.valid) return ctx_fail(ctx, VMS_ERR_STATE, "no state uploaded");
  Scales sc;
  for (int c = 0; c < NO; ++c) sc.out[c] = scale_out ? scale_out[c] : 1.f;
  cudaSetDevice(ctx_device(ctx));
  const unsigned blocks = (unsigned)((m.n_nodes + 255) / 256);
  apply_increment_kernel<<<blocks, 256, 0, ctx_stream(ctx)>>>(s.u, m.n_nodes, sc, D);
  launch_impose(m, s.u, ctx_stream(ctx));
  ctx_work(ctx).assembled = false;
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? VMS_OK : ctx_fail(ctx, VMS_ERR_CUDA, cudaGetErrorString(e));
}

int vms_shift_time(vms_ctx* ctx) {
  if (!ctx) return VMS_ERR_INVALID_ARG;
  const Mesh& m = ctx_mesh(ctx);
  State& s = ctx_state(ctx);
  if (!s.valid) return ctx_fail(ctx, VMS_ERR_STATE, "no state uploaded");
  cudaSetDevice(ctx_device(ctx));
  const cudaError_t e = cudaMemcpyAsync(s.u_prev, s.u, sizeof(double4_32a) * m.n_nodes,
                                        cudaMemcpyDeviceToDevice, ctx_stream(ctx));
  ctx_work(ctx).assembled = false;
  return e == cudaSuccess ? VMS_OK : ctx_fail(ctx, VMS_ERR_CUDA, cudaGetErrorString(e));
}

}  // extern "C"
