// Capacity predictor: a small FP32 MLP (n_in -> hidden x layers -> n_out, ReLU)
// trained with a pinball (quantile) loss and Adam, plus the capacity sizing
// that turns its prediction into per-model slab capacities. The paper has no
// learned component; its Section 4 notes that the maximum number of agents
// must be known in advance, which is what this predicts.
//
// Everything is plain FP32 FFMA with shared-memory tiles: the matrices are at
// most 128 wide, so tensor cores would idle on the operand staging (and TF32
// would drop mantissa bits that the FP32 interface keeps).
//
// Nets whose weights fit one CTA's shared memory (hidden and input width up to
// 128, outputs up to 8: every capacity predictor) run fused: k_rows takes a
// slab of rows through all layers and back, k_wgrad turns the activations it
// leaves into weight gradients and applies Adam. Wider nets take one GEMM per
// matrix product (k_gemm).
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "common.cuh"

namespace abm {

constexpr int kGT = 64;   // GEMM tile (rows and columns)
constexpr int kGK = 16;   // GEMM k-step
constexpr int kGThreads = 256;

// C[m][n] (+)= sum_k opA(m,k) * opB(k,n), with opA(m,k) = TA ? A[k*lda + m] : A[m*lda + k]
// and opB(k,n) = TB ? B[n*ldb + k] : B[k*ldb + n]. Epilogue: + bias[n], ReLU,
// or multiply by (mask[m*ldm + n] > 0). Rows of A may be gathered through an
// affine permutation of [0, rows): row(m) = (pa * (m0 + m) + pc) % rows.
struct GemmArgs {
  int M, N, K;
  const float* A;
  int lda;
  const float* B;
  int ldb;
  float* C;
  int ldc;
  const float* bias;
  const float* mask;
  int ldm;
  int relu;
  // optional row gather of A (only when !TA): 0 = none
  long long gather_rows, gather_a, gather_c, gather_m0;
  // split-K: grid.z slices of K, each writing its own C slice (C + z * split_stride)
  int k_per_split;
  long long split_stride;
};

template <bool TA, bool TB>
__global__ void __launch_bounds__(kGThreads) k_gemm(GemmArgs g) {
  __shared__ float sA[kGK][kGT + 4];
  __shared__ float sB[kGK][kGT + 4];
  const int m0 = blockIdx.y * kGT, n0 = blockIdx.x * kGT;
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;  // 16 x 16 threads, 4 x 4 outputs each
  const int kbeg = blockIdx.z * g.k_per_split;
  const int kend = min(g.K, kbeg + g.k_per_split);
  float acc[4][4] = {};
  for (int k0 = kbeg; k0 < kend; k0 += kGK) {
    // stage A tile (kGK x kGT) and B tile (kGK x kGT)
    for (int i = threadIdx.x; i < kGK * kGT; i += kGThreads) {
      const int kk = i / kGT, mm = i % kGT;
      const int m = m0 + mm, k = k0 + kk;
      float va = 0.f;
      if (m < g.M && k < kend) {
        if (TA) {
          va = g.A[(size_t)k * g.lda + m];
        } else {
          long long row = m;
          if (g.gather_rows) row = (g.gather_a * (g.gather_m0 + m) + g.gather_c) % g.gather_rows;
          va = g.A[(size_t)row * g.lda + k];
        }
      }
      sA[kk][mm] = va;
      const int n = n0 + mm;
      float vb = 0.f;
      if (n < g.N && k < kend) vb = TB ? g.B[(size_t)n * g.ldb + k] : g.B[(size_t)k * g.ldb + n];
      sB[kk][mm] = vb;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < kGK; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = sA[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = sB[kk][tx * 4 + j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  float* C = g.C + (size_t)blockIdx.z * g.split_stride;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int m = m0 + ty * 4 + i;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n >= g.N) continue;
      float v = acc[i][j];
      if (g.bias) v += g.bias[n];
      if (g.relu) v = fmaxf(v, 0.f);
      if (g.mask && !(g.mask[(size_t)m * g.ldm + n] > 0.f)) v = 0.f;
      C[(size_t)m * g.ldc + n] = v;
    }
  }
}

// out[i] = sum over z of part[z * stride + i] (fixed order: deterministic)
__global__ void k_sum_splits(const float* part, int nsplit, long long stride, int n, float* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    float s = 0.f;
    for (int z = 0; z < nsplit; ++z) s += part[(size_t)z * stride + i];
    out[i] = s;
  }
}

// column sums of a [rows x cols] matrix, one thread per column, fixed order
__global__ void k_colsum(const float* d, int rows, int cols, float* out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  float s = 0.f;
  for (int r = 0; r < rows; ++r) s += d[(size_t)r * cols + c];
  out[c] = s;
}

// pinball loss at quantile tau: e = y - yhat, loss = max(tau e, (tau - 1) e),
// averaged over all entries; dyhat = d loss / d yhat. Targets are gathered
// with the same row permutation as the inputs.
__global__ void k_pinball(const float* yhat, const float* y, int B, int n_out, float tau, long long grows,
                          long long ga, long long gc, long long gm0, float* dyhat, float* loss_part) {
  __shared__ float s[256];
  float acc = 0.f;
  const float scale = 1.f / (float)(B * n_out);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B * n_out; i += gridDim.x * blockDim.x) {
    const int r = i / n_out, o = i % n_out;
    long long row = r;
    if (grows) row = (ga * (gm0 + r) + gc) % grows;
    const float e = y[(size_t)row * n_out + o] - yhat[i];
    acc += e > 0.f ? tau * e : (tau - 1.f) * e;
    dyhat[i] = (e > 0.f ? -tau : 1.f - tau) * scale;
  }
  s[threadIdx.x] = acc;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) loss_part[blockIdx.x] = s[0];
}

__global__ void k_loss_final(const float* part, int n, float scale, float* out) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    float s = 0.f;
    for (int i = 0; i < n; ++i) s += part[i];
    *out = s * scale;
  }
}

// Adam (Kingma & Ba, 2015) with bias correction
__global__ void k_adam(float* p, const float* g, float* m, float* v, int n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / c1, vh = vi / c2;
    p[i] -= lr * mh / (sqrtf(vh) + eps);
  }
}

// He-uniform initialisation from Philox: W ~ U(-sqrt(6/fan_in), +sqrt(6/fan_in)), b = 0
__global__ void k_mlp_init(float* p, long long n, const long long* off, const int* fan_in, int nlayers, u32 seed) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    int l = 0;
    while (l + 1 < 2 * nlayers && off[l + 1] <= i) ++l;
    if (l & 1) {  // bias block
      p[i] = 0.f;
    } else {
      const u32 u = draw(seed, 0x4D4C50u, (u32)(i >> 32), (u32)i, 15u, (u32)l);
      const float r = ((float)(u >> 8) + 0.5f) * (1.f / 16777216.f);  // (0, 1)
      const float lim = sqrtf(6.f / (float)fan_in[l >> 1]);
      p[i] = (2.f * r - 1.f) * lim;
    }
  }
}

// ---------------------------------------------------------------------------
// Fused path. A training step is two launches instead of 23: the layers are so
// small (0.2 GFLOP a step at 1024 rows of the 12-128-128-128-2 predictor) that
// the chain of separate kernels costs launches and drained pipelines, not
// arithmetic.
//
// Between the two kernels (and for the backward pass) activations and their
// gradients live in row-slab blocks: layer l's block is [slab][unit][R], R rows
// of one unit contiguous, the same image that k_rows keeps in shared memory,
// so that both kernels move it in whole 16-byte runs and k_wgrad reads four
// rows of a unit per load.
constexpr int kMaxLin = 9;       // linear maps: up to 8 hidden layers + the output
constexpr int kFusedWidth = 128; // widest layer of the fused path
constexpr int kFusedOut = 8;     // most outputs
constexpr int kRowThreads = 512;
constexpr int kTrainRows = 8;    // rows of a training slab
constexpr int kLd = 132;         // row stride of weights, gradients and partial sums: 4 words past 128, so that rows
                                 // that are read side by side fall into different banks

struct FusedNet {
  int nlin;
  int din[kMaxLin], dout[kMaxLin];
  int offW[kMaxLin], offb[kMaxLin];      // in the flat parameters
  int sW[kMaxLin], sB[kMaxLin];          // shared memory: weights [din][kLd] (columns past dout zero; the output
                                         // layer's [din][kFusedOut]), biases
  int sA[kMaxLin];                       // shared memory: activations, (x, x) pairs [width][R]
  int sD, sRed;                          // shared memory: gradients [R][kLd], partial sums [splits][R][kLd]
  long long offA[kMaxLin + 1];           // global row-slab blocks
  int nparams;
};

struct RowArgs {
  FusedNet net;
  const float* p;
  const float* x;
  const float* y;   // training: targets
  float* act;       // training: activations for k_wgrad
  float* dact;      // training: gradients of the layers' outputs
  float* out;       // forward: yhat
  float* lossp;     // training: one partial sum per CTA
  int B;
  float tau, scale;
  long long grows, ga, gc, gm0;  // row permutation (grows = 0: none)
};

// two FP32 FMAs in one instruction (each rounded as fmaf)
typedef unsigned long long f32x2;
__device__ __forceinline__ void fma2(f32x2& c, f32x2 a, f32x2 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
__device__ __forceinline__ float2 split2(f32x2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}

// One CTA takes R rows at a time through the net, weights resident in shared
// memory. Bound by instruction issue (a step at 1024 rows is 8 rows per CTA),
// so the inner loops are packed FMAs on operands that need no shuffling:
// forward, a thread's tile is 4 columns x 4 rows, two columns to a packed FMA,
// and activations are kept twice over ((x, x) pairs); backward, it is 4 inputs x
// 4 rows, even and odd outputs in the two halves, from gradients kept row by
// row. The threads left over split the sum over the inputs (outputs), and the
// partial sums meet in shared memory (fixed order: the result does not depend
// on the launch). Weight rows are 132 words apart whatever the layer's width
// (constant offsets; the backward pass, whose lanes walk the rows, reads 16 bytes
// per lane without bank conflicts).
// R: 8 rows give every SM work at the usual batch of 1024; inference takes 16 once
// there are more than 16 rows per SM. One step at 1024 rows of the 12-128-128-128-2
// net: scalar FMAs and strides by width 16.5 us, this 13.3 (of 26,000 cycles the weights take
// 5,900, 24 bytes a cycle and SM: what L2 delivers to 128 SMs at once; the rest is twelve
// dependent stages). Inference of 16384 rows 54 us.
template <int R, bool TRAIN>
__global__ void __launch_bounds__(kRowThreads, 1) k_rows(const __grid_constant__ RowArgs a) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float s_loss[R * kFusedOut];
  __shared__ float s_dout[kFusedOut * R];       // d loss / d yhat, [output][R]
  constexpr int NT = kRowThreads;
  constexpr int RG = R / 4;                     // row groups of a tile row
  constexpr int KS = NT / (32 * RG);            // splits of a sum
  const FusedNet& net = a.net;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int L = net.nlin, n_in = net.din[0], n_out = net.dout[L - 1];
  griddep_wait();  // the parameters (and, on a reused handle, the blocks) belong to the previous launch until here
  for (int l = 0; l < L; ++l) {
    const int din = net.din[l], dout = net.dout[l];
    const float* W = a.p + net.offW[l];
    float* s = sm + net.sW[l];
    if (l == L - 1) {  // [din][kFusedOut]
      for (int i = tid; i < din * dout; i += NT) cp_async4(s + (i / dout) * kFusedOut + i % dout, W + i);
    } else if ((dout & 3) == 0 && (net.offW[l] & 3) == 0) {  // a warp per row
      if (4 * lane < dout)
        for (int k = warp; k < din; k += NT / 32) cp_async16(s + k * kLd + 4 * lane, W + k * dout + 4 * lane);
    } else {
      for (int k = warp; k < din; k += NT / 32)
        for (int c = lane; c < ((dout + 3) & ~3); c += 32)
          if (c < dout) cp_async4(s + k * kLd + c, W + k * dout + c);
          else s[k * kLd + c] = 0.f;
    }
    for (int i = tid; i < dout; i += NT) cp_async4(sm + net.sB[l] + i, a.p + net.offb[l] + i);
  }
  cp_async_commit();
  float* const red = sm + net.sRed;
  float* const drow = sm + net.sD;  // gradients of the current layer's outputs, [R][kLd]
  const int rg = warp % RG, ks = warp / RG;
  const int nslab = (a.B + R - 1) / R;
  float loss = 0.f;
  // inference: the next slab's inputs are fetched beside this one's layers
  constexpr int NX = TRAIN ? 1 : kFusedWidth * R / NT;
  float xn[NX] = {};
  const auto fetch = [&](int slab) {
#pragma unroll
    for (int j = 0; j < NX; ++j) {
      const int i = tid + j * NT, r = i % R, k = i / R;
      const long long row = (long long)slab * R + r;
      xn[j] = k < n_in && row < a.B ? a.x[(size_t)row * n_in + k] : 0.f;
    }
  };
  if (!TRAIN) fetch(blockIdx.x);
  for (int slab = blockIdx.x; slab < nslab; slab += gridDim.x) {
    const int r0 = slab * R;
    const int nr = min(R, a.B - r0);  // rows of this slab; the others stay zero in every block
    float2* const s = reinterpret_cast<float2*>(sm + net.sA[0]);
    float target = 0.f;  // training: y of the (row, output) whose loss this thread takes
    if (TRAIN) {
      const auto source = [&](int r) -> long long {  // the row of the data set that is row r of the slab
        const long long row = r0 + r;
        return a.grows ? (a.ga * (a.gm0 + row) + a.gc) % a.grows : row;
      };
      if (tid < R * n_out && tid % R < nr) target = a.y[(size_t)source(tid % R) * n_out + tid / R];
      float* out = a.act + net.offA[0] + (long long)slab * n_in * R;
      for (int i = tid; i < n_in * R; i += NT) {
        const int r = i % R, k = i / R;
        const float v = r < nr ? a.x[(size_t)source(r) * n_in + k] : 0.f;
        s[i] = make_float2(v, v);
        out[i] = v;
      }
    } else {
#pragma unroll
      for (int j = 0; j < NX; ++j)
        if (tid + j * NT < n_in * R) s[tid + j * NT] = make_float2(xn[j], xn[j]);
      fetch(slab + gridDim.x);
    }
    cp_async_wait_0();
    __syncthreads();
    // forward through the hidden layers
    for (int l = 0; l + 1 < L; ++l) {
      const int din = net.din[l], dout = net.dout[l];
      if (4 * lane < dout) {
        const int per = (din + KS - 1) / KS, k0 = ks * per, n = min(din - k0, per);
        const float* W = sm + net.sW[l] + k0 * kLd + 4 * lane;
        const float* X = sm + net.sA[l] + 2 * (k0 * R + 4 * rg);
        f32x2 acc[4][2] = {};
#pragma unroll 4
        for (int k = 0; k < n; ++k) {
          const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(W + k * kLd);
          const ulonglong2 xa = *reinterpret_cast<const ulonglong2*>(X + k * (2 * R));
          const ulonglong2 xb = *reinterpret_cast<const ulonglong2*>(X + k * (2 * R) + 4);
          fma2(acc[0][0], xa.x, w.x);
          fma2(acc[0][1], xa.x, w.y);
          fma2(acc[1][0], xa.y, w.x);
          fma2(acc[1][1], xa.y, w.y);
          fma2(acc[2][0], xb.x, w.x);
          fma2(acc[2][1], xb.x, w.y);
          fma2(acc[3][0], xb.y, w.x);
          fma2(acc[3][1], xb.y, w.y);
        }
        float* o = red + (ks * R + 4 * rg) * kLd + 4 * lane;
#pragma unroll
        for (int r = 0; r < 4; ++r) *reinterpret_cast<ulonglong2*>(o + r * kLd) = make_ulonglong2(acc[r][0], acc[r][1]);
      }
      __syncthreads();
      float2* Y = reinterpret_cast<float2*>(sm + net.sA[l + 1]);
      float* out = TRAIN ? a.act + net.offA[l + 1] + (long long)slab * dout * R : nullptr;
      const float* bias = sm + net.sB[l];
      for (int i = tid; i < dout * R; i += NT) {
        const int r = i % R, c = i / R;
        const float* p = red + r * kLd + c;
        float v = 0.f;
#pragma unroll
        for (int z = 0; z < KS; ++z) v += p[z * R * kLd];
        v = r < nr ? fmaxf(v + bias[c], 0.f) : 0.f;
        Y[i] = make_float2(v, v);
        if (TRAIN) out[i] = v;
      }
      __syncthreads();
    }
    // output layer: the inputs split over the warps, and over a warp's 32 / R lanes of a row; the partial sums of the
    // warps meet in `red`. (A warp per row and output, lanes over the inputs, read the activations R banks apart.)
    {
      const int l = L - 1, din = net.din[l], r = lane % R;
      const float* W = sm + net.sW[l];
      const float* X = sm + net.sA[l];
      const int per = (din + NT / 32 - 1) / (NT / 32), k0 = warp * per, k1 = min(din, k0 + per);
      for (int o = 0; o < n_out; ++o) {
        float v = 0.f;
        for (int k = k0 + lane / R; k < k1; k += 32 / R) v = fmaf(X[2 * (k * R + r)], W[k * kFusedOut + o], v);
#pragma unroll
        for (int m = R; m < 32; m <<= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, m);
        if (lane < R) red[(warp * kFusedOut + o) * R + r] = v;
      }
    }
    __syncthreads();
    if (tid < R * n_out) {
      const int r = tid % R, o = tid / R;
      float v = 0.f;
#pragma unroll
      for (int z = 0; z < NT / 32; ++z) v += red[(z * kFusedOut + o) * R + r];
      v += sm[net.sB[L - 1] + o];
      if (!TRAIN) {
        if (r < nr) a.out[(size_t)(r0 + r) * n_out + o] = v;
      } else {
        // pinball loss at quantile tau: e = y - yhat, max(tau e, (tau - 1) e), averaged over all entries
        float d = 0.f, le = 0.f;
        if (r < nr) {
          const float er = target - v;
          le = er > 0.f ? a.tau * er : (a.tau - 1.f) * er;
          d = (er > 0.f ? -a.tau : 1.f - a.tau) * a.scale;
        }
        s_loss[tid] = le;
        s_dout[tid] = d;
        a.dact[net.offA[L] + (long long)slab * n_out * R + tid] = d;
      }
    }
    if (!TRAIN) continue;  // (`red` is written again behind the next slab's first barrier)
    __syncthreads();
    if (warp == 0) {
      float v = 0.f;
      for (int e = lane; e < R * n_out; e += 32) v += s_loss[e];
#pragma unroll
      for (int m = 16; m > 0; m >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, m);
      loss += v;
    }
    // backward: the gradients of layer l's input, from those of its outputs (drow; s_dout for the output layer)
    for (int l = L - 1; l > 0; --l) {
      const int din = net.din[l], dout = net.dout[l];
      const float2* X = reinterpret_cast<const float2*>(sm + net.sA[l]);
      float* dst = a.dact + net.offA[l] + (long long)slab * din * R;
      if (l == L - 1) {  // at most 8 outputs: one thread per (input, row)
        const float* W = sm + net.sW[l];
        for (int i = tid; i < din * R; i += NT) {
          const int r = i % R, k = i / R;
          float v = 0.f;
          for (int o = 0; o < dout; ++o) v = fmaf(s_dout[o * R + r], W[k * kFusedOut + o], v);
          v = X[i].x > 0.f ? v : 0.f;
          drow[r * kLd + k] = v;
          dst[i] = v;
        }
        // columns up to the next multiple of 4, which the next layer down reads against zero weights
        if (tid < R)
          for (int k = din; k < ((din + 3) & ~3); ++k) drow[tid * kLd + k] = 0.f;
        __syncthreads();
        continue;
      }
      // lanes take the inputs lane, lane + 32, ...; the outputs are taken four at a time and split over the warps
      {
        const int nq = (dout + 3) >> 2, per = (nq + KS - 1) / KS, q0 = ks * per, n = min(nq - q0, per);
        const float* W[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) W[i] = sm + net.sW[l] + min(lane + 32 * i, din - 1) * kLd + 4 * q0;
        const float* D = drow + 4 * rg * kLd + 4 * q0;
        f32x2 acc[4][4] = {};  // [input][row]: even | odd outputs
#pragma unroll 2
        for (int q = 0; q < n; ++q) {
          ulonglong2 d[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) d[r] = *reinterpret_cast<const ulonglong2*>(D + r * kLd + 4 * q);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const ulonglong2 w = *reinterpret_cast<const ulonglong2*>(W[i] + 4 * q);
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              fma2(acc[i][r], d[r].x, w.x);
              fma2(acc[i][r], d[r].y, w.y);
            }
          }
        }
        float* o = red + (ks * R + 4 * rg) * kLd + lane;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (lane + 32 * i < din)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              const float2 v = split2(acc[i][r]);
              o[r * kLd + 32 * i] = v.x + v.y;
            }
      }
      __syncthreads();
      for (int i = tid; i < din * R; i += NT) {
        const int r = i % R, k = i / R;
        const float* p = red + r * kLd + k;
        float v = 0.f;
#pragma unroll
        for (int z = 0; z < KS; ++z) v += p[z * R * kLd];
        v = X[i].x > 0.f ? v : 0.f;
        drow[r * kLd + k] = v;
        dst[i] = v;
      }
      if (tid < R)
        for (int k = din; k < ((din + 3) & ~3); ++k) drow[tid * kLd + k] = 0.f;
      __syncthreads();
    }
  }
  if (TRAIN && tid == 0) a.lossp[blockIdx.x] = loss;
}

struct WgradArgs {
  FusedNet net;
  const float* act;
  const float* dact;
  float *g, *p, *m, *v;
  int nslab, slabs_per_split;
  const float* lossp;
  int nloss;
  float loss_scale;
  float* loss_out;  // nullable
  int adam;
  float lr, b1, b2, eps, c1, c2;
};

constexpr int kWT = 32;         // inputs and outputs of a weight-gradient tile
constexpr int kWRows = 128;     // rows staged at a time
constexpr int kWThreads = 256;
constexpr int kMaxRuns = 8;     // runs of rows = CTAs of a cluster (the portable size), at most

__host__ __device__ inline int wgrad_tiles(const FusedNet& net, int l) {
  return ((net.din[l] + kWT - 1) / kWT) * ((net.dout[l] + kWT - 1) / kWT);
}

// Weight gradients X^T dY of every layer in one launch: a cluster owns a 32 x
// 32 tile of one layer's gradient, its CTAs a run of rows each. 64 threads cover
// the tile with 4 x 4 outputs each and four such groups take a quarter of the
// staged rows each (128 rows a stage: 32 KB of shared memory). The tiles of the
// first inputs also sum the bias gradients. The CTAs' tiles meet in distributed
// shared memory: after one cluster barrier each CTA adds up its share of the
// tile in run order (so the sums do not depend on timing) and applies Adam to
// those parameters. (Partial tiles in global memory, added by the last CTA to
// finish, took 15.9 us a step at 1024 rows; this 8.8.)
constexpr int kTileEntries = kWT * kWT + kWT;  // the tile and, below it, the bias row

__global__ void __launch_bounds__(kWThreads) k_wgrad(const __grid_constant__ WgradArgs a) {
  __shared__ __align__(16) float s_x[kWRows / 4][kWT][4];   // [row quad][unit][row]
  __shared__ __align__(16) float s_d[kWRows / 4][kWT][4];
  __shared__ float s_b[8][kWT];
  __shared__ float s_sum[kTileEntries];
  const FusedNet& net = a.net;
  const int tid = threadIdx.x;
  int l = 0, tile = blockIdx.x;
  while (tile >= wgrad_tiles(net, l)) tile -= wgrad_tiles(net, l++);
  const int din = net.din[l], dout = net.dout[l];
  const int tn = (dout + kWT - 1) / kWT;
  const int k0 = (tile / tn) * kWT, n0 = (tile % tn) * kWT;
  const int nk = min(kWT, din - k0), nn = min(kWT, dout - n0);
  const int s0 = blockIdx.y * a.slabs_per_split, s1 = min(a.nslab, s0 + a.slabs_per_split);
  constexpr int R = kTrainRows;
  constexpr int SS = kWRows / R;  // slabs per stage
  constexpr int RQ = R / 4;
  const int grp = tid >> 6, kg = (tid & 63) >> 3, ng = tid & 7;
  float acc[4][4] = {}, bacc = 0.f;
  griddep_wait();
  const float* X = a.act + net.offA[l];
  const float* D = a.dact + net.offA[l + 1];
  for (int s = s0; s < s1; s += SS) {
    // [slab][unit][R] -> [row quad][unit][4]; missing units and slabs are zero
#pragma unroll
    for (int i = tid; i < SS * kWT * RQ; i += kWThreads) {
      const int q = i % RQ, u = (i / RQ) % kWT, j = i / (RQ * kWT);
      float4 x = make_float4(0.f, 0.f, 0.f, 0.f), d = x;
      if (s + j < s1) {
        if (u < nk) x = *reinterpret_cast<const float4*>(X + ((long long)(s + j) * din + k0 + u) * R + 4 * q);
        if (u < nn) d = *reinterpret_cast<const float4*>(D + ((long long)(s + j) * dout + n0 + u) * R + 4 * q);
      }
      *reinterpret_cast<float4*>(s_x[j * RQ + q][u]) = x;
      *reinterpret_cast<float4*>(s_d[j * RQ + q][u]) = d;
    }
    __syncthreads();
#pragma unroll 2
    for (int q = 8 * grp; q < 8 * grp + 8; ++q) {
      float4 x[4], d[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float4*>(s_x[q][kg + 8 * i]);
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] = *reinterpret_cast<const float4*>(s_d[q][ng + 8 * i]);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fmaf(x[i].x, d[j].x, acc[i][j]);
          acc[i][j] = fmaf(x[i].y, d[j].y, acc[i][j]);
          acc[i][j] = fmaf(x[i].z, d[j].z, acc[i][j]);
          acc[i][j] = fmaf(x[i].w, d[j].w, acc[i][j]);
        }
    }
    if (k0 == 0) {  // bias: output tid % 32, every eighth quad
#pragma unroll
      for (int q = tid >> 5; q < kWRows / 4; q += 8) {
        const float4 d = *reinterpret_cast<const float4*>(s_d[q][tid & 31]);
        bacc += (d.x + d.y) + (d.z + d.w);
      }
    }
    __syncthreads();
  }
  // the four row groups' tiles meet in shared memory (the staging arrays, 1024 floats each)
  float* s_t = &s_x[0][0][0];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) s_t[grp * kWT * kWT + (kg + 8 * i) * kWT + ng + 8 * j] = acc[i][j];
  s_b[tid >> 5][tid & 31] = bacc;
  __syncthreads();
#pragma unroll
  for (int i = tid; i < kWT * kWT; i += kWThreads)
    s_sum[i] = (s_t[i] + s_t[i + kWT * kWT]) + (s_t[i + 2 * kWT * kWT] + s_t[i + 3 * kWT * kWT]);
  if (tid < kWT) {
    float b = 0.f;
#pragma unroll
    for (int z = 0; z < 8; ++z) b += s_b[z][tid];
    s_sum[kWT * kWT + tid] = b;
  }
  const int S = gridDim.y;  // = the cluster's CTAs
  cluster_arrive();
  cluster_wait();
  // this CTA's share of the tile's entries
  const int entries = k0 == 0 ? kTileEntries : kWT * kWT;
  const int share = (entries + S - 1) / S;
  const int e0 = blockIdx.y * share, e1 = min(entries, e0 + share);
  for (int i = e0 + tid; i < e1; i += kWThreads) {
    const int k = i / kWT, n = i % kWT;  // k = 32: the bias row
    if (n >= nn || (k < kWT && k >= nk)) continue;
    const int e = k < kWT ? net.offW[l] + (k0 + k) * dout + n0 + n : net.offb[l] + n0 + n;
    float v[kMaxRuns];
#pragma unroll
    for (int z = 0; z < kMaxRuns; ++z) v[z] = z < S ? ld_cluster_f32(&s_sum[i], (u32)z) : 0.f;
    float gi = 0.f;
#pragma unroll
    for (int z = 0; z < kMaxRuns; ++z) gi += v[z];
    a.g[e] = gi;
    if (a.adam) {  // Adam (Kingma & Ba, 2015) with bias correction
      const float mi = a.b1 * a.m[e] + (1.f - a.b1) * gi;
      const float vi = a.b2 * a.v[e] + (1.f - a.b2) * gi * gi;
      a.m[e] = mi;
      a.v[e] = vi;
      a.p[e] -= a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
    }
  }
  if (blockIdx.x == 0 && blockIdx.y == 0 && a.loss_out && tid < 32) {
    float v = 0.f;
    for (int i = tid; i < a.nloss; i += 32) v += a.lossp[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    if (tid == 0) *a.loss_out = v * a.loss_scale;
  }
  cluster_arrive();  // no CTA leaves while another reads its sums
  cluster_wait();
}

// features of a model: log1p(side), log1p(n0 sheep), log1p(n0 wolves), the 8
// rule params over their nominal values, horizon / 500
__global__ void k_features(const int32_t* tab, int B, const int32_t* nominal, float* x) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B; i += gridDim.x * blockDim.x) {
    const int32_t* t = tab + (size_t)i * 12;
    float* o = x + (size_t)i * 12;
    o[0] = log1pf((float)t[0]);
    o[1] = log1pf((float)t[1]);
    o[2] = log1pf((float)t[2]);
    for (int j = 0; j < 8; ++j) o[3 + j] = (float)(u32)t[3 + j] / (float)(u32)nominal[j];
    o[11] = (float)t[11] / 500.f;
  }
}

// capacity from a predicted log peak: min(cap_max, roundup(ceil(exp(yhat) * (1 + margin)), round_to)),
// never below the initial population and never below round_to
__global__ void k_capacity(const float* yhat, int B, float margin, int round_to, const int32_t* cap_max,
                           const int32_t* n0, int32_t* cap) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < 2 * B; i += gridDim.x * blockDim.x) {
    const double want = ceil(exp((double)yhat[i]) * (1.0 + (double)margin));
    long long c = (long long)fmin(want, 2147483647.0);
    if (c < n0[i]) c = n0[i];
    c = ((c + round_to - 1) / round_to) * round_to;
    if (c < round_to) c = round_to;
    if (c > cap_max[i]) c = cap_max[i];
    cap[i] = (int32_t)c;
  }
}

}  // namespace abm

// ============================================================================
using namespace abm;

struct abm_mlp {
  int n_in, hidden, layers, n_out, max_batch;  // layers = hidden layers
  int nlin;                                    // linear maps = layers + 1
  std::vector<int> din, dout;
  std::vector<long long> offW, offb;
  long long nparams;
  float *p, *g, *m, *v;
  float* act;    // activations: [nlin + 1] blocks of max_batch x width
  std::vector<long long> offA;
  float* dact;   // gradients of activations, same layout
  float* part;   // split-K partials
  float* lossp;  // loss partial sums
  long long* d_off;
  int* d_fan;
  int adam_t;
  // fused path (fused = 0: a GEMM per product)
  int fused;
  FusedNet net;          // shared-memory offsets filled in per launch shape
};

static void mlp_free(abm_mlp* n) {
  cudaFree(n->p);
  cudaFree(n->g);
  cudaFree(n->m);
  cudaFree(n->v);
  cudaFree(n->act);
  cudaFree(n->dact);
  cudaFree(n->part);
  cudaFree(n->lossp);
  cudaFree(n->d_off);
  cudaFree(n->d_fan);
  delete n;
}

static const int kSplits = 32;
constexpr size_t kMaxSmem = 227 * 1024 - 2048;  // dynamic shared memory of a CTA, less the static arrays

// Shared-memory layout of k_rows<R, train>: weights, biases, activations
// (training keeps every layer's, inference two that take turns), partial sums.
// Returns the bytes.
static size_t fused_layout(FusedNet& f, int R, bool train) {
  int at = 0;
  const auto take = [&](int n) {
    const int o = at;
    at += (n + 3) & ~3;
    return o;
  };
  for (int l = 0; l < f.nlin; ++l) {
    f.sW[l] = take(f.din[l] * (l == f.nlin - 1 ? kFusedOut : kLd));
    f.sB[l] = take(f.dout[l]);
  }
  if (train) {
    for (int l = 0; l < f.nlin; ++l) f.sA[l] = take(2 * f.din[l] * R);
    f.sD = take(R * kLd);
  } else {
    int w[2] = {1, 1};  // widest of the layers that take turns
    for (int l = 0; l < f.nlin; ++l) w[l & 1] = std::max(w[l & 1], f.din[l]);
    const int o[2] = {take(2 * w[0] * R), take(2 * w[1] * R)};
    for (int l = 0; l < f.nlin; ++l) f.sA[l] = o[l & 1];
    f.sD = at;
  }
  f.sRed = take((kRowThreads / (32 * (R / 4))) * R * kLd);  // KS splits of k_rows
  return (size_t)at * sizeof(float);
}

// nets whose widths the fused tiles cover and whose shared memory fits with
// the largest slabs (8 rows in training, 16 in inference)
static bool fused_fits(FusedNet f) {
  for (int l = 0; l < f.nlin; ++l)
    if (f.din[l] > kFusedWidth || f.dout[l] > kFusedWidth) return false;
  return f.dout[f.nlin - 1] <= kFusedOut && fused_layout(f, kTrainRows, true) <= kMaxSmem &&
         fused_layout(f, 16, false) <= kMaxSmem;
}

extern "C" abm_status abm_mlp_destroy(abm_mlp* n) {
  if (!n) return ABM_ERR_ARG;
  mlp_free(n);
  return ABM_OK;
}

extern "C" abm_status abm_mlp_create(int32_t n_in, int32_t hidden, int32_t layers, int32_t n_out, uint32_t seed,
                                     int32_t max_batch, void* stream, abm_mlp** out) {
  if (!out || n_in < 1 || n_in > 1024 || hidden < 1 || hidden > 1024 || layers < 1 || layers > 8 || n_out < 1 ||
      n_out > 1024 || max_batch < 1)
    return ABM_ERR_ARG;
  abm_mlp* n = new (std::nothrow) abm_mlp();
  if (!n) return ABM_ERR_OOM;
  n->n_in = n_in;
  n->hidden = hidden;
  n->layers = layers;
  n->n_out = n_out;
  n->max_batch = max_batch;
  n->nlin = layers + 1;
  long long off = 0;
  std::vector<long long> offs;
  std::vector<int> fan;
  for (int l = 0; l < n->nlin; ++l) {
    const int di = l == 0 ? n_in : hidden, dd = l == n->nlin - 1 ? n_out : hidden;
    n->din.push_back(di);
    n->dout.push_back(dd);
    n->offW.push_back(off);
    offs.push_back(off);
    off += (long long)di * dd;
    n->offb.push_back(off);
    offs.push_back(off);
    off += dd;
    fan.push_back(di);
  }
  n->nparams = off;
  const long long rows_pad = ((long long)max_batch + 31) / 32 * 32;  // whole row slabs
  long long aoff = 0;
  for (int l = 0; l <= n->nlin; ++l) {
    n->offA.push_back(aoff);
    const int w = l == 0 ? n_in : n->dout[l - 1];
    aoff += rows_pad * w;
  }
  n->net.nlin = n->nlin;
  n->net.nparams = (int)n->nparams;
  for (int l = 0; l < n->nlin; ++l) {
    n->net.din[l] = n->din[l];
    n->net.dout[l] = n->dout[l];
    n->net.offW[l] = (int)n->offW[l];
    n->net.offb[l] = (int)n->offb[l];
    n->net.offA[l] = n->offA[l];
  }
  n->net.offA[n->nlin] = n->offA[n->nlin];
  n->fused = fused_fits(n->net);
  const size_t P = (size_t)n->nparams;
  bool ok = cudaMalloc(&n->p, P * 4) == cudaSuccess && cudaMalloc(&n->g, P * 4) == cudaSuccess &&
            cudaMalloc(&n->m, P * 4) == cudaSuccess && cudaMalloc(&n->v, P * 4) == cudaSuccess &&
            cudaMalloc(&n->act, (size_t)aoff * 4) == cudaSuccess && cudaMalloc(&n->dact, (size_t)aoff * 4) == cudaSuccess &&
            cudaMalloc(&n->part, (size_t)kSplits * std::max(hidden, n_in) * std::max(hidden, n_out) * 4) == cudaSuccess &&
            cudaMalloc(&n->lossp, 1024 * 4) == cudaSuccess &&
            cudaMalloc(&n->d_off, offs.size() * sizeof(long long)) == cudaSuccess &&
            cudaMalloc(&n->d_fan, fan.size() * sizeof(int)) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
    mlp_free(n);
    return ABM_ERR_OOM;
  }
  cudaStream_t st = (cudaStream_t)stream;
  if (cudaMemcpyAsync(n->d_off, offs.data(), offs.size() * sizeof(long long), cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemcpyAsync(n->d_fan, fan.data(), fan.size() * sizeof(int), cudaMemcpyHostToDevice, st) != cudaSuccess ||
      cudaMemsetAsync(n->m, 0, P * 4, st) != cudaSuccess || cudaMemsetAsync(n->v, 0, P * 4, st) != cudaSuccess) {
    mlp_free(n);
    return ABM_ERR_CUDA;
  }
  k_mlp_init<<<num_sms() * 4, 256, 0, st>>>(n->p, n->nparams, n->d_off, n->d_fan, n->nlin, seed);
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(st) != cudaSuccess) {
    mlp_free(n);
    return ABM_ERR_CUDA;
  }
  n->adam_t = 0;
  *out = n;
  return ABM_OK;
}

template <bool TA, bool TB>
static void gemm(const GemmArgs& a, cudaStream_t st, int splits = 1) {
  dim3 grid((unsigned)((a.N + kGT - 1) / kGT), (unsigned)((a.M + kGT - 1) / kGT), (unsigned)splits);
  k_gemm<TA, TB><<<grid, kGThreads, 0, st>>>(a);
}

static GemmArgs gargs(int M, int N, int K) {
  GemmArgs a;
  std::memset(&a, 0, sizeof(a));
  a.M = M;
  a.N = N;
  a.K = K;
  a.k_per_split = K;
  return a;
}

struct Perm {
  long long rows, a, c, m0;
};

// forward through all layers; the output lands in act block nlin
static abm_status mlp_forward(abm_mlp* n, const float* x, int B, const Perm& pm, cudaStream_t st) {
  for (int l = 0; l < n->nlin; ++l) {
    GemmArgs a = gargs(B, n->dout[l], n->din[l]);
    if (l == 0) {
      a.A = x;
      a.gather_rows = pm.rows;
      a.gather_a = pm.a;
      a.gather_c = pm.c;
      a.gather_m0 = pm.m0;
    } else {
      a.A = n->act + n->offA[l];
    }
    a.lda = n->din[l];
    a.B = n->p + n->offW[l];
    a.ldb = n->dout[l];
    a.C = n->act + n->offA[l + 1];
    a.ldc = n->dout[l];
    a.bias = n->p + n->offb[l];
    a.relu = l < n->nlin - 1;
    gemm<false, false>(a, st);
  }
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

// loss + gradients of all parameters into n->g (loss_out: device float, nullable)
static abm_status mlp_backward(abm_mlp* n, const float* x, const float* y, int B, float tau, const Perm& pm,
                               float* loss_out, cudaStream_t st) {
  const int L = n->nlin;
  const int nblk = std::min(1024, std::max(1, (B * n->n_out + 255) / 256));
  k_pinball<<<nblk, 256, 0, st>>>(n->act + n->offA[L], y, B, n->n_out, tau, pm.rows, pm.a, pm.c, pm.m0,
                                  n->dact + n->offA[L], n->lossp);
  if (loss_out) k_loss_final<<<1, 32, 0, st>>>(n->lossp, nblk, 1.f / (float)(B * n->n_out), loss_out);
  for (int l = L - 1; l >= 0; --l) {
    const float* dY = n->dact + n->offA[l + 1];  // [B x dout]
    // dW = X^T dY  (din x dout), split over the batch, summed in fixed order
    const int per = (((B + kSplits - 1) / kSplits) + kGK - 1) / kGK * kGK;
    const int splits = (B + per - 1) / per;
    GemmArgs a = gargs(n->din[l], n->dout[l], B);
    a.A = n->act + n->offA[l];  // block 0 holds the gathered input rows
    a.lda = n->din[l];
    a.B = dY;
    a.ldb = n->dout[l];
    a.C = n->part;
    a.ldc = n->dout[l];
    a.k_per_split = per;
    a.split_stride = (long long)n->din[l] * n->dout[l];
    gemm<true, false>(a, st, splits);
    k_sum_splits<<<std::max(1, std::min(256, (n->din[l] * n->dout[l] + 255) / 256)), 256, 0, st>>>(
        n->part, splits, a.split_stride, n->din[l] * n->dout[l], n->g + n->offW[l]);
    k_colsum<<<(n->dout[l] + 127) / 128, 128, 0, st>>>(dY, B, n->dout[l], n->g + n->offb[l]);
    if (l > 0) {
      // dX = (dY W^T) * (X > 0)
      GemmArgs d = gargs(B, n->din[l], n->dout[l]);
      d.A = dY;
      d.lda = n->dout[l];
      d.B = n->p + n->offW[l];
      d.ldb = n->dout[l];
      d.C = n->dact + n->offA[l];
      d.ldc = n->din[l];
      d.mask = n->act + n->offA[l];
      d.ldm = n->din[l];
      gemm<false, true>(d, st);
    }
  }
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

// copy the (gathered) input rows into act block 0 so that the first layer's
// weight gradient can read them transposed
__global__ void k_gather_rows(const float* x, int B, int w, long long rows, long long ga, long long gc, long long gm0,
                              float* out) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B * w; i += gridDim.x * blockDim.x) {
    const int r = i / w, c = i % w;
    long long row = r;
    if (rows) row = (ga * (gm0 + r) + gc) % rows;
    out[i] = x[(size_t)row * w + c];
  }
}

static Perm make_perm(int64_t rows, int64_t a, int64_t c, int64_t m0) {
  Perm p;
  p.rows = rows;
  p.a = a;
  p.c = c;
  p.m0 = m0;
  return p;
}

// ---- fused path, host side
template <int R, bool TRAIN>
static abm_status rows_launch(abm_mlp* n, RowArgs& ra, cudaStream_t st, int& grid) {
  static std::atomic<unsigned long long> attr{0};
  ra.net = n->net;
  const size_t smem = fused_layout(ra.net, R, TRAIN);
  ABM_CUDA_TRY(smem_attr_once(k_rows<R, TRAIN>, (int)kMaxSmem, attr));
  grid = std::min((ra.B + R - 1) / R, num_sms());
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kRowThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  ABM_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_rows<R, TRAIN>, ra));
  return ABM_OK;
}

struct AdamStep {
  int on;
  float lr, b1, b2, eps, c1, c2;
};

static abm_status fused_train(abm_mlp* n, RowArgs& ra, const AdamStep& ad, float* loss_out, cudaStream_t st) {
  constexpr int R = kTrainRows;
  int grid = 0;
  abm_status e = rows_launch<R, true>(n, ra, st, grid);
  if (e != ABM_OK) return e;
  WgradArgs wa;
  std::memset(&wa, 0, sizeof(wa));
  wa.net = ra.net;
  wa.act = n->act;
  wa.dact = n->dact;
  wa.g = n->g;
  wa.p = n->p;
  wa.m = n->m;
  wa.v = n->v;
  wa.nslab = (ra.B + R - 1) / R;
  // runs of whole stages (128 rows each up to 1024 rows), one CTA of the cluster each
  const int stages = (wa.nslab * R + kWRows - 1) / kWRows;
  static std::atomic<int> known[64];
  const int most = std::min(kMaxRuns, cluster_limit(k_wgrad, kWThreads, known));
  const int per = (stages + most - 1) / most, runs = (stages + per - 1) / per;
  wa.slabs_per_split = per * (kWRows / R);
  wa.lossp = n->lossp;
  wa.nloss = grid;
  wa.loss_scale = ra.scale;
  wa.loss_out = loss_out;
  wa.adam = ad.on;
  wa.lr = ad.lr;
  wa.b1 = ad.b1;
  wa.b2 = ad.b2;
  wa.eps = ad.eps;
  wa.c1 = ad.c1;
  wa.c2 = ad.c2;
  int tiles = 0;
  for (int l = 0; l < n->nlin; ++l) tiles += wgrad_tiles(n->net, l);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)tiles, (unsigned)runs);
  cfg.blockDim = dim3(kWThreads);
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = at[1].val.clusterDim.z = 1;
  at[1].val.clusterDim.y = (unsigned)runs;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  ABM_CUDA_TRY(cudaLaunchKernelEx(&cfg, k_wgrad, wa));
  return ABM_OK;
}

static abm_status fused_gradients(abm_mlp* n, const float* x, const float* y, int B, float tau, const Perm& pm,
                                  const AdamStep& ad, float* loss_out, cudaStream_t st) {
  RowArgs ra;
  std::memset(&ra, 0, sizeof(ra));
  ra.p = n->p;
  ra.x = x;
  ra.y = y;
  ra.act = n->act;
  ra.dact = n->dact;
  ra.lossp = n->lossp;
  ra.B = B;
  ra.tau = tau;
  ra.scale = 1.f / (float)(B * n->n_out);
  ra.grows = pm.rows;
  ra.ga = pm.a;
  ra.gc = pm.c;
  ra.gm0 = pm.m0;
  return fused_train(n, ra, ad, loss_out, st);
}

static abm_status fused_forward(abm_mlp* n, const float* x, int B, float* y, cudaStream_t st) {
  RowArgs ra;
  std::memset(&ra, 0, sizeof(ra));
  ra.p = n->p;
  ra.x = x;
  ra.out = y;
  ra.B = B;
  int grid;
  return B <= 16 * num_sms() ? rows_launch<8, false>(n, ra, st, grid) : rows_launch<16, false>(n, ra, st, grid);
}

extern "C" abm_status abm_mlp_forward(abm_mlp* n, const float* x, int32_t B, float* y, void* stream) {
  if (!n || !x || !y || B < 1 || B > n->max_batch) return ABM_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  if (n->fused) return fused_forward(n, x, B, y, st);
  abm_status e = mlp_forward(n, x, B, make_perm(0, 0, 0, 0), st);
  if (e != ABM_OK) return e;
  ABM_CUDA_TRY(cudaMemcpyAsync(y, n->act + n->offA[n->nlin], sizeof(float) * (size_t)B * n->n_out,
                               cudaMemcpyDeviceToDevice, st));
  return ABM_OK;
}

static bool grad_args_ok(abm_mlp* n, const float* x, const float* y, int32_t B, int64_t perm_rows, int64_t perm_a) {
  return n && x && y && B >= 1 && B <= n->max_batch && perm_rows >= 0 && (perm_rows == 0 || perm_a >= 1);
}

static abm_status gemm_gradients(abm_mlp* n, const float* x, const float* y, int B, float tau, const Perm& pm,
                                 float* loss_out, cudaStream_t st) {
  abm_status e = mlp_forward(n, x, B, pm, st);
  if (e != ABM_OK) return e;
  k_gather_rows<<<std::max(1, std::min(1024, (B * n->n_in + 255) / 256)), 256, 0, st>>>(
      x, B, n->n_in, pm.rows, pm.a, pm.c, pm.m0, n->act);
  return mlp_backward(n, x, y, B, tau, pm, loss_out, st);
}

extern "C" abm_status abm_mlp_gradients(abm_mlp* n, const float* x, const float* y, int32_t B, float tau,
                                        int64_t perm_rows, int64_t perm_a, int64_t perm_c, int64_t perm_m0,
                                        float* loss_out, void* stream) {
  if (!grad_args_ok(n, x, y, B, perm_rows, perm_a)) return ABM_ERR_ARG;
  const Perm pm = make_perm(perm_rows, perm_a, perm_c, perm_m0);
  if (n->fused) return fused_gradients(n, x, y, B, tau, pm, AdamStep{}, loss_out, (cudaStream_t)stream);
  return gemm_gradients(n, x, y, B, tau, pm, loss_out, (cudaStream_t)stream);
}

extern "C" abm_status abm_mlp_train_step(abm_mlp* n, const float* x, const float* y, int32_t B, float tau, float lr,
                                         int64_t perm_rows, int64_t perm_a, int64_t perm_c, int64_t perm_m0,
                                         float* loss_out, void* stream) {
  if (!grad_args_ok(n, x, y, B, perm_rows, perm_a)) return ABM_ERR_ARG;
  const Perm pm = make_perm(perm_rows, perm_a, perm_c, perm_m0);
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const int t = n->adam_t + 1;
  const float c1 = (float)(1.0 - std::pow((double)b1, t));
  const float c2 = (float)(1.0 - std::pow((double)b2, t));
  if (n->fused) {
    const abm_status e =
        fused_gradients(n, x, y, B, tau, pm, AdamStep{1, lr, b1, b2, eps, c1, c2}, loss_out, (cudaStream_t)stream);
    if (e == ABM_OK) n->adam_t = t;
    return e;
  }
  const abm_status e = gemm_gradients(n, x, y, B, tau, pm, loss_out, (cudaStream_t)stream);
  if (e != ABM_OK) return e;
  n->adam_t = t;
  k_adam<<<std::max(1, std::min(1024, (int)((n->nparams + 255) / 256))), 256, 0, (cudaStream_t)stream>>>(
      n->p, n->g, n->m, n->v, (int)n->nparams, lr, b1, b2, eps, c1, c2);
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

extern "C" abm_status abm_mlp_params(abm_mlp* n, float** params, float** grads, int64_t* count) {
  if (!n) return ABM_ERR_ARG;
  if (params) *params = n->p;
  if (grads) *grads = n->g;
  if (count) *count = n->nparams;
  return ABM_OK;
}

extern "C" abm_status abm_mlp_set_params(abm_mlp* n, const float* src, int64_t count, void* stream) {
  if (!n || !src || count != n->nparams) return ABM_ERR_ARG;
  ABM_CUDA_TRY(cudaMemcpyAsync(n->p, src, sizeof(float) * (size_t)count, cudaMemcpyDeviceToDevice,
                               (cudaStream_t)stream));
  return ABM_OK;
}

extern "C" abm_status abm_mlp_get_params(abm_mlp* n, float* dst, int64_t count, void* stream) {
  if (!n || !dst || count != n->nparams) return ABM_ERR_ARG;
  ABM_CUDA_TRY(cudaMemcpyAsync(dst, n->p, sizeof(float) * (size_t)count, cudaMemcpyDeviceToDevice,
                               (cudaStream_t)stream));
  return ABM_OK;
}

extern "C" abm_status abm_mlp_get_grads(abm_mlp* n, float* dst, int64_t count, void* stream) {
  if (!n || !dst || count != n->nparams) return ABM_ERR_ARG;
  ABM_CUDA_TRY(cudaMemcpyAsync(dst, n->g, sizeof(float) * (size_t)count, cudaMemcpyDeviceToDevice,
                               (cudaStream_t)stream));
  return ABM_OK;
}

extern "C" abm_status abm_mlp_reset_adam(abm_mlp* n, void* stream) {
  if (!n) return ABM_ERR_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  ABM_CUDA_TRY(cudaMemsetAsync(n->m, 0, sizeof(float) * (size_t)n->nparams, st));
  ABM_CUDA_TRY(cudaMemsetAsync(n->v, 0, sizeof(float) * (size_t)n->nparams, st));
  n->adam_t = 0;
  return ABM_OK;
}

extern "C" abm_status abm_capacity_features(const int32_t* table, int32_t B, const int32_t* nominal, float* x,
                                            void* stream) {
  if (!table || !nominal || !x || B < 1) return ABM_ERR_ARG;
  k_features<<<std::max(1, std::min(1024, (B + 255) / 256)), 256, 0, (cudaStream_t)stream>>>(table, B, nominal, x);
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}

extern "C" abm_status abm_capacity_from_prediction(const float* yhat, int32_t B, float margin, int32_t round_to,
                                                   const int32_t* cap_max, const int32_t* n0, int32_t* cap,
                                                   void* stream) {
  if (!yhat || !cap_max || !n0 || !cap || B < 1 || round_to < 1 || margin < 0.f) return ABM_ERR_ARG;
  k_capacity<<<std::max(1, std::min(1024, (2 * B + 255) / 256)), 256, 0, (cudaStream_t)stream>>>(
      yhat, B, margin, round_to, cap_max, n0, cap);
  ABM_LAUNCH_CHECK();
  return ABM_OK;
}
