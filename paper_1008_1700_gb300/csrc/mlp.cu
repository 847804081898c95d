// Learned initial guess for the reduced solve of Fig. 3 (6.3): a multilayer
// perceptron with ReLU hidden layers and a linear output, trained with Adam
// on reduced solutions that the solver itself produced.  The paper has no
// network; it solves 6.3 iteratively from a starting vector, which is what
// the network predicts.  Forward, backward and the optimiser step are FP32 CUDA
// kernels: tiled GEMMs with fused epilogues (bias, ReLU and its mask, the loss
// and its gradient, the bias gradient).
#include <cuda_runtime.h>

#include <cstdint>

#include "ddps.h"
#include "tri.h"

namespace {

constexpr int kThreads = 256;

// One product C(i,j) = sum_k A(i,k) B(k,j) with arbitrary element strides (a
// unit stride on either side of each operand) and its epilogue.
enum Mode {
  MODE_STORE = 0,      // C = acc; with rowsum: rowsum[i] = sum_k A(i,k) as well
  MODE_BIAS = 1,       // C = acc + bias[j]
  MODE_BIAS_RELU = 2,  // C = relu(acc + bias[j])
  MODE_MASK = 3,       // C = acc where mask > 0, else 0 (mask: the layer's ReLU output)
  MODE_LOSS = 4,       // C = (acc + bias[j] - target) scale, and per CTA the sum of
                       // (acc + bias[j] - target)^2 in partial[]
  MODE_SPLIT = 5       // C[split] = acc of the CTA's part of K
};
struct GemmArgs {
  const float* A;
  int64_t sa0, sa1;
  const float* B;
  int64_t sb0, sb1;
  float* C;
  int64_t ldc;
  int M, N, K;
  int mode;
  const float* bias;
  const float* aux;  // mask or target, laid out as C
  float* rowsum;
  double* partial;
  float scale;
  int kper;  // MODE_SPLIT: K taken by one split
};

// A sum of squares of floats as an unevaluated sum of three (tri.h): FP64's digits and more
// without the FP64 pipe, whose rate is 1/64 here and held the loss epilogue of a 64 x 128 tile
// for 4 us.  Squares that FP32's range does not hold to the last bit are left out and noted.
struct SquareSum {
  ddps::Tri t = {0.f, 0.f, 0.f};
  bool left_out = false;
  __device__ static __forceinline__ bool in_range(float d) {
    return d == 0.f || (fabsf(d) >= 0x1p-48f && fabsf(d) <= 0x1p60f);
  }
  __device__ __forceinline__ void add(float d) {
    const bool in = in_range(d);
    const float v = in ? d : 0.f;
    t = ddps::sum(t, ddps::mul(v, v));
    left_out |= !in;
  }
  __device__ __forceinline__ double total() const { return ((double)t.l + t.m) + t.h; }
};

__device__ __forceinline__ float finish(const GemmArgs& g, float v, int64_t o, int j, SquareSum& sq) {
  if (g.mode == MODE_BIAS) return v + g.bias[j];
  if (g.mode == MODE_BIAS_RELU) return fmaxf(v + g.bias[j], 0.f);
  if (g.mode == MODE_MASK) return g.aux[o] > 0.f ? v : 0.f;
  if (g.mode == MODE_LOSS) {
    const float d = v + g.bias[j] - g.aux[o];
    sq.add(d);
    return d * g.scale;
  }
  return v;
}

// Wide products (the output layer: 32,256 x 256 weights at a batch of 100):
// 64 x 128 tiles, K in steps of 16 through two shared-memory buffers, the
// next step's loads in registers meanwhile, 4 x 8 results per thread.  Bound
// by FP32 arithmetic.  The rows of a batch of about 100 are the short side,
// so the tile is 64 high: two tiles waste less of it than one of 128 and a
// remainder.  MODE_SPLIT: blockIdx.z takes K range z of kper.  At a batch of 100
// and 256 x 32,256 weights: output layer with loss 79 us (a 64 x 64 tile kernel
// with a separate loss pass took 197), weight gradient 57 us (99 with the bias
// pass), input gradient 53 + 10 us in 75 splits (5,650 us in 8 CTAs without).
constexpr int BM = 64, BN = 128, BK = 16;

// Loads ROWS x BK values of an operand into registers: KC: k contiguous
// (element (r, k) at p[r * ld + k]), else r contiguous (p[r + k * ld]); `vec`:
// 16-byte loads are aligned.
template <int ROWS>
__device__ __forceinline__ void load_tile(const float* __restrict__ p, int64_t ld, bool kc,
                                          bool vec, int r0, int nr, int k0, int k1,
                                          float (&v)[ROWS * BK / kThreads]) {
  constexpr int NV = ROWS * BK / kThreads / 4;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const int e = threadIdx.x + q * kThreads;
    const int r = r0 + (kc ? e / (BK / 4) : (e % (ROWS / 4)) * 4);
    const int k = k0 + (kc ? (e % (BK / 4)) * 4 : e / (ROWS / 4));
    float* d = v + 4 * q;
    if (kc) {
      const float* s = p + r * ld + k;
      if (vec && r < nr && k + 4 <= k1) {
        const float4 t = __ldg(reinterpret_cast<const float4*>(s));
        d[0] = t.x, d[1] = t.y, d[2] = t.z, d[3] = t.w;
      } else {
#pragma unroll
        for (int t = 0; t < 4; ++t) d[t] = (r < nr && k + t < k1) ? __ldg(s + t) : 0.f;
      }
    } else {
      const float* s = p + r + k * ld;
      if (vec && r + 4 <= nr && k < k1) {
        const float4 t = __ldg(reinterpret_cast<const float4*>(s));
        d[0] = t.x, d[1] = t.y, d[2] = t.z, d[3] = t.w;
      } else {
#pragma unroll
        for (int t = 0; t < 4; ++t) d[t] = (r + t < nr && k < k1) ? __ldg(s + t) : 0.f;
      }
    }
  }
}
template <int ROWS>
__device__ __forceinline__ void store_tile(float (*S)[ROWS + 4], bool kc,
                                           const float (&v)[ROWS * BK / kThreads]) {
  constexpr int NV = ROWS * BK / kThreads / 4;
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    const int e = threadIdx.x + q * kThreads;
    if (kc) {
#pragma unroll
      for (int t = 0; t < 4; ++t) S[(e % (BK / 4)) * 4 + t][e / (BK / 4)] = v[4 * q + t];
    } else {
      *reinterpret_cast<float4*>(&S[e / (ROWS / 4)][(e % (ROWS / 4)) * 4]) =
          make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    }
  }
}

template <bool ROWSUM>
__global__ void __launch_bounds__(kThreads) k_gemm_wide(GemmArgs g) {
  __shared__ __align__(16) float As[2][BK][BM + 4];
  __shared__ __align__(16) float Bs[2][BK][BN + 4];
  __shared__ double red[kThreads / 32];
  const int i0 = blockIdx.y * BM, j0 = blockIdx.x * BN;
  const int tid = threadIdx.x, ty = tid / 16, tx = tid % 16;
  const bool akc = g.sa1 == 1, bkc = g.sb0 == 1;
  const int64_t lda = akc ? g.sa0 : g.sa1, ldb = bkc ? g.sb1 : g.sb0;
  const bool avec = lda % 4 == 0 && ((uintptr_t)g.A & 15) == 0;
  const bool bvec = ldb % 4 == 0 && ((uintptr_t)g.B & 15) == 0;
  const int kb = g.mode == MODE_SPLIT ? blockIdx.z * g.kper : 0;
  const int ke = g.mode == MODE_SPLIT ? min(g.K, kb + g.kper) : g.K;
  float va[BM * BK / kThreads], vb[BN * BK / kThreads];
  float acc[4][8] = {}, rs[4] = {};
  load_tile<BM>(g.A, lda, akc, avec, i0, g.M, kb, ke, va);
  load_tile<BN>(g.B, ldb, bkc, bvec, j0, g.N, kb, ke, vb);
  int st = 0;
  for (int k0 = kb; k0 < ke; k0 += BK, st ^= 1) {
    store_tile<BM>(As[st], akc, va);
    store_tile<BN>(Bs[st], bkc, vb);
    __syncthreads();
    if (k0 + BK < ke) {
      load_tile<BM>(g.A, lda, akc, avec, i0, g.M, k0 + BK, ke, va);
      load_tile<BN>(g.B, ldb, bkc, bvec, j0, g.N, k0 + BK, ke, vb);
    }
#pragma unroll
    for (int k = 0; k < BK; ++k) {
      const float4 a4 = *reinterpret_cast<const float4*>(&As[st][k][ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[st][k][tx * 4]);
      const float4 b1 = *reinterpret_cast<const float4*>(&Bs[st][k][BN / 2 + tx * 4]);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (ROWSUM) rs[u] += a[u];
#pragma unroll
        for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
      }
    }
    // the buffer written next was last read before the barrier above
  }
  float* __restrict__ C = g.C + (g.mode == MODE_SPLIT ? (int64_t)blockIdx.z * g.M * g.N : 0);
  const bool cvec = g.ldc % 4 == 0 && ((uintptr_t)C & 15) == 0;
  SquareSum sum;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int i = i0 + ty * 4 + u;
    if (i >= g.M) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int j = j0 + h * (BN / 2) + tx * 4;
      const int64_t o = i * g.ldc + j;
      float v[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) v[t] = j + t < g.N ? finish(g, acc[u][4 * h + t], o + t, j + t, sum) : 0.f;
      if (cvec && j + 4 <= g.N) {
        *reinterpret_cast<float4*>(C + o) = make_float4(v[0], v[1], v[2], v[3]);
      } else {
#pragma unroll
        for (int t = 0; t < 4; ++t)
          if (j + t < g.N) C[o + t] = v[t];
      }
    }
    if (ROWSUM && blockIdx.x == 0 && tx == 0) g.rowsum[i] = rs[u];
  }
  if (g.mode == MODE_LOSS) {
    double sq = sum.total();
    if (sum.left_out) {  // rare
      for (int u = 0; u < 4; ++u)
        for (int v = 0; v < 8; ++v) {
          const int i = i0 + ty * 4 + u, j = j0 + v / 4 * (BN / 2) + tx * 4 + v % 4;
          if (i >= g.M || j >= g.N) continue;
          const float d = acc[u][v] + g.bias[j] - g.aux[i * g.ldc + j];
          if (!SquareSum::in_range(d)) sq += (double)d * d;
        }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if ((tid & 31) == 0) red[tid >> 5] = sq;
    __syncthreads();
    if (tid == 0) {
      for (int q = 1; q < kThreads / 32; ++q) sq += red[q];
      g.partial[(int64_t)blockIdx.y * gridDim.x + blockIdx.x] = sq;
    }
  }
}

// C = sum over the splits, in order, where mask > 0.
__global__ void __launch_bounds__(kThreads)
    k_split_sum(const float* __restrict__ P, int nsplit, int64_t cnt, const float* __restrict__ mask,
                float* __restrict__ C) {
  const int64_t i = blockIdx.x * (int64_t)kThreads + threadIdx.x;
  if (i >= cnt) return;
  float s = 0.f;
#pragma unroll 8
  for (int q = 0; q < nsplit; ++q) s += P[q * cnt + i];
  C[i] = !mask || mask[i] > 0.f ? s : 0.f;
}

// Small products (the hidden layers: 256 x 256 at a batch of 100): 32 x 32
// tiles, so that the layer fills 32 SMs instead of 8; the CTA stages up to 256
// values of K at once and its eight warps split them (4 x 8 results per lane,
// summed over the warps in shared memory): a chain of one load, one barrier and
// 32 steps in place of 16 rounds of them.  Latency-bound.  Two problems (a
// layer's weight and input gradients) may share a launch: problem 1 takes the
// CTAs from n0 on.
constexpr int SM_T = 32, SM_K = 256;
constexpr int kSmallSmem = 2 * SM_K * (SM_T + 4) * (int)sizeof(float);
__global__ void __launch_bounds__(kThreads) k_gemm_small(GemmArgs g0, GemmArgs g1, int n0) {
  extern __shared__ __align__(16) float sm[];
  float(*As)[SM_T + 4] = reinterpret_cast<float(*)[SM_T + 4]>(sm);
  float(*Bs)[SM_T + 4] = As + SM_K;
  const bool second = (int)blockIdx.x >= n0;
  const GemmArgs g = second ? g1 : g0;
  const int t = second ? blockIdx.x - n0 : blockIdx.x;
  const int nj = (g.N + SM_T - 1) / SM_T;
  const int i0 = t / nj * SM_T, j0 = t % nj * SM_T;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int li = (lane >> 2) * 4, lj = (lane & 3) * 8;
  const bool akc = g.sa1 == 1, bkc = g.sb0 == 1;
  float acc[4][8] = {}, rs[4] = {};
  for (int k0 = 0; k0 < g.K; k0 += SM_K) {
    const int kn = min(SM_K, g.K - k0);
    if (k0) __syncthreads();
    // 32 loads per thread and operand, 16 in flight, lanes along the unit stride
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float va[16], vb[16];
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int e = tid + (h * 16 + q) * kThreads;
        const int ra = akc ? e / SM_K : e % SM_T, ka = akc ? e % SM_K : e / SM_T;
        const int rb = bkc ? e / SM_K : e % SM_T, kb = bkc ? e % SM_K : e / SM_T;
        va[q] = ka < kn && i0 + ra < g.M ? __ldg(g.A + (i0 + ra) * g.sa0 + (k0 + ka) * g.sa1) : 0.f;
        vb[q] = kb < kn && j0 + rb < g.N ? __ldg(g.B + (k0 + kb) * g.sb0 + (j0 + rb) * g.sb1) : 0.f;
      }
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        const int e = tid + (h * 16 + q) * kThreads;
        As[akc ? e % SM_K : e / SM_T][akc ? e / SM_K : e % SM_T] = va[q];
        Bs[bkc ? e % SM_K : e / SM_T][bkc ? e / SM_K : e % SM_T] = vb[q];
      }
    }
    __syncthreads();
    for (int k = warp; k < kn; k += kThreads / 32) {
      const float4 a4 = *reinterpret_cast<const float4*>(&As[k][li]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[k][lj]);
      const float4 b1 = *reinterpret_cast<const float4*>(&Bs[k][lj + 4]);
      const float a[4] = {a4.x, a4.y, a4.z, a4.w};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        rs[u] += a[u];
#pragma unroll
        for (int v = 0; v < 8; ++v) acc[u][v] = fmaf(a[u], b[v], acc[u][v]);
      }
    }
  }
  __syncthreads();
  // partial tiles of the warps (8 x 32 x 36) over the staged operands
  float(*P)[SM_T][SM_T + 4] = reinterpret_cast<float(*)[SM_T][SM_T + 4]>(sm);
  float* R = sm + (kThreads / 32) * SM_T * (SM_T + 4);  // row sums of the warps
#pragma unroll
  for (int u = 0; u < 4; ++u) {
#pragma unroll
    for (int v = 0; v < 8; v += 4)
      *reinterpret_cast<float4*>(&P[warp][li + u][lj + v]) =
          make_float4(acc[u][v], acc[u][v + 1], acc[u][v + 2], acc[u][v + 3]);
    if ((lane & 3) == 0) R[warp * SM_T + li + u] = rs[u];
  }
  __syncthreads();
  SquareSum sq;  // no small product takes MODE_LOSS
  for (int e = tid; e < SM_T * SM_T; e += kThreads) {
    const int r = e / SM_T, c = e % SM_T, i = i0 + r, j = j0 + c;
    if (i >= g.M || j >= g.N) continue;
    float s = P[0][r][c];
#pragma unroll
    for (int q = 1; q < kThreads / 32; ++q) s += P[q][r][c];
    const int64_t o = i * g.ldc + j;
    g.C[o] = finish(g, s, o, j, sq);
  }
  if (g.rowsum && j0 == 0 && tid < SM_T && i0 + tid < g.M) {
    float s = R[tid];
    for (int q = 1; q < kThreads / 32; ++q) s += R[q * SM_T + tid];
    g.rowsum[i0 + tid] = s;
  }
}

// A layer for NB <= 4 input vectors (a prediction): one warp per four rows of
// W, 16-byte loads along the row, all of them issued before they are used; bound by
// reading W once (33 MB at 32,256 outputs).
template <int NB>
__global__ void __launch_bounds__(kThreads)
    k_layer_vec(const float* __restrict__ W, const float* __restrict__ bias,
                const float* __restrict__ X, int K, int N, int relu, float* __restrict__ Y) {
  const int lane = threadIdx.x & 31;
  const int j0 = (blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * 4;
  if (j0 >= N) return;
  float acc[4][NB] = {};
  if (K % 4 == 0 && (((uintptr_t)W | (uintptr_t)X) & 15) == 0) {
    for (int k = lane * 4; k < K; k += 128) {
      float4 w[4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
        w[r] = __ldcs(reinterpret_cast<const float4*>(W + (int64_t)min(j0 + r, N - 1) * K + k));
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(X + (int64_t)b * K + k));
#pragma unroll
        for (int r = 0; r < 4; ++r)
          acc[r][b] = fmaf(w[r].x, x.x, fmaf(w[r].y, x.y, fmaf(w[r].z, x.z, fmaf(w[r].w, x.w, acc[r][b]))));
      }
    }
  } else {
    for (int k = lane; k < K; k += 32)
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float w = W[(int64_t)min(j0 + r, N - 1) * K + k];
#pragma unroll
        for (int b = 0; b < NB; ++b) acc[r][b] = fmaf(w, X[(int64_t)b * K + k], acc[r][b]);
      }
  }
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int b = 0; b < NB; ++b)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[r][b] += __shfl_xor_sync(0xffffffffu, acc[r][b], o);
  if (lane == 0)
    for (int r = 0; r < 4 && j0 + r < N; ++r)
#pragma unroll
      for (int b = 0; b < NB; ++b) {
        const float v = acc[r][b] + bias[j0 + r];
        Y[(int64_t)b * N + j0 + r] = relu ? fmaxf(v, 0.f) : v;
      }
}

__global__ void __launch_bounds__(kThreads)
    k_loss_final(const double* __restrict__ partial, int n, double scale, float* __restrict__ loss) {
  __shared__ double red[kThreads];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += kThreads) s += partial[i];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = kThreads / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = (float)(red[0] * scale);
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int64_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float mh = mi / c1, vh = vi / c2;
    p[i] -= lr * mh / (sqrtf(vh) + eps);
  }
}

struct Layout {
  int L;  // number of affine layers = layers + 1
  int64_t woff[16], boff[16];
  int din[16], dout[16];
};

bool make_layout(int32_t d_in, int32_t hidden, int32_t layers, int32_t d_out, Layout& lay) {
  if (d_in <= 0 || hidden <= 0 || layers <= 0 || layers > 14 || d_out <= 0) return false;
  lay.L = layers + 1;
  int64_t off = 0;
  for (int l = 0; l < lay.L; ++l) {
    lay.din[l] = l == 0 ? d_in : hidden;
    lay.dout[l] = l == lay.L - 1 ? d_out : hidden;
    lay.woff[l] = off;
    off += (int64_t)lay.din[l] * lay.dout[l];
    lay.boff[l] = off;
    off += lay.dout[l];
  }
  return true;
}

// Splits of K for a product of few output tiles (at most 304: about two CTAs per
// SM, at least 256 values of K each; a fixed rule, so that the workspace can be
// sized and the summation order does not depend on the device).
constexpr int kSplitCtas = 304;
int split_count(int M, int N, int K) {
  const int tiles = ((M + BM - 1) / BM) * ((N + BN - 1) / BN);
  int s = kSplitCtas / tiles;
  if (s > K / 256) s = K / 256;
  return s < 1 ? 1 : s;
}
int loss_blocks(int B, int d_out) { return ((B + BM - 1) / BM) * ((d_out + BN - 1) / BN); }

// workspace: A_l (B x hidden, the ReLU outputs) of the hidden layers, dY
// (B x d_out), two B x hidden gradient buffers, the K splits of the output
// layer's input gradient, the loss partial sums.
struct Work {
  float* Aact[16];
  float* dY;
  float* dA0;
  float* dA1;
  float* split;
  double* partial;
};

int64_t up4(int64_t n) { return (n + 3) / 4 * 4; }

// Floats of the split sums of any batch up to B: a batch one above a multiple of 64 takes fewer
// splits and so less than the one before it, but a buffer for the full batch also has to hold
// the ragged last one.
int64_t split_floats(int32_t hidden, int32_t d_out, int32_t B) {
  const int K = d_out > hidden ? d_out : hidden;
  int64_t most = up4((int64_t)B * hidden);
  for (int64_t b = BM;; b += BM) {
    const int32_t rows = (int32_t)(b < B ? b : B);
    const int ns = split_count(rows, hidden, K);
    const int64_t n = ns * up4((int64_t)rows * hidden);
    if (n > most) most = n;
    if (rows == B || ns == 1) return most;
  }
}

int64_t work_bytes(int32_t hidden, int32_t layers, int32_t d_out, int32_t B) {
  const int64_t hb = up4((int64_t)B * hidden);
  return 4 * ((layers + 2) * hb + split_floats(hidden, d_out, B) + up4((int64_t)B * d_out)) +
         8 * (int64_t)loss_blocks(B, d_out) + 256;
}

Work carve(void* ws, int32_t hidden, int32_t layers, int32_t d_out, int32_t B) {
  Work w{};
  float* p = (float*)(((uintptr_t)ws + 15) & ~(uintptr_t)15);
  const int64_t hb = up4((int64_t)B * hidden);
  for (int l = 0; l < layers; ++l) {
    w.Aact[l] = p;
    p += hb;
  }
  w.dY = p;
  p += up4((int64_t)B * d_out);
  w.dA0 = p;
  p += hb;
  w.dA1 = p;
  p += hb;
  w.split = p;
  p += split_floats(hidden, d_out, B);
  w.partial = (double*)p;
  return w;
}

int small_ctas(const GemmArgs& g) { return ((g.M + SM_T - 1) / SM_T) * ((g.N + SM_T - 1) / SM_T); }

// Products of at most 128 32 x 32 tiles (less than one per SM) and K within two
// stages take the small kernel, others the wide one.  At 100 x 256 x 256 the small
// kernel takes 11 us and the wide one (4 CTAs) 22; a layer's two gradients take
// 11 us in one small launch and 13 + 25 in two wide ones.
bool is_small(const GemmArgs& g) { return small_ctas(g) <= 128 && g.K <= 2 * SM_K; }

void gemm_small(const GemmArgs& g0, const GemmArgs* g1, cudaStream_t s) {
  cudaFuncSetAttribute(k_gemm_small, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmallSmem);
  const int n0 = small_ctas(g0), n1 = g1 ? small_ctas(*g1) : 0;
  k_gemm_small<<<n0 + n1, kThreads, kSmallSmem, s>>>(g0, g1 ? *g1 : g0, n0);
}
void gemm(const GemmArgs& g, cudaStream_t s) {
  if (is_small(g) && g.mode != MODE_LOSS) {
    gemm_small(g, nullptr, s);
    return;
  }
  dim3 grid((g.N + BN - 1) / BN, (g.M + BM - 1) / BM);
  if (g.rowsum)
    k_gemm_wide<true><<<grid, kThreads, 0, s>>>(g);
  else
    k_gemm_wide<false><<<grid, kThreads, 0, s>>>(g);
}
// C (M x N contiguous) = A B where mask > 0, K split over CTAs
void gemm_masked(GemmArgs g, float* split, cudaStream_t s) {
  const int ns = split_count(g.M, g.N, g.K);
  if (is_small(g) || ns == 1) {
    gemm(g, s);
    return;
  }
  const float* mask = g.aux;
  float* C = g.C;
  g.mode = MODE_SPLIT;
  g.C = split;
  g.kper = ((g.K + ns - 1) / ns + BK - 1) / BK * BK;
  const int nz = (g.K + g.kper - 1) / g.kper;
  k_gemm_wide<false><<<dim3((g.N + BN - 1) / BN, (g.M + BM - 1) / BM, nz), kThreads, 0, s>>>(g);
  const int64_t cnt = (int64_t)g.M * g.N;
  k_split_sum<<<(unsigned)((cnt + kThreads - 1) / kThreads), kThreads, 0, s>>>(split, nz, cnt, mask, C);
}

// The network's layers; with T, the last one leaves dY = (Y - T) / B and the
// loss partial sums instead of Y.
void forward(const float* P, const Layout& lay, const float* X, int B, const Work& w, float* Y,
             const float* T, cudaStream_t s) {
  const float* a = X;
  for (int l = 0; l < lay.L; ++l) {
    const bool last = l == lay.L - 1;
    float* out = !last ? w.Aact[l] : T ? w.dY : Y;
    if (B <= 4 && !(last && T)) {
      const unsigned grid = (unsigned)((lay.dout[l] + kThreads / 8 - 1) / (kThreads / 8));
      const float *W = P + lay.woff[l], *bias = P + lay.boff[l];
      auto kern = B == 1 ? k_layer_vec<1> : B == 2 ? k_layer_vec<2> : B == 3 ? k_layer_vec<3> : k_layer_vec<4>;
      kern<<<grid, kThreads, 0, s>>>(W, bias, a, lay.din[l], lay.dout[l], !last, out);
    } else {
      GemmArgs g{};
      g.A = a;
      g.sa0 = lay.din[l];
      g.sa1 = 1;
      g.B = P + lay.woff[l];  // W is [out x in] row-major; B(k, j) = W[j, k]
      g.sb0 = 1;
      g.sb1 = lay.din[l];
      g.M = B;
      g.N = lay.dout[l];
      g.K = lay.din[l];
      g.bias = P + lay.boff[l];
      g.C = out;
      g.ldc = lay.dout[l];
      g.mode = !last ? MODE_BIAS_RELU : T ? MODE_LOSS : MODE_BIAS;
      g.aux = T;
      g.scale = 1.f / B;
      g.partial = w.partial;
      gemm(g, s);
    }
    a = out;
  }
}

}  // namespace

extern "C" {

int64_t ddps_mlp_param_count(int32_t d_in, int32_t hidden, int32_t layers, int32_t d_out) {
  Layout lay;
  if (!make_layout(d_in, hidden, layers, d_out, lay)) return -1;
  return lay.boff[lay.L - 1] + lay.dout[lay.L - 1];
}

int64_t ddps_mlp_workspace_bytes(int32_t d_in, int32_t hidden, int32_t layers, int32_t d_out,
                                 int32_t B) {
  Layout lay;
  if (!make_layout(d_in, hidden, layers, d_out, lay) || B <= 0) return -1;
  return work_bytes(hidden, layers, d_out, B);
}

ddps_status ddps_mlp_forward(const float* params, int32_t d_in, int32_t hidden, int32_t layers,
                             int32_t d_out, const float* X, int32_t B, float* Y, void* workspace,
                             void* stream) {
  Layout lay;
  if (!params || !X || !Y || !workspace || B <= 0 || !make_layout(d_in, hidden, layers, d_out, lay))
    return DDPS_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  Work w = carve(workspace, hidden, layers, d_out, B);
  forward(params, lay, X, B, w, Y, nullptr, s);
  return cudaGetLastError() == cudaSuccess ? DDPS_OK : DDPS_ERR_CUDA;
}

ddps_status ddps_mlp_backward(const float* params, int32_t d_in, int32_t hidden, int32_t layers,
                              int32_t d_out, const float* X, const float* T, int32_t B,
                              float* grads, float* loss, void* workspace, void* stream) {
  Layout lay;
  if (!params || !X || !T || !grads || !loss || !workspace || B <= 0 ||
      !make_layout(d_in, hidden, layers, d_out, lay))
    return DDPS_ERR_INVALID_ARG;
  cudaStream_t s = (cudaStream_t)stream;
  Work w = carve(workspace, hidden, layers, d_out, B);
  forward(params, lay, X, B, w, nullptr, T, s);
  k_loss_final<<<1, kThreads, 0, s>>>(w.partial, loss_blocks(B, d_out), 0.5 / B, loss);
  const float* d = w.dY;  // gradient w.r.t. the pre-activation of layer l
  for (int l = lay.L - 1; l >= 0; --l) {
    // dW_l[o, i] = sum_b d[b, o] ain[b, i], db_l[o] = sum_b d[b, o]
    GemmArgs g{};
    g.A = d;
    g.sa0 = 1;
    g.sa1 = lay.dout[l];
    g.B = l == 0 ? X : w.Aact[l - 1];
    g.sb0 = lay.din[l];
    g.sb1 = 1;
    g.C = grads + lay.woff[l];
    g.ldc = lay.din[l];
    g.M = lay.dout[l];
    g.N = lay.din[l];
    g.K = B;
    g.mode = MODE_STORE;
    g.rowsum = grads + lay.boff[l];
    if (l == 0) {
      gemm(g, s);
      break;
    }
    // dA_{l-1} = d W_l where the layer's ReLU passed (its output is positive)
    float* dst = (d == w.dA0) ? w.dA1 : w.dA0;
    GemmArgs h{};
    h.A = d;
    h.sa0 = lay.dout[l];
    h.sa1 = 1;
    h.B = params + lay.woff[l];
    h.sb0 = lay.din[l];
    h.sb1 = 1;
    h.C = dst;
    h.ldc = lay.din[l];
    h.M = B;
    h.N = lay.din[l];
    h.K = lay.dout[l];
    h.mode = MODE_MASK;
    h.aux = w.Aact[l - 1];
    if (is_small(g) && is_small(h)) {
      gemm_small(g, &h, s);
    } else {
      gemm(g, s);
      gemm_masked(h, w.split, s);
    }
    d = dst;
  }
  return cudaGetLastError() == cudaSuccess ? DDPS_OK : DDPS_ERR_CUDA;
}

ddps_status ddps_mlp_adam(float* params, const float* grads, float* m, float* v, int64_t count,
                          float lr, float beta1, float beta2, float eps, int32_t step,
                          void* stream) {
  if (!params || !grads || !m || !v || count <= 0 || step < 1) return DDPS_ERR_INVALID_ARG;
  const float c1 = 1.f - powf(beta1, (float)step);
  const float c2 = 1.f - powf(beta2, (float)step);
  int64_t g = (count + kThreads - 1) / kThreads;
  if (g > 152 * 16) g = 152 * 16;
  k_adam<<<(int)g, kThreads, 0, (cudaStream_t)stream>>>(params, grads, m, v, count, lr, beta1,
                                                        beta2, eps, c1, c2);
  return cudaGetLastError() == cudaSuccess ? DDPS_OK : DDPS_ERR_CUDA;
}

}  // extern "C"
