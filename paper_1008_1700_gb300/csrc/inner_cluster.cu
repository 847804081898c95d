// Fig. 3 step 6.3 for systems whose rows of G^ fit the shared memory of a
// cluster: the whole inner BiCGStab (Sec. 4) of every system of the handle in one
// launch (one per size class), one cluster of up to eight CTAs per system.
//
// The launch-per-step loop spends five launches on an iteration (two products
// with G^, three vector steps), each a chain of latencies when a system has a few
// hundred to a few thousand reduced rows: 31 us an iteration for one system of
// 384 rows, 130 us for a batch of 256 systems of 1,100.  Here a CTA copies its
// rows of G^ into shared memory once per solve, its slices of all vectors live there
// too, and the CTAs of a cluster exchange the product's input vector and the partial
// sums through distributed shared memory, one cluster barrier per reduction.  The
// steps are those of the loop: products accumulate in FP32 (FP64 for FP64 storage),
// vectors are rounded to the inner precision after each update, sums and scalars are
// kept to FP64 or more (see Tri).  Sums are taken over threads, warps and
// CTAs in a fixed order: two solves are bitwise equal.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "inner_cluster.h"
#include "launch.h"
#include "tri.h"

namespace ddps {
namespace cg = cooperative_groups;

namespace {

constexpr int kMaxCs = 8;
constexpr size_t kSmemMax = 220 * 1024;  // dynamic shared memory of a CTA
// G^ bytes of a system that one cluster streams by every product: at 2.9 MB (200 x 200
// grid, 10 blocks) a re-solve takes 6.0 ms, with the launch-per-step loop 9.5; at 7.9 MB
// (256 x 256, 16 blocks) 16.8 against 12.6, where the loop's products use every SM.
constexpr int64_t kStreamMax = 4 << 20;

__host__ __device__ constexpr size_t up16(size_t n) { return (n + 15) / 16 * 16; }

// Sixteen bytes of a stored row in shared memory, as accumulator values.
template <typename TG>
struct Vec;
template <>
struct Vec<double> {
  using acc = double;
  static constexpr int n = 2;
  static __device__ __forceinline__ void load(const double* p, double* o) {
    const double2 v = *reinterpret_cast<const double2*>(p);
    o[0] = v.x, o[1] = v.y;
  }
};
template <>
struct Vec<float> {
  using acc = float;
  static constexpr int n = 4;
  static __device__ __forceinline__ void load(const float* p, float* o) {
    const float4 v = *reinterpret_cast<const float4*>(p);
    o[0] = v.x, o[1] = v.y, o[2] = v.z, o[3] = v.w;
  }
};
template <>
struct Vec<__half> {
  using acc = float;
  static constexpr int n = 8;
  static __device__ __forceinline__ void load(const __half* p, float* o) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[i]));
      o[2 * i] = f.x, o[2 * i + 1] = f.y;
    }
  }
};
template <>
struct Vec<__nv_bfloat16> {
  using acc = float;
  static constexpr int n = 8;
  static __device__ __forceinline__ void load(const __nv_bfloat16* p, float* o) {
    const uint4 v = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      o[2 * i] = __uint_as_float(w[i] << 16);
      o[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
    }
  }
};

// Scalars and sums.  FP64 vectors take FP64.  For FP32 vectors they are unevaluated sums of
// three floats (tri.h: about 70 bits, more than FP64 holds), because the FP64 pipe runs a warp
// instruction in 64 cycles here: with FP64 sums, scalars and updates an iteration of a 384-row
// system took 18 us at first, with pairs of floats (48 bits) 12, and 7.8 with fewer barriers,
// too; the third float adds 1.1.  They have FP32's range, so the system is scaled by the power of
// two that brings ||g|| to [2^20, 2^21): squares of vectors up to 10^13 ||g|| stay finite, and
// those of 10^-17 ||g|| keep FP64's digits.
__device__ __forceinline__ Tri shfl_xor(Tri x, int o) {
  return {__shfl_xor_sync(0xffffffffu, x.h, o), __shfl_xor_sync(0xffffffffu, x.m, o),
          __shfl_xor_sync(0xffffffffu, x.l, o)};
}
__device__ __forceinline__ Tri bcast(Tri x) {
  return {__shfl_sync(0xffffffffu, x.h, 0), __shfl_sync(0xffffffffu, x.m, 0),
          __shfl_sync(0xffffffffu, x.l, 0)};
}
__device__ __forceinline__ double bcast(double x) { return __shfl_sync(0xffffffffu, x, 0); }
__device__ __forceinline__ double shfl_xor(double x, int o) {
  return __shfl_xor_sync(0xffffffffu, x, o);
}

template <typename TI>
struct Wide;
template <>
struct Wide<float> {
  using W = Tri;
  static __device__ __forceinline__ Tri make(double x) {
    const float h = (float)x;
    x -= (double)h;
    const float m = (float)x;
    return {h, m, (float)(x - (double)m)};
  }
};
template <>
struct Wide<double> {
  using W = double;
  static __device__ __forceinline__ double make(double x) { return x; }
};

// Shared memory of another CTA of the cluster.
__device__ __forceinline__ uint32_t peer(const void* p, uint32_t rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;"
      : "=r"(a)
      : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ float ld_peer(const float* p, uint32_t rank) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(peer(p, rank)) : "memory");
  return v;
}
__device__ __forceinline__ double ld_peer(const double* p, uint32_t rank) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(peer(p, rank)) : "memory");
  return v;
}
__device__ __forceinline__ void st_peer(Tri* p, uint32_t rank, Tri v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %3};" ::"r"(peer(p, rank)), "f"(v.h),
               "f"(v.m), "f"(v.l)
               : "memory");
}
__device__ __forceinline__ void st_peer(double* p, uint32_t rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(peer(p, rank)), "d"(v) : "memory");
}

// Eight warps for FP32 vectors; four for FP64, one per quarter of the SM: every warp
// forms the scalars for itself, and two warps' FP64 instructions would queue.
constexpr int inner_threads(size_t size_i) { return size_i == 8 ? 128 : 256; }

// Position of a gathered column: the CTA that holds it and its place in the slice.
constexpr int kRankShift = 28;

// Products of VN stored entries with VN vector entries added to a row's sums.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(reinterpret_cast<uint64_t&>(d))
      : "l"(reinterpret_cast<uint64_t&>(a)), "l"(reinterpret_cast<uint64_t&>(b)),
        "l"(reinterpret_cast<uint64_t&>(c)));
  return d;
}
struct Acc32 {  // FP32: two sums, two products per instruction
  float2 s = {0.f, 0.f};
  template <int N>
  __device__ __forceinline__ void add(const float* g, const float* x) {
#pragma unroll
    for (int w = 0; w < N; w += 2)
      s = fma2(make_float2(g[w], g[w + 1]), make_float2(x[w], x[w + 1]), s);
  }
  __device__ __forceinline__ void add1(float g, float x) { s.x = fmaf(g, x, s.x); }
  __device__ __forceinline__ float total() const { return s.x + s.y; }
};
struct Acc64 {
  double s = 0.0;
  template <int N>
  __device__ __forceinline__ void add(const double* g, const double* x) {
#pragma unroll
    for (int w = 0; w < N; ++w) s = fma(g[w], x[w], s);
  }
  __device__ __forceinline__ void add1(double g, double x) { s = fma(g, x, s); }
  __device__ __forceinline__ double total() const { return s; }
};

// HELD: the CTA's rows of G^ are copied to shared memory; else they are streamed by
// every product (from L2 when the batch's G^ fits it).
template <typename TG, typename TI, bool HELD, int T>
__global__ void __launch_bounds__(T, sizeof(TI) == 4 ? 768 / T : 1)
    k_inner_cluster(const InnerCta* __restrict__ ctas, const InnerGroup* __restrict__ groups,
                    const int32_t* __restrict__ cols, InnerClass C, const TG* __restrict__ ghat,
                    const double* __restrict__ g64, const double* __restrict__ z064,
                    double* __restrict__ z64, KScal* __restrict__ sc,
                    const KScal* __restrict__ outer, double tol, int maxit) {
  using AT = typename Vec<TG>::acc;
  using Sums = typename std::conditional<sizeof(AT) == 8, Acc64, Acc32>::type;
  using W = typename Wide<TI>::W;
  constexpr int VN = Vec<TG>::n, R = kInnerRows;
  constexpr int NW = T / 32;
  // the next size class is independent of this one: it may start at once
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  cg::cluster_group cl = cg::this_cluster();
  const int cs = (int)cl.num_blocks(), rank = (int)cl.block_rank();
  const InnerCta c = ctas[C.cta0 + blockIdx.x];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* at = smem;
  auto take = [&](size_t bytes) {
    unsigned char* p = at;
    at += up16(bytes);
    return p;
  };
  TG* G = HELD ? (TG*)take((size_t)C.g_elems * sizeof(TG)) : nullptr;
  AT* xs = (AT*)take((size_t)C.cols * sizeof(AT));  // the product's input on the coupling columns
  TI* r = (TI*)take((size_t)C.rows * sizeof(TI));
  TI* rh = (TI*)take((size_t)C.rows * sizeof(TI));
  TI* sv = (TI*)take((size_t)C.rows * sizeof(TI));
  TI* t = (TI*)take((size_t)C.rows * sizeof(TI));
  TI* z = (TI*)take((size_t)C.rows * sizeof(TI));
  // p and v alternate between two arrays: the other CTAs form the new p on their
  // coupling columns from the old p and v while this one already writes the new ones
  TI* pbuf = (TI*)take((size_t)2 * C.rows * sizeof(TI));
  TI* vbuf = (TI*)take((size_t)2 * C.rows * sizeof(TI));
  int32_t* ci = (int32_t*)take((size_t)C.cols * sizeof(int32_t));
  InnerGroup* gr = (InnerGroup*)take((size_t)C.groups * sizeof(InnerGroup));
  __shared__ __align__(16) W wsum[2][3][NW];       // the warps' partial sums
  __shared__ __align__(16) W csum[4][3][kMaxCs];   // the CTAs', per step of an iteration
  __shared__ double part64[kMaxCs * NW];

  for (int i = tid; i < c.ngrp; i += T) gr[i] = groups[c.grp0 + i];
  for (int i = tid; i < c.ncol; i += T) ci[i] = cols[c.col0 + i];
  const int64_t q = c.q0 + c.row0;
  double ref2 = 0.0;
  for (int i = tid; i < c.nrows; i += T) {
    const double gv = g64[q + i];
    ref2 += gv * gv;
  }
  __syncthreads();
  for (int gi = warp; HELD && gi < c.ngrp; gi += NW) {  // the rows of G^, 16 bytes per load
    const InnerGroup& e = gr[gi];
    const int n16 = (int)((size_t)e.nrows * e.ld * sizeof(TG) / 16);
    const uint4* __restrict__ src = reinterpret_cast<const uint4*>(ghat + e.gsrc);
    uint4* dst = reinterpret_cast<uint4*>(G + e.goff);
#pragma unroll 8
    for (int i = lane; i < n16; i += 32) dst[i] = __ldcs(src + i);
  }

  auto barrier = [&]() {
    if (cs > 1)
      cl.sync();
    else
      __syncthreads();
  };
  // out = x + G x on the own rows; at(rank, i) gives entry i of CTA rank's slice of x
  // (formed from vectors that stand since the last barrier)
  auto product = [&](const TI* x, TI* out, auto at) {
    for (int i = tid; i < c.ncol; i += T) {
      const int32_t e = ci[i];
      xs[i] = (AT)at((uint32_t)e >> kRankShift, e & ((1 << kRankShift) - 1));
    }
    __syncthreads();
    for (int gi = warp; gi < c.ngrp; gi += NW) {
      const InnerGroup e = gr[gi];
      const TG* __restrict__ g0 = HELD ? G + e.goff : ghat + e.gsrc;
      const AT* xe = xs + e.xoff;
      Sums acc[R];
      const int nvec = e.nc / VN;
      for (int k = lane; k < nvec; k += 32) {
        AT xv[VN];
#pragma unroll
        for (int w = 0; w < VN; w += 16 / (int)sizeof(AT)) Vec<AT>::load(xe + k * VN + w, xv + w);
#pragma unroll
        for (int u = 0; u < R; ++u) {
          AT gv[VN];
          Vec<TG>::load(g0 + min(u, e.nrows - 1) * e.ld + k * VN, gv);
          acc[u].template add<VN>(gv, xv);
        }
      }
      for (int j = nvec * VN + lane; j < e.nc; j += 32) {
#pragma unroll
        for (int u = 0; u < R; ++u) acc[u].add1((AT)g0[min(u, e.nrows - 1) * e.ld + j], xe[j]);
      }
      AT s[R];
#pragma unroll
      for (int u = 0; u < R; ++u) s[u] = acc[u].total();
      // the R sums over the lanes, halving the rows a lane carries in the first
      // steps: lane l ends with row l / (32 / R)
#pragma unroll
      for (int h = R / 2, o = 16; h >= 1; h /= 2, o /= 2) {
        const bool up = lane & o;
#pragma unroll
        for (int u = 0; u < h; ++u) {
          const AT give = up ? s[u] : s[u + h];
          const AT keep = up ? s[u + h] : s[u];
          s[u] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
      }
#pragma unroll
      for (int o = 16 / R; o > 0; o >>= 1) s[0] += __shfl_xor_sync(0xffffffffu, s[0], o);
      const int u = lane / (32 / R);
      if (lane % (32 / R) == 0 && u < e.nrows) out[e.row + u] = (TI)((AT)x[e.row + u] + s[0]);
    }
    __syncthreads();
  };
  // N sums over the cluster: over the lanes, over the CTA's warps (one warp), written
  // to every CTA, one cluster barrier, and over the CTAs by every warp for itself, in
  // one fixed order: all threads hold the sums and form the same scalars.  `slot`:
  // the step's own exchange slot, so that a fast CTA's next sums never meet a
  // slow CTA's reads.
  auto reduce = [&](int slot, auto& a) {
    constexpr int N = sizeof(a) / sizeof(W);
    if (c.nrows > warp * 32) {  // warps without rows hold zeros
#pragma unroll
      for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int n = 0; n < N; ++n) a[n] = sum(a[n], shfl_xor(a[n], o));
    }
    if (lane == 0)
#pragma unroll
      for (int n = 0; n < N; ++n) wsum[slot & 1][n][warp] = a[n];
    __syncthreads();
    if (warp == 0 || cs == 1) {
#pragma unroll
      for (int n = 0; n < N; ++n) a[n] = lane < NW ? wsum[slot & 1][n][lane] : W{};
#pragma unroll
      for (int o = NW / 2; o > 0; o >>= 1)
#pragma unroll
        for (int n = 0; n < N; ++n) a[n] = sum(a[n], shfl_xor(a[n], o));
#pragma unroll
      for (int n = 0; n < N; ++n) a[n] = bcast(a[n]);
    }
    if (cs > 1) {
      if (warp == 0 && lane < cs)
#pragma unroll
        for (int n = 0; n < N; ++n) st_peer(&csum[slot][n][rank], lane, a[n]);
      cl.sync();
#pragma unroll
      for (int n = 0; n < N; ++n) a[n] = lane < cs ? csum[slot][n][lane] : W{};
      for (int o = cs / 2; o > 0; o >>= 1)
#pragma unroll
        for (int n = 0; n < N; ++n) a[n] = sum(a[n], shfl_xor(a[n], o));
#pragma unroll
      for (int n = 0; n < N; ++n) a[n] = bcast(a[n]);
    }
#pragma unroll
    for (int n = 0; n < N; ++n) a[n] = settle(a[n]);
  };

  barrier();  // every CTA of the cluster runs before its shared memory is written
  {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ref2 += __shfl_xor_sync(0xffffffffu, ref2, o);
    if (lane < cs) st_peer(&part64[rank * NW + warp], lane, ref2);
    barrier();
    ref2 = 0.0;
    for (int d = lane; d < cs * NW; d += 32) ref2 += part64[d];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ref2 += __shfl_xor_sync(0xffffffffu, ref2, o);
  }
  const double ref = sqrt(ref2);
  // power of two that brings ||g|| to [2^20, 2^21) (FP32 vectors only)
  int ex = 0;
  if (sizeof(TI) == 4 && ref > 0.0 && ref < 1e300) ex = max(-1000, min(1000, ilogb(ref) - 20));
  const double down = scalbn(1.0, -ex);
  W rr[1] = {};  // ||r||^2 in the vectors' precision
  for (int i = tid; i < c.nrows; i += T) {
    const TI gv = (TI)(g64[q + i] * down);
    r[i] = gv;
    z[i] = TI(0);
    rr[0] = sum(rr[0], mul(gv, gv));
  }
  reduce(0, rr);
  // stop when ||r|| <= tol ||g||, as squares
  const W lim = Wide<TI>::make(tol * tol * (down * down) * ref2);
  bool active = ref > 0.0 && !(outer && !outer[c.sys].active), guess = false;
  if (z064 && active) {  // the guess is taken when its residual is smaller than that of zero
    const W r0 = rr[0];
    for (int i = tid; i < c.nrows; i += T) z[i] = (TI)(z064[q + i] * down);
    barrier();
    product(z, t, [&](uint32_t rk, int i) { return ld_peer(z + i, rk); });
    rr[0] = W{};
    for (int i = tid; i < c.nrows; i += T) {
      const TI rv = r[i] - t[i];
      sv[i] = rv;
      rr[0] = sum(rr[0], mul(rv, rv));
    }
    reduce(1, rr);
    guess = less(rr[0], r0);
    if (guess && at_most(rr[0], lim)) active = false;
    for (int i = tid; i < c.nrows; i += T) {
      if (guess)
        r[i] = sv[i];
      else
        z[i] = TI(0);
    }
    if (!guess) rr[0] = r0;
  }
  // rho = (rh, r) with rh = r; the first p is r (beta = 0)
  W rho = rr[0], alpha = Wide<TI>::make(1.0), omega = alpha, beta{}, bo{};  // bo = -beta omega
  bool breakdown = value(rho) == TI(0);
  double iters = 0.0;
  for (int i = tid; i < c.nrows; i += T) rh[i] = r[i];
  if (active) barrier();
  for (int it = 1; active; ++it) {
    const TI *p0 = pbuf + (it & 1) * C.rows, *v0 = vbuf + (it & 1) * C.rows;
    TI *p = pbuf + (~it & 1) * C.rows, *v = vbuf + (~it & 1) * C.rows;
    auto next_p = [&](TI rv, TI pv, TI vv) { return lin(rv, beta, pv, bo, vv); };
    for (int i = tid; i < c.nrows; i += T) p[i] = it == 1 ? r[i] : next_p(r[i], p0[i], v0[i]);
    product(p, v, [&](uint32_t rk, int i) {
      const TI rv = ld_peer(r + i, rk);
      return it == 1 ? rv : next_p(rv, ld_peer(p0 + i, rk), ld_peer(v0 + i, rk));
    });
    W a[1] = {};
    for (int i = tid; i < c.nrows; i += T) a[0] = sum(a[0], mul(rh[i], v[i]));
    reduce(1, a);
    if (value(a[0]) == TI(0)) {
      breakdown = true;
      alpha = W{};
    } else {
      alpha = quot(rho, a[0]);
    }
    const W na = neg(alpha);
    auto next_s = [&](TI rv, TI vv) { return lin(rv, na, vv); };
    for (int i = tid; i < c.nrows; i += T) sv[i] = next_s(r[i], v[i]);
    product(sv, t, [&](uint32_t rk, int i) { return next_s(ld_peer(r + i, rk), ld_peer(v + i, rk)); });
    // (t, s), (t, t) and ||s||^2 with one barrier: the half-step check comes after
    // the second product, which its last iteration then does not use
    W b[3] = {};
    for (int i = tid; i < c.nrows; i += T) {
      b[0] = sum(b[0], mul(t[i], sv[i]));
      b[1] = sum(b[1], mul(t[i], t[i]));
      b[2] = sum(b[2], mul(sv[i], sv[i]));
    }
    reduce(2, b);
    if (at_most(b[2], lim)) {  // the half step
      for (int i = tid; i < c.nrows; i += T) z[i] = lin(z[i], alpha, p[i]);
      iters = it - 0.5;
      break;
    }
    if (breakdown) {
      iters = it;
      break;
    }
    omega = value(b[1]) != TI(0) ? quot(b[0], b[1]) : W{};
    const W ao = quot(alpha, omega);  // not used if omega is zero
    W d[2] = {};
    for (int i = tid; i < c.nrows; i += T) {
      z[i] = lin(z[i], alpha, p[i], omega, sv[i]);
      const TI rv = lin(sv[i], neg(omega), t[i]);
      r[i] = rv;
      d[0] = sum(d[0], mul(rv, rv));
      d[1] = sum(d[1], mul(rh[i], rv));
    }
    reduce(3, d);
    iters = it;
    if (at_most(d[0], lim) || value(omega) == TI(0) || it >= maxit) break;
    breakdown = value(d[1]) == TI(0);
    const W ratio = quot(d[1], rho);
    beta = mul(ratio, ao);
    bo = neg(mul(ratio, alpha));
    rho = d[1];
  }
  const double up = scalbn(1.0, ex);
  for (int i = tid; i < c.nrows; i += T) z64[q + i] = (double)z[i] * up;
  if (rank == 0 && tid == 0) {
    KScal k{};
    k.ref = ref;
    k.iters = iters;
    k.flag = guess;
    sc[c.sys] = k;
  }
  barrier();  // no CTA leaves while another may still read from it
  // the launch that follows the last class must find every class finished
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace

static void plan_mode(const InnerInput& in, bool held, InnerPlan& P) {
  P.classes.clear();
  P.h_ctas.clear();
  P.h_groups.clear();
  P.h_cols.clear();
  struct Sys {
    int cs = 0;
    size_t smem = 0;
    std::vector<InnerCta> ctas;
    std::vector<InnerGroup> groups;
    std::vector<int32_t> cols;
  };
  auto need = [&](int64_t g, int64_t cols, int64_t rows, int64_t grp) {
    return up16(held ? g * in.size_g : 0) + up16(cols * in.size_acc) + 5 * up16(rows * in.size_i) +
           2 * up16(2 * rows * in.size_i) +
           up16(cols * 4) + up16(grp * (int64_t)sizeof(InnerGroup));
  };
  // system s over cs CTAs, by entries of G^ and (32 each) rows
  auto split = [&](int32_t s, int cs, int64_t total, Sys& y) {
    const int64_t q0 = in.sys_c_ptr[s], m = in.sys_c_ptr[s + 1] - q0;
    y = Sys();
    int64_t done = 0, row = 0;
    int32_t b = in.sys_block_ptr[s];
    std::vector<int32_t> first;
    for (int rk = 0; rk < cs; ++rk) {
      InnerCta c{};
      c.sys = s;
      c.q0 = (int32_t)q0;
      c.row0 = (int32_t)row;
      c.grp0 = (int32_t)y.groups.size();
      c.col0 = (int32_t)y.cols.size();
      first.push_back((int32_t)row);
      const int64_t upto = total * (rk + 1) / cs;
      int64_t gel = 0;
      while (row < m && (done < upto || rk == cs - 1)) {
        while (q0 + row >= in.gq1[b]) ++b;
        const int64_t ld = in.gld[b], nc = in.gcol_ptr[b + 1] - in.gcol_ptr[b];
        int64_t n = 0;  // rows of block b up to the share's end
        while (q0 + row + n < in.gq1[b] && (done < upto || rk == cs - 1)) {
          done += ld + 32;
          ++n;
        }
        const int32_t xoff = (int32_t)(y.cols.size() - c.col0);
        for (int64_t j = in.gcol_ptr[b]; j < in.gcol_ptr[b + 1]; ++j)
          y.cols.push_back((int32_t)(in.gcols_panel[j] - q0));
        for (int64_t i = 0; i < n; i += kInnerRows) {
          InnerGroup g{};
          g.nrows = (int32_t)std::min<int64_t>(kInnerRows, n - i);
          g.gsrc = in.ghat_off[b] + (q0 + row + i - in.gq0[b]) * ld;
          g.goff = (int32_t)gel;
          g.row = (int32_t)(row + i - c.row0);
          g.xoff = xoff;
          g.nc = (int32_t)nc;
          g.ld = (int32_t)ld;
          gel += g.nrows * ld;
          y.groups.push_back(g);
        }
        // the next block's gathered vector starts on a 16-byte boundary (16-byte loads)
        while ((y.cols.size() - c.col0) % 4) y.cols.push_back(0);
        row += n;
      }
      c.nrows = (int32_t)row - c.row0;
      c.ngrp = (int32_t)y.groups.size() - c.grp0;
      c.ncol = (int32_t)y.cols.size() - c.col0;
      y.smem = std::max(y.smem, need(gel, c.ncol, c.nrows, c.ngrp));
      y.ctas.push_back(c);
    }
    for (int32_t& j : y.cols) {  // column -> CTA and place in its slice
      const int rk = (int)(std::upper_bound(first.begin(), first.end(), j) - first.begin()) - 1;
      j = (int32_t)(((uint32_t)rk << kRankShift) | (uint32_t)(j - first[rk]));
    }
  };
  std::vector<Sys> all;
  for (int32_t s = 0; s < in.nsys; ++s) {
    const int64_t m = in.sys_c_ptr[s + 1] - in.sys_c_ptr[s];
    int64_t total = 0, ent = 0;
    for (int32_t b = in.sys_block_ptr[s]; b < in.sys_block_ptr[s + 1]; ++b) {
      total += (in.gq1[b] - in.gq0[b]) * (in.gld[b] + 32);
      ent += (in.gq1[b] - in.gq0[b]) * in.gld[b];
    }
    if (ent * in.size_g > (held ? (int64_t)(kMaxCs * kSmemMax) : kStreamMax)) return;
    // CTAs per system.  Held: about 128 rows each (two rounds of row groups for eight
    // warps), with FP64 products also about 1,024 entries; more where the rows
    // would not fit.  Streamed: as many as a cluster takes.
    int cs = held ? 1 : kMaxCs;
    while (cs < kMaxCs && (m > 128 * cs || (in.size_acc == 8 && ent > 1024 * cs))) cs *= 2;
    Sys y;
    for (;; cs *= 2) {
      split(s, cs, total, y);
      if (y.smem <= kSmemMax || cs == kMaxCs) break;
    }
    if (y.smem > kSmemMax) return;
    y.cs = cs;
    all.push_back(std::move(y));
  }
  // Launches by cluster size and by how many CTAs fit an SM, the largest first (its
  // systems run longest; the others fill in behind them).
  const size_t tier[5] = {kSmemMax, 107 * 1024, 69 * 1024, 50 * 1024, 0};
  for (int k = 0; k < 4; ++k)
    for (int cs = kMaxCs; cs >= 1; cs /= 2) {
      InnerClass C{};
      C.cs = cs;
      C.cta0 = (int32_t)P.h_ctas.size();
      for (const Sys& y : all) {
        if (y.cs != cs || y.smem > tier[k] || y.smem <= tier[k + 1]) continue;
        const int32_t g0 = (int32_t)P.h_groups.size(), c0 = (int32_t)P.h_cols.size();
        for (InnerCta c : y.ctas) {
          int32_t gel = 0;
          for (int32_t i = c.grp0; i < c.grp0 + c.ngrp; ++i) gel += y.groups[i].nrows * y.groups[i].ld;
          C.g_elems = std::max(C.g_elems, gel);
          C.cols = std::max(C.cols, c.ncol);
          C.rows = std::max(C.rows, c.nrows);
          C.groups = std::max(C.groups, c.ngrp);
          c.grp0 += g0;
          c.col0 += c0;
          P.h_ctas.push_back(c);
        }
        P.h_groups.insert(P.h_groups.end(), y.groups.begin(), y.groups.end());
        P.h_cols.insert(P.h_cols.end(), y.cols.begin(), y.cols.end());
      }
      C.ncta = (int32_t)P.h_ctas.size() - C.cta0;
      if (!C.ncta) continue;
      C.smem = need(C.g_elems, C.cols, C.rows, C.groups);
      if (C.smem > kSmemMax) return;
      C.held = held;
      P.classes.push_back(C);
    }
  P.ok = held || (int64_t)P.h_ctas.size() <= in.nsm;
}

// Held in shared memory if every system of the handle fits a cluster (1.7 MB), however
// many there are: G^ is read once per solve.  One system of 384 rows takes 8.9 us an
// iteration (loop 31); 256 systems of 1,100 rows 9.4 ms per five reduced solves (loop
// 20.2; streamed with all systems resident it was the slower, 8.9 ms where held took 8.0,
// bound by reading 98 MB per product).
// Otherwise streamed, when there are so few systems that all run at once; else
// the plan is not ok and the loop takes them.
void plan_inner_cluster(const InnerInput& in, InnerPlan& P) {
  P.ok = false;
  for (int held = 1; held >= 0 && !P.ok; --held) plan_mode(in, held != 0, P);
}


template <typename TG, typename TI>
int launch_inner_cluster(const InnerPlan& P, const TG* ghat, const double* g64, const double* z064,
                         double* z64, KScal* sc, const KScal* outer, double tol, int maxit,
                         cudaStream_t s) {
  constexpr int T = inner_threads(sizeof(TI));
  for (size_t k = 0; k < P.classes.size(); ++k) {
    const InnerClass& C = P.classes[k];
    auto kern = C.held ? k_inner_cluster<TG, TI, true, T> : k_inner_cluster<TG, TI, false, T>;
    record_launch_error(
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)C.ncta);
    cfg.blockDim = dim3((unsigned)T);
    cfg.dynamicSmemBytes = C.smem;
    cfg.stream = s;
    cudaLaunchAttribute a[2];
    a[0].id = cudaLaunchAttributeClusterDimension;
    a[0].val.clusterDim.x = (unsigned)C.cs;
    a[0].val.clusterDim.y = 1;
    a[0].val.clusterDim.z = 1;
    a[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = a;
    cfg.numAttrs = k ? 2 : 1;  // the first class waits for the work before it
    record_launch_error(
        cudaLaunchKernelEx(&cfg, kern, P.ctas, P.groups, P.cols, C, ghat, g64, z064, z64, sc, outer, tol,
                           maxit));
  }
  return (int)P.classes.size();
}

#define DDPS_INST(TG, TI)                                                                         \
  template int launch_inner_cluster<TG, TI>(const InnerPlan&, const TG*, const double*,          \
                                            const double*, double*, KScal*, const KScal*, double, \
                                            int, cudaStream_t);
DDPS_INST(double, double)
DDPS_INST(float, double)
DDPS_INST(float, float)
DDPS_INST(__nv_bfloat16, float)
DDPS_INST(__nv_bfloat16, double)
DDPS_INST(__half, float)
DDPS_INST(__half, double)

}  // namespace ddps
