// Incomplete LU with zero fill, ILU(0), of every diagonal block (Sec. 3: the
// block factors of Fig. 2 step 2 may be approximate; the paper names
// incomplete LU as that choice), and the triangular solves that use it:
// the block solves of Fig. 3 (6.1, 6.5) and the multi-right-hand-side spike
// solves of Fig. 2 step 4.
//
// The factors live on the pattern of the blocks, in their own row order:
// one CSR array (values in the factor precision) holds L below the diagonal
// (unit diagonal implied) and U on and above it.  Row i of L depends on the
// rows k < i that it references; rows are grouped in levels (a row's level is
// one more than the largest level of those rows) so that each launch handles
// rows that are independent of one another, all blocks of all systems at
// once.  The backward solves use the levels of the U dependencies (a row's
// level is one more than the largest level of the rows j > i it references,
// so level 0 holds the rows that reference none and is solved first).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "launch.h"

namespace ddps {

namespace {

constexpr int kT = 256;

template <typename T>
__device__ __forceinline__ double to_d(T v) {
  return (double)v;
}

// Row i of the factorisation (IKJ elimination with updates outside the
// pattern left out), one thread per row of the level; small pivots are
// reported (code 1, the row) and replaced by pivot_tol * max|a_i.|.
template <typename T>
__global__ void k_ilu0_rows(const int32_t* __restrict__ rows, int32_t nrows,
                            const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                            const int32_t* __restrict__ diag, T* __restrict__ a,
                            const double* __restrict__ rownorm, double pivot_tol,
                            long long* __restrict__ err) {
  const int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nrows) return;
  const int32_t i = rows[t];
  const int32_t e0 = rp[i], e1 = rp[i + 1], di = diag[i];
  for (int32_t e = e0; e < di; ++e) {
    const int32_t k = col[e];
    const T lik = a[e] / a[diag[k]];
    a[e] = lik;
    // a_ij -= l_ik u_kj for j > k in both patterns (both rows sorted)
    int32_t p = e + 1;
    for (int32_t u = diag[k] + 1; u < rp[k + 1] && p < e1; ++u) {
      const int32_t j = col[u];
      while (p < e1 && col[p] < j) ++p;
      if (p < e1 && col[p] == j) a[p] -= lik * a[u];
    }
  }
  const double piv = to_d(a[di]);
  const double thr = pivot_tol * rownorm[i];
  if (!(fabs(piv) >= thr)) {
    if (atomicCAS((unsigned long long*)&err[0], 0ull, 1ull) == 0ull) {
      err[1] = -1;
      err[2] = i;
    }
    a[di] = (T)(piv < 0 ? -thr : thr);
  }
}

// One right-hand side: forward x_i -= sum_{k<i} l_ik x_k (unit diagonal), or
// backward x_i = (x_i - sum_{j>i} u_ij x_j) / u_ii, over the rows of a level.
template <typename T, bool FWD>
__global__ void k_ilu_vec(const int32_t* __restrict__ rows, int32_t nrows,
                          const int32_t* __restrict__ rp, const int32_t* __restrict__ col,
                          const int32_t* __restrict__ diag, const T* __restrict__ a,
                          T* __restrict__ x) {
  const int32_t t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nrows) return;
  const int32_t i = rows[t];
  T s = x[i];
  if (FWD) {
    for (int32_t e = rp[i]; e < diag[i]; ++e) s -= a[e] * x[col[e]];
    x[i] = s;
  } else {
    for (int32_t e = diag[i] + 1; e < rp[i + 1]; ++e) s -= a[e] * x[col[e]];
    x[i] = s / a[diag[i]];
  }
}

// A whole block solve g = (L~ U~)^-1 y in one launch, one CTA per block (the blocks are
// independent), instead of one launch per level and sweep: the levels are a chain of
// dependent steps of a few hundred rows each (158 of them for a 37 x 37 x 7 slab), and a
// launch costs far more than a step.  A step is one block barrier: thread t takes row t of
// the level, whose packed row (see IluSweep) it has copied asynchronously, 16 bytes at a
// time, into its own places of a ring in shared memory some steps before; the vector is
// in shared memory too (in its block of `w` where it does not fit).  The sums run in the
// order of the rows' entries, as in k_ilu_vec: bitwise the same result.  Bound by the
// chain of steps.  On the 37^3 grid in five slabs a solve takes 73 us against 770 for
// the launches (120 with 4-byte copies of each row's parts: twenty copies a step and
// thread kept the load unit busy longer than the step).
template <typename T, int Q, int NT>
struct IluRing {
  static constexpr int row_bytes = Q * 4 * (4 + (int)sizeof(T));
  static constexpr int fit = 64 * 1024 / (NT * row_bytes);
  static constexpr int ahead = fit < 2 ? 2 : fit > 6 ? 6 : fit;
  int4 c[ahead][Q][NT];
  T v[ahead][Q][NT][4];
};
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}

// Q: packed groups of four (row number or diagonal, then entries) in the ring; longer
// rows read their further groups from global memory.
template <typename T, int Q, int NT, bool SMEM>
__global__ void __launch_bounds__(NT)
    k_ilu_solve(IluSweep L, IluSweep U, const T* __restrict__ lval, const T* __restrict__ uval,
                int64_t n, const int64_t* __restrict__ block_ptr, int32_t lev_bytes,
                const double* __restrict__ y, T* __restrict__ w, double* __restrict__ g) {
  using Ring = IluRing<T, Q, NT>;
  constexpr int kAhead = Ring::ahead;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Ring& R = *reinterpret_cast<Ring*>(smem_raw);
  const int b = blockIdx.x, tid = threadIdx.x;
  const int64_t r0 = block_ptr[b];
  const int32_t nb = (int32_t)(block_ptr[b + 1] - r0);
  // the level starts of both sweeps (their loads would stall every step), then the vector
  int32_t* slev = reinterpret_cast<int32_t*>(smem_raw + sizeof(Ring));
  T* x = SMEM ? reinterpret_cast<T*>(smem_raw + sizeof(Ring) + lev_bytes) : w + r0;
  const int32_t nlev[2] = {L.lev_off[b + 1] - L.lev_off[b], U.lev_off[b + 1] - U.lev_off[b]};
  if (lev_bytes)
    for (int32_t i = tid; i < nlev[0] + nlev[1]; i += NT)
      slev[i] = i < nlev[0] ? L.lev[L.lev_off[b] + i] : U.lev[U.lev_off[b] + i - nlev[0]];
#pragma unroll 8
  for (int32_t i = tid; i < nb; i += NT) x[i] = (T)y[r0 + i];
  __syncthreads();
#pragma unroll
  for (int dir = 0; dir < 2; ++dir) {
    const IluSweep& S = dir ? U : L;
    const int4* __restrict__ col = reinterpret_cast<const int4*>(S.col);
    const T* __restrict__ val = dir ? uval : lval;
    const int nl = nlev[dir] - 1, ng = S.groups;
    auto level = [&](int32_t l) {
      return lev_bytes ? slev[dir * nlev[0] + l] : S.lev[S.lev_off[b] + l];
    };
    int32_t ct0 = level(0);  // start of the next level to copy
    auto copy = [&](int32_t l, int q) {  // one group of copies per step, empty past the end
      if (l < nl) {
        const int32_t t = ct0 + tid;
        ct0 = level(l + 1);
        if (t < ct0) {
#pragma unroll
          for (int k = 0; k < Q; ++k)
            if (k < ng) {
              copy16(&R.c[q][k][tid], col + (int64_t)k * n + t);
              const T* v = val + ((int64_t)k * n + t) * 4;
#pragma unroll
              for (int h = 0; h < (int)sizeof(T) / 4; ++h)
                copy16(&R.v[q][k][tid][h * 16 / (int)sizeof(T)], v + h * 16 / (int)sizeof(T));
            }
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    // s minus the entries of one packed group from entry k0 on (no entry: 0 times 0)
    auto take = [&](T s, int4 c, const T* v, int k0) {
      const T x0 = k0 == 0 && c.x >= 0 ? x[c.x] : T(0), x1 = c.y >= 0 ? x[c.y] : T(0);
      const T x2 = c.z >= 0 ? x[c.z] : T(0), x3 = c.w >= 0 ? x[c.w] : T(0);
      if (k0 == 0) s -= v[0] * x0;
      s -= v[1] * x1;
      s -= v[2] * x2;
      s -= v[3] * x3;
      return s;
    };
    auto rest = [&](int32_t t, T s, int k) {  // groups from k on, from global memory
      for (; k < ng; ++k) {
        const int4 c = col[(int64_t)k * n + t];
        if (c.x < 0) break;
        s = take(s, c, val + ((int64_t)k * n + t) * 4, 0);
      }
      return s;
    };
    for (int q = 0; q < kAhead - 1; ++q) copy(q, q);
    int slot = 0, next = kAhead - 1;
    int32_t t1 = level(0);
    for (int32_t l = 0; l < nl; ++l) {
      copy(l + kAhead - 1, next);
      const int32_t t0 = t1;
      t1 = level(l + 1);
      asm volatile("cp.async.wait_group %0;" ::"n"(kAhead - 1) : "memory");
      if (t0 + tid < t1) {  // a thread reads what it has copied itself
        const int4 c = R.c[slot][0][tid];
        T s = take(x[c.x], c, R.v[slot][0][tid], 1);
#pragma unroll
        for (int k = 1; k < Q; ++k)
          if (k < ng) s = take(s, R.c[slot][k][tid], R.v[slot][k][tid], 0);
        if (ng > Q) s = rest(t0 + tid, s, Q);
        x[c.x] = dir ? s / R.v[slot][0][tid][0] : s;
      }
      for (int32_t t = t0 + NT + tid; t < t1; t += NT) {  // rows beyond the CTA's threads
        const int4 c = col[t];
        const T* v = val + (int64_t)t * 4;
        const T s = rest(t, take(x[c.x], c, v, 1), 1);
        x[c.x] = dir ? s / v[0] : s;
      }
      slot = slot + 1 == kAhead ? 0 : slot + 1;
      next = next + 1 == kAhead ? 0 : next + 1;
      __syncthreads();
    }
  }
#pragma unroll 8
  for (int32_t i = tid; i < nb; i += NT) g[r0 + i] = (double)x[i];
}

// Packed coefficients of a sweep from the factor's values (src < 0: padding).
template <typename T>
__global__ void k_ilu_pack(const T* __restrict__ a, const int32_t* __restrict__ src, int64_t cnt,
                           T* __restrict__ out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = src[i] >= 0 ? a[src[i]] : T(0);
}

// The same on the spike panel X (row-major, NR columns): one CTA per (row,
// 256 columns); a row of block b touches the columns [0, ncols_b - j0) of
// the chunk that hold its coupling columns.
template <typename T, bool FWD>
__global__ void __launch_bounds__(kT)
    k_ilu_panel(const int32_t* __restrict__ rows, const int32_t* __restrict__ rp,
                const int32_t* __restrict__ col, const int32_t* __restrict__ diag,
                const T* __restrict__ a, const int32_t* __restrict__ row_block,
                const int64_t* __restrict__ block_ncols, int64_t j0, int32_t NR, int32_t nchunk,
                T* __restrict__ X) {
  const int32_t t = blockIdx.x / nchunk;
  const int32_t c = (blockIdx.x - t * nchunk) * kT + threadIdx.x;
  const int32_t i = rows[t];
  const int64_t nc = min((int64_t)NR, block_ncols[row_block[i]] - j0);
  if (c >= nc) return;
  T s = X[(int64_t)i * NR + c];
  if (FWD) {
    for (int32_t e = rp[i]; e < diag[i]; ++e) s -= a[e] * X[(int64_t)col[e] * NR + c];
    X[(int64_t)i * NR + c] = s;
  } else {
    for (int32_t e = diag[i] + 1; e < rp[i + 1]; ++e) s -= a[e] * X[(int64_t)col[e] * NR + c];
    X[(int64_t)i * NR + c] = s / a[diag[i]];
  }
}

inline int blocks_for(int64_t n) { return (int)((n + kT - 1) / kT); }

}  // namespace

template <typename T>
void launch_ilu0_level(const int32_t* rows, int32_t nrows, const IluDev& L, T* a,
                       const double* rownorm, double pivot_tol, long long* err, cudaStream_t s) {
  if (nrows <= 0) return;
  k_ilu0_rows<T><<<blocks_for(nrows), kT, 0, s>>>(rows, nrows, L.rp, L.col, L.diag, a, rownorm,
                                                  pivot_tol, err);
}

template <typename T>
void launch_ilu_vec_level(bool fwd, const int32_t* rows, int32_t nrows, const IluDev& L,
                          const T* a, T* x, cudaStream_t s) {
  if (nrows <= 0) return;
  if (fwd)
    k_ilu_vec<T, true><<<blocks_for(nrows), kT, 0, s>>>(rows, nrows, L.rp, L.col, L.diag, a, x);
  else
    k_ilu_vec<T, false><<<blocks_for(nrows), kT, 0, s>>>(rows, nrows, L.rp, L.col, L.diag, a, x);
}

template <typename T>
void launch_ilu_panel_level(bool fwd, const int32_t* rows, int32_t nrows, const IluDev& L,
                            const T* a, const int64_t* block_ncols, int64_t j0, int32_t NR, T* X,
                            cudaStream_t s) {
  if (nrows <= 0) return;
  const int32_t nchunk = (NR + kT - 1) / kT;
  const int64_t grid = (int64_t)nrows * nchunk;
  if (fwd)
    k_ilu_panel<T, true><<<(unsigned)grid, kT, 0, s>>>(rows, L.rp, L.col, L.diag, a, L.row_block,
                                                       block_ncols, j0, NR, nchunk, X);
  else
    k_ilu_panel<T, false><<<(unsigned)grid, kT, 0, s>>>(rows, L.rp, L.col, L.diag, a, L.row_block,
                                                        block_ncols, j0, NR, nchunk, X);
}

template <typename T>
void launch_ilu_pack(const T* a, const int32_t* src, int64_t cnt, T* out, cudaStream_t s) {
  if (cnt > 0) k_ilu_pack<T><<<(int)std::min<int64_t>(blocks_for(cnt), 152 * 16), kT, 0, s>>>(a, src, cnt, out);
}

constexpr size_t kIluSmem = 220 * 1024;
// level starts in shared memory; very many of them stay in global memory
static size_t lev_bytes(int32_t max_starts) {
  const size_t lev = ((size_t)max_starts * 4 + 15) / 16 * 16;
  return lev > kIluSmem / 8 ? 0 : lev;
}

template <typename T, int Q, int NT>
static void launch_solve(int32_t nblocks, int64_t max_rows, int32_t max_starts, const IluSweep& L,
                         const IluSweep& U, const T* lval, const T* uval, int64_t n,
                         const int64_t* block_ptr, const double* y, T* w, double* g, cudaStream_t s) {
  const size_t lev = lev_bytes(max_starts), ring = sizeof(IluRing<T, Q, NT>);
  const size_t sm = ring + lev + (size_t)max_rows * sizeof(T);
  if (sm <= kIluSmem) {
    record_launch_error(cudaFuncSetAttribute(k_ilu_solve<T, Q, NT, true>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kIluSmem));
    k_ilu_solve<T, Q, NT, true><<<nblocks, NT, sm, s>>>(L, U, lval, uval, n, block_ptr,
                                                        (int32_t)lev, y, w, g);
  } else {
    record_launch_error(cudaFuncSetAttribute(k_ilu_solve<T, Q, NT, false>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kIluSmem));
    k_ilu_solve<T, Q, NT, false><<<nblocks, NT, ring + lev, s>>>(L, U, lval, uval, n, block_ptr,
                                                          (int32_t)lev, y, w, g);
  }
}

// A CTA walks its block alone: a step of at most as many rows as it has threads takes 0.4 us
// (vector in shared memory) or 1.5 (in global memory), every further round of a wider level,
// whose rows were not copied ahead, 1 or 2.6; FP64 half as much again.  A launch per level
// takes 5.5 us, and its rows spread over all SMs.  Measured, one launch against a launch per
// level in us, FP32: 64^3 in 16 slabs 88 / 1,434, in two 1,240 / 1,679; 96^3 in eight 1,346 /
// 2,354, in two 4,579 / 2,709; 128^3 in two 10,956 / 4,037; a 1000 x 1000 grid in two 4,392 /
// 16,255; eight levels of 62,500 rows 2,805 / 67, of 625 rows 21 / 46.
template <typename T>
bool ilu_one_launch(int32_t nblocks, int64_t max_rows, int32_t max_starts, int32_t groups,
                    int threads, const int32_t* steps, const int64_t* rounds, int32_t launches) {
  const size_t ring = groups <= 1 ? (threads == 256 ? sizeof(IluRing<T, 1, 256>) : sizeof(IluRing<T, 1, 512>))
                                  : (threads == 256 ? sizeof(IluRing<T, 2, 256>) : sizeof(IluRing<T, 2, 512>));
  size_t sm = ring + lev_bytes(max_starts) + (size_t)max_rows * sizeof(T);
  const bool shared = sm <= kIluSmem;
  if (!shared) sm = ring + lev_bytes(max_starts);
  const double step = shared ? 0.4 : 1.5, more = shared ? 1.0 : 2.6;
  double longest = 0.0;
  for (int32_t b = 0; b < nblocks; ++b)
    longest = std::max(longest, step * steps[b] + more * (double)(rounds[b] - steps[b]));
  if (sizeof(T) == 8) longest *= 1.5;
  const int per_sm = (int)std::max<size_t>(1, std::min<size_t>(1024 / threads, 227 * 1024 / (sm + 1024)));
  const int at_once = per_sm * device_sm_count();
  return longest * ((nblocks + at_once - 1) / at_once) <= 5.5 * launches;
}

// max_level: rows of the widest level of a block.  256 threads while two rounds
// cover it (a barrier of eight warps is cheaper), else 512; three entries a row in the
// ring for the 5- and 7-point grids, else seven.
template <typename T>
void launch_ilu_solve(int32_t nblocks, int64_t max_rows, int32_t max_level, int32_t max_starts,
                      const IluSweep& L, const IluSweep& U, const T* lval, const T* uval, int64_t n,
                      const int64_t* block_ptr, const double* y, T* w, double* g, cudaStream_t s) {
  auto run = [&](auto fn) { fn(nblocks, max_rows, max_starts, L, U, lval, uval, n, block_ptr, y, w, g, s); };
  const bool narrow = std::max(L.groups, U.groups) <= 1, small = ilu_threads(max_level) == 256;
  if (narrow)
    run(small ? launch_solve<T, 1, 256> : launch_solve<T, 1, 512>);
  else
    run(small ? launch_solve<T, 2, 256> : launch_solve<T, 2, 512>);
}

#define DDPS_INST_ILU(T)                                                                         \
  template void launch_ilu0_level<T>(const int32_t*, int32_t, const IluDev&, T*, const double*, \
                                     double, long long*, cudaStream_t);                         \
  template void launch_ilu_pack<T>(const T*, const int32_t*, int64_t, T*, cudaStream_t);         \
  template bool ilu_one_launch<T>(int32_t, int64_t, int32_t, int32_t, int, const int32_t*,       \
                                  const int64_t*, int32_t);                                      \
  template void launch_ilu_solve<T>(int32_t, int64_t, int32_t, int32_t, const IluSweep&,         \
                                    const IluSweep&,                                             \
                                    const T*, const T*, int64_t, const int64_t*,                 \
                                    const double*, T*, double*, cudaStream_t);                   \
  template void launch_ilu_vec_level<T>(bool, const int32_t*, int32_t, const IluDev&, const T*, \
                                        T*, cudaStream_t);                                      \
  template void launch_ilu_panel_level<T>(bool, const int32_t*, int32_t, const IluDev&,         \
                                          const T*, const int64_t*, int64_t, int32_t, T*,       \
                                          cudaStream_t);
DDPS_INST_ILU(double)
DDPS_INST_ILU(float)

}  // namespace ddps
