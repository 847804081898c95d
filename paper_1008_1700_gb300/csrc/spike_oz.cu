// The four spike GEMM ops of spike.cu for FP64 factors on the tensor cores, in fixed
// point (the splitting scheme of Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 2012).
//
// FP64 runs at 1/64 of the FP32 rate here: on the FP64 pipe these products took 262 ms of a
// 300 ms step (48^3, eight slabs), at three quarters of that pipe's peak.  Instead every row
// of A and every column of B is scaled by its own power of two to a 55-bit integer (which
// holds the 53-bit significand of its largest entry exactly) and cut into seven signed 8-bit
// digits.  Digits are exact in bf16; their products and the sums of a level (the digit pairs
// of one weight) over 128 values of K stay below 2^24 and so are exact in the FP32
// accumulators.  34 MMAs per 16 values of K give the eight upper levels; what is left out is
// below 2^-58 of the row's times the column's largest entry.  Every 128 values of K the levels
// are added, exactly, to a pair of 64-bit integers, and one rounding at the end turns them
// into an FP64 number.  G^ of 24^2 .. 96^2 and 12^3 .. 20^3 grids against a refined
// long-double solution: 1.8e-16 .. 2.8e-16 relative (2.5e-16 .. 3.7e-16 with FP64 FMAs).
//
// The products are bound by latency and issue slots, not by the MMAs (13% of the tensor
// pipe at the roots, 3 to 8% below them): cutting an entry costs some 50 instructions, rounding a
// result 80, and most fronts have one to four 32-column stages.  So a CTA of 512 threads takes
// 32 front rows (N of the MMA) times 128 panel columns (M: a thread holds a column, its
// accesses are coalesced), with 64 registers and 256 tensor-memory columns, and two CTAs
// share an SM: one's loads and rounding run beside the other's products.  A's digits are cut
// once per factorisation (k_oz_pack) and come with one bulk copy per stage; B's are cut by
// all threads from the panel, in integer arithmetic.  48^3, eight slabs, FP64: forward and
// backward products 54.7 + 207 -> 12.0 + 34.7 ms, the packing (0.9 ms) included (the zero
// halves of the triangles skipped; 12.5 + 36.2 with them); tiles of 64 rows, one CTA per SM:
// 12.7 + 40.7 ms with 1,024 threads, 14.2 + 45.2 with 512; 128 rows by 64 columns: 18.9 + 67.4.
// Every wait is bounded; a wait that runs out records error code 2.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "launch.h"
#include "tc_common.cuh"

namespace ddps {

namespace {

constexpr int OZ_D = 7, OZ_L = 8;           // digits, levels
constexpr int OZ_R = oz_tile_m(), OZ_C = 128, OZ_T = 512;  // front rows (N) and panel columns (M) of a tile
constexpr int OZ_RPT = OZ_R * OZ_C / OZ_T, OZ_KPT = TC_BK * OZ_C / OZ_T;  // rows of C, of a stage of B per thread
static_assert(OZ_R % TC_BK == 0, "a tile's first row starts a stage of K");
static_assert(OZ_RPT == 8 && OZ_KPT % 4 == 0, "shares of a thread");
constexpr int OZ_GROUP = 4;                 // stages of 32 between two drains: 128 values of K
constexpr uint32_t OZ_ATILE = OZ_R * TC_BK * 2, OZ_BTILE = OZ_C * TC_BK * 2;
constexpr uint32_t OZ_ABLK = OZ_D * OZ_ATILE, OZ_BBLK = OZ_D * OZ_BTILE;
constexpr uint32_t OZ_SMEM = 2 * OZ_ABLK + OZ_BBLK;
constexpr int OZ_NONE = -8192, OZ_INF = 1 << 20;  // exponents of zero and of infinity or NaN
static_assert(OZ_C == TC_BM, "lanes of the tensor memory: panel columns");
static_assert(OZ_D * 128 * 128 * OZ_GROUP * TC_BK < (1 << 24), "a level's sum is exact in FP32");

// Biased exponent of x (denormals: 1), OZ_NONE of zero, OZ_INF of infinity and NaN.
__device__ __forceinline__ int expo(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x) << 1;
  const int e = (int)(b >> 53);
  return b == 0ull ? OZ_NONE : e == 0x7ff ? OZ_INF : max(e, 1);
}

// x 2^(53 + sh) / 2^(e_max) as an integer, where sh = 1 - (largest biased exponent): below
// 2^54; biased by 128 in each of seven bytes, so that byte q minus 128 is digit q.
__device__ __forceinline__ unsigned long long fixed(double x, int sh) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = (b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0ull);
  const int p = min(max(e, 1) + sh, 1);  // 1 for the largest binade
  unsigned long long v;
  if (p >= 0)
    v = m << p;
  else
    v = p < -60 ? 0ull : (m + (1ull << (-p - 1))) >> -p;
  return (b >> 63 ? 0ull - v : v) + 0x0080808080808080ull;
}

// Digit bytes of two values as a pair of bf16: byte q of w0 (low half) and of w1.
__device__ __forceinline__ uint32_t digit_pair(unsigned long long w0, unsigned long long w1, int q) {
  const uint32_t a = q < 4 ? (uint32_t)w0 : (uint32_t)(w0 >> 32);
  const uint32_t b = q < 4 ? (uint32_t)w1 : (uint32_t)(w1 >> 32);
  // 2^23 + byte as a float, minus 2^23 + 128
  const float f = __uint_as_float(__byte_perm(a, 0x4B000000u, 0x7540u | (q & 3))) - 8388736.f;
  const float g = __uint_as_float(__byte_perm(b, 0x4B000000u, 0x7540u | (q & 3))) - 8388736.f;
  return __byte_perm(__float_as_uint(f), __float_as_uint(g), 0x7632);
}

// M rows and K of an op for front f, and A's entry (row, column); zero outside.
template <int OP>
struct OzA {
  const double* __restrict__ A;
  int32_t m, k, M, K;
  __device__ __forceinline__ OzA(const DevFronts& F, int32_t f, const double* arena)
      : A(arena + F.arena[f]), m(F.m[f]), k(F.k[f]) {
    M = OP == OP_FWD_L21 ? m - k : k;
    K = OP == OP_BWD_U12 ? m - k : k;
  }
  __device__ __forceinline__ double at(int i, int j) const {
    if (i >= M || j >= K) return 0.0;
    if (OP == OP_FWD_LINV) return i > j ? A[i + (int64_t)j * m] : (i == j ? 1.0 : 0.0);
    if (OP == OP_BWD_UINV) return i <= j ? A[i + (int64_t)j * m] : 0.0;
    return A[(OP == OP_FWD_L21 ? k + i : i) + (int64_t)(OP == OP_BWD_U12 ? k + j : j) * m];
  }
};

// Units of the equations (r) and the unknowns (c): the exponents with which the entries
// 2^-(r_i + c_j) a_ij of the matrix come closest to 1 (Curtis and Reid, J. IMA 1972), by
// turns over rows and columns, in sixteenths, as integers (their sums are the same in any
// order).  A first row sweep starts from c = 0.
constexpr int OZ_SWEEPS = 3;
__global__ void k_oz_rows(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ colind,
                          const double* __restrict__ vals, const int32_t* __restrict__ iperm,
                          int64_t n, const int32_t* __restrict__ c, unsigned long long* __restrict__ csum,
                          int32_t* __restrict__ ccnt, int32_t* __restrict__ r) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t a = rowptr[i], b = rowptr[i + 1];
  long long s = 0;
  int cnt = 0;
  for (int32_t t = a; t < b; ++t) {
    const int e = expo(vals[t]);
    if (e != OZ_NONE) s += 16 * (min(e, 0x7ff) - 1023) - c[colind[t]], ++cnt;
  }
  const int ri = cnt ? (int)(s / cnt) : 0;
  r[iperm[i]] = (int32_t)(ri >= 0 ? ri + 8 : ri - 8) / 16;
  for (int32_t t = a; t < b; ++t) {
    const int e = expo(vals[t]);
    if (e == OZ_NONE) continue;
    atomicAdd(&csum[colind[t]], (unsigned long long)(long long)(16 * (min(e, 0x7ff) - 1023) - ri));
    atomicAdd(&ccnt[colind[t]], 1);
  }
}

__global__ void k_oz_cols(int64_t n, const int32_t* __restrict__ iperm,
                          unsigned long long* __restrict__ csum,
                          int32_t* __restrict__ ccnt, int32_t* __restrict__ c16, int32_t* __restrict__ c) {
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= n) return;
  const int cj = ccnt[j] ? (int)((long long)csum[j] / ccnt[j]) : 0;
  csum[j] = 0ull;
  ccnt[j] = 0;
  c16[j] = cj;
  c[iperm[j]] = (cj >= 0 ? cj + 8 : cj - 8) / 16;
}

// The unit of row gk of an op's B (a panel of equations or of unknowns); A's columns have
// its inverse, so that the digits of both need not span different units.  Without it random
// units of 10^-3 .. 10^3 cost four of G^'s sixteen digits (2e-12); with it, none (3e-16).
template <int OP>
__device__ __forceinline__ int oz_unit(const OzUnits& U, const int32_t* idx, int64_t row0, int k, int gk) {
  return OP == OP_BWD_U12 ? -U.c[idx[k + gk]] : U.r[row0 + gk];
}

// A packed tile: the exponents of its 64 rows, then per 32 columns of K seven digit tiles,
// the largest digit first, each 64 x 32 K-major.
constexpr int OZ_HEAD = OZ_R * 4;

template <int OP>
__global__ void __launch_bounds__(256)
    k_oz_scale(DevFronts F, OzUnits U, const int32_t* __restrict__ tile_front,
               const int32_t* __restrict__ tile_m0, const int64_t* __restrict__ tile_aoff,
               const double* __restrict__ arena, unsigned char* __restrict__ out) {
  __shared__ int ex[OZ_R];
  const int32_t f = tile_front[blockIdx.x];
  const OzA<OP> A(F, f, arena);
  const int32_t* idx = F.idx + F.idx_off[f];
  const int64_t row0 = F.row0[f];
  const int m0 = tile_m0[blockIdx.x], tid = threadIdx.x, row = tid % OZ_R;
  if (tid < OZ_R) ex[tid] = OZ_NONE;
  __syncthreads();
  int e = OZ_NONE;
#pragma unroll 4
  for (int j = tid / OZ_R; j < A.K; j += 256 / OZ_R) {
    const int x = expo(A.at(m0 + row, j));
    if (x != OZ_NONE) e = max(e, x + oz_unit<OP>(U, idx, row0, A.k, j));
  }
  atomicMax(&ex[row], e);
  __syncthreads();
  if (tid < OZ_R) reinterpret_cast<int*>(out + tile_aoff[blockIdx.x])[tid] = ex[tid];
}

template <int OP>
__global__ void __launch_bounds__(OZ_R * 4)
    k_oz_pack(DevFronts F, OzUnits U, const int32_t* __restrict__ tile_front,
              const int32_t* __restrict__ tile_m0, const int64_t* __restrict__ tile_aoff,
              const double* __restrict__ arena, unsigned char* __restrict__ out) {
  const int32_t f = tile_front[blockIdx.x];
  const OzA<OP> A(F, f, arena);
  const int32_t* idx = F.idx + F.idx_off[f];
  const int64_t row0 = F.row0[f];
  const int nk = (A.K + TC_BK - 1) / TC_BK;
  const int m0 = tile_m0[blockIdx.x], row = threadIdx.x % OZ_R, kc = threadIdx.x / OZ_R;
  unsigned char* dst = out + tile_aoff[blockIdx.x];
  const int e = reinterpret_cast<const int*>(dst)[row];
  for (int kt = blockIdx.y; kt < nk; kt += gridDim.y) {
    const int g0 = kt * TC_BK + kc * 8;
    unsigned char* blk = dst + OZ_HEAD + (int64_t)kt * OZ_ABLK;
    unsigned long long w[8];
#pragma unroll
    for (int t = 0; t < 8; ++t)
      w[t] = g0 + t < A.K ? fixed(A.at(m0 + row, g0 + t), 1 - e + oz_unit<OP>(U, idx, row0, A.k, g0 + t))
                          : fixed(0.0, 0);
#pragma unroll
    for (int q = 0; q < OZ_D; ++q)
      *reinterpret_cast<uint4*>(blk + (OZ_D - 1 - q) * OZ_ATILE + chunk_off(row, kc)) =
          make_uint4(digit_pair(w[0], w[1], q), digit_pair(w[2], w[3], q),
                     digit_pair(w[4], w[5], q), digit_pair(w[6], w[7], q));
  }
}

// (hi 2^32 + lo) 2^s rounded to FP64 (nearest, ties to even).
__device__ __forceinline__ double to_double(long long hi, long long lo, int s) {
  hi += lo >> 32;
  uint32_t l = (uint32_t)lo;
  const bool neg = hi < 0;
  if (neg) {
    l = 0u - l;
    hi = ~hi + (l == 0u);
  }
  unsigned long long h = (unsigned long long)hi, m;
  int z;
  uint32_t sticky = 0u;
  if (h) {
    z = __clzll((long long)h);
    m = z <= 32 ? (h << z) | ((unsigned long long)l >> (32 - z)) : (h << z) | ((unsigned long long)l << (z - 32));
    if (z < 32) sticky = l << z;
  } else {
    if (!l) return 0.0;
    z = 32 + __clz((int)l);
    m = (unsigned long long)l << z;
    z += 32;
  }
  unsigned long long r = m >> 11;
  const uint32_t rem = ((uint32_t)m & 0x7ffu) | (sticky ? 1u : 0u);
  r += rem > 0x400u || (rem == 0x400u && (r & 1ull));
  int e = 1023 + 95 - z + s;  // biased exponent of r's leading bit (2^52)
  if (r >> 53) {
    r >>= 1;
    ++e;
  }
  if (e <= 0 || e >= 0x7ff) {  // outside the normal range
    const double d = ldexp((double)r, e - 1075);
    return neg ? -d : d;
  }
  return __longlong_as_double((long long)((r & 0xfffffffffffffull) | ((unsigned long long)e << 52) |
                                          (neg ? 1ull << 63 : 0ull)));
}

template <int OP>
__global__ void __launch_bounds__(OZ_T, 2)
    k_spike_gemm_oz(DevFronts F, OzUnits U, const int32_t* __restrict__ tile_front,
                    const int32_t* __restrict__ tile_m0, const int64_t* __restrict__ tile_aoff,
                    const unsigned char* __restrict__ packed, const int64_t* __restrict__ block_ncols,
                    int64_t j0, int32_t NR, double* __restrict__ X, double* __restrict__ Tb,
                    long long* __restrict__ err) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[2], empty[2];
  __shared__ uint32_t tmem_slot;
  __shared__ int cex[OZ_C], rex[OZ_R];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int32_t f = tile_front[blockIdx.x];
  const int32_t m0 = tile_m0[blockIdx.x];
  const int n0 = blockIdx.y * OZ_C;
  const unsigned char* head = packed + tile_aoff[blockIdx.x];
  const int32_t k = F.k[f], m = F.m[f];
  const int64_t row0 = F.row0[f], tb0 = F.idx_off[f];
  const int64_t ncols = min((int64_t)NR, block_ncols[F.block[f]] - j0);
  if (n0 >= ncols) return;  // uniform over the CTA, before any tcgen05 work
  const int M = OP == OP_FWD_L21 ? m - k : k, K = OP == OP_BWD_U12 ? m - k : k;
  const int rows = min(OZ_R, M - m0);
  const int32_t* __restrict__ idx = F.idx + tb0;
  // the triangles' columns of these rows: up to the last row's (L11^-1), from the first (U11^-1)
  const int k0 = OP == OP_BWD_UINV ? m0 : 0, k1 = OP == OP_FWD_LINV ? min(K, m0 + OZ_R) : K;
  int nk = (k1 - k0 + TC_BK - 1) / TC_BK;
  const unsigned char* apk = head + OZ_HEAD + (int64_t)(k0 / TC_BK) * OZ_ABLK;
  const uint32_t sbase = smem_u32(smem);
  int issued = 0, committed = 0;  // thread 0
  auto fetch_a = [&](int kt) {
    const uint32_t bar = smem_u32(&full[kt & 1]);
    mbar_expect_tx(bar, OZ_ABLK);
    bulk_g2s(sbase + (kt & 1) * OZ_ABLK, apk + (int64_t)kt * OZ_ABLK, OZ_ABLK, bar);
    issued = kt + 1;
  };
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[i])));
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int kt = 0; kt < min(nk, 2); ++kt) fetch_a(kt);
  }
  if (tid < OZ_C) cex[tid] = OZ_NONE - 4096;
  if (tid < OZ_R) rex[tid] = reinterpret_cast<const int*>(head)[tid];

  const double* Bp = (OP == OP_FWD_L21 || OP == OP_BWD_U12) ? X : Tb;
  auto brow = [&](int gk) -> int64_t {
    return OP == OP_FWD_L21 ? row0 + gk : OP == OP_BWD_U12 ? (int64_t)idx[k + gk] : tb0 + gk;
  };
  // this thread's panel column, and rows OZ_KPT bk .. of a stage
  const int bc = tid % OZ_C, bk = tid / OZ_C;
  const bool live = n0 + bc < ncols;
  double breg[OZ_KPT];
  int ureg[OZ_KPT];
  auto load_b = [&](int kt) {
    const int g0 = k0 + kt * TC_BK + bk * OZ_KPT;
#pragma unroll
    for (int t = 0; t < OZ_KPT; ++t) {
      const bool in = g0 + t < k1;
      breg[t] = live && in ? Bp[brow(g0 + t) * NR + n0 + bc] : 0.0;
      ureg[t] = in ? oz_unit<OP>(U, idx, row0, k, g0 + t) : 0;
    }
  };
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"((uint32_t)(OZ_L * OZ_R)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;

  // the columns' exponents over all of K; stage 0 stays in registers
  int be = OZ_NONE - 4096;
  for (int kt = nk - 1; kt >= 0; --kt) {
    load_b(kt);
#pragma unroll
    for (int t = 0; t < OZ_KPT; ++t)
      if (breg[t] != 0.0) be = max(be, expo(breg[t]) - ureg[t]);
  }
  if (be > OZ_NONE - 4096) atomicMax(&cex[bc], be);
  // a tile of zeros (fronts that these columns' right-hand sides do not reach) has no products
  if (!__syncthreads_or(be > OZ_NONE)) nk = 0;
  be = cex[bc];

  // this thread's results: panel column 32 quarter + lane, front rows r1 .. r1 + 7
  const int quarter = warp & 3, r1 = (warp >> 2) * OZ_RPT;
  long long hi[OZ_RPT], lo[OZ_RPT];
#pragma unroll
  for (int u = 0; u < OZ_RPT; ++u) hi[u] = lo[u] = 0;
  auto drain = [&]() {  // the levels' exact sums into hi 2^32 + lo
    if (r1 >= rows) return;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
    for (int l = 0; l < OZ_L; ++l) {
      uint32_t rv[8];
      const uint32_t taddr = tmem + (uint32_t)(l * OZ_R + r1) + ((uint32_t)(quarter * 32) << 16);
      asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                   : "=r"(rv[0]), "=r"(rv[1]), "=r"(rv[2]), "=r"(rv[3]), "=r"(rv[4]), "=r"(rv[5]),
                     "=r"(rv[6]), "=r"(rv[7])
                   : "r"(taddr));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int u = 0; u < OZ_RPT; ++u) {
        const long long v = __float2int_rn(__uint_as_float(rv[u]));
        if (l < 4)
          hi[u] += v << (8 * (3 - l));
        else
          lo[u] += v << (8 * (7 - l));
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  };

  // N: the rows of this tile in steps of 16
  const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(((rows + 15) / 16 * 16) >> 3) << 17) |
                         ((uint32_t)(OZ_C >> 4) << 24);
  bool timed_out = false;
  for (int kt = 0; kt < nk; ++kt) {
    const int st = kt & 1;
    if (kt > 0 && !timed_out)
      timed_out = !mbar_wait(smem_u32(&empty[st ^ 1]), ((kt - 1) >> 1) & 1, err);
    const uint32_t aS = sbase + st * OZ_ABLK, bS = sbase + 2 * OZ_ABLK;
    unsigned char* sB = smem + 2 * OZ_ABLK;
    if (tid == 0 && kt >= 2 && !timed_out) fetch_a(kt);
#pragma unroll
    for (int g = 0; g < OZ_KPT / 4; ++g) {
      unsigned long long w[4];
#pragma unroll
      for (int t = 0; t < 4; ++t) w[t] = fixed(breg[g * 4 + t], 1 - be - ureg[g * 4 + t]);
      const int k4 = bk * OZ_KPT / 4 + g;
      const uint32_t off = chunk_off(bc, k4 >> 1) + (k4 & 1) * 8;
#pragma unroll
      for (int q = 0; q < OZ_D; ++q)
        *reinterpret_cast<uint2*>(sB + (OZ_D - 1 - q) * OZ_BTILE + off) =
            make_uint2(digit_pair(w[0], w[1], q), digit_pair(w[2], w[3], q));
    }
    if (kt + 1 < nk) load_b(kt + 1);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    const bool first = kt % OZ_GROUP == 0;
    timed_out = __syncthreads_or(timed_out);  // all threads give up together
    if (timed_out) break;
    if (first && kt > 0) {
      drain();
      __syncthreads();
    }
    if (tid == 0) {
      timed_out = !mbar_wait(smem_u32(&full[st]), (kt >> 1) & 1, err);
      if (!timed_out) {  // else the others learn of it at the next barrier
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t dA = make_desc(aS, 128, kSBO), dB = make_desc(bS, 128, kSBO);
#pragma unroll
        for (int kk = 0; kk < TC_BK / 16; ++kk) {
#pragma unroll
          for (int l = 0; l < OZ_L; ++l)
#pragma unroll
            for (int i = 0; i < OZ_D; ++i) {
              const int j = l - i;
              if (j < 0 || j >= OZ_D) continue;
              const bool start = i == (l < OZ_D ? 0 : l - OZ_D + 1) && first && kk == 0;
              mma_bf16_n(tmem + (uint32_t)(l * OZ_R), dB + ((j * OZ_BTILE + kk * 256) >> 4),
                         dA + ((i * OZ_ATILE + kk * 256) >> 4), idesc, start ? 0u : 1u);
            }
        }
        mma_commit(smem_u32(&empty[st]));
        committed = kt + 1;
      }
    }
  }
  if (nk > 0 && !timed_out)
    timed_out = !mbar_wait(smem_u32(&empty[(nk - 1) & 1]), ((nk - 1) >> 1) & 1, err);
  timed_out = __syncthreads_or(timed_out);
  if (timed_out) {
    if (tid == 0) atomicCAS((unsigned long long*)&err[0], 0ull, 2ull);
  } else if (nk > 0) {
    drain();
  }
  if (tid == 0 && (timed_out || nk == 0)) {  // let this thread's copies and MMAs complete
    for (int g = max(0, issued - 2); g < issued; ++g) mbar_drain(smem_u32(&full[g & 1]), (g >> 1) & 1);
    for (int g = max(0, committed - 2); g < committed; ++g)
      mbar_drain(smem_u32(&empty[g & 1]), (g >> 1) & 1);
  }
  const int c = quarter * 32 + lane;
  if (n0 + c < ncols && r1 < rows && !timed_out) {
    const int64_t r0 = row0 + m0 + r1, t0 = tb0 + m0 + r1;
    double* out;
    const double* cin = nullptr;
    if (OP == OP_FWD_LINV || OP == OP_BWD_UINV) {
      out = X + r0 * NR + n0 + c;
    } else if (OP == OP_FWD_L21) {
      out = Tb + (t0 + k) * NR + n0 + c;
      cin = out;
    } else {
      out = Tb + t0 * NR + n0 + c;
      cin = X + r0 * NR + n0 + c;
    }
    const int ce = cex[c];
#pragma unroll
    for (int u = 0; u < OZ_RPT; ++u) {
      if (r1 + u >= rows) break;
      const int re = rex[r1 + u];
      // units: 2^(re - 1022 - 54) 2^(ce - 1022 - 54) 2^40
      double v = to_double(hi[u], lo[u], re + ce - 2 * 1022 - 2 * 54 + 40);
      if (re >= OZ_INF || ce > OZ_INF / 2) v = __longlong_as_double(0x7ff8000000000000ll);
      out[(int64_t)u * NR] = cin ? cin[(int64_t)u * NR] - v : v;
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"((uint32_t)(OZ_L * OZ_R)));
}

template <int OP>
void pack_one(DevFronts F, OzUnits U, const int32_t* tf, const int32_t* tm, const int64_t* ta, int32_t nt,
              int32_t max_kt, const double* arena, unsigned char* out, cudaStream_t s) {
  k_oz_scale<OP><<<nt, 256, 0, s>>>(F, U, tf, tm, ta, arena, out);
  k_oz_pack<OP><<<dim3(nt, std::min(max_kt, 8)), OZ_R * 4, 0, s>>>(F, U, tf, tm, ta, arena, out);
}

template <int OP>
void gemm_one(DevFronts F, OzUnits U, const int32_t* tf, const int32_t* tm, const int64_t* ta,
              const unsigned char* packed, int32_t nt, const int64_t* block_ncols, int64_t j0,
              int32_t NR, double* X, double* Tb, long long* err, cudaStream_t s) {
  const size_t sm = OZ_SMEM;
  record_launch_error(
      cudaFuncSetAttribute(k_spike_gemm_oz<OP>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
  k_spike_gemm_oz<OP><<<dim3(nt, (NR + OZ_C - 1) / OZ_C), OZ_T, sm, s>>>(F, U, tf, tm, ta, packed,
                                                                         block_ncols, j0, NR, X, Tb, err);
}

}  // namespace

int64_t oz_tile_bytes(int K) {
  const int nk = (K + TC_BK - 1) / TC_BK;
  return OZ_HEAD + (int64_t)nk * OZ_ABLK;
}

void launch_oz_units(const int32_t* rowptr, const int32_t* colind, const double* vals,
                     const int32_t* iperm, int64_t n, int32_t* work, OzUnits U, cudaStream_t s) {
  unsigned long long* csum = reinterpret_cast<unsigned long long*>(work);
  int32_t *c16 = work + 2 * n, *ccnt = work + 3 * n;
  record_launch_error(cudaMemsetAsync(work, 0, 4 * n * sizeof(int32_t), s));
  const unsigned g = (unsigned)((n + 255) / 256);
  for (int q = 0; q < OZ_SWEEPS; ++q) {
    k_oz_rows<<<g, 256, 0, s>>>(rowptr, colind, vals, iperm, n, c16, csum, ccnt, U.r);
    k_oz_cols<<<g, 256, 0, s>>>(n, iperm, csum, ccnt, c16, U.c);
  }
}

void launch_oz_pack(int op, DevFronts F, OzUnits U, const int32_t* tile_front, const int32_t* tile_m0,
                    const int64_t* tile_aoff, int32_t ntiles, int32_t max_kt, const double* arena,
                    unsigned char* packed, cudaStream_t s) {
  if (ntiles <= 0 || max_kt <= 0) return;
  auto f = op == OP_FWD_LINV ? pack_one<OP_FWD_LINV> : op == OP_FWD_L21 ? pack_one<OP_FWD_L21>
           : op == OP_BWD_U12 ? pack_one<OP_BWD_U12> : pack_one<OP_BWD_UINV>;
  f(F, U, tile_front, tile_m0, tile_aoff, ntiles, max_kt, arena, packed, s);
}

void launch_spike_gemm_oz(int op, DevFronts F, OzUnits U, const int32_t* tile_front, const int32_t* tile_m0,
                          const int64_t* tile_aoff, const unsigned char* packed, int32_t ntiles,
                          const int64_t* block_ncols, int64_t j0, int32_t NR, double* X, double* Tb,
                          long long* err, cudaStream_t s) {
  if (ntiles <= 0) return;
  auto f = op == OP_FWD_LINV ? gemm_one<OP_FWD_LINV> : op == OP_FWD_L21 ? gemm_one<OP_FWD_L21>
           : op == OP_BWD_U12 ? gemm_one<OP_BWD_U12> : gemm_one<OP_BWD_UINV>;
  f(F, U, tile_front, tile_m0, tile_aoff, packed, ntiles, block_ncols, j0, NR, X, Tb, err, s);
}

}  // namespace ddps
