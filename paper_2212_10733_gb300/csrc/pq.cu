// Product quantisation of the latent space (Sec. III Stage 3, Sec. V-B):
// per subdomain and latent dimension, K-means with k clusters; a latent value
// is stored as the index of its nearest centroid and decoded as the centroid.
//
// Training runs Lloyd iterations from k centroids evenly spaced in the
// column's range.  Each iteration is one pass over the latents: the nearest
// centroid is chosen in float32 (ties to the lowest index), and the members'
// sum is accumulated as a 64-bit fixed-point integer (value * 2^s with s set
// from the column's largest magnitude and the group's row count, so that no
// sum can overflow).  Integer sums are order-independent, so the result does
// not depend on scheduling; each value is rounded to 2^-s, at most 2^-(s+1)
// away, which moves a mean by far less than half a float32 ulp of the column's
// range.  The new centroid is the sum over the count, rounded to float32; a
// centroid without members stays.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <type_traits>

#include "aeqc_internal.cuh"
#include "workspace.cuh"

namespace aeqc {
namespace {

constexpr int PQ_THREADS = 256;

__device__ __forceinline__ float load_z(const void* z, int bf16, long long i) {
  if (bf16) return __bfloat162float(static_cast<const __nv_bfloat16*>(z)[i]);
  return static_cast<const float*>(z)[i];
}

__device__ __forceinline__ void store_z(void* z, int bf16, long long i, float v) {
  if (bf16) static_cast<__nv_bfloat16*>(z)[i] = __float2bfloat16_rn(v);
  else static_cast<float*>(z)[i] = v;
}

// float <-> int32 key with the same order (finite values)
__device__ __forceinline__ int order_key(float v) {
  const int b = __float_as_int(v);
  return b >= 0 ? b : b ^ 0x7FFFFFFF;
}
__device__ __forceinline__ float key_value(int k) {
  return __int_as_float(k >= 0 ? k : k ^ 0x7FFFFFFF);
}

__device__ __forceinline__ long long group_lo(const long long* off, int g, long long n) {
  return off ? off[g] : 0;
}
__device__ __forceinline__ long long group_hi(const long long* off, int g, long long n) {
  return off ? off[g + 1] : n;
}

// The table of one group in shared memory as [k][L] (the lanes of a warp are
// consecutive dimensions: any centroid indices they read lie in different
// banks for L = 32), padded with +infinity to k2 rows (k2 >= k), and per
// dimension lim: the distance up to which the bisection below may replace
// the k distances.
// The table goes through `stage` (L (k + 1) words) where there is one: written
// straight to its place, a warp's 32 centroids of a dimension fall into one bank
// (2,048 cycles of a block at L k = 2,048).
__device__ __forceinline__ void load_table(const float* table, int L, int k, int k2, float* c,
                                           int* lim, float* stage = nullptr) {
  if (stage) {
    const int ks = k | 1;  // odd: the lanes of both copies in different banks
    for (int t = threadIdx.x; t < L * k; t += blockDim.x) {
      const int dd = t / k;
      stage[dd * ks + (t - dd * k)] = table[t];
    }
    __syncthreads();
    for (int t = threadIdx.x; t < L * k; t += blockDim.x) {
      const int j = t / L;
      c[t] = stage[(t - j * L) * ks + j];
    }
  } else {
    for (int t = threadIdx.x; t < L * k; t += blockDim.x) {
      const int dd = t / k, j = t - dd * k;
      c[j * L + dd] = table[t];
    }
  }
  for (int t = L * k + threadIdx.x; t < L * k2; t += blockDim.x) c[t] = INFINITY;
  for (int t = threadIdx.x; t < L; t += blockDim.x) lim[t] = 0x7F000000;  // 2^127
  __syncthreads();
  for (int t = threadIdx.x; t < L * (k - 1); t += blockDim.x) {
    const float g = c[t + L] - c[t];  // centroid j + 1 minus centroid j of dimension t % L
    atomicMin(&lim[t % L], g > 0.f ? __float_as_int(fminf(g * 2097152.f, 1.7e38f)) : 0);
  }
  __syncthreads();
}

// Index of the nearest of the k centroids cd[j L] (float32 distances, lowest
// index on ties), by bisection in STEPS steps where that gives the same
// index.  Let gap be the smallest difference of neighbouring centroids
// (positive: they ascend) and every distance below lim = 2^21 gap.  A float
// below 2^22 gap has an ulp of at most gap / 2, so the float32 distances to
// two centroids on the same side of v, at least gap apart, round to different
// values in their own order: only the last centroid at or below v and the
// first above it can be nearest, and of these two the lower index wins a
// tie.  Anything else (equal or descending centroids, values far outside,
// NaN) takes the full search, as does STEPS = 0; the table is padded to
// 2^STEPS + 1 rows.  At k = 16: six reads instead of sixteen distances and
// selects, 176 -> 87 us for 2^20 x 32 latents (pq_encode, bound by issue).
struct Range {
  float lo, hi;  // bisection for lo < v < hi
};

// |v - c| < lim for the first and the last centroid, with room for the
// rounding of these two sums (2^-24 of 2^21 gap and of the centroids); empty
// for a table that does not ascend or is not finite
__device__ __forceinline__ Range bisect_range(const float* cd, int L, int k, int lim) {
  const float l = __int_as_float(lim), a = cd[0], b = cd[(k - 1) * L];
  const float m = l - 1e-6f * (l + fabsf(a) + fabsf(b));
  if (!(m > 0.f)) return {0.f, 0.f};
  return {b - m, a + m};
}

template <int STEPS>
__device__ __forceinline__ int nearest(float v, const float* cd, int L, int k, Range in) {
  if (STEPS > 0 && v > in.lo && v < in.hi) {
    int j = 0;
#pragma unroll
    for (int st = 1 << (STEPS > 0 ? STEPS - 1 : 0); st > 0; st >>= 1)
      j = v >= cd[(j + st) * L] ? j + st : j;
    return fabsf(v - cd[(j + 1) * L]) < fabsf(v - cd[j * L]) ? j + 1 : j;
  }
  float best = fabsf(v - cd[0]);
  int arg = 0;
  for (int j = 1; j < k; ++j) {
    const float e = fabsf(v - cd[j * L]);
    if (e < best) {
      best = e;
      arg = j;
    }
  }
  return arg;
}

// bisection steps for k centroids (2^steps >= k), rows of the padded table
inline int bisect_steps(int k) {
  int s = 1;
  while ((1 << s) < k) ++s;
  return s;
}
inline int padded_rows(int k, int steps) { return steps ? (1 << steps) + 1 : k; }

// f(std::integral_constant<int, steps>) for steps in 0..8
template <typename F>
void with_steps(int steps, F f) {
  switch (steps) {
    case 1: f(std::integral_constant<int, 1>()); break;
    case 2: f(std::integral_constant<int, 2>()); break;
    case 3: f(std::integral_constant<int, 3>()); break;
    case 4: f(std::integral_constant<int, 4>()); break;
    case 5: f(std::integral_constant<int, 5>()); break;
    case 6: f(std::integral_constant<int, 6>()); break;
    case 7: f(std::integral_constant<int, 7>()); break;
    case 8: f(std::integral_constant<int, 8>()); break;
    default: f(std::integral_constant<int, 0>()); break;
  }
}

// rn(v 2^s) for a finite float, to nearest even, on the integer pipe: the
// conversions and the product of the FP64 form are three instructions of the
// FP64 pipe, which takes one in ~64 cycles per quarter of an SM (they were
// 160 of the 226 us of a pass over 2^20 x 32 latents).  |v 2^s| < 2^62.
__device__ __forceinline__ long long fixed_of(float v, int s) {
  const unsigned u = __float_as_uint(v);
  const int E = (int)((u >> 23) & 0xffu);
  const long long m = (long long)((u & 0x7fffffu) | (E ? 0x800000u : 0u));
  const int sh = (E ? E : 1) - 150 + s;
  long long r;
  if (sh >= 0) {
    r = m << min(sh, 62);
  } else if (sh > -26) {
    r = (m + (1ll << (-sh - 1)) - 1 + ((m >> -sh) & 1)) >> -sh;
  } else {
    r = 0;  // below a quarter
  }
  return (u >> 31) ? -r : r;
}

// start centroid j of a column with the range [lo, hi]
__device__ __forceinline__ float start_centroid(double lo, double hi, int j, int k) {
  return __double2float_rn(lo + (j + 0.5) * (hi - lo) / k);
}

// scale 2^s of the fixed-point sums: |value| < 2^e, so the sum of ng values
// stays below 2^62
__device__ __forceinline__ int fixed_shift(double lo, double hi, long long ng) {
  const double amax = fmax(fabs(lo), fabs(hi));
  if (!(amax > 0.0)) return 0;
  int e = 0, lg = 0;
  frexp(amax, &e);
  while (lg < 40 && (1ll << lg) < ng) ++lg;
  return min(62 - lg - e, 1000);
}

// mean of a cluster from its fixed-point sum, rounded to float32
__device__ __forceinline__ float moved_centroid(long long sum, unsigned long long cnt, int s) {
  return __double2float_rn(ldexp((double)sum / (double)cnt, -s));
}

// The block's elements of group g: rows off[g] + blockIdx.x R + tr + i gridDim.x R
// of dimension d (R = rows per block step), PQ_UNROLL loads in flight per
// thread: a row of 2 to 4 bytes per lane is far from filling a load.
constexpr int PQ_UNROLL = 4;

template <typename F>
__device__ __forceinline__ void for_elements(const void* z, int bf16, long long n, int L,
                                             const long long* off, F body) {
  const int g = blockIdx.y;
  const long long r1 = group_hi(off, g, n);
  const int R = PQ_THREADS / L;
  const int d = threadIdx.x % L, tr = threadIdx.x / L;
  if (tr >= R) return;
  const long long step = (long long)gridDim.x * R, estep = step * L;
  long long r = group_lo(off, g, n) + (long long)blockIdx.x * R + tr;
  long long e = r * L + d;
  for (; r + (PQ_UNROLL - 1) * step < r1; r += PQ_UNROLL * step, e += PQ_UNROLL * estep) {
    float v[PQ_UNROLL];
#pragma unroll
    for (int i = 0; i < PQ_UNROLL; ++i) v[i] = load_z(z, bf16, e + i * estep);
#pragma unroll
    for (int i = 0; i < PQ_UNROLL; ++i) body(e + i * estep, d, v[i]);
  }
  for (; r < r1; r += step, e += estep) body(e, d, load_z(z, bf16, e));
}

// True in every thread of the last of the group's blocks to arrive at its
// counter; what the others wrote before is then visible.  The counter is left at
// zero.
__device__ __forceinline__ bool last_block_of_group(int* counter) {
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    last = atomicAdd(counter, 1) == (int)gridDim.x - 1;
    if (last) *counter = 0;
  }
  __syncthreads();
  if (last) __threadfence();
  return last;
}

__global__ void pq_clear_kernel(int* keys, long long* acc, unsigned long long* cnt, int GL,
                                int k) {
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < GL * k; t += gridDim.x * blockDim.x) {
    acc[t] = 0;
    cnt[t] = 0;
    if (t < GL) {
      keys[2 * t] = 0x7FFFFFFF;    // running minimum
      keys[2 * t + 1] = (int)0x80000000;  // running maximum
    }
  }
}

// Range of each column; the group's last block then sets the start centroids
// and the fixed-point scale of each dimension (one launch, and one thread per
// centroid: as a kernel of its own with a thread per column it took 11 us).  The
// group's counter is the low word of its first member count, zero until the
// iterations; theirs is its first key, which is read here for the last time.
__global__ void pq_minmax_init_kernel(const void* z, int bf16, long long n, int L,
                                      const long long* off, int* keys,
                                      unsigned long long* cnt, int k, float* table,
                                      int* shift) {
  __shared__ int smin[PQ_THREADS], smax[PQ_THREADS];
  int mn = 0x7FFFFFFF, mx = (int)0x80000000;
  for_elements(z, bf16, n, L, off, [&](long long, int, float v) {
    if (isfinite(v)) {  // a non-finite latent takes no part in training
      mn = min(mn, order_key(v));
      mx = max(mx, order_key(v));
    }
  });
  smin[threadIdx.x] = mn;
  smax[threadIdx.x] = mx;
  __syncthreads();
  if ((int)threadIdx.x < L) {  // fold the block's rows of dimension threadIdx.x
    const int R = PQ_THREADS / L;
    for (int t = 1; t < R; ++t) {
      mn = min(mn, smin[threadIdx.x + t * L]);
      mx = max(mx, smax[threadIdx.x + t * L]);
    }
    const int gd = blockIdx.y * L + threadIdx.x;
    atomicMin(&keys[2 * gd], mn);
    atomicMax(&keys[2 * gd + 1], mx);
  }
  const int g = blockIdx.y;
  if (!last_block_of_group(reinterpret_cast<int*>(&cnt[(long long)g * L * k]))) return;
  const long long ng = group_hi(off, g, n) - group_lo(off, g, n);
  for (int t = threadIdx.x; t < L * k; t += blockDim.x) {
    const int gd = g * L + t / k, j = t % k;
    const int klo = __ldcg(&keys[2 * gd]), khi = __ldcg(&keys[2 * gd + 1]);
    // an empty group, or no finite value in the column
    const bool none = ng <= 0 || klo > khi;
    const double lo = none ? 0.0 : (double)key_value(klo), hi = none ? 0.0 : (double)key_value(khi);
    table[(long long)g * L * k + t] = none ? 0.f : start_centroid(lo, hi, j, k);
    if (j == 0) shift[gd] = fixed_shift(lo, hi, ng);
  }
  __syncthreads();
  if (threadIdx.x == 0) keys[2 * g * L] = 0;
}

// One Lloyd iteration: every value is assigned to its nearest centroid and
// added to the cluster's fixed-point sum (shared-memory totals of the block,
// then one global add per cluster), and the group's last block moves the
// centroids.  The totals are pairs of 32-bit words with the carry taken from
// the value that the low word's add returns: 64-bit adds in shared memory are
// compare-and-swap loops.  Training on float32 latents of 32 dimensions, before
// (64-bit adds, FP64 conversion, full search) and now: 10^6 rows, k = 16, four
// iterations 957 and 500 us; 100,000 rows, ten iterations, k = 16 428 and 302, k =
// 64 658 and 404 us; bound by instruction issue.
template <int STEPS>
__global__ void __launch_bounds__(PQ_THREADS) pq_accum_kernel(
    const void* z, int bf16, long long n, int L, const long long* off, int k, int k2,
    float* table, const int* shift, long long* acc, unsigned long long* cnt, int* keys) {
  extern __shared__ __align__(16) unsigned char sm[];
  float* c = reinterpret_cast<float*>(sm);                     // [k2][L]
  unsigned* slo = reinterpret_cast<unsigned*>(c + L * k2);     // [k][L]
  unsigned* shi = slo + L * k;                                 // [k][L]
  unsigned* scnt = shi + L * k;                                // [k][L]
  int* lim = reinterpret_cast<int*>(scnt + L * k);             // [L]
  const int g = blockIdx.y;
  // (the sums' room, 3 L k words, for the table on its way in)
  load_table(table + (long long)g * L * k, L, k, k2, c, lim, reinterpret_cast<float*>(slo));
  for (int t = threadIdx.x; t < L * k; t += blockDim.x) slo[t] = shi[t] = scnt[t] = 0u;
  __syncthreads();
  const int s = shift[g * L + threadIdx.x % L];
  const Range in = bisect_range(c + threadIdx.x % L, L, k, lim[threadIdx.x % L]);
  for_elements(z, bf16, n, L, off, [&](long long, int d, float v) {
    if (isfinite(v)) {
      const int j = nearest<STEPS>(v, c + d, L, k, in) * L + d;
      const unsigned long long x = (unsigned long long)fixed_of(v, s);
      const unsigned lo = (unsigned)x;
      const unsigned old = atomicAdd(&slo[j], lo);
      atomicAdd(&shi[j], (unsigned)(x >> 32) + (old + lo < lo ? 1u : 0u));
      atomicAdd(&scnt[j], 1u);
    }
  });
  __syncthreads();
  // global sums in the same order [k][L]: a warp's adds fall into whole lines
  // (as [L][k], each lane's add was a transaction of its own)
  const long long g0 = (long long)g * L * k;
  for (int t = threadIdx.x; t < L * k; t += blockDim.x) {
    if (scnt[t]) {
      atomicAdd(reinterpret_cast<unsigned long long*>(&acc[g0 + t]),
                (unsigned long long)shi[t] << 32 | slo[t]);
      atomicAdd(&cnt[g0 + t], (unsigned long long)scnt[t]);
    }
  }
  if (!keys || !last_block_of_group(&keys[2 * g * L])) return;
  for (int t = threadIdx.x; t < L * k; t += blockDim.x) {
    const unsigned long long ct = __ldcg(&cnt[g0 + t]);
    const int j = t / L, gd = g * L + t - j * L;
    if (ct) table[(long long)gd * k + j] = moved_centroid(__ldcg(&acc[g0 + t]), ct, shift[gd]);
    acc[g0 + t] = 0;
    cnt[g0 + t] = 0;
  }
}

// The move of the centroids as a launch of its own, where a group has too many of
// them for one block (the division is FP64 work): 64 x 16 centroids in the block,
// 104 -> 112 us for four iterations over 10,000 rows and 138 -> 163 over 30,000.
constexpr int PQ_MOVE_IN_BLOCK = 512;

__global__ void pq_move_kernel(int G, int L, int k, const int* shift, long long* acc,
                               unsigned long long* cnt, float* table) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)G * L * k) return;
  const unsigned long long ct = cnt[t];
  const long long g = t / (L * k);
  const int u = (int)(t - g * L * k), j = u / L;
  const long long gd = g * L + u - j * L;
  if (ct) table[gd * k + j] = moved_centroid(acc[t], ct, shift[gd]);
  acc[t] = 0;
  cnt[t] = 0;
}

// ---- Lloyd on value counts (bfloat16 latents) -----------------------------------
// A bfloat16 column has at most 65,536 different values, a few thousand in
// practice (2^20 normal values: about 5,000), so it is read once, counting how
// often each bit pattern occurs, and every iteration walks the patterns: the
// member sums are integers, count * rn(v 2^s) is exactly the sum over the
// members.  One pass over the latents instead of one per iteration and one
// for the range.
constexpr int PQ_BINS = 65536;

// counts [G][L][PQ_BINS], zeroed before; elements of group g are contiguous
// in z.  VEC = 8: 16-byte loads (rows and their dimensions aligned to eight
// elements).  Bound by the rate of the L2's atomic adds.
template <int VEC>
__global__ void __launch_bounds__(256) pq_count_kernel(const uint16_t* z, long long n, int L,
                                                       const long long* off, unsigned* counts) {
  const int g = blockIdx.y;
  const long long e1 = group_hi(off, g, n) * L;
  unsigned* cg = counts + (long long)g * L * PQ_BINS;
  const long long step = (long long)gridDim.x * blockDim.x * VEC;
  long long e = group_lo(off, g, n) * L + ((long long)blockIdx.x * blockDim.x + threadIdx.x) * VEC;
  int d = (int)(e % L);
  const int dstep = (int)(step % L);
  for (; e < e1; e += step) {
    if (VEC == 8) {
      const uint4 w = __ldg(reinterpret_cast<const uint4*>(z + e));
      const unsigned u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        atomicAdd(&cg[((d + 2 * i) << 16) + (u[i] & 0xffffu)], 1u);
        atomicAdd(&cg[((d + 2 * i + 1) << 16) + (u[i] >> 16)], 1u);
      }
    } else {
      atomicAdd(&cg[(d << 16) + z[e]], 1u);
    }
    d += dstep;
    if (d >= L) d -= L;
  }
}

// The same counts with the adds in shared memory first: a block takes eight
// dimensions of a share of the rows and holds 16-bit counters for the sign,
// the mantissa and a window of PQ_WEXP exponents per dimension (its top from
// the block's first rows); values outside the window go to global memory
// directly, and the counters are added there every 65,535 rows at the
// latest.  2^20 x 32 latents: 362 us with every add in the L2 (about 93 G
// adds/s), 41 us here.
constexpr int PQ_CT = 1024;                       // threads
constexpr int PQ_WEXP = 48;                       // exponents of the window
constexpr int PQ_WBINS = 2 * PQ_WEXP * 128;       // counters per dimension
constexpr int PQ_CSMEM = 8 * PQ_WBINS * 2;        // bytes
constexpr long long PQ_CROWS = 65535 / PQ_CT * PQ_CT;  // rows between two write-outs

__global__ void __launch_bounds__(PQ_CT, 1) pq_count_window_kernel(const uint16_t* z, long long n,
                                                                   int L, const long long* off,
                                                                   unsigned* counts) {
  extern __shared__ __align__(16) unsigned char sm[];
  unsigned* w = reinterpret_cast<unsigned*>(sm);  // [8][PQ_WBINS / 2], two counters a word
  __shared__ int top[8];
  const int g = blockIdx.z, d0 = blockIdx.y * 8, tid = threadIdx.x;
  const long long g0 = group_lo(off, g, n), g1 = group_hi(off, g, n);
  const long long share = (g1 - g0 + gridDim.x - 1) / gridDim.x;
  const long long lo = g0 + blockIdx.x * share, hi = lo + share < g1 ? lo + share : g1;
  if (lo >= hi) return;
  unsigned* cg = counts + ((long long)g * L + d0) * PQ_BINS;
  for (int t = tid; t < PQ_CSMEM / 16; t += PQ_CT)
    reinterpret_cast<uint4*>(sm)[t] = make_uint4(0, 0, 0, 0);
  if (tid < 8) top[tid] = 0;
  __syncthreads();
  if (lo + tid < hi) {
    const uint4 q = __ldg(reinterpret_cast<const uint4*>(z + (lo + tid) * L + d0));
    const unsigned u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
    for (int i = 0; i < 8; ++i)
      atomicMax(&top[i], (int)((u[i >> 1] >> (16 * (i & 1) + 7)) & 0xffu));
  }
  __syncthreads();
  int base[8];  // pattern (exponent and mantissa) of the window's first counter
#pragma unroll
  for (int i = 0; i < 8; ++i) base[i] = (top[i] + 2 - PQ_WEXP) * 128;
  for (long long c0 = lo; c0 < hi; c0 += PQ_CROWS) {
    const long long c1 = c0 + PQ_CROWS < hi ? c0 + PQ_CROWS : hi;
#pragma unroll 2
    for (long long r = c0 + tid; r < c1; r += PQ_CT) {
      const uint4 q = __ldg(reinterpret_cast<const uint4*>(z + r * L + d0));
      const unsigned u[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const unsigned bits = (u[i >> 1] >> (16 * (i & 1))) & 0xffffu;
        const int m = (int)(bits & 0x7fffu) - base[i];
        if ((unsigned)m < (unsigned)(PQ_WBINS / 2)) {
          // counter m of the sign's half: the word m / 2 of it
          const int b = (int)(bits >> 15) * (PQ_WBINS / 4) + (m >> 1);
          atomicAdd(&w[i * (PQ_WBINS / 2) + b], 1u << (16 * (m & 1)));
        } else {
          atomicAdd(&cg[(i << 16) + bits], 1u);
        }
      }
    }
    __syncthreads();
    for (int t = tid; t < 8 * (PQ_WBINS / 2); t += PQ_CT) {
      const unsigned v = w[t];
      if (v == 0u) continue;
      w[t] = 0u;
      const int i = t / (PQ_WBINS / 2), b = t % (PQ_WBINS / 2);
      const int sgn = b / (PQ_WBINS / 4), m = b % (PQ_WBINS / 4) * 2;
      const int bits = (sgn << 15) + base[i] + m;
      if (v & 0xffffu) atomicAdd(&cg[(i << 16) + bits], v & 0xffffu);
      if (v >> 16) atomicAdd(&cg[(i << 16) + bits + 1], v >> 16);
    }
    __syncthreads();
  }
}

constexpr int PQ_LT = 1024;         // threads of the kernel below
constexpr int PQ_LCAP = 24 * 1024;  // distinct values held in shared memory

// All iterations of one column (a block per group and dimension): range,
// start centroids, then per iteration every distinct value (its pattern and
// count in shared memory; a column with more than PQ_LCAP of them re-reads
// its counts) to its nearest centroid.  Neighbouring lanes hold neighbouring
// values, so a warp's 32 values mostly belong to one cluster and are summed
// by shuffles before one shared-memory add.  Ten iterations over 32 columns
// of 2^20 values, k = 16: 82 us, bound by the latency of one block's steps.
__global__ void __launch_bounds__(PQ_LT, 1) pq_lloyd_counts_kernel(
    const unsigned* counts, long long n, int L, const long long* off, int k, int iters,
    float* table) {
  extern __shared__ __align__(16) unsigned char sm[];
  unsigned* ecnt = reinterpret_cast<unsigned*>(sm);                            // [PQ_LCAP]
  uint16_t* ebits = reinterpret_cast<uint16_t*>(ecnt + PQ_LCAP);               // [PQ_LCAP]
  unsigned long long* ssum = reinterpret_cast<unsigned long long*>(ebits + PQ_LCAP);  // [k]
  unsigned long long* scnt = ssum + k;                                         // [k]
  float* c = reinterpret_cast<float*>(scnt + k);                               // [k]
  __shared__ int skey[2], swarp[PQ_LT / 32];
  const int gd = blockIdx.x, g = gd / L, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const unsigned* cb = counts + (long long)gd * PQ_BINS;
  const long long ng = group_hi(off, g, n) - group_lo(off, g, n);
  if (tid == 0) {
    skey[0] = 0x7FFFFFFF;
    skey[1] = (int)0x80000000;
  }
  __syncthreads();
  // the column's finite values: range, number of distinct ones, and their
  // list in the order of their patterns (64 consecutive patterns per thread)
  constexpr int PER = PQ_BINS / PQ_LT;
  const uint4* mine = reinterpret_cast<const uint4*>(cb + tid * PER);
  int found = 0, mn = 0x7FFFFFFF, mx = (int)0x80000000;
  const auto finite = [](int bits) { return (bits & 0x7F80) != 0x7F80; };
  for (int i = 0; i < PER / 4; ++i) {
    const uint4 w = __ldg(mine + i);
    const unsigned u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int bits = tid * PER + 4 * i + q;
      if (u[q] && finite(bits)) {
        const int key = order_key(__uint_as_float((unsigned)bits << 16));
        mn = min(mn, key);
        mx = max(mx, key);
        ++found;
      }
    }
  }
  int inc = found;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) swarp[warp] = inc;
  if (found) {
    atomicMin(&skey[0], mn);
    atomicMax(&skey[1], mx);
  }
  __syncthreads();
  int at = inc - found, total = 0;
  for (int w = 0; w < PQ_LT / 32; ++w) {
    if (w < warp) at += swarp[w];
    total += swarp[w];
  }
  const bool listed = total <= PQ_LCAP;
  if (listed && found) {
    for (int i = 0; i < PER / 4; ++i) {
      const uint4 w = __ldg(mine + i);
      const unsigned u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int bits = tid * PER + 4 * i + q;
        if (u[q] && finite(bits)) {
          ecnt[at] = u[q];
          ebits[at] = (uint16_t)bits;
          ++at;
        }
      }
    }
  }
  const double lo = total ? (double)key_value(skey[0]) : 0.0;
  const double hi = total ? (double)key_value(skey[1]) : 0.0;
  const int s = fixed_shift(lo, hi, ng);
  for (int j = tid; j < k; j += PQ_LT) {
    c[j] = total ? start_centroid(lo, hi, j, k) : 0.f;
    ssum[j] = scnt[j] = 0ull;
  }
  __syncthreads();
  const int ne = listed ? total : PQ_BINS;
  for (int it = 0; it < iters && total; ++it) {
    for (int e0 = warp * 32; e0 < ne; e0 += PQ_LT) {
      const int e = e0 + lane;
      unsigned ct = 0;
      int bits = 0;
      if (e < ne) {
        bits = listed ? ebits[e] : e;
        ct = listed ? ecnt[e] : (finite(e) ? __ldg(cb + e) : 0u);
      }
      const float v = __uint_as_float((unsigned)bits << 16);
      const int j = ct ? nearest<0>(v, c, 1, k, Range{0.f, 0.f}) : -1;
      unsigned long long x = ct ? (unsigned long long)fixed_of(v, s) * ct : 0ull;
      unsigned todo = __ballot_sync(0xffffffffu, ct != 0);
      while (todo) {  // the clusters among the warp's values
        const int jl = __shfl_sync(0xffffffffu, j, __ffs((int)todo) - 1);
        unsigned long long xs = j == jl ? x : 0ull, cs = j == jl ? ct : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          xs += __shfl_xor_sync(0xffffffffu, xs, o);
          cs += __shfl_xor_sync(0xffffffffu, cs, o);
        }
        if (lane == 0) {
          atomicAdd(&ssum[jl], xs);
          atomicAdd(&scnt[jl], cs);
        }
        todo &= ~__ballot_sync(0xffffffffu, j == jl);
      }
    }
    __syncthreads();
    for (int j = tid; j < k; j += PQ_LT) {
      if (scnt[j]) c[j] = moved_centroid((long long)ssum[j], scnt[j], s);
      ssum[j] = scnt[j] = 0ull;
    }
    __syncthreads();
  }
  for (int j = tid; j < k; j += PQ_LT) table[(long long)gd * k + j] = c[j];
}

size_t lloyd_smem(int k) { return 6 * (size_t)PQ_LCAP + 20 * (size_t)k; }

// Rows per group from which the counters in shared memory pay for being
// cleared and written out: at 100,000 x 32 the counting takes 11 us with them
// and 37 us without, at 2^20 rows 41 and 362 us.
constexpr int64_t PQ_WINDOW_ROWS = 32768;

// Counts are possible for bfloat16 latents while the counts of all columns stay
// within 16 MB (64 columns) and fit 32 bits.  Ten iterations over n x 32
// latents, counted / one by one: n = 1,000 58 / 125 us, 10,000 68 / 214 us,
// 100,000 93 / 302 us.
bool use_counts(int G, int L) { return (long long)G * L <= 64; }

// The counts cost a pass of their own, so the start table alone is made without
// (100,000 x 7 latents, k = 16: 20 us, counted 50), and one iteration up to
// 2^21 values (100,000 x 7 32 / 55 us; 100,000 x 32 59 / 53 us).
bool counts_pay(int64_t n, int L, int iters) {
  return iters >= 2 || (iters == 1 && n * L >= (1 << 21));
}

template <int STEPS>
__global__ void __launch_bounds__(PQ_THREADS) pq_encode_kernel(
    const void* z, int bf16, long long n, int L, const long long* off, int k, int k2,
    const float* table, int staged, uint8_t* codes, void* zq) {
  extern __shared__ __align__(16) unsigned char sm[];
  float* c = reinterpret_cast<float*>(sm);            // [k2][L]
  int* lim = reinterpret_cast<int*>(c + L * k2);      // [L]
  load_table(table + (long long)blockIdx.y * L * k, L, k, k2, c, lim,
             staged ? reinterpret_cast<float*>(lim + L) : nullptr);
  const Range in = bisect_range(c + threadIdx.x % L, L, k, lim[threadIdx.x % L]);
  for_elements(z, bf16, n, L, off, [&](long long e, int d, float v) {
    const int j = nearest<STEPS>(v, c + d, L, k, in);
    if (codes) codes[e] = (uint8_t)j;
    if (zq) store_z(zq, bf16, e, c[j * L + d]);
  });
}

__global__ void pq_decode_kernel(const uint8_t* codes, long long n, int L, const long long* off,
                                 int k, const float* table, int bf16, void* z) {
  const int g = blockIdx.y;
  const long long r0 = group_lo(off, g, n), r1 = group_hi(off, g, n);
  const int R = PQ_THREADS / L;
  const int d = threadIdx.x % L, tr = threadIdx.x / L;
  if (tr >= R) return;
  for (long long r = r0 + (long long)blockIdx.x * R + tr; r < r1; r += (long long)gridDim.x * R) {
    const long long e = r * L + d;
    const int j = codes[e];
    store_z(z, bf16, e, j < k ? table[((long long)g * L + d) * k + j] : 0.f);
  }
}

int pq_check(int32_t latent_dtype, int64_t n, int32_t L, int32_t G, int32_t k) {
  AEQC_CHECK_ARG(latent_dtype == AEQC_DTYPE_F32 || latent_dtype == AEQC_DTYPE_BF16,
                 "pq: latent dtype %d", latent_dtype);
  AEQC_CHECK_ARG(n >= 0, "pq: n < 0");
  AEQC_CHECK_ARG(L >= 1 && L <= PQ_THREADS, "pq: L=%d out of range", L);
  AEQC_CHECK_ARG(G >= 1 && G <= 65535, "pq: G=%d out of range", G);
  AEQC_CHECK_ARG(k >= 2 && k <= AEQC_PQ_MAX_K, "pq: k=%d out of range", k);
  return AEQC_OK;
}

int pq_sms() {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// blocks per group: eight per SM over all groups, no more than give each of
// the average group's blocks one step of its unrolled rows
dim3 pq_grid(int G, int64_t n, int L) {
  const int rows = PQ_THREADS / L * PQ_UNROLL;
  const int64_t most = (n / G + rows - 1) / rows;
  int64_t c = (8 * pq_sms() + G - 1) / G;
  if (c > most) c = most;
  if (c < 1) c = 1;
  if (c > 4096) c = 4096;
  return dim3((unsigned)c, (unsigned)G);
}

// what the calls accept (L k at most about 10 K for training, 51 K for encoding)
size_t accum_limit(int L, int k) {
  const size_t e = (size_t)L * (k + 1);
  return sizeof(float) * ((e + 1) & ~(size_t)1) + 16 * e;
}
size_t accum_smem(int L, int k, int k2) { return 4 * (size_t)L * (3 * (size_t)k + k2 + 1); }
size_t encode_smem(int L, int k2) { return 4 * (size_t)L * ((size_t)k2 + 1); }

}  // namespace
}  // namespace aeqc

using namespace aeqc;

static size_t counts_bytes(int32_t G, int32_t L) {
  return use_counts(G, L) ? sizeof(unsigned) * (size_t)G * L * PQ_BINS : 0;
}

// what every call needs: the sums of the iterations
static size_t sums_bytes(int32_t G, int32_t L, int32_t k) {
  WsSize w;
  const size_t GL = (size_t)G * L;
  w.add<int>(2 * GL);
  w.add<int>(GL);
  w.add<long long>(GL * k);
  w.add<unsigned long long>(GL * k);
  return w.bytes;
}

extern "C" size_t pq_train_workspace_size(int32_t G, int32_t L, int32_t k) {
  if (G < 1 || L < 1 || k < 2) return 0;
  return sums_bytes(G, L, k) + counts_bytes(G, L);
}

extern "C" int pq_train(const void* z, int32_t latent_dtype, int64_t n, int32_t L,
                        const int64_t* group_offsets, int32_t G, int32_t k, int32_t iters,
                        float* table, void* workspace, size_t workspace_bytes, void* stream) {
  clear_error();
  int rc = pq_check(latent_dtype, n, L, G, k);
  if (rc) return rc;
  AEQC_CHECK_ARG(table && workspace && (z || n == 0), "pq_train: null pointer");
  AEQC_CHECK_ARG(G == 1 || group_offsets, "pq_train: G > 1 needs group_offsets");
  AEQC_CHECK_ARG(iters >= 0 && iters <= 10000, "pq_train: iters=%d", iters);
  AEQC_CHECK_ARG(workspace_bytes >= sums_bytes(G, L, k), "pq_train: workspace too small");
  AEQC_CHECK_ARG(accum_limit(L, k) <= 200 * 1024, "pq_train: L * k = %d too large", L * k);

  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const long long* off = reinterpret_cast<const long long*>(group_offsets);
  const int GL = G * L, bf16 = latent_dtype == AEQC_DTYPE_BF16;
  WsCarver c(static_cast<char*>(workspace), workspace_bytes);
  int* keys = c.take<int>(2 * (size_t)GL);
  int* shift = c.take<int>(GL);
  long long* acc = c.take<long long>((size_t)GL * k);
  unsigned long long* cnt = c.take<unsigned long long>((size_t)GL * k);
  AEQC_CHECK_ARG(c.ok(), "pq_train: workspace not 256-byte aligned");
  // the counts where the workspace has room for them
  const size_t cb = counts_bytes(G, L);
  unsigned* counts = cb && c.left >= cb ? c.take<unsigned>((size_t)GL * PQ_BINS) : nullptr;
  const dim3 grid = pq_grid(G, n, L);
  if (bf16 && counts && n < (1ll << 32) && counts_pay(n, L, iters)) {
    AEQC_CUDA_TRY(cudaMemsetAsync(counts, 0, cb, s));
    const uint16_t* zb = static_cast<const uint16_t*>(z);
    // 16-byte loads: every row starts at a multiple of eight elements
    const bool vec = L % 8 == 0 && reinterpret_cast<uintptr_t>(z) % 16 == 0;
    if (vec && n / G >= PQ_WINDOW_ROWS) {
      rc = raise_smem_limit((const void*)pq_count_window_kernel, PQ_CSMEM);
      if (rc) return rc;
      // one block per SM, of them at least one per group and eight dimensions
      const int per = pq_sms() / (G * (L / 8));
      pq_count_window_kernel<<<dim3(per > 1 ? per : 1, L / 8, G), PQ_CT, PQ_CSMEM, s>>>(
          zb, n, L, off, counts);
    } else if (vec)
      pq_count_kernel<8><<<grid, 256, 0, s>>>(zb, n, L, off, counts);
    else
      pq_count_kernel<1><<<grid, 256, 0, s>>>(zb, n, L, off, counts);
    rc = check_launch("pq_count_kernel");
    if (rc) return rc;
    const size_t lsm = lloyd_smem(k);
    rc = raise_smem_limit((const void*)pq_lloyd_counts_kernel, (int)lsm);
    if (rc) return rc;
    pq_lloyd_counts_kernel<<<GL, PQ_LT, lsm, s>>>(counts, n, L, off, k, iters, table);
    return check_launch("pq_lloyd_counts_kernel");
  }
  const int nb = (GL * k + 255) / 256;
  pq_clear_kernel<<<nb, 256, 0, s>>>(keys, acc, cnt, GL, k);
  pq_minmax_init_kernel<<<grid, PQ_THREADS, 0, s>>>(z, bf16, n, L, off, keys, cnt, k, table,
                                                    shift);
  rc = check_launch("pq_minmax_init_kernel");
  if (rc) return rc;
  int steps = bisect_steps(k);
  if (accum_smem(L, k, padded_rows(k, steps)) > 200 * 1024) steps = 0;  // no room to pad
  const int k2 = padded_rows(k, steps);
  const size_t sm = accum_smem(L, k, k2);
  with_steps(steps, [&](auto st) {
    const auto kernel = pq_accum_kernel<decltype(st)::value>;
    if (sm > 48 * 1024) rc = raise_smem_limit((const void*)kernel, (int)sm);
    // rows of a block: at least twice as many as centroids to load and add up
    const int64_t least = (pq_sms() + G - 1) / G, fit = n / (2 * (int64_t)G * k);
    dim3 blocks = grid;
    blocks.x = (unsigned)std::min<int64_t>(grid.x, std::max(least, fit));
    const bool apart = L * k > PQ_MOVE_IN_BLOCK;
    for (int it = 0; it < iters && !rc; ++it) {
      kernel<<<blocks, PQ_THREADS, sm, s>>>(z, bf16, n, L, off, k, k2, table, shift, acc, cnt,
                                          apart ? nullptr : keys);
      if (apart)
        pq_move_kernel<<<(GL * k + 127) / 128, 128, 0, s>>>(G, L, k, shift, acc, cnt, table);
    }
  });
  return rc ? rc : check_launch("pq_accum_kernel");
}

extern "C" int pq_encode(const void* z, int32_t latent_dtype, int64_t n, int32_t L,
                         const int64_t* group_offsets, int32_t G, int32_t k, const float* table,
                         uint8_t* codes, void* zq, void* stream) {
  clear_error();
  int rc = pq_check(latent_dtype, n, L, G, k);
  if (rc) return rc;
  AEQC_CHECK_ARG(table && (z || n == 0) && (codes || zq), "pq_encode: null pointer");
  AEQC_CHECK_ARG(G == 1 || group_offsets, "pq_encode: G > 1 needs group_offsets");
  if (n == 0) return AEQC_OK;
  AEQC_CHECK_ARG(sizeof(float) * (size_t)L * (k + 1) <= 200 * 1024,
                 "pq_encode: L * k = %d too large", L * k);
  int steps = bisect_steps(k);
  if (encode_smem(L, padded_rows(k, steps)) > 200 * 1024) steps = 0;  // no room to pad
  const int k2 = padded_rows(k, steps);
  size_t sm = encode_smem(L, k2);
  // a large table through room of its own (10,000 x 64 latents, k = 64: 29 -> 23 us;
  // tables below 2,048 entries lose 2 us to the additional step)
  const size_t room = sizeof(float) * (size_t)L * (k + 1);
  const int staged = L * k >= 2048 && sm + room <= 48 * 1024;
  if (staged) sm += room;
  with_steps(steps, [&](auto st) {
    const auto kernel = pq_encode_kernel<decltype(st)::value>;
    if (sm > 48 * 1024) rc = raise_smem_limit((const void*)kernel, (int)sm);
    if (!rc)
      kernel<<<pq_grid(G, n, L), PQ_THREADS, sm, static_cast<cudaStream_t>(stream)>>>(
          z, latent_dtype == AEQC_DTYPE_BF16, n, L,
          reinterpret_cast<const long long*>(group_offsets), k, k2, table, staged, codes, zq);
  });
  return rc ? rc : check_launch("pq_encode_kernel");
}

extern "C" int pq_decode(const uint8_t* codes, int64_t n, int32_t L, const int64_t* group_offsets,
                         int32_t G, int32_t k, const float* table, int32_t latent_dtype, void* z,
                         void* stream) {
  clear_error();
  int rc = pq_check(latent_dtype, n, L, G, k);
  if (rc) return rc;
  AEQC_CHECK_ARG(table && ((codes && z) || n == 0), "pq_decode: null pointer");
  AEQC_CHECK_ARG(G == 1 || group_offsets, "pq_decode: G > 1 needs group_offsets");
  if (n == 0) return AEQC_OK;
  pq_decode_kernel<<<pq_grid(G, n, L), PQ_THREADS, 0, static_cast<cudaStream_t>(stream)>>>(
      codes, n, L, reinterpret_cast<const long long*>(group_offsets), k, table,
      latent_dtype == AEQC_DTYPE_BF16, z);
  return check_launch("pq_decode_kernel");
}
