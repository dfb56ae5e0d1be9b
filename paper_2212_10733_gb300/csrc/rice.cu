// Entropy coding of the residual codes (the lossless stage the paper leaves to
// MGARD's Huffman/Zstd, Sec. III Stage 4; its output is part of the buffer of
// Stage 5): one Golomb-Rice code per histogram.
//
// Symbols: the zero-level code -> 0, a level q -> zigzag(q) + 1, the escape
// code -> 65535.  Per histogram the parameter k in 0..15 with the fewest bits
// (ties to the smaller k).  Per symbol s: u = s >> k; if u < 24: u one-bits, a
// zero-bit, the k low bits of s (least significant first); else 24 one-bits
// and the 16 bits of s.  Bit i of a histogram's stream is bit (i mod 32) of
// 32-bit word i / 32, unused high bits zero; streams are stored back to back
// at word offsets given by an exclusive prefix sum.
//
// rice_measure: warp per histogram, the symbols in registers, two to a word;
// only the candidates that can still be the shortest are summed.
// rice_pack: warp per histogram.  Rows of 993 codes and more (rice_pack_seg):
// every lane appends the patterns of a run of consecutive symbols, placed by one
// prefix sum of the runs' lengths.  Shorter rows (rice_pack): each 32-symbol step
// places its patterns with a prefix sum of their lengths and ORs them into the
// histogram's stream in shared memory.  Both copy the stream out from there.
// rice_unpack: one thread per histogram reads its stream through a 64-bit buffer
// filled from words copied ahead (reads never leave the histogram's words) and
// the warp writes the decoded codes through shared memory in contiguous rows.
#include "aeqc_internal.cuh"
#include "workspace.cuh"

namespace aeqc {
namespace {

constexpr int RW = 4;           // warps per CTA (measure, pack)
constexpr int RCAP = 24;        // unary prefix cap
constexpr int RMAXBITS = 40;    // longest code
constexpr int RSLOT = (AEQC_MAX_P * RMAXBITS + 31) / 32;  // words of the longest stream
constexpr int SCAN_B = 1024;    // elements per scan block

__device__ __forceinline__ unsigned rice_symbol(int code) {
  if (code == AEQC_CODE_ZERO) return 0u;
  if (code == AEQC_CODE_ESCAPE) return 65535u;
  return (code >= 0 ? 2u * (unsigned)code : 2u * (unsigned)(-code) - 1u) + 1u;
}

__device__ __forceinline__ int rice_code(unsigned s) {
  const unsigned z = s - 1u;
  const int q = (int)(z >> 1) ^ -(int)(z & 1u);
  return s == 0u ? AEQC_CODE_ZERO : (s == 65535u ? AEQC_CODE_ESCAPE : q);
}

// ---- two symbols per 32-bit word --------------------------------------------------

__device__ __forceinline__ unsigned min_u16x2(unsigned a, unsigned b) {
  unsigned r;
  asm("min.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ unsigned max_u16x2(unsigned a, unsigned b) {
  unsigned r;
  asm("max.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ unsigned add_u16x2(unsigned a, unsigned b) {
  unsigned r;
  asm("add.u16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// A row of P codes as the aligned words it touches: code p is half (p + par) % 2
// of word (p + par) / 2, par the row's parity (rows of an odd P start on 2-byte
// boundaries every other time).  The first and last word's other half belongs
// to a neighbouring row, or lies outside the array (edge): there each half is
// read by itself.  Halves outside the row are not meaningful.
constexpr int RNW = (AEQC_MAX_P / 2 + 1 + 31) / 32;  // words per lane of the longest row

struct RowWords {
  const int16_t* row;
  int par, words;  // words touched
  bool edge;       // first or last row of the array
};

__device__ __forceinline__ RowWords row_words(const int16_t* codes, long long b, long long n,
                                              int P) {
  RowWords r;
  r.row = codes + b * P;
  r.par = (int)((reinterpret_cast<uintptr_t>(r.row) >> 1) & 1);
  r.words = (r.par + P + 1) / 2;
  r.edge = b == 0 || b + 1 == n;
  return r;
}

// word lane + 32 i into w[i] (zero-level codes past the row; NW words a lane hold
// the row), every load in flight at once
template <int NW>
__device__ __forceinline__ void load_words(const RowWords& r, int P, int lane,
                                           unsigned (&w)[NW]) {
  const unsigned* base = reinterpret_cast<const unsigned*>(r.row - r.par) + lane;
  if (!r.edge) {
#pragma unroll
    for (int i = 0; i < NW; ++i)
      w[i] = lane + 32 * i < r.words ? __ldg(base + 32 * i) : 0x80018001u;
  } else {
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      const int p = 2 * (lane + 32 * i) - r.par;
      const unsigned lo = p >= 0 && p < P ? (uint16_t)__ldg(r.row + p) : 0x8001u;
      const unsigned hi = p + 1 < P ? (uint16_t)__ldg(r.row + p + 1) : 0x8001u;
      w[i] = lo | (hi << 16);
    }
  }
}

// symbols of two codes, per half modulo 2^16: z = zigzag (2q, or -2q - 1 below 0),
// then z + 1; the escape code (z = 65535) stays there and the zero level
// (z = 65533) goes to 0
__device__ __forceinline__ unsigned symbols_of(unsigned c) {
  const unsigned neg = ((c >> 15) & 0x00010001u) * 0xFFFFu;
  const unsigned z = ((c << 1) & 0xFFFEFFFEu) ^ neg;
  const unsigned s = add_u16x2(z, min_u16x2(add_u16x2(z, 0x00010001u), 0x00010001u));
  return s & (min_u16x2(s ^ 0xFFFEFFFEu, 0x00010001u) * 0xFFFFu);
}

// bits of the symbols in a word beyond 1 + k each: the prefixes (capped), as
// a packed sum, and the number of capped ones
__device__ __forceinline__ unsigned prefixes(unsigned s, int k) {
  return min_u16x2((s >> k) & ((0xFFFFu >> k) * 0x00010001u), RCAP * 0x00010001u);
}
__device__ __forceinline__ unsigned capped(unsigned t) {  // t from prefixes(): halves at RCAP
  return ((t + (0x8000u - RCAP) * 0x00010001u) >> 15) & 0x00010001u;
}
__device__ __forceinline__ int halves(unsigned v) { return (int)(v & 0xFFFFu) + (int)(v >> 16); }

// The parameter with the fewest bits.  T_k, the row's length with parameter k,
// is summed for k0 (from the mean symbol) and then outwards while another k
// can be shorter:
//  * above: a symbol takes at least 1 + k bits, so no k > hi is shorter than
//    the best once P (hi + 2) reaches it;
//  * below: c_i(s) - c_(i+1)(s) is at least -1, and that only for s < 2^i
//    (a symbol capped at i + 1 stays at 40 bits, one capped at i only had at
//    most 39, else the difference is ceil((s >> i) / 2) - 1).  So T_j >= T_lo -
//    lo N for every j < lo with N the number of symbols below 2^(lo-1).
// A tie goes to the smaller k.  Residual codes take four or five sums of the
// sixteen, two symbols an instruction: 811 -> 300 us for 131,072 rows
// of 1,521 codes.  NW words a lane hold a row: rows of up to RSMALL codes take the
// form with four of them instead of twenty-five (20,000 rows of 10, measured and
// packed: 103 -> 95 us).
constexpr int RSMALL = 4 * 64 - 2;  // the row's words with one half at either end

template <int NW>
__global__ void __launch_bounds__(RW * 32) rice_measure_kernel(const int16_t* codes, long long n,
                                                               int P, uint8_t* kparam,
                                                               uint32_t* nbits,
                                                               long long* wcount) {
  const int lane = threadIdx.x & 31;
  const long long nw = (long long)gridDim.x * RW;
  long long b = (long long)blockIdx.x * RW + (threadIdx.x >> 5);
  if (b >= n) return;
  RowWords r = row_words(codes, b, n, P);
  unsigned ahead[NW];  // the next row, loaded while this one is summed
  load_words(r, P, lane, ahead);
  for (; b < n; b += nw) {
    unsigned s[NW], sum = 0, mx = 0;
    const int words = r.words;
    // the half past an odd end becomes the zero level: symbol 0 adds no prefix
    const int odd = (r.par + P) & 1 ? words - 1 - lane : -1;
    if (lane == 0 && r.par) ahead[0] = (ahead[0] & 0xFFFF0000u) | 0x8001u;
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      if (32 * i >= words) break;
      if (32 * i == odd) ahead[i] = (ahead[i] & 0xFFFFu) | 0x80010000u;
      const unsigned v = symbols_of(ahead[i]);
      s[i] = v;
      sum += (v & 0xFFFFu) + (v >> 16);
      mx = max_u16x2(mx, v);
    }
    if (b + nw < n) {
      r = row_words(codes, b + nw, n, P);
      load_words(r, P, lane, ahead);
    }
    const unsigned total = __reduce_add_sync(0xffffffffu, sum);  // <= 1536 * 65535
    const unsigned smax = __reduce_max_sync(0xffffffffu, max(mx & 0xFFFFu, mx >> 16));
    const unsigned mean = total / (unsigned)P * 11u / 16u;
    int lo = mean ? min(31 - __clz(mean), 15) : 0, hi = lo, k = lo;
    int best = 0x7FFFFFFF, arg = 0, tlo = 0;
    for (;;) {
      unsigned acc = 0, cap = 0;
      if (smax >= ((unsigned)RCAP << k)) {
#pragma unroll
        for (int i = 0; i < NW; ++i) {
          if (32 * i >= words) break;
          const unsigned t = prefixes(s[i], k);
          acc += t;
          cap += capped(t);
        }
      } else {
#pragma unroll
        for (int i = 0; i < NW; ++i) {
          if (32 * i >= words) break;
          acc += prefixes(s[i], k);
        }
      }
      // a capped symbol takes RCAP + 16 bits: 15 - k more than 1 + k + RCAP
      const int T = P * (1 + k) + (int)__reduce_add_sync(
                                      0xffffffffu, (unsigned)(halves(acc) + halves(cap) * (15 - k)));
      if (T < best || (T == best && k < arg)) {
        best = T;
        arg = k;
      }
      if (k == lo) tlo = T;
      if (hi < 15 && P * (hi + 2) < best) {
        k = ++hi;
        continue;
      }
      if (lo == 0) break;
      unsigned ge = 0;
#pragma unroll
      for (int i = 0; i < NW; ++i) {
        if (32 * i >= words) break;
        ge += min_u16x2((s[i] >> (lo - 1)) & ((0xFFFFu >> (lo - 1)) * 0x00010001u), 0x00010001u);
      }
      const int below = P - (int)__reduce_add_sync(0xffffffffu, (unsigned)halves(ge));
      if (tlo - lo * below > best) break;
      k = --lo;
    }
    if (lane == 0) {
      kparam[b] = (uint8_t)arg;
      nbits[b] = (uint32_t)best;
      wcount[b] = (best + 31) / 32;
    }
  }
}

// exclusive prefix sum of wcount [n] into off [n + 1], three passes
__global__ void scan_block_sums(const long long* v, long long n, long long* bsum) {
  __shared__ long long s[32];
  const long long i0 = (long long)blockIdx.x * SCAN_B;
  long long acc = 0;
  for (int t = threadIdx.x; t < SCAN_B; t += blockDim.x)
    if (i0 + t < n) acc += v[i0 + t];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    long long t = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += s[w];
    bsum[blockIdx.x] = t;
  }
}

// one block of SCAN_B threads: the block sums to their exclusive prefix sums, a
// SCAN_B piece at a time
__global__ void scan_sums(long long* bsum, long long nb) {
  __shared__ long long wsum[SCAN_B / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  long long run = 0;
  for (long long i0 = 0; i0 < nb; i0 += SCAN_B) {
    const long long i = i0 + threadIdx.x;
    const long long x = i < nb ? bsum[i] : 0;
    long long inc = x;
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wsum[w] = inc;
    __syncthreads();
    long long before = 0, all = 0;
    for (int v = 0; v < SCAN_B / 32; ++v) {
      if (v < w) before += wsum[v];
      all += wsum[v];
    }
    if (i < nb) bsum[i] = run + before + inc - x;
    run += all;
    __syncthreads();
  }
}

// SCAN_B threads: one element each
__global__ void scan_apply(const long long* v, long long n, const long long* bsum, long long* off) {
  __shared__ long long wsum[SCAN_B / 32];
  const long long i = (long long)blockIdx.x * SCAN_B + threadIdx.x;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const long long x = i < n ? v[i] : 0;
  long long inc = x;
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wsum[w] = inc;
  __syncthreads();
  if (w == 0) {
    long long t = wsum[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const long long y = __shfl_up_sync(0xffffffffu, t, o);
      if (lane >= o) t += y;
    }
    wsum[lane] = t;  // inclusive over warps
  }
  __syncthreads();
  const long long before = (w ? wsum[w - 1] : 0) + inc - x;
  if (i < n) off[i] = bsum[blockIdx.x] + before;
  if (i == n - 1) off[n] = bsum[blockIdx.x] + before + x;
}

__global__ void __launch_bounds__(RW * 32) rice_pack_kernel(const int16_t* codes, long long n,
                                                            int P, const uint8_t* kparam,
                                                            const long long* off, uint32_t* words,
                                                            long long capacity) {
  __shared__ uint32_t slot[RW][RSLOT];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  uint32_t* st = slot[wi];
  const long long nw = (long long)gridDim.x * RW;
  for (long long b = (long long)blockIdx.x * RW + wi; b < n; b += nw) {
    const int16_t* cb = codes + b * P;
    const int k = kparam[b] & 15;
    const int nwords = (P * RMAXBITS + 31) / 32;
    for (int t = lane; t < nwords; t += 32) st[t] = 0u;
    __syncwarp();
    long long base = 0;
    for (int p0 = 0; p0 < P; p0 += 32) {
      const int p = p0 + lane;
      int len = 0;
      unsigned long long v = 0ull;
      if (p < P) {
        const unsigned s = rice_symbol(cb[p]);
        const unsigned u = s >> k;
        if (u < (unsigned)RCAP) {
          len = (int)u + 1 + k;
          v = ((1ull << u) - 1ull) | ((unsigned long long)(s & ((1u << k) - 1u)) << (u + 1));
        } else {
          len = RCAP + 16;
          v = ((1ull << RCAP) - 1ull) | ((unsigned long long)s << RCAP);
        }
      }
      int inc = len;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      const long long at = base + inc - len;
      if (len) {
        const int w0 = (int)(at >> 5), sh = (int)(at & 31);
        atomicOr(&st[w0], (uint32_t)(v << sh));
        const unsigned long long rest = sh ? (v >> (32 - sh)) : (v >> 32);
        if (rest) {
          atomicOr(&st[w0 + 1], (uint32_t)rest);
          if (rest >> 32) atomicOr(&st[w0 + 2], (uint32_t)(rest >> 32));
        }
      }
      base += __shfl_sync(0xffffffffu, inc, 31);
    }
    __syncwarp();
    const long long w0 = off[b], wc = (base + 31) >> 5;
    if (w0 >= 0 && w0 + wc <= capacity)
      for (int t = lane; t < (int)wc; t += 32) words[w0 + t] = st[t];
    __syncwarp();
  }
}

// Pack with every lane coding its own run of R consecutive halves, R = 2 mod 4
// and at least 34 (so a run that is not the last has 33 symbols and more than
// 32 bits, a 32-bit word is shared by at most two neighbouring runs, and the
// runs lie an odd number of words apart in shared memory: no bank conflicts): one prefix
// sum of the run lengths per histogram, then each lane appends its patterns
// to a 64-bit buffer and stores whole words; the word it shares with the
// previous lane is merged after the run.  The stream is put together in
// shared memory and written out in whole lines (streams beyond RSTREAM words
// go to global memory word by word).  723 -> 386 us for 131,072 rows of 1,521
// codes, bound by instruction issue.
constexpr int RSTREAM = 1024;  // words of the staged stream

__host__ __device__ constexpr int rice_run(int P) {  // smallest R = 2 mod 4, 32 R > P
  const int r = P / 32 + 1;
  return r + ((2 - r % 4) + 4) % 4;
}
constexpr int RSYMW = 32 * RNW > 16 * rice_run(AEQC_MAX_P) ? 32 * RNW : 16 * rice_run(AEQC_MAX_P);

// One lane's run of symbols sym[q0 .. q1) (two a word), whose first bit is bit S
// of the stream, into words of arr: the first goes to index `first`, the next
// ones from index `rest` on.  Returns the bits of the unfinished last word (0 if
// there is none) and its index in *at.
__device__ __forceinline__ uint32_t code_run(const uint32_t* run, int q0, int q1, int k, int S,
                                             uint32_t* arr, int first, int rest, int* at) {
  const unsigned low = (1u << k) - 1u;
  unsigned long long buf = 0ull;
  int cnt = S & 31, dst = first, nx = rest;
  auto put = [&](uint32_t v, int l) {  // l <= 32 bits; cnt < 32 before and after
    buf |= (unsigned long long)v << cnt;
    cnt += l;
    const bool full = cnt >= 32;
    if (full) arr[dst] = (uint32_t)buf;
    dst = full ? nx : dst;
    nx += full;
    buf = full ? buf >> 32 : buf;
    cnt &= 31;
  };
  auto code = [&](unsigned s) {
    const unsigned u = s >> k;
    int l = (int)u + 1 + k;
    unsigned v;
    if (u >= (unsigned)RCAP || l > 32) {  // in two pieces
      const bool c = u >= (unsigned)RCAP;
      put(c ? (1u << RCAP) - 1u : (1u << u) - 1u, c ? RCAP : (int)u + 1);
      v = c ? s : s & low;
      l = c ? 16 : k;
    } else {
      v = ((s & low) << (u + 1)) | ((1u << u) - 1u);
    }
    put(v, l);
  };
  int q = q0;
  if (q & 1) code(run[q++ >> 1] >> 16);
  for (; q + 1 < q1; q += 2) {
    const unsigned s = run[q >> 1];
    code(s & 0xFFFFu);
    code(s >> 16);
  }
  if (q < q1) code(run[q >> 1] & 0xFFFFu);
  *at = cnt ? dst : -1;
  return (uint32_t)buf;
}

__global__ void __launch_bounds__(RW * 32) rice_pack_seg_kernel(const int16_t* codes,
                                                                long long n, int P,
                                                                const uint8_t* kparam,
                                                                const long long* off,
                                                                uint32_t* words,
                                                                long long capacity) {
  // the stream behind the 32 lanes' shared first words
  __shared__ uint32_t sym[RW][RSYMW], stream[RW][32 + RSTREAM], tail[RW][32];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const int R = rice_run(P);
  const uint32_t* run = &sym[wi][lane * (R / 2)];
  uint32_t* st = stream[wi];
  const long long nw = (long long)gridDim.x * RW;
  long long b = (long long)blockIdx.x * RW + wi;
  if (b >= n) return;
  RowWords r = row_words(codes, b, n, P);
  unsigned ahead[RNW];  // the next row, loaded while this one is coded
  load_words(r, P, lane, ahead);
  for (; b < n; b += nw) {
    // symbol p at half p + par; the run: halves q0 to q1 of this lane's R
    const int end = P + r.par;  // halves in use
#pragma unroll
    for (int i = 0; i < RNW; ++i) sym[wi][lane + 32 * i] = symbols_of(ahead[i]);
    __syncwarp();
    // the halves either side of the row: symbol 0, which adds no prefix
    if (lane == 0) {
      if (r.par) sym[wi][0] &= 0xFFFF0000u;
      if (end & 1) sym[wi][end >> 1] &= 0xFFFFu;
    }
    __syncwarp();
    const int q0 = lane == 0 ? r.par : 0, q1 = min(R, end - lane * R);
    const bool any = q1 > q0, last = any && lane * R + q1 == end;
    const long long w0 = off[b];
    const int k = kparam[b] & 15;
    if (b + nw < n) {
      r = row_words(codes, b + nw, n, P);
      load_words(r, P, lane, ahead);
    }
    unsigned acc = 0, cap = 0;
    for (int q = 0; q < q1; q += 2) {
      const unsigned t = prefixes(run[q >> 1], k);
      acc += t;
      cap += capped(t);
    }
    const int len = any ? (q1 - q0) * (1 + k) + halves(acc) + halves(cap) * (15 - k) : 0;
    int inc = len;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    const int S = inc - len, wc = (__shfl_sync(0xffffffffu, inc, 31) + 31) >> 5;
    if (w0 >= 0 && w0 + wc <= capacity) {  // the same for the whole warp
      uint32_t* out = words + w0;
      const bool shared_head = any && (S & 31) != 0;
      // a run's unfinished last word: the stream's last one (which may be the
      // shared first word of the run itself), else shared with the next run
      if (wc <= RSTREAM) {
        const int own = 32 + (S >> 5);
        int at = -1;
        const uint32_t rem =
            any ? code_run(run, q0, q1, k, S, st, shared_head ? lane : own, own + 1, &at) : 0u;
        if (at >= 0) {
          if (last) st[at] = rem;
          else tail[wi][lane] = rem;
        }
        __syncwarp();
        if (shared_head) st[own] = st[lane] | tail[wi][lane - 1];
        __syncwarp();
        for (int t = lane; t < wc; t += 32) out[t] = st[32 + t];
      } else {
        // the same straight into global memory; a lane adds the previous run's
        // bits to its own first word
        const int own = S >> 5;
        int at = -1;
        uint32_t rem = 0u;
        if (any) rem = code_run(run, q0, q1, k, S, out, own, own + 1, &at);
        if (at >= 0) {
          if (last) out[at] = rem;
          else tail[wi][lane] = rem;
        }
        __syncwarp();
        if (shared_head) out[own] |= tail[wi][lane - 1];
      }
    }
    __syncwarp();
  }
}

// One thread per histogram decodes 32 symbols at a time into shared memory;
// the warp then writes each of its 32 histograms' 32 codes as one contiguous
// 64-byte store (instead of 32 scattered 2-byte stores per instruction).  The
// bit buffer is topped up once per symbol from words copied asynchronously
// RRING - 1 refills ahead (a load into a register is waited for at the next
// refill, before it has come from HBM), and a symbol of at most 32 bits is
// taken out in one step: 1271 -> 513 us
// for 131,072 rows of 1,521 codes.  Launched with 128 threads (4 warps) per
// block.
constexpr int RRING = 8;

__global__ void __launch_bounds__(128, 8) rice_unpack_kernel(const uint32_t* words,
                                                          long long total_words,
                                                          const long long* off,
                                                          const uint8_t* kparam, long long n,
                                                          int P, int16_t* codes) {
  __shared__ uint16_t stage[4][32][34];  // rows 17 words apart: no bank conflicts
  __shared__ uint32_t ring[RRING][128];
  const int lane = threadIdx.x & 31, wi = threadIdx.x >> 5;
  const long long b0 = ((long long)blockIdx.x * 4 + wi) * 32;  // the warp's first histogram
  const long long b = b0 + lane;
  const int hist = (int)min(32ll, n - b0);  // histograms of this warp (<= 0 past the end)
  const uint32_t* w = words;
  int left = 0;  // words of the stream not yet asked for
  int k = 0;
  if (lane < hist) {
    long long o0 = off[b], o1 = off[b + 1];
    if (o0 < 0) o0 = 0;
    if (o1 > total_words) o1 = total_words;
    if (o0 < o1) {
      w = words + o0;
      left = (int)min(o1 - o0, 0x7FFFFFFFll);
    }
    k = kparam[b] & 15;
  }
  const unsigned low = (1u << k) - 1u;
  unsigned long long buf = 0ull;
  int have = 0;  // valid bits in buf
  // slot (the thread's column of the ring) <- the stream's next word; zeros
  // follow the last one
  auto ask = [&](int slot) {
    uint32_t* d = &ring[slot][threadIdx.x];
    if (left > 0)
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(
                       (unsigned)__cvta_generic_to_shared(d)),
                   "l"(w)
                   : "memory");
    else
      *d = 0u;
    asm volatile("cp.async.commit_group;" ::: "memory");
    ++w;
    --left;
  };
#pragma unroll
  for (int i = 0; i < RRING - 1; ++i) ask(i);
  int slot = 0;
  auto refill = [&]() {  // to more than 32 bits
    if (have <= 32) {
      asm volatile("cp.async.wait_group %0;" ::"n"(RRING - 2) : "memory");  // the oldest is there
      buf |= (unsigned long long)ring[slot][threadIdx.x] << have;
      have += 32;
      ask((slot + RRING - 1) % RRING);  // the slot read before this one
      slot = (slot + 1) % RRING;
    }
  };
  auto drop = [&](int l) {
    buf >>= l;
    have -= l;
  };
  refill();
  for (int c0 = 0; c0 < P; c0 += 32) {
    const int m = min(32, P - c0);
    if (lane < hist) {
#pragma unroll 2
      for (int i = 0; i < m; ++i) {
        refill();
        // unary prefix: count of trailing ones, at most RCAP
        const unsigned z = ~(unsigned)buf;
        const int u = z ? __ffs((int)z) - 1 : 32;
        unsigned sy;
        if (u < RCAP && u + 1 + k <= 32) {
          sy = ((unsigned)u << k) | ((unsigned)(buf >> (u + 1)) & low);
          drop(u + 1 + k);
        } else if (u < RCAP) {
          drop(u + 1);
          refill();
          sy = ((unsigned)u << k) | ((unsigned)buf & low);
          drop(k);
        } else {
          drop(RCAP);
          refill();
          sy = (unsigned)buf & 0xFFFFu;
          drop(16);
        }
        stage[wi][lane][i] = (uint16_t)rice_code(sy);
      }
    }
    __syncwarp();
    if (lane < m) {
      int16_t* dst = codes + b0 * P + c0 + lane;
#pragma unroll 4
      for (int h = 0; h < hist; ++h, dst += P) *dst = (int16_t)stage[wi][h][lane];
    }
    __syncwarp();
  }
  // the words asked for and not needed any more
  asm volatile("cp.async.wait_all;" ::: "memory");
}

}  // namespace
}  // namespace aeqc

using namespace aeqc;

extern "C" size_t rice_workspace_size(int64_t n) {
  if (n < 0) return 0;
  WsSize w;
  w.add<long long>((size_t)n + 1);
  w.add<long long>((size_t)(n + SCAN_B - 1) / SCAN_B + 1);
  w.add<long long>(1);
  return w.bytes;
}

extern "C" int rice_measure(const int16_t* codes, int64_t n, int32_t P, uint8_t* kparam,
                            uint32_t* nbits, int64_t* offsets, void* workspace,
                            size_t workspace_bytes, void* stream) {
  clear_error();
  AEQC_CHECK_ARG(n >= 0 && P >= 1 && P <= AEQC_MAX_P, "rice_measure: bad sizes");
  AEQC_CHECK_ARG((n == 0 || (codes && kparam && nbits)) && offsets && workspace,
                 "rice_measure: null pointer");
  AEQC_CHECK_ARG(workspace_bytes >= rice_workspace_size(n), "rice_measure: workspace too small");
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  WsCarver c(static_cast<char*>(workspace), workspace_bytes);
  long long* wc = c.take<long long>((size_t)n + 1);
  const long long nb = (n + SCAN_B - 1) / SCAN_B;
  long long* bsum = c.take<long long>((size_t)nb + 1);
  AEQC_CHECK_ARG(c.ok(), "rice_measure: workspace not 256-byte aligned");
  long long* off = reinterpret_cast<long long*>(offsets);
  if (n == 0) {
    AEQC_CUDA_TRY(cudaMemsetAsync(off, 0, sizeof(long long), s));
    return AEQC_OK;
  }
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  long long blocks = (n + RW - 1) / RW;
  if (blocks > (long long)sms * 16) blocks = (long long)sms * 16;
  const auto measure = P <= RSMALL ? rice_measure_kernel<4> : rice_measure_kernel<RNW>;
  measure<<<(unsigned)blocks, RW * 32, 0, s>>>(codes, n, P, kparam, nbits, wc);
  scan_block_sums<<<(unsigned)nb, 256, 0, s>>>(wc, n, bsum);
  scan_sums<<<1, SCAN_B, 0, s>>>(bsum, nb);
  scan_apply<<<(unsigned)nb, SCAN_B, 0, s>>>(wc, n, bsum, off);
  return check_launch("rice_measure");
}

extern "C" int rice_pack(const int16_t* codes, int64_t n, int32_t P, const uint8_t* kparam,
                         const int64_t* offsets, uint32_t* words, int64_t capacity, void* stream) {
  clear_error();
  AEQC_CHECK_ARG(n >= 0 && P >= 1 && P <= AEQC_MAX_P && capacity >= 0, "rice_pack: bad sizes");
  AEQC_CHECK_ARG(n == 0 || (codes && kparam && offsets && words), "rice_pack: null pointer");
  if (n == 0) return AEQC_OK;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  long long blocks = (n + RW - 1) / RW;
  const long long* off = reinterpret_cast<const long long*>(offsets);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (P >= 32 * 31 + 1) {  // runs of at least 32 symbols per lane
    if (blocks > (long long)sms * 8) blocks = (long long)sms * 8;
    rice_pack_seg_kernel<<<(unsigned)blocks, RW * 32, 0, s>>>(codes, n, P, kparam, off, words,
                                                               capacity);
    return check_launch("rice_pack_seg_kernel");
  }
  if (blocks > (long long)sms * 7) blocks = (long long)sms * 7;
  rice_pack_kernel<<<(unsigned)blocks, RW * 32, 0, s>>>(codes, n, P, kparam, off, words,
                                                          capacity);
  return check_launch("rice_pack_kernel");
}

extern "C" int rice_unpack(const uint32_t* words, int64_t total_words, const int64_t* offsets,
                           const uint8_t* kparam, int64_t n, int32_t P, int16_t* codes,
                           void* stream) {
  clear_error();
  AEQC_CHECK_ARG(n >= 0 && P >= 1 && P <= AEQC_MAX_P && total_words >= 0,
                 "rice_unpack: bad sizes");
  AEQC_CHECK_ARG(n == 0 || (offsets && kparam && codes && (words || total_words == 0)),
                 "rice_unpack: null pointer");
  if (n == 0) return AEQC_OK;
  rice_unpack_kernel<<<(unsigned)((n + 127) / 128), 128, 0, static_cast<cudaStream_t>(stream)>>>(
      words, total_words, reinterpret_cast<const long long*>(offsets), kparam, n, P, codes);
  // 128 threads = 4 warps x 32 histograms per block
  return check_launch("rice_unpack_kernel");
}
