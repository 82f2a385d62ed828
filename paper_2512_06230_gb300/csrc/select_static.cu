// glmb_select_top_static: top-H selection of child log-weights that makes no
// device allocation.  Its scratch is the file-scope array below (41,216
// bytes, sized for at most kMaxBlocks blocks); every GPU that loads the
// library holds it until the process exits.
//
// Who needs it: callers that may not allocate device memory while they run,
// such as a tracking loop with a fixed memory budget and a hard frame
// deadline (cudaMalloc can synchronise the device and stall for
// milliseconds), or code embedded in a host application whose memory policy
// forbids raw cudaMalloc.  The caller still passes the inputs and outputs.
//
// The steps are those of the selection inside glmb_prune: log-weights are
// converted to int64 with 2^-32 resolution, normalised by their log-sum-exp,
// children below tau are dropped, the h_max largest are kept (ties by
// index), the kept ones are listed in index order and their log-weights
// renormalised.  The log-sum-exp is summed differently (exponentials to
// 2^-54 here, FP32 exponentials with compensated sums there), so the two
// agree up to its rounding: a child whose normalised weight lies within that
// rounding of tau may land on either side of the cut.
//
// What bounds it: at a million children the 8 MB of log-weights stay in L2,
// so a pass is a few microseconds and the cost is the FP64 pipe (about two
// operations a clock on an SM) and the number of launches.  Therefore the
// keys and the exponentials are formed in integer arithmetic (fx_math.cuh), and
// what one block has to decide between two passes is done by the last block
// of the first (six launches instead of twelve).  Measured, 10^6 children,
// h_max 20000: 413 us with an FP64 exponential per child and per kept child
// in one block (twelve launches), 66 us with these.
#include <algorithm>
#include <cmath>
#include <mutex>

#include "../../include/glmb.h"
#include "fx_math.cuh"
#include "glmb_dev.cuh"

namespace {

using namespace glmb;

constexpr int kMaxBlocks = 1024;
constexpr int kThreads = 256;
constexpr int kDigitS = 12, kBinsS = 1 << kDigitS;
constexpr long long kMaxN = 1LL << 30;

// scratch layout (bytes)
constexpr size_t kOffBlkM = 0;                                   // long long[kMaxBlocks]
constexpr size_t kOffBlkS = kOffBlkM + 8 * kMaxBlocks;           // double[kMaxBlocks]
constexpr size_t kOffBlkGt = kOffBlkS + 8 * kMaxBlocks;          // uint32[kMaxBlocks]
constexpr size_t kOffBlkEq = kOffBlkGt + 4 * kMaxBlocks;         // uint32[kMaxBlocks]
constexpr size_t kOffHist = kOffBlkEq + 4 * kMaxBlocks;          // uint32[kBinsS], then the boundary list
constexpr size_t kOffScal = kOffHist + 4 * kBinsS;               // Scal
constexpr size_t kScratchBytes = kOffScal + 256;
// the size glmb.h states for the scratch array
static_assert(kScratchBytes == 41216, "scratch size changed: update glmb.h");
// keys of the boundary bin that fit in the histogram's place
constexpr unsigned kListS = kBinsS / 2;
// A boundary bin with no more keys than that is listed and finished by one
// block.  A bin with more (equal or nearly equal weights, or a cap that
// crowds it) takes its next digits, of up to 13 bits, from histograms over
// the grid until it does fit: the passes for them are always launched and
// return at once when the list was enough (1 us of a call).  One block that
// read all the children again for each digit took 1.4 ms for a million and
// 5.6 ms for four million equal weights; now 65 and 138 us, as other weights.
constexpr int kWideBits = 13, kWideBins = 1 << kWideBits;
static_assert(4 * kWideBins <= kOffScal, "the wide histogram takes the place of the partials and the first one");
// Up to this many children one block does read them again, and the passes are
// not launched: 5000 children, equal or smooth weights, 37.2 and 34.3 us with
// one block and 38.3 and 35.0 with the passes; 16384, 50.2 and 36.5 against
// 40.6 and 37.3.
constexpr long long kSoloN = 1LL << 13;

struct SelScal {
  unsigned done[3];     // last-block counters (histogram, boundary, count)
  unsigned n_list;      // keys in the boundary list
  unsigned n_bin;       // keys in the boundary bin
  int left;             // bits of the boundary key still to be found
  double lse;           // log-sum-exp over valid children
  double lse_kept;      // log-sum-exp of the kept log-weights less lse
  long long thr;        // fixed-point threshold
  long long top;        // largest key
  long long prefix;     // radix prefix
  long long need;       // elements still needed at the boundary key
  long long bound;      // boundary key
  long long mode;       // 0 running, 1 keep all candidates, 2 nothing valid
};

__device__ __align__(256) unsigned char g_select_scratch[kScratchBytes];

struct Ptrs {
  long long* blk_m;
  double* blk_s;
  unsigned* blk_gt;
  unsigned* blk_eq;
  unsigned* hist;
  unsigned* wide;
  long long* list;
  SelScal* sc;
};

__host__ __device__ inline Ptrs ptrs_of(unsigned char* base) {
  return Ptrs{(long long*)(base + kOffBlkM), (double*)(base + kOffBlkS), (unsigned*)(base + kOffBlkGt),
              (unsigned*)(base + kOffBlkEq), (unsigned*)(base + kOffHist), (unsigned*)base, (long long*)(base + kOffHist),
              (SelScal*)(base + kOffScal)};
}

// The log-weight times 2^32, rounded to nearest (ties to even), from its
// bits: the FP64 conversion runs at a small fraction of the integer rate.
// Log-weights outside (-2^30, 2^30) -- -inf, +inf and NaN among them -- mark
// children without weight; inside, every key is below 2^62 in magnitude, so
// the difference of two keys cannot overflow.
__device__ __forceinline__ long long key_of(double lw) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(lw);
  const int e = (int)((b >> 52) & 0x7FFull);
  if (e >= 1023 + 30) return kKeyInvalid;
  const unsigned long long m = (b & 0xFFFFFFFFFFFFFull) | 0x10000000000000ull;   // |lw| = m 2^(e - 1075)
  const int r = 1043 - e;   // right shift that leaves |lw| 2^32 (subnormals give 0 too)
  unsigned long long v;
  if (r <= 0) {
    v = m << -r;
  } else if (r > 54) {
    v = 0ull;
  } else {
    v = m >> r;
    const unsigned long long rem = m << (64 - r);   // the part dropped, as a fraction of 2^64
    v += (rem > 0x8000000000000000ull || (rem == 0x8000000000000000ull && (v & 1ull))) ? 1ull : 0ull;
  }
  return (b >> 63) ? -(long long)v : (long long)v;
}

__device__ const fx::Tables kFx{};
// the block's copy of 2^(-j/64) (lanes read different entries); every kernel
// that forms exponentials fills it first
__device__ __forceinline__ unsigned long long* exp_tab() {
  __shared__ unsigned long long t[64];
  return t;
}
__device__ __forceinline__ void load_exp_tab() {
  if (threadIdx.x < 64) exp_tab()[threadIdx.x] = kFx.exp2[threadIdx.x];
  __syncthreads();
}

__device__ __forceinline__ long long warp_max_ll(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = max(v, __shfl_xor_sync(0xFFFFFFFFu, v, o));
  return v;
}
template <typename T>
__device__ __forceinline__ T warp_sum_of(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}
// inclusive scan over a warp
template <typename T>
__device__ __forceinline__ T warp_incl(T x) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  return x;
}

// The maximum and the sum of exp(key - maximum) over a block's (m, s) pairs
// (a pair with m = kKeyInvalid is empty), in every thread.
struct LseS {
  long long m;
  double s;
};
__device__ LseS block_lse(LseS v) {
  __shared__ long long sm[32];
  __shared__ double ss[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
  const long long wm = warp_max_ll(v.m);
  if (lane == 0) sm[w] = wm;
  __syncthreads();
  const long long M = warp_max_ll(lane < nw ? sm[lane] : kKeyInvalid);
  const double r = v.m == kKeyInvalid ? 0.0
                   : v.m == M         ? v.s
                                      : v.s * fx::exp_fixed((unsigned long long)(M - v.m), exp_tab());
  const double ws = warp_sum_of(r);
  if (lane == 0) ss[w] = ws;
  __syncthreads();
  return LseS{M, warp_sum_of(lane < nw ? ss[lane] : 0.0)};
}

__device__ __forceinline__ void chunk_of(long long n, long long& lo, long long& hi) {
  const long long per = (n + gridDim.x - 1) / gridDim.x;
  lo = min(n, (long long)blockIdx.x * per);
  hi = min(n, lo + per);
}

// Pass 1: per-block maximum and sum of exponentials.  Each warp takes eight
// keys per lane at a time and sums them against its running maximum, so only
// a new maximum costs FP64 work.  Block 0 clears what the later passes count
// in (the previous call's contents).
__global__ void __launch_bounds__(kThreads) sel_lse(const double* __restrict__ lw, long long n, int h_max,
                                                    unsigned char* base) {
  load_exp_tab();
  pdl_enter();
  Ptrs p = ptrs_of(base);
  if (blockIdx.x == 0) {
    for (int b = threadIdx.x; b < kBinsS; b += blockDim.x) p.hist[b] = 0u;
    if (threadIdx.x == 0) {
      p.sc->done[0] = p.sc->done[1] = p.sc->done[2] = 0u;
      p.sc->n_list = 0u;
      p.sc->n_bin = 0u;
      p.sc->left = 0;
      p.sc->need = h_max;
      p.sc->prefix = 0;
      p.sc->bound = 0;
      p.sc->mode = 0;
    }
  }
  long long lo, hi;
  chunk_of(n, lo, hi);
  LseS v{kKeyInvalid, 0.0};
  constexpr int kU = 8;
  for (long long j0 = lo; j0 < hi; j0 += kU * kThreads) {
    double x[kU];
    long long k[kU], m = v.m;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const long long j = j0 + u * kThreads + threadIdx.x;
      x[u] = j < hi ? lw[j] : -INFINITY;
    }
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      k[u] = key_of(x[u]);
      m = max(m, k[u]);
    }
    m = warp_max_ll(m);
    if (m == kKeyInvalid) continue;
    if (m != v.m) {
      if (v.m != kKeyInvalid) v.s *= fx::exp_fixed((unsigned long long)(m - v.m), exp_tab());
      v.m = m;
    }
    fx::ExpSum s;
#pragma unroll
    for (int u = 0; u < kU; ++u)
      if (k[u] != kKeyInvalid) s.add((unsigned long long)(m - k[u]), exp_tab());
    if (s.any()) v.s += s.value();
  }
  v = block_lse(v);
  if (threadIdx.x == 0) {
    p.blk_m[blockIdx.x] = v.m;
    p.blk_s[blockIdx.x] = v.s;
  }
}

// Boundary digit of histogram h (BINS bins, shared memory) by a block of 1024
// threads: the digit, the elements in its bin and those still needed of them;
// `all`: the whole histogram is within `need`.
struct Digit {
  int digit;
  unsigned count;
  long long need;
  bool all;
};
template <int BINS>
__device__ Digit find_digit(const unsigned* h, long long need) {
  constexpr int kPer = BINS / 1024;
  __shared__ unsigned wsum[32];
  __shared__ int s_digit;
  __shared__ unsigned s_count;
  __shared__ long long s_need;
  const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
  unsigned b[kPer], mine = 0;
#pragma unroll
  for (int k = 0; k < kPer; ++k) {
    b[k] = h[kPer * t + k];
    mine += b[k];
  }
  const unsigned x = warp_incl(mine);
  if (lane == 31) wsum[wp] = x;
  __syncthreads();
  const unsigned ws = warp_incl(wsum[lane]);
  const unsigned total = __shfl_sync(0xFFFFFFFFu, ws, 31);
  const unsigned before = __shfl_sync(0xFFFFFFFFu, ws, max(wp - 1, 0));
  const unsigned above = total - x - (wp > 0 ? before : 0u), upto = above + mine;
  if ((long long)above < need && (long long)upto >= need) {
    unsigned cum = above, in = 0;
    int at = 0;
    bool found = false;
#pragma unroll
    for (int k = kPer - 1; k >= 0; --k) {
      if (found) continue;
      if ((long long)(cum + b[k]) >= need) {
        found = true;
        at = k;
        in = b[k];
      } else {
        cum += b[k];
      }
    }
    s_digit = kPer * t + at;
    s_count = in;
    s_need = need - cum;
  }
  __syncthreads();
  const Digit d{s_digit, s_count, s_need, (long long)total <= need};
  __syncthreads();
  return d;
}

// one more key in bin `bin` (< 0: none) of a histogram in shared memory; a
// warp whose keys share their bin (equal weights) adds them at once
__device__ __forceinline__ void hist_add(unsigned* hist, int bin) {
  const unsigned act = __ballot_sync(__activemask(), bin >= 0);
  if (bin < 0) return;
  int same;
  __match_all_sync(act, bin, &same);
  if (!same) atomicAdd(&hist[bin], 1u);
  else if ((int)(threadIdx.x & 31) == __ffs(act) - 1) atomicAdd(&hist[bin], (unsigned)__popc(act));
}

// true in every thread of the grid's last block to get here
__device__ bool last_block(unsigned* done) {
  __shared__ bool last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (last) __threadfence();
  return last;
}

// Pass 2: histogram of the first digit, of `width` bits at `shift`, of the
// keys at or above the threshold; the last block finds the boundary digit.
// Every block forms the log-sum-exp and the threshold from pass 1's partials
// (the same in all).
__global__ void __launch_bounds__(1024) sel_hist(const double* __restrict__ lw, long long n, int shift, int width,
                                                 int nblk_lse, double log_tau, unsigned char* base) {
  load_exp_tab();
  pdl_enter();
  __shared__ unsigned hist[kBinsS];
  __shared__ long long s_thr;
  Ptrs p = ptrs_of(base);
  for (int b = threadIdx.x; b < kBinsS; b += blockDim.x) hist[b] = 0;
  {
    const int b = threadIdx.x;   // one partial per thread (kMaxBlocks = blockDim)
    const LseS u = block_lse(b < nblk_lse ? LseS{p.blk_m[b], p.blk_s[b]} : LseS{kKeyInvalid, 0.0});
    const bool none = u.m == kKeyInvalid || !(u.s > 0.0);
    if (threadIdx.x == 0) {
      double lse = -INFINITY;
      long long thr = LLONG_MAX;
      if (!none) {
        lse = (double)u.m * kFxInv + log(u.s);
        thr = (long long)ceil((lse + log_tau) * 4294967296.0);
      }
      s_thr = thr;
      if (blockIdx.x == 0) {
        p.sc->lse = lse;
        p.sc->thr = thr;
        p.sc->top = u.m;
      }
    }
  }
  __syncthreads();
  const long long thr = s_thr;
  long long lo, hi;
  chunk_of(n, lo, hi);
#pragma unroll 4
  for (long long j = lo + threadIdx.x; j < hi; j += blockDim.x) {
    const long long k = key_of(lw[j]);
    if (k == kKeyInvalid || k < thr) continue;
    const unsigned long long v = (unsigned long long)(k - thr);
    if ((v >> (shift + width)) != 0ull) continue;
    atomicAdd(&hist[(v >> shift) & ((1u << width) - 1u)], 1u);
  }
  __syncthreads();
  for (int b = threadIdx.x; b < kBinsS; b += blockDim.x)
    if (hist[b]) atomicAdd(&p.hist[b], hist[b]);
  if (!last_block(&p.sc->done[0])) return;
  for (int b = threadIdx.x; b < kBinsS; b += blockDim.x) hist[b] = __ldcg(&p.hist[b]);
  __syncthreads();
  const Digit d = find_digit<kBinsS>(hist, p.sc->need);
  // the next digit's bins, in place of the partials and of this histogram
  if (d.count > kListS)
    for (int b = threadIdx.x; b < kWideBins; b += blockDim.x) p.wide[b] = 0u;
  if (threadIdx.x != 0) return;
  if (thr == LLONG_MAX) {
    p.sc->mode = 2;
  } else if (d.all) {
    p.sc->mode = 1;
    p.sc->bound = thr - 1;
    p.sc->need = 0;
  } else {
    p.sc->prefix = d.digit;
    p.sc->need = d.need;
    p.sc->n_bin = d.count;
    p.sc->left = shift;
    if (shift == 0) p.sc->bound = thr + d.digit;
  }
}

// Pass 3, once or, for more than kSoloN children, once per kWideBits bits that
// may be left: the rest of the boundary key.  A boundary bin that fits the
// list is listed, and the last block finds the key among its keys digit by
// digit in shared memory; a larger one takes one digit from a histogram over
// the grid (`solo`: the last block reads the children again for each digit).
// A million children, whole call: h_max 20000 of smooth, equal, nearly equal
// weights 66, 65, 73 us, h_max 400000 of smooth ones 70 us; four million,
// h_max a million 177 us (in one block 5.3 ms).
__global__ void __launch_bounds__(1024) sel_boundary(const double* __restrict__ lw, long long n, int solo,
                                                     unsigned char* base) {
  pdl_enter();
  __shared__ unsigned hist[kWideBins];
  Ptrs p = ptrs_of(base);
  const int left = p.sc->left;
  if (p.sc->mode != 0 || left == 0) return;
  const long long thr = p.sc->thr;
  unsigned long long prefix = (unsigned long long)p.sc->prefix;
  const int lane = threadIdx.x & 31;
  const bool listed = p.sc->n_bin <= kListS, wide = !listed && !solo;
  const int width_w = min(kWideBits, left), shift_w = left - width_w;   // a wide digit
  long long lo, hi;
  chunk_of(n, lo, hi);
  if (wide) {
    for (int b = threadIdx.x; b < kWideBins; b += blockDim.x) hist[b] = 0u;
    __syncthreads();
#pragma unroll 4
    for (long long j = lo + threadIdx.x; j < hi; j += blockDim.x) {
      const long long k = key_of(lw[j]);
      if (k == kKeyInvalid || k < thr) continue;
      const unsigned long long v = (unsigned long long)(k - thr);
      if ((v >> left) != prefix) continue;
      atomicAdd(&hist[(v >> shift_w) & ((1u << width_w) - 1u)], 1u);
    }
    __syncthreads();
    for (int b = threadIdx.x; b < kWideBins; b += blockDim.x)
      if (hist[b]) atomicAdd(&p.wide[b], hist[b]);
  } else if (listed) {
    for (long long j0 = lo; j0 < hi; j0 += blockDim.x) {
      const long long j = j0 + threadIdx.x;
      const long long k = j < hi ? key_of(lw[j]) : kKeyInvalid;
      const bool in = k != kKeyInvalid && k >= thr && ((unsigned long long)(k - thr) >> left) == prefix;
      const unsigned bal = __ballot_sync(0xFFFFFFFFu, in);
      if (!bal) continue;
      unsigned at = 0;
      if (lane == __ffs(bal) - 1) at = atomicAdd(&p.sc->n_list, (unsigned)__popc(bal));
      at = __shfl_sync(0xFFFFFFFFu, at, __ffs(bal) - 1) + __popc(bal & ((1u << lane) - 1u));
      if (in && at < kListS) p.list[at] = k;
    }
  }
  if (!last_block(&p.sc->done[1])) return;
  long long need = p.sc->need;
  if (wide) {
    for (int b = threadIdx.x; b < kWideBins; b += blockDim.x) {
      hist[b] = __ldcg(&p.wide[b]);
      p.wide[b] = 0u;   // for the next digit
    }
    __syncthreads();
    const Digit d = find_digit<kWideBins>(hist, need);
    if (threadIdx.x == 0) {
      prefix = (prefix << width_w) | (unsigned)d.digit;
      p.sc->done[1] = 0u;
      p.sc->prefix = (long long)prefix;
      p.sc->need = d.need;
      p.sc->n_bin = d.count;
      p.sc->left = shift_w;
      if (shift_w == 0) p.sc->bound = thr + (long long)prefix;
    }
    return;
  }
  const long long total = listed ? (long long)min(__ldcg(&p.sc->n_list), kListS) : n;
  for (int above = left; above > 0;) {
    const int width = min(kWideBits, above), sh = above - width;
    for (int b = threadIdx.x; b < kWideBins; b += blockDim.x) hist[b] = 0u;
    __syncthreads();
    for (long long j0 = 0; j0 < total; j0 += blockDim.x) {
      const long long j = j0 + threadIdx.x;
      const long long k = j >= total ? kKeyInvalid : listed ? __ldcg(&p.list[j]) : key_of(lw[j]);
      const unsigned long long v = (unsigned long long)(k - thr);
      const bool in = k != kKeyInvalid && k >= thr && (v >> above) == prefix;
      hist_add(hist, in ? (int)((v >> sh) & ((1u << width) - 1u)) : -1);
    }
    __syncthreads();
    const Digit d = find_digit<kWideBins>(hist, need);
    prefix = (prefix << width) | (unsigned)d.digit;
    need = d.need;
    above = sh;
  }
  if (threadIdx.x == 0) {
    p.sc->need = need;
    p.sc->bound = thr + (long long)prefix;
    p.sc->left = 0;
  }
}

__device__ __forceinline__ void keep_kind(long long k, const SelScal& s, bool& gt, bool& eq) {
  gt = eq = false;
  if (s.mode == 2 || k == kKeyInvalid || k < s.thr) return;
  if (k > s.bound) gt = true;
  else if (k == s.bound && s.need > 0) eq = true;
}

// Pass 4: per-block counts above and at the boundary, and the sum of
// exp(key - largest key) above it; the last block turns the counts into
// offsets and forms the kept children's log-sum-exp (the largest key is
// always kept).
__global__ void __launch_bounds__(kThreads) sel_count(const double* __restrict__ lw, long long n, int h_max,
                                                      int* n_out, unsigned char* base) {
  load_exp_tab();
  pdl_enter();
  __shared__ unsigned long long wc[kThreads / 32];
  __shared__ double wd[kThreads / 32];
  Ptrs p = ptrs_of(base);
  const SelScal s = *p.sc;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  constexpr int kWarps = kThreads / 32;
  long long lo, hi;
  chunk_of(n, lo, hi);
  unsigned long long c = 0;   // above | at << 32
  double sum = 0.0;
  constexpr int kU = 4;
  for (long long j0 = lo; j0 < hi; j0 += kU * kThreads) {
    fx::ExpSum f;
#pragma unroll
    for (int u = 0; u < kU; ++u) {
      const long long j = j0 + u * kThreads + threadIdx.x;
      const long long k = j < hi ? key_of(lw[j]) : kKeyInvalid;
      bool gt, eq;
      keep_kind(k, s, gt, eq);
      c += (gt ? 1ull : 0ull) + (eq ? 1ull << 32 : 0ull);
      if (gt) f.add((unsigned long long)(s.top - k), exp_tab());
    }
    if (f.any()) sum += f.value();
  }
  c = warp_sum_of(c);
  sum = warp_sum_of(sum);
  if (lane == 0) {
    wc[wp] = c;
    wd[wp] = sum;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kWarps; ++w) {
      c += wc[w];
      sum += wd[w];
    }
    p.blk_gt[blockIdx.x] = (unsigned)(c & 0xFFFFFFFFull);
    p.blk_eq[blockIdx.x] = (unsigned)(c >> 32);
    p.blk_s[blockIdx.x] = sum;
  }
  if (!last_block(&p.sc->done[2])) return;
  // exclusive offsets over the blocks, four per thread
  unsigned long long v[4], mine = 0;
  sum = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const unsigned b = 4 * threadIdx.x + q;
    v[q] = b < gridDim.x ? ((unsigned long long)__ldcg(&p.blk_eq[b]) << 32) | __ldcg(&p.blk_gt[b]) : 0ull;
    if (b < gridDim.x) sum += __ldcg(&p.blk_s[b]);
    mine += v[q];
  }
  const unsigned long long x = warp_incl(mine);
  sum = warp_sum_of(sum);
  if (lane == 31) wc[wp] = x;
  if (lane == 0) wd[wp] = sum;
  __syncthreads();
  unsigned long long excl = x - mine, total = 0;
  for (int w = 0; w < kWarps; ++w) {
    if (w < wp) excl += wc[w];
    total += wc[w];
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const unsigned b = 4 * threadIdx.x + q;
    if (b < gridDim.x) {
      p.blk_gt[b] = (unsigned)(excl & 0xFFFFFFFFull);
      p.blk_eq[b] = (unsigned)(excl >> 32);
    }
    excl += v[q];
  }
  if (threadIdx.x == 0) {
    const long long gt = (long long)(total & 0xFFFFFFFFull), eq = (long long)(total >> 32);
    long long kept = s.mode == 2 ? 0 : gt + min(eq, s.need);
    if (kept > h_max) kept = h_max;
    *n_out = (int)kept;
    for (int w = 1; w < kWarps; ++w) sum += wd[w];
    if (s.mode == 0 && s.need > 0)
      sum += (double)min(eq, s.need) * fx::exp_fixed((unsigned long long)(s.top - s.bound), exp_tab());
    p.sc->lse_kept = kept > 0 ? ((double)s.top * kFxInv - s.lse) + log(sum) : 0.0;
  }
}

// Pass 5: kept children in index order, their log-weights normalised over
// all children and then over the kept ones
__global__ void __launch_bounds__(kThreads) sel_write(const double* __restrict__ lw, long long n, int h_max,
                                                      long long* idx_out, double* lw_out, unsigned char* base) {
  pdl_enter();
  __shared__ unsigned wg[2][kThreads / 32], we[2][kThreads / 32];
  Ptrs p = ptrs_of(base);
  const SelScal s = *p.sc;
  long long lo, hi;
  chunk_of(n, lo, hi);
  unsigned run_g = p.blk_gt[blockIdx.x], run_e = p.blk_eq[blockIdx.x];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  int par = 0;
  for (long long base_j = lo; base_j < hi; base_j += kThreads, par ^= 1) {
    const long long j = base_j + threadIdx.x;
    bool gt = false, eq = false;
    long long k = kKeyInvalid;
    if (j < hi) {
      k = key_of(lw[j]);
      keep_kind(k, s, gt, eq);
    }
    const unsigned bg = __ballot_sync(0xFFFFFFFFu, gt), be = __ballot_sync(0xFFFFFFFFu, eq);
    if (lane == 0) { wg[par][wp] = __popc(bg); we[par][wp] = __popc(be); }
    __syncthreads();
    unsigned og = run_g, oe = run_e;
    for (int w = 0; w < kThreads / 32; ++w) {
      if (w < wp) { og += wg[par][w]; oe += we[par][w]; }
      run_g += wg[par][w];
      run_e += we[par][w];
    }
    og += __popc(bg & ((1u << lane) - 1u));
    oe += __popc(be & ((1u << lane) - 1u));
    if (gt || (eq && (long long)oe < s.need)) {
      const long long pos = (long long)og + ((long long)oe < s.need ? (long long)oe : s.need);
      if (pos < h_max) {
        idx_out[pos] = j;
        lw_out[pos] = ((double)k * kFxInv - s.lse) - s.lse_kept;
      }
    }
  }
}

// a launch whose blocks may start while the previous kernel of the stream
// finishes (every kernel waits for it in pdl_enter)
template <typename... KArgs, typename... Args>
void launch_sel(void (*k)(KArgs...), int grid, int block, cudaStream_t s, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, static_cast<KArgs>(args)...);
}

// device address of the scratch array, looked up once per device
std::mutex g_setup_mutex;
unsigned char* g_scratch_ptr[128] = {};

glmb_status scratch_for_current_device(unsigned char** out) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 128) return GLMB_E_CUDA;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_scratch_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_select_scratch) != cudaSuccess || !p) return GLMB_E_CUDA;
    g_scratch_ptr[dev] = (unsigned char*)p;
  }
  *out = g_scratch_ptr[dev];
  return GLMB_OK;
}

}  // namespace

extern "C" glmb_status glmb_select_top_static(const double* logw_dev, int64_t n, int32_t h_max,
                                              double tau, int64_t* idx_out_dev, double* logw_out_dev,
                                              int32_t* n_out_dev, void* stream) {
  if (n < 0 || h_max < 1 || !(tau > 0.0) || !n_out_dev || (n > 0 && (!logw_dev || !idx_out_dev ||
                                                                      !logw_out_dev)))
    return GLMB_E_INVALID;
  if (n > kMaxN || h_max > (1 << 30)) return GLMB_E_CAPACITY;
  unsigned char* base = nullptr;
  const glmb_status st = scratch_for_current_device(&base);
  if (st != GLMB_OK) return st;
  cudaStream_t s = (cudaStream_t)stream;
  // blocks of the passes whose partials are kept per block, and of the
  // passes with a histogram per block (one of 1024 threads per SM: each
  // block adds its bins to global memory once)
  const int nblk = (int)(n == 0 ? 1 : std::min<long long>((n + 4 * kThreads - 1) / (4 * kThreads), kMaxBlocks));
  const int hblk = (int)std::max<long long>(1, std::min<long long>((n + 1023) / 1024, 152));
  const double log_tau = std::log(tau);
  const double vmax = std::max(1.0, -log_tau) * 4294967296.0 + 2.0;
  const int nbits = std::max(1, (int)std::ceil(std::log2(vmax)));
  // digits from the top of the nbits bits of key - threshold
  const int width = std::min(kDigitS, nbits), top = nbits - width;
  launch_sel(sel_lse, nblk, kThreads, s, logw_dev, n, h_max, base);
  launch_sel(sel_hist, hblk, 1024, s, logw_dev, n, top, width, nblk, log_tau, base);
  const int solo = n <= kSoloN ? 1 : 0;
  for (int above = top; above > 0; above -= solo ? above : kWideBits)
    launch_sel(sel_boundary, hblk, 1024, s, logw_dev, n, solo, base);
  launch_sel(sel_count, nblk, kThreads, s, logw_dev, n, h_max, n_out_dev, base);
  launch_sel(sel_write, nblk, kThreads, s, logw_dev, n, h_max, (long long*)idx_out_dev, logw_out_dev, base);
  return cudaGetLastError() == cudaSuccess ? GLMB_OK : GLMB_E_CUDA;
}
