// Alg. 2 on small windows: one block runs a whole window in shared memory.
//
// A window of a few thousand tokens leaves the many kernels of the general
// path (suffix.cu, repeats.cu: about 60 launches and six host reads per call)
// with nothing but their latencies: 580-630 us for 4,096 tokens of which no
// kernel needs more than a few.  Here one launch does every stage of every
// window, one block each, and the host reads the counts once at the end.  The
// online finder's slices (250 to 5,000 tokens) and the batches a server forms
// of them are such calls.
//
//  codes    the window's tokens sorted by an in-block LSD radix sort (only the
//           digits in which they differ) become dense order-preserving codes;
//           that order is also the doubling's level 0.
//  SA       prefix doubling: round r sorts each group of equal first h tokens
//           by the rank at distance h.  Groups are contiguous, so a suffix's new
//           slot is its group's first slot plus the number of smaller keys in
//           the group, counted directly -- sum g^2 comparisons in all, two per
//           instruction on the keys' bits read as halves; when that exceeds what a
//           radix sort of the whole window costs (long runs, short periods), the
//           sort is taken instead.
//  LCP      Phi / PLCP over a few positions per thread by direct comparison of
//           the codes; a match that keeps going is finished by lifting over the
//           level ranks (kept in global memory).
//  rest     candidates, their ids by block minima of the LCP array, one in-block sort of
//           (length, id, start) keys, deduplication, the greedy loop in rounds
//           that start small (the first long candidates cover most of the
//           window, so that later rounds drop most of theirs unsettled), R, and
//           the selected intervals by a scan over positions.
// Windows learn where their outputs go from a decoupled look-back over their
// counts, in ticket order.  Every result equals the general path's: the order
// of candidates is total, and the doubling-round count is derived from the
// longest LCP (a round r runs iff some LCP is at least h0 * 2^(r-1)).
//
// What bounds it: the instructions one SM can issue (1,024 threads, one block
// per SM; fewer threads were slower, 158 against 144 us at 4,096 tokens) and
// barriers; the data never leaves the SM between the stages.  At 4,096 tokens
// (period 50, 5% noise; 122 us in the kernel): token order 11 us, seven rounds
// 46, LCP 13, candidates 12, their sort 15, greedy 19, R and outputs 5.
// Measured per call, before (general path) and now: 4,096 u32 tokens 581-629
// -> 144-149 us; 40 windows of 250 to 5,000 u64 tokens 830 -> 176-186 us.
#include <algorithm>
#include <cstring>
#include <vector>

#include <cuda_fp16.h>

#include "apo_internal.cuh"
#include "device_util.cuh"

namespace apo {

namespace {

constexpr int kRowPad = 258;     // digit counters per warp, padded against bank conflicts
constexpr uint32_t kHalfBase = 0x400;  // minor keys 0 .. 8192 plus this are the bits of normal halves, in order
constexpr uint32_t kDirectCost = 320;  // comparisons per suffix that cost what a radix sort of the window costs
constexpr int kSharedLevels = 8;  // level ranks that fit the sort keys' 16 bytes per token
constexpr uint32_t kDirect = 8;  // tokens compared directly before lifting
constexpr uint64_t kSetEmpty = ~0ull;

// Device words of a call (zeroed ahead of it): see small_find_repeats.
enum : int { kSwTicket = 0, kSwCand, kSwSel, kSwTrace, kSwMaxLcp, kSwSigma, kSwMaxTok /* u64 */, kSwWords = 8 };

struct SmallArgs {
  const void *tokens;
  const uint32_t *off;     // [W + 1] window offsets, null for one window
  uint32_t W, n;           // windows; tokens of the single window
  uint32_t min_len;
  uint16_t *snaps;         // level ranks: window w's level L at (off[w] * levels, up to a multiple of 8) + 8 w + L * n_w
                           // (16-byte boundaries, and no window reaches into the next one's)
  int levels;
  uint32_t *sa, *lcp;      // outputs as apo_repeats_out (null: not wanted)
  uint32_t *cl, *cid, *cs;
  uint8_t *acc;
  uint64_t cand_cap, sel_cap, trace_cap;
  uint32_t *ss, *sl, *st;
  uint32_t *tl, *ts;
  uint32_t *offs;          // [3 (W + 1)] where each window's candidates, intervals, traces start
  uint32_t *words;         // kSw*
  uint64_t *status;        // [3 W] look-back words
  uint64_t *set;           // distinct tokens of all windows (null: not wanted)
  uint64_t set_mask;
  uint32_t epoch;
  uint32_t *err;
};

__device__ __forceinline__ int sm_bits(uint32_t v) { return v ? 32 - __clz(v) : 0; }

// One stable LSD radix pass after another over bits [lo, hi) of buf[0, cnt)
// (and of the values in vbuf).  A thread keeps its keys in registers between
// the read and the scatter, so the sort is in place.  Digits in which `diff`
// has no bit set are skipped (all keys agree there).
template <int TPB, int ITEMS, bool VAL>
__device__ void block_sort(uint64_t *buf, uint16_t *vbuf, uint32_t cnt, int lo, int hi, uint64_t diff,
                           uint16_t *wc, WarpScan<TPB / 32> &scan) {
  constexpr int NW = TPB / 32, PARTS = TPB / 256, WPP = NW / PARTS;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lt = lanemask_lt();
  const int per = (int)((cnt + TPB - 1) / TPB);  // rows of 32 per warp
  const uint32_t seg = (uint32_t)warp * per * 32 + lane;
  uint16_t *my = wc + warp * kRowPad;
  for (int sh = lo; sh < hi; sh += 8) {
    if (((diff >> sh) & 255) == 0) continue;
    for (int d = lane; d < kRowPad / 2; d += 32) reinterpret_cast<uint32_t *>(my)[d] = 0;
    __syncwarp();
    uint64_t k[ITEMS];
    uint16_t v[VAL ? ITEMS : 1];
    uint32_t rk[(ITEMS + 1) / 2];  // two 16-bit ranks per word
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      if (j >= per) break;
      const uint32_t p = seg + j * 32;
      const bool ok = p < cnt;
      k[j] = ok ? buf[p] : 0;
      if (VAL) v[j] = ok ? vbuf[p] : 0;
      const uint32_t d = (uint32_t)(k[j] >> sh) & 255u;
      const uint32_t peers = __match_any_sync(0xffffffffu, ok ? d : 256u);
      const uint32_t b = my[d];
      __syncwarp();
      const uint32_t r = b + __popc(peers & lt);
      if (ok && (peers & lt) == 0) my[d] = (uint16_t)(b + __popc(peers));
      __syncwarp();
      if (j & 1) rk[j / 2] |= r << 16;
      else rk[j / 2] = r;
    }
    __syncthreads();
    {  // digit-major, warp-minor prefixes: PARTS threads per digit, WPP warps each
      const int d = tid / PARTS, w0 = (tid % PARTS) * WPP;
      uint32_t run = 0, c[WPP];
#pragma unroll
      for (int w = 0; w < WPP; ++w) {
        c[w] = wc[(w0 + w) * kRowPad + d];
        run += c[w];
      }
      const uint32_t inc = warp_inclusive(run, OpSum());
      uint32_t tot;
      uint32_t at = scan.run(__shfl_sync(0xffffffffu, inc, 31), OpSum(), &tot) + inc - run;
#pragma unroll
      for (int w = 0; w < WPP; ++w) {
        wc[(w0 + w) * kRowPad + d] = (uint16_t)at;
        at += c[w];
      }
    }
    __syncthreads();
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      if (j >= per) break;
      if (seg + j * 32 < cnt) {
        const uint32_t q = my[(uint32_t)(k[j] >> sh) & 255u] + ((j & 1) ? rk[j / 2] >> 16 : rk[j / 2] & 0xffffu);
        buf[q] = k[j];
        if (VAL) vbuf[q] = v[j];
      }
    }
    __syncthreads();
  }
}

// Adds a token to the call's set of distinct tokens and counts it when it is
// new (all-ones, the empty mark, is not counted).  Past half the table's
// entries the count only says "more than that", and insertion stops.
__device__ __forceinline__ void set_insert(uint64_t *set, uint64_t mask, uint64_t t, uint32_t *count) {
  if (t == kSetEmpty || *(volatile uint32_t *)count > mask / 2 + 1) return;
  uint64_t x = t;
  x ^= x >> 33;
  x *= 0xff51afd7ed558ccdull;
  x ^= x >> 33;
  uint64_t slot = x & mask;
  for (uint64_t probe = 0; probe <= mask; ++probe) {
    const uint64_t cur =
        atomicCAS((unsigned long long *)&set[slot], (unsigned long long)kSetEmpty, (unsigned long long)t);
    if (cur == kSetEmpty) {
      atomicAdd(count, 1u);
      return;
    }
    if (cur == t) return;
    slot = (slot + 1) & mask;
  }
}

template <class T>
__global__ void k_small_set(const T *__restrict__ tokens, uint32_t n, uint64_t *set, uint64_t mask,
                            uint32_t *count) {
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
    if (i == 0 || tokens[i] != tokens[i - 1]) set_insert(set, mask, tokens[i], count);
}

// How many of mk[b, e) are below x (all of them bits of positive halves):
// eight keys per load, two per comparison; entries of the first and last load
// that lie outside are turned into NaNs, which compare as not below.
__device__ __forceinline__ uint32_t count_less(const uint16_t *mk, uint32_t b, uint32_t e, uint32_t x) {
  const __half2 xx = __halves2half2(__ushort_as_half((unsigned short)x), __ushort_as_half((unsigned short)x));
  uint32_t total = 0;
  const uint32_t v1 = (e + 7) >> 3;
  for (uint32_t v = b >> 3; v < v1;) {
    __half2 acc = __float2half2_rn(0.f);
    const uint32_t stop = min(v1, v + 256);  // sums of at most 1,024 per half: exact
    for (; v < stop; ++v) {
      uint4 z = *reinterpret_cast<const uint4 *>(mk + 8 * v);
      const uint32_t p = 8 * v;
      if (p < b || p + 8 > e) {
        uint32_t *w = &z.x;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          if (p + 2 * q < b || p + 2 * q >= e) w[q] |= 0x7fffu;
          if (p + 2 * q + 1 < b || p + 2 * q + 1 >= e) w[q] |= 0x7fff0000u;
        }
      }
      const __half2 *hh = reinterpret_cast<const __half2 *>(&z);
      acc = __hadd2(acc, __hadd2(__hadd2(__hlt2(hh[0], xx), __hlt2(hh[1], xx)),
                                 __hadd2(__hlt2(hh[2], xx), __hlt2(hh[3], xx))));
    }
    total += (uint32_t)(__low2float(acc) + __high2float(acc));
  }
  return total;
}

// Largest j < k with a0[j] < l, or -1 (meaningful for lanes with `want`), for
// the 32 entries k = base + lane of a warp (base a multiple of 32, v = a0[k]);
// a1[x] = the minimum of a0[32 x .. 32 x + 31].  The block of 32 is in the
// warp's registers; the blocks before it are the same for every lane, so their
// minima are read eight at a time by all lanes at once; then each lane looks
// through its own block.
__device__ __forceinline__ int prev_less_warp(const uint16_t *a0, const uint16_t *a1, uint32_t base, uint32_t v,
                                              uint32_t l, bool want) {
  const int lane = threadIdx.x & 31;
  int f = -1;
#pragma unroll
  for (int d = 31; d >= 1; --d) {
    const uint32_t x = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d && x < l) f = lane - d;  // the nearest one is met last
  }
  int blk = -1;
  bool open = want && f < 0;
  for (int x = ((int)(base >> 5) - 1) | 7; x >= 0 && __any_sync(0xffffffffu, open); x -= 8) {
    const uint4 z = *reinterpret_cast<const uint4 *>(a1 + (x & ~7));
    const uint32_t w[4] = {z.x, z.y, z.z, z.w};
    if (open) {
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int y = (x & ~7) + q;
        if (y < (int)(base >> 5) && ((w[q >> 1] >> (16 * (q & 1))) & 0xffffu) < l) blk = y;
      }
      open = blk < 0;
    }
  }
  if (f >= 0) return (int)base + f;
  if (blk < 0) return -1;
  int r = -1;
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    const uint4 z = *reinterpret_cast<const uint4 *>(a0 + blk * 32 + g * 8);
    const uint32_t w[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (((w[q >> 1] >> (16 * (q & 1))) & 0xffffu) < l) r = g * 8 + q;
  }
  return blk * 32 + r;
}

__device__ __forceinline__ void pair_cand_small(uint32_t s1, uint32_t s2, uint32_t p, uint32_t *l, uint32_t *a,
                                                uint32_t *b) {
  const uint32_t lo = min(s1, s2), d = max(s1, s2) - lo;
  if (d >= p) {
    *l = p;
    *a = s1;
    *b = s2;
  } else {  // the common prefix is a run of S[lo, lo + d)
    uint32_t h = (p + d) / 2;
    h -= h % d;
    *l = h;
    *a = lo;
    *b = lo + h;
  }
}

template <int TPB, int ITEMS>
struct SmallShape {
  static constexpr int kMaxN = TPB * ITEMS / 2;  // 2n candidates, ITEMS per thread
  static constexpr size_t kSmem = (size_t)2 * kMaxN * 8               // sort keys
                                  + (size_t)(TPB / 32) * kRowPad * 2 + 16  // digit counters
                                  + (size_t)(kMaxN + 64) * 2            // codes
                                  + (size_t)kMaxN * 2 * 3               // sa, rank, lcp
                                  + (size_t)(kMaxN / 32 + 32) * 2       // LCP minima
                                  + (size_t)(kMaxN / 32 + 4) * 4        // mark bitmap
                                  + (size_t)(2 * kMaxN / 32) * 4;       // accepted candidates
  static_assert(kMaxN <= 8192, "slots, ranks and minor keys fit 13 bits");
};

template <class T, int TPB, int ITEMS>
__global__ void __launch_bounds__(TPB, 1) k_small(const SmallArgs a) {
  using S = SmallShape<TPB, ITEMS>;
  constexpr int NW = TPB / 32, NMAX = S::kMaxN, HI = ITEMS / 2;  // HI: suffixes per thread
  extern __shared__ __align__(16) uint8_t smem[];
  uint64_t *buf = reinterpret_cast<uint64_t *>(smem);                // [2 NMAX]
  uint16_t *wc = reinterpret_cast<uint16_t *>(buf + 2 * NMAX);       // [NW][kRowPad]
  uint16_t *code = wc + NW * kRowPad + 8;                            // [NMAX + 64], 0 past the end
  uint16_t *sa = code + NMAX + 64, *rank = sa + NMAX, *lcp = rank + NMAX;
  uint16_t *t1 = lcp + NMAX;                                         // [NMAX / 32 + 32]
  uint32_t *bits = reinterpret_cast<uint32_t *>(t1 + NMAX / 32 + 32);  // [NMAX / 32 + 4]
  uint32_t *accw = bits + NMAX / 32 + 4;                             // [2 NMAX / 32] accepted candidates, as bits
  // while the doubling runs, in the half of buf that its sorts leave free:
  uint16_t *mk = reinterpret_cast<uint16_t *>(buf + NMAX);           // [NMAX] minor keys of a round, by slot
  uint16_t *act = mk + NMAX;                                         // [NMAX] active slots
  uint32_t *cnt = reinterpret_cast<uint32_t *>(act + NMAX);          // [NMAX] a group's size, at its first slot
  __shared__ uint32_t scr[2 * NW], s_win, s_cnt, s_sum, s_tot[3], s_base[3];
  __shared__ uint64_t s_or[NW], s_and[NW];
  WarpScan<NW> scan{scr, 0};
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t lt = lanemask_lt();
  if (tid == 0) {
    s_win = a.off ? atomicAdd(&a.words[kSwTicket], 1u) : 0u;
    s_cnt = 0;
  }
  __syncthreads();
  const uint32_t w = s_win;
  const uint32_t o0 = a.off ? a.off[w] : 0u;
  const uint32_t n = a.off ? a.off[w + 1] - o0 : a.n;
  if (n > (uint32_t)NMAX) {  // (the host launches a shape that holds the longest window)
    if (tid == 0) atomicExch(a.err, kDevRange);
    return;
  }
  const int nb = max(1, sm_bits(n ? n - 1 : 0));
  uint32_t m = 0, K = 0, Tn = 0;  // candidates, accepted, traces
  uint32_t maxl = 0;
  uint16_t *snap = a.snaps + (((size_t)o0 * a.levels + 7) & ~(size_t)7) + (size_t)w * 8;

  if (n) {
    // ---- dense codes: the tokens in order
    {
      const T *tok = static_cast<const T *>(a.tokens) + o0;
      uint64_t orv = 0, andv = ~0ull, mx = 0;
#pragma unroll
      for (int j = 0; j < HI; ++j) {
        const uint32_t i = tid + j * TPB;
        if (i < n) {
          const uint64_t t = tok[i];
          buf[i] = t;
          rank[i] = (uint16_t)i;
          orv |= t;
          andv &= t;
          mx = t > mx ? t : mx;
        }
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        orv |= __shfl_xor_sync(0xffffffffu, orv, o);
        andv &= __shfl_xor_sync(0xffffffffu, andv, o);
        const uint64_t x = __shfl_xor_sync(0xffffffffu, mx, o);
        mx = x > mx ? x : mx;
      }
      if (lane == 0) {
        s_or[warp] = orv;
        s_and[warp] = andv;
        atomicMax(reinterpret_cast<unsigned long long *>(a.words + kSwMaxTok), (unsigned long long)mx);
      }
    }
    __syncthreads();
    uint64_t diff;  // bits in which the tokens differ
    {
      uint64_t x = lane < NW ? s_or[lane] : 0, y = lane < NW ? s_and[lane] : ~0ull;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        x |= __shfl_xor_sync(0xffffffffu, x, o);
        y &= __shfl_xor_sync(0xffffffffu, y, o);
      }
      diff = x ^ y;
    }
    block_sort<TPB, HI, true>(buf, rank, n, 0, 8 * (int)sizeof(T), diff, wc, scan);
    // level 0: sorted element k is suffix rank[k]; its group starts at the
    // last token change at or before k, its code is the number of changes
    const int per = (int)((n + TPB - 1) / TPB);
    const uint32_t seg = (uint32_t)warp * per * 32 + lane;
    uint32_t hb = 0, wmax = 0, wsum = 0;  // bit j: element seg + 32 j starts a group
#pragma unroll
    for (int j = 0; j < HI; ++j) {
      if (j >= per) break;
      const uint32_t k = seg + j * 32;
      const bool h = k < n && (k == 0 || buf[k] != buf[k - 1]);
      if (h) hb |= 1u << j;
      const uint32_t b = __ballot_sync(0xffffffffu, h);
      if (b) wmax = (uint32_t)(warp * per + j) * 32 + (31 - __clz(b)) + 1;
      wsum += __popc(b);
      if (h && a.set) set_insert(a.set, a.set_mask, buf[k], a.words + kSwSigma);
    }
    uint32_t tot;
    uint32_t rmax = scan.run(wmax, OpMax(), &tot);
    uint32_t rsum = scan.run(wsum, OpSum(), &tot);
    if (!a.off && tid == 0) a.words[kSwSigma] = tot - (n && buf[n - 1] == kSetEmpty ? 1u : 0u);
    uint16_t id_[HI], hd_[HI], cd_[HI];
#pragma unroll
    for (int j = 0; j < HI; ++j) {
      if (j >= per) break;
      const uint32_t k = seg + j * 32;
      const uint32_t b = __ballot_sync(0xffffffffu, (hb >> j) & 1u);
      const uint32_t le = b & (lt | (1u << lane));
      const uint32_t row = (uint32_t)(warp * per + j) * 32;
      hd_[j] = (uint16_t)((le ? row + (31 - __clz(le)) + 1 : rmax) - 1);
      cd_[j] = (uint16_t)(rsum + __popc(le));
      id_[j] = k < n ? rank[k] : 0;
      if (b) rmax = row + (31 - __clz(b)) + 1;
      rsum += __popc(b);
    }
    __syncthreads();  // rank[] held the sorted suffixes
#pragma unroll
    for (int j = 0; j < HI; ++j) {
      if (j >= per) break;
      const uint32_t k = seg + j * 32;
      if (k < n) {
        sa[k] = id_[j];
        rank[id_[j]] = hd_[j];
        code[id_[j]] = cd_[j];
        if (k + 1 == n || buf[k + 1] != buf[k]) cnt[hd_[j]] = k + 1 - hd_[j];  // a group's size
      }
    }
    if (tid < 64) code[n + tid] = 0;
    __syncthreads();

    // The active slots (in groups of two or more) of the list `act`, or of
    // all slots: kept in order, their number in na, sum of group sizes in s_sum.
    uint32_t na = n;
    auto keep_active = [&](bool all) {
      const int rows = (int)((na + TPB - 1) / TPB);
      const uint32_t sg = (uint32_t)warp * rows * 32 + lane;
      uint32_t fb = 0, ws = 0, sq = 0;
      uint16_t kk[HI];
#pragma unroll
      for (int j = 0; j < HI; ++j) {
        if (j >= rows) break;
        const uint32_t x = sg + j * 32;
        uint32_t k = 0, g = 0;
        if (x < na) {
          k = all ? x : act[x];
          g = cnt[rank[sa[k]]];
        }
        kk[j] = (uint16_t)k;
        if (g > 1) {
          fb |= 1u << j;
          sq += g;
        }
        ws += __popc(__ballot_sync(0xffffffffu, g > 1));
      }
      sq = __reduce_add_sync(0xffffffffu, sq);
      if (lane == 0 && sq) atomicAdd(&s_sum, sq);
      uint32_t total;
      uint32_t at = scan.run(ws, OpSum(), &total);  // (its barrier: every act[] entry is read)
#pragma unroll
      for (int j = 0; j < HI; ++j) {
        if (j >= rows) break;
        const uint32_t b = __ballot_sync(0xffffffffu, (fb >> j) & 1u);
        if ((fb >> j) & 1u) act[at + __popc(b & lt)] = kk[j];
        at += __popc(b);
      }
      na = total;
      __syncthreads();
    };
    if (tid == 0) s_sum = 0;
    for (uint32_t i = tid; i < n; i += TPB) snap[i] = rank[i];
    __syncthreads();
    keep_active(true);

    // ---- doubling rounds
    int level = 0;
    for (uint32_t h = 1; na && level + 1 < a.levels; h *= 2) {
      const bool direct = s_sum <= kDirectCost * n;
      ++level;
      if (direct) {
        // the minor keys in slot order, as halves (see kHalfBase)
        uint16_t id[HI];
        uint32_t nh[HI] = {};
#pragma unroll
        for (int j = 0; j < HI; ++j) {
          const uint32_t x = tid + j * TPB;
          if (x >= na) break;
          const uint32_t k = act[x], i = sa[k];
          id[j] = (uint16_t)i;
          mk[k] = (uint16_t)((i + h < n ? rank[i + h] + 1u : 0u) + kHalfBase);
        }
        __syncthreads();
        if (tid == 0) s_sum = 0;
#pragma unroll
        for (int j = 0; j < HI; ++j) {
          if (tid + j * TPB >= na) break;
          const uint32_t i = id[j], hd = rank[i];
          nh[j] = hd + count_less(mk, hd, hd + cnt[hd], (i + h < n ? rank[i + h] + 1u : 0u) + kHalfBase);
        }
        __syncthreads();  // ranks, sizes and keys of the round before are read
#pragma unroll
        for (int j = 0; j < HI; ++j) {
          const uint32_t x = tid + j * TPB;
          if (x >= na) break;
          cnt[act[x]] = 0;
          rank[id[j]] = (uint16_t)nh[j];
        }
        __syncthreads();
        // a subgroup's members take its slots in any order (later rounds sort them)
#pragma unroll
        for (int j = 0; j < HI; ++j) {
          if (warp * 32 + j * TPB >= na) break;  // (the whole warp)
          const bool ok = tid + j * TPB < na;
          const uint32_t peers = __match_any_sync(0xffffffffu, ok ? nh[j] : ~0u);
          uint32_t q = 0;
          if (ok && (peers & lt) == 0) q = atomicAdd(&cnt[nh[j]], (uint32_t)__popc(peers));
          q = __shfl_sync(0xffffffffu, q, __ffs(peers) - 1) + __popc(peers & lt);
          if (ok) sa[nh[j] + q] = id[j];
        }
      } else {
        // (group's first slot, minor key, suffix), sorted over all slots
#pragma unroll
        for (int j = 0; j < HI; ++j) {
          const uint32_t k = tid + j * TPB;
          if (k < n) {
            const uint32_t i = sa[k];
            const uint64_t mi = i + h < n ? rank[i + h] + 1u : 0u;
            buf[k] = ((uint64_t)rank[i] << 27) | (mi << 13) | i;  // minor keys take 14 bits
          }
        }
        __syncthreads();
        if (tid == 0) s_sum = 0;  // (every thread has read it above)
        block_sort<TPB, HI, false>(buf, nullptr, n, 13, 27 + nb, ~0ull, wc, scan);
        uint32_t sb = 0, wm = 0;
#pragma unroll
        for (int j = 0; j < HI; ++j) {
          if (j >= per) break;
          const uint32_t k = seg + j * 32;
          const bool st = k < n && (k == 0 || (buf[k] >> 13) != (buf[k - 1] >> 13));
          if (st) sb |= 1u << j;
          const uint32_t b = __ballot_sync(0xffffffffu, st);
          if (b) wm = (uint32_t)(warp * per + j) * 32 + (31 - __clz(b)) + 1;
        }
        uint32_t t3;
        uint32_t rm = scan.run(wm, OpMax(), &t3);
#pragma unroll
        for (int j = 0; j < HI; ++j) {
          if (j >= per) break;
          const uint32_t k = seg + j * 32, row = (uint32_t)(warp * per + j) * 32;
          const uint32_t b = __ballot_sync(0xffffffffu, (sb >> j) & 1u);
          const uint32_t le = b & (lt | (1u << lane));
          const uint32_t hd = (le ? row + (31 - __clz(le)) + 1 : rm) - 1;
          if (b) rm = row + (31 - __clz(b)) + 1;
          if (k < n) {
            const uint32_t i = (uint32_t)buf[k] & 8191u;
            sa[k] = (uint16_t)i;
            rank[i] = (uint16_t)hd;
            if (k + 1 == n || (buf[k + 1] >> 13) != (buf[k] >> 13)) cnt[hd] = k + 1 - hd;
          }
        }
      }
      __syncthreads();
      for (uint32_t i = tid; i < n; i += TPB) snap[(size_t)level * n + i] = rank[i];
      keep_active(false);
    }
    if (na && tid == 0) atomicExch(a.err, kDevRange);  // levels bound the rounds: cannot happen
    if (a.sa)
      for (uint32_t k = tid; k < n; k += TPB) a.sa[o0 + k] = sa[k];

    // ---- LCP[rank[i] - 1] = lcp(i, the suffix before it), a few positions per thread
    // (the sorts are done: buf holds the first eight levels' ranks)
    uint16_t *lev_s = reinterpret_cast<uint16_t *>(buf);
    {
      const uint32_t total = n * (uint32_t)min(level + 1, kSharedLevels);
      for (uint32_t x = tid; x < (total + 7) / 8; x += TPB)
        reinterpret_cast<uint4 *>(lev_s)[x] = reinterpret_cast<const uint4 *>(snap)[x];
    }
    __syncthreads();
    {
      const uint32_t i0 = (uint32_t)tid * per, i1 = min(n, i0 + per);
      uint32_t l = 0;
      for (uint32_t i = i0; i < i1; ++i) {
        const uint32_t r = rank[i];
        if (r == 0) {
          l = 0;
          continue;
        }
        const uint32_t j = sa[r - 1];
        const uint32_t lim = n - max(i, j);
        uint32_t steps = 0;
        bool go = true;
        while (go && steps < kDirect) {  // codes are 0 past the end, and i != j: a mismatch stops there
          const uint32_t a0 = code[i + l], a1 = code[i + l + 1], a2 = code[i + l + 2], a3 = code[i + l + 3];
          const uint32_t b0 = code[j + l], b1 = code[j + l + 1], b2 = code[j + l + 2], b3 = code[j + l + 3];
          uint32_t c = a0 != b0 ? 0u : a1 != b1 ? 1u : a2 != b2 ? 2u : a3 != b3 ? 3u : 4u;
          if (l + c >= lim) {
            c = lim - l;
            go = false;
          } else if (c < 4) {
            go = false;
          }
          l += c;
          steps += 4;
        }
        if (go) {
          // level L ranks are equal iff the next 2^L tokens are
          for (int lev = level; lev >= 0; --lev) {
            const uint32_t x = i + l, y = j + l;
            if (x >= n || y >= n) continue;
            const uint16_t *lv = lev < kSharedLevels ? lev_s + (size_t)lev * n : snap + (size_t)lev * n;
            if (lv[x] == lv[y]) l += 1u << lev;
          }
        }
        lcp[r - 1] = (uint16_t)l;
        maxl = max(maxl, l);
        l = l ? l - 1 : 0;
      }
      if (tid == 0) lcp[n - 1] = 0;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) maxl = max(maxl, __shfl_xor_sync(0xffffffffu, maxl, o));
    if (lane == 0) scr[warp] = maxl;
    __syncthreads();
    maxl = 0;
#pragma unroll
    for (int x = 0; x < NW; ++x) maxl = max(maxl, scr[x]);
    if (a.lcp)
      for (uint32_t k = tid; k < n; k += TPB) a.lcp[o0 + k] = lcp[k];

    // ---- minima of 32 entries of LCP
    for (uint32_t b = warp; b * 32 < n; b += NW) {
      const uint32_t x = b * 32 + lane;
      const uint32_t v = __reduce_min_sync(0xffffffffu, x < n ? (uint32_t)lcp[x] : 0xffffu);
      if (lane == 0) t1[b] = (uint16_t)v;
    }
    __syncthreads();

    // ---- candidates: ((maxl - l) << 2 nb) | (id << nb) | start
    if (maxl >= a.min_len) {
      for (uint32_t base = warp * 32; base < n - 1; base += TPB) {
        const uint32_t k = base + lane;
        bool ok = false, ok_b = false;
        uint32_t l = 0, x = 0, y = 0;
        if (k < n - 1) {
          pair_cand_small(sa[k], sa[k + 1], lcp[k], &l, &x, &y);
          ok = ok_b = l >= a.min_len && l > 0;
          if (ok && k + 1 < n - 1) {  // often the next pair's first candidate
            uint32_t l2, x2, y2;
            pair_cand_small(sa[k + 1], sa[k + 2], lcp[k + 1], &l2, &x2, &y2);
            if (l2 == l && x2 == y) ok_b = false;
          }
        }
        const int pl = prev_less_warp(lcp, t1, base, k < n ? lcp[k] : 0u, l, ok);
        const uint32_t ba = __ballot_sync(0xffffffffu, ok), bb = __ballot_sync(0xffffffffu, ok_b);
        if (ba == 0) continue;
        uint32_t s0 = 0;
        if (lane == 0) s0 = atomicAdd(&s_cnt, (uint32_t)(__popc(ba) + __popc(bb)));
        s0 = __shfl_sync(0xffffffffu, s0, 0);
        if (ok) {
          const uint32_t q = s0 + __popc(ba & lt) + __popc(bb & lt);
          const uint64_t id = (uint64_t)(pl + 1);
          const uint64_t hi = ((uint64_t)(maxl - l) << (2 * nb)) | (id << nb);
          buf[q] = hi | x;  // at most two per pair: q + 1 < 2 NMAX
          if (ok_b) buf[q + 1] = hi | y;
        }
      }
      __syncthreads();
      const uint32_t mraw = s_cnt;
      block_sort<TPB, ITEMS, false>(buf, nullptr, mraw, 0, 2 * nb + sm_bits(maxl), ~0ull, wc, scan);
      // ---- equal candidates kept once
      {
        const int rows = (int)((mraw + TPB - 1) / TPB);
        const uint32_t sg = (uint32_t)warp * rows * 32 + lane;
        uint64_t kk[ITEMS];
        uint32_t fb = 0, wsum2 = 0;
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
          if (j >= rows) break;
          const uint32_t p = sg + j * 32;
          kk[j] = p < mraw ? buf[p] : 0;
          const bool f = p < mraw && (p == 0 || buf[p - 1] != kk[j]);
          if (f) fb |= 1u << j;
          wsum2 += __popc(__ballot_sync(0xffffffffu, f));
        }
        uint32_t at = scan.run(wsum2, OpSum(), &m);  // (its barrier: every key is read)
#pragma unroll
        for (int j = 0; j < ITEMS; ++j) {
          if (j >= rows) break;
          const uint32_t b = __ballot_sync(0xffffffffu, (fb >> j) & 1u);
          if ((fb >> j) & 1u) buf[at + __popc(b & lt)] = kk[j];
          at += __popc(b);
        }
      }
    }
  }

  if (m) {
    // ---- greedy: rounds of growing size; survivors (ends unmarked) settled
    // 32 at a time by warp 0, as in k_greedy
    const uint64_t smask = (1ull << nb) - 1;
    // the lists lie over the codes, suffixes and ranks, which are used up (not
    // over lcp, which the accepted starts take over below)
    static_assert(3 * TPB * sizeof(uint32_t) <= (NMAX + 64 + 2 * NMAX) * sizeof(uint16_t), "the greedy's lists end before lcp");
    uint32_t *list = reinterpret_cast<uint32_t *>(code);  // [TPB] survivors: (start << 16) | end
    uint32_t *lk = list + TPB;                             // [TPB] their candidates
    uint32_t *lov = lk + TPB;                              // [TPB] overlap masks
    __syncthreads();
    for (uint32_t x = tid; x < n / 32 + 1; x += TPB) bits[x] = 0;
    for (uint32_t x = tid; x < 2 * NMAX / 32; x += TPB) accw[x] = 0;
    __syncthreads();
    uint32_t size = 32;
    for (uint32_t base = 0; base < m; base += size, size = min(size * 2, (uint32_t)TPB)) {
      const uint32_t k = base + tid;
      uint32_t st = 0, en = 0;
      bool sv = false;
      if ((uint32_t)tid < size && k < m) {
        const uint64_t key = buf[k];
        st = (uint32_t)(key & smask);
        en = st + maxl - (uint32_t)(key >> (2 * nb)) - 1;
        sv = !(((bits[st >> 5] >> (st & 31)) | (bits[en >> 5] >> (en & 31))) & 1u);
      }
      const uint32_t bal = __ballot_sync(0xffffffffu, sv);
      uint32_t total;
      const uint32_t q = scan.run((uint32_t)__popc(bal), OpSum(), &total) + __popc(bal & lt);
      if (total == 0) continue;
      if (sv) {
        list[q] = (st << 16) | en;
        lk[q] = k;
      }
      __syncthreads();
      if ((uint32_t)tid < total) {
        const uint32_t q0 = tid & ~31u, nbt = min(32u, total - q0);
        const uint32_t me = list[tid], ms = me >> 16, mend = me & 0xffffu;
        uint32_t ov = 0;
        for (uint32_t j = 0; j < nbt; ++j) {
          const uint32_t z = list[q0 + j];
          if (j < (uint32_t)lane && (z >> 16) <= mend && ms <= (z & 0xffffu)) ov |= 1u << j;
        }
        lov[tid] = ov;
      }
      __syncthreads();
      if (warp == 0) {
        uint32_t pe = (uint32_t)lane < total ? list[lane] : 0u, po = (uint32_t)lane < total ? lov[lane] : 0u,
                 pk = (uint32_t)lane < total ? lk[lane] : 0u;
        for (uint32_t q0 = 0; q0 < total; q0 += 32) {
          const uint32_t qs = pe >> 16, qe = pe & 0xffffu, ov = po, ck = pk;
          const uint32_t nq = q0 + 32 + lane;
          if (nq < total) {  // the next batch's survivors, read ahead
            pe = list[nq];
            po = lov[nq];
            pk = lk[nq];
          }
          const bool free = q0 + lane < total &&
                            !(((bits[qs >> 5] >> (qs & 31)) | (bits[qe >> 5] >> (qe & 31))) & 1u);
          uint32_t und = __ballot_sync(0xffffffffu, free), accm = 0;
          while (und) {
            const uint32_t take = __ballot_sync(0xffffffffu, ((und >> lane) & 1u) && (ov & (und | accm)) == 0);
            accm |= take;
            und &= ~take;
            und &= ~__ballot_sync(0xffffffffu, ((und >> lane) & 1u) && (ov & accm) != 0);
          }
          bool lng = false;
          if ((accm >> lane) & 1u) {
            atomicOr(&accw[ck >> 5], 1u << (ck & 31));
            const uint32_t w0 = qs >> 5, w1 = qe >> 5;
            if (w1 - w0 < 4) {
              for (uint32_t x = w0; x <= w1; ++x) {
                uint32_t msk = 0xffffffffu;
                if (x == w0) msk &= 0xffffffffu << (qs & 31);
                if (x == w1) msk &= 0xffffffffu >> (31 - (qe & 31));
                atomicOr(&bits[x], msk);
              }
            } else {
              lng = true;
            }
          }
          for (uint32_t am = __ballot_sync(0xffffffffu, lng); am; am &= am - 1) {
            const int j = __ffs(am) - 1;
            const uint32_t js = __shfl_sync(0xffffffffu, qs, j), je = __shfl_sync(0xffffffffu, qe, j);
            for (uint32_t x = (js >> 5) + lane; x <= (je >> 5); x += 32) {
              uint32_t msk = 0xffffffffu;
              if (x == (js >> 5)) msk &= 0xffffffffu << (js & 31);
              if (x == (je >> 5)) msk &= 0xffffffffu >> (31 - (je & 31));
              atomicOr(&bits[x], msk);
            }
          }
          K += __popc(accm);
          __syncwarp();
        }
      }
      __syncthreads();
    }
    // ---- accepted candidates in order; a new trace where (length, id) changes
    uint16_t *al = sa, *tr = rank, *at_pos = lcp;  // (the suffix array is out)
    for (uint32_t x = tid; x < n; x += TPB) at_pos[x] = 0;
    uint32_t done = 0;
    for (uint32_t base = 0; base < m; base += TPB) {
      const uint32_t k = base + tid;
      const uint32_t b = base + warp * 32 < m ? accw[base / 32 + warp] : 0u;
      const bool f = (b >> lane) & 1u;
      uint32_t total;
      const uint32_t q1 = done + scan.run((uint32_t)__popc(b), OpSum(), &total) + __popc(b & lt);
      if (f) al[q1] = (uint16_t)k;  // accepted intervals are disjoint: at most n
      done += total;
    }
    K = done;
    __syncthreads();
    for (uint32_t base = 0; base < K; base += TPB) {
      const uint32_t q = base + tid;
      bool f = false;
      if (q < K) {
        const uint64_t key = buf[al[q]];
        f = q == 0 || (key >> nb) != (buf[al[q - 1]] >> nb);
        at_pos[(uint32_t)(key & smask)] = (uint16_t)(q + 1);
      }
      const uint32_t b = __ballot_sync(0xffffffffu, f);
      uint32_t total;
      const uint32_t p = scan.run((uint32_t)__popc(b), OpSum(), &total);
      const uint32_t t = Tn + p + __popc(b & (lt | (1u << lane))) - 1;
      if (q < K) tr[q] = (uint16_t)(t | (f ? 0x8000u : 0u));  // t < 8192
      Tn += total;
    }
    __syncthreads();
  }

  // ---- where this window's outputs start
  if (tid == 0) {
    s_tot[0] = m;
    s_tot[1] = K;
    s_tot[2] = Tn;
    if (maxl) atomicMax(&a.words[kSwMaxLcp], maxl);
  }
  __syncthreads();
  if (warp < 3) {
    const uint32_t v = s_tot[warp];
    uint32_t base = 0;
    if (a.off) {
      uint64_t *st = a.status + (size_t)warp * a.W;
      if (lane == 0) lb_store(&st[w], lb_pack(w == 0 ? kLbInclusive : kLbAggregate, a.epoch, v));
      if (w > 0) {
        base = lb_exclusive_warp(st, 1, w, a.epoch, OpSum(), 0u, a.err);
        if (lane == 0) lb_store(&st[w], lb_pack(kLbInclusive, a.epoch, base + v));
      }
      if (lane == 0) {
        a.offs[(size_t)warp * (a.W + 1) + w] = base;
        if (w + 1 == a.W) a.offs[(size_t)warp * (a.W + 1) + a.W] = base + v;
      }
    }
    if (lane == 0) {
      s_base[warp] = base;
      if (!a.off || w + 1 == a.W) a.words[kSwCand + warp] = base + v;
    }
  }
  __syncthreads();
  if (m) {
    const uint64_t smask = (1ull << nb) - 1;
    const uint64_t b0 = s_base[0], b1 = s_base[1], b2 = s_base[2];
    if (a.cl || a.cid || a.cs || a.acc)
      for (uint32_t k = tid; k < m; k += TPB) {
        if (b0 + k >= a.cand_cap) break;
        const uint64_t key = buf[k];
        if (a.cl) a.cl[b0 + k] = maxl - (uint32_t)(key >> (2 * nb));
        if (a.cid) a.cid[b0 + k] = (uint32_t)((key >> nb) & smask) + o0;
        if (a.cs) a.cs[b0 + k] = (uint32_t)(key & smask);
        if (a.acc) a.acc[b0 + k] = (accw[k >> 5] >> (k & 31)) & 1u;
      }
    const uint16_t *al = sa, *tr = rank, *at_pos = lcp;
    for (uint32_t q = tid; q < K; q += TPB) {
      const uint32_t t = tr[q];
      if ((t & 0x8000u) && b2 + (t & 0x7fffu) < a.trace_cap) {
        const uint64_t key = buf[al[q]];
        if (a.tl) a.tl[b2 + (t & 0x7fffu)] = maxl - (uint32_t)(key >> (2 * nb));
        if (a.ts) a.ts[b2 + (t & 0x7fffu)] = (uint32_t)(key & smask);
      }
    }
    // selected intervals by start
    uint32_t done = 0;
    for (uint32_t base = 0; base < n; base += TPB) {
      const uint32_t x = base + tid;
      const uint32_t q = x < n ? at_pos[x] : 0u;
      const uint32_t b = __ballot_sync(0xffffffffu, q != 0);
      uint32_t total;
      const uint64_t at = b1 + done + scan.run((uint32_t)__popc(b), OpSum(), &total) + __popc(b & lt);
      if (q && at < a.sel_cap) {
        if (a.ss) a.ss[at] = x;
        if (a.sl) a.sl[at] = maxl - (uint32_t)(buf[al[q - 1]] >> (2 * nb));
        if (a.st) a.st[at] = tr[q - 1] & 0x7fffu;
      }
      done += total;
    }
  }
}

struct SmallKernel {
  void (*fn[2])(const SmallArgs);  // u32, u64 tokens
  int threads;
  uint32_t max_n;
  size_t smem;
};
template <int TPB, int ITEMS>
SmallKernel small_kernel() {
  return SmallKernel{{k_small<uint32_t, TPB, ITEMS>, k_small<uint64_t, TPB, ITEMS>},
                     TPB,
                     (uint32_t)SmallShape<TPB, ITEMS>::kMaxN,
                     SmallShape<TPB, ITEMS>::kSmem};
}
// A call takes the first shape that holds its longest window.
const SmallKernel kSmall[] = {small_kernel<256, 4>(), small_kernel<1024, 4>(), small_kernel<1024, 8>(),
                              small_kernel<1024, 16>()};
constexpr int kSmallShapes = sizeof(kSmall) / sizeof(kSmall[0]);

// Host reads of the call: device words into host[], answered from the tape
// while the call is captured.
int read_words(apo_ctx *c, const uint32_t *dev, uint32_t *host, int words, cudaStream_t s) {
  if (capturing(c)) {
    uint32_t e = 0;
    APO_TRY(tape_take(c, dev, host, words, s));
    return tape_take(c, c->ps.err, &e, 1, s);
  }
  APO_CUDA_TRY(cudaMemcpyAsync(c->host_pinned, dev, (size_t)words * 4, cudaMemcpyDeviceToHost, s));
  APO_CUDA_TRY(cudaMemcpyAsync(c->host_pinned + kPinnedErr, c->ps.err, 4, cudaMemcpyDeviceToHost, s));
  APO_CUDA_TRY(cudaStreamSynchronize(s));
  memcpy(host, c->host_pinned, (size_t)words * 4);
  if (recording(c)) {
    tape_put(c, host, words);
    tape_put(c, c->host_pinned + kPinnedErr, 1);
  }
  return device_error_status(c, s);
}

}  // namespace

// Whether a call's windows go through k_small: each at most 8,192 tokens (what fits a
// block's shared memory), and not so many that the general path, which shares its
// launches among any number of windows, is the faster one.  Both sides' times are
// modelled from measurements (152 SMs), on the contents that favour the general path
// most -- four tokens at random, whose groups are gone after a few rounds -- so that
// hardly a call is slower here than there: a block of 1,024 threads holds an SM for
// about 24 us + 25 ns per token of the longest window, one of 256 threads (windows of
// up to 512 tokens; eight are resident) for 10.3 us + 18.5 ns, u32 tokens 15% less;
// the general path takes about 750 us + 0.24 ns per token, a little more per token of
// longer windows.  Windows below 64 tokens, with fewer rounds, cost both sides less:
// 8.5 us + 47 ns per token here, 410 us (u64 tokens 470) + 4.7 us per token there.
// Measured (here / general path, us), u64 tokens, loops with noise and four tokens at
// random: 10,000 x 64 933 / 1,010 and 834 / 887; 5,000 x 513 1,607 / 1,929 and 1,340 /
// 1,381; 5,000 x 600 1,671 / 2,051 and 1,395 / 1,486; 10,000 x 1,000 3,862 / 4,751 and
// 3,237 / 3,305; 3,000 x 8,192 5,486 / 10,639 and 4,538 / 9,156; past the line: 12,000
// x 8 678 / 554 and 758 / 522; 20,000 x 128 2,038 / 1,794 and 1,709 / 1,360; 50,000 x
// 250 5,706 / 5,537 and 4,553 / 3,634; 10,000 x 600 3,196 / 3,232 and 2,669 / 2,226;
// 50,000 x 513 14,510 / 10,626 and 11,994 / 6,883.
// Of 516 batches measured on both sides the line takes the slower one (by 3% or more)
// for 41: 7 run here, at most 1.08 times slower; given up are loops at up to 1.13 times
// (20,000 x 1,000 u64) and random u64 tokens at up to 1.7.
bool small_windows(int sms, uint64_t total, uint64_t windows, uint64_t longest, int token_bytes) {
  if (longest > kSmall[kSmallShapes - 1].max_n) return false;
  const double len = (double)longest;
  const double block = longest > kSmall[0].max_n ? 24.0 + 0.0252 * len
                       : longest >= 64           ? 10.3 + 0.0185 * len
                                                 : 8.5 + 0.047 * len;
  const double general = longest >= 64 ? 750.0 : (token_bytes == 4 ? 410.0 : 470.0) + 4.7 * len;
  return (double)windows * block * (token_bytes == 4 ? 0.85 : 1.0) / sms <
         general + (0.00024 + 1.3e-8 * len) * (double)total;
}

int small_init() {
  for (const auto &k : kSmall)
    for (auto f : k.fn)
      APO_CUDA_TRY(cudaFuncSetAttribute((const void *)f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)k.smem));
  return APO_OK;
}

int small_find_repeats(apo_ctx *c, const void *tokens, int tb, const uint64_t *win_off, uint32_t W,
                       uint32_t longest, const apo_repeats_params *p, apo_repeats_out *out, cudaStream_t s) {
  const uint32_t total = (uint32_t)win_off[W];
  int shape = 0;
  while (kSmall[shape].max_n < longest) ++shape;
  const SmallKernel &k = kSmall[shape];
  uint32_t *words = c->ps.counters + kCtrMisc + kMiscSmall;
  SmallArgs a{};
  a.tokens = tokens;
  a.W = W;
  a.n = total;
  a.min_len = p->min_len;
  a.levels = bits_for(longest) + 2;
  a.snaps = c->arena.take_n<uint16_t>((size_t)total * a.levels + 8 * (size_t)W + 16);
  bool ok = a.snaps != nullptr;
  uint32_t *off = nullptr;
  // the distinct tokens of all windows are counted for the rounds reported
  // (see below): on the way for 64-bit tokens, which are mostly hashes
  const uint64_t cap = [&] {
    uint64_t x = 1;
    while (x < 2ull * total && x < (1ull << 23)) x <<= 1;
    return x;
  }();
  uint64_t *set = nullptr;
  if (W > 1) {
    off = c->arena.take_n<uint32_t>(W + 1);
    a.offs = c->arena.take_n<uint32_t>(3 * (size_t)(W + 1));
    a.status = c->arena.take_n<uint64_t>(3 * (size_t)W);
    set = total >= 4096 ? c->arena.take_n<uint64_t>(cap) : nullptr;
    ok = ok && off && a.offs && a.status && (set || total < 4096);
  }
  if (!ok) {
    set_error("find_repeats: workspace too small");
    return APO_ENOMEM;
  }
  if (W > 1) {
    std::vector<uint32_t> pageable;
    uint32_t *h;
    if (capturing(c)) {
      h = c->tape->upload;  // a graph copies from a pinned buffer that outlives this call
    } else if (3 * (size_t)(W + 1) <= kPinnedOffs) {
      h = c->host_pinned + kPinnedWords;  // (the call ends synchronised: free again)
    } else {
      pageable.resize(W + 1);
      h = pageable.data();
    }
    for (uint32_t w = 0; w <= W; ++w) h[w] = (uint32_t)win_off[w];
    APO_CUDA_TRY(cudaMemcpyAsync(off, h, (size_t)(W + 1) * 4, cudaMemcpyHostToDevice, s));
    if (!pageable.empty()) APO_CUDA_TRY(cudaStreamSynchronize(s));
    APO_CUDA_TRY(cudaMemsetAsync(a.status, 0, 3 * (size_t)W * 8, s));
    a.off = off;
    if (set && tb == 8) {
      APO_CUDA_TRY(cudaMemsetAsync(set, 0xff, cap * 8, s));
      a.set = set;
      a.set_mask = cap - 1;
    }
  }
  APO_CUDA_TRY(cudaMemsetAsync(words, 0, kSwWords * 4, s));
  a.sa = out->sa;
  a.lcp = out->lcp;
  a.cl = out->cand_len;
  a.cid = out->cand_id;
  a.cs = out->cand_start;
  a.acc = out->cand_accepted;
  a.cand_cap = out->cand_cap;
  a.ss = out->sel_start;
  a.sl = out->sel_len;
  a.st = out->sel_trace;
  a.sel_cap = out->sel_cap;
  a.tl = out->trace_len;
  a.ts = out->trace_start;
  a.trace_cap = out->trace_cap;
  a.words = words;
  a.epoch = next_epoch(c);
  a.err = c->ps.err;
  {
    Launch lp_(c, kKSmall, total, s);
    k.fn[tb == 8]<<<W, k.threads, k.smem, s>>>(a);
  }
  APO_CUDA_TRY(cudaGetLastError());
  const bool want_off = W > 1 && (out->cand_off || out->sel_off || out->trace_off);
  const size_t owords = 3 * (size_t)(W + 1);
  std::vector<uint32_t> oh;
  const uint32_t *offs_host = nullptr;
  if (W > 1 && capturing(c)) {
    // a replay copies the offsets to the tape's pinned stage
    APO_CUDA_TRY(cudaMemcpyAsync(c->tape->stage, a.offs, owords * 4, cudaMemcpyDeviceToHost, s));
  } else if (want_off) {
    uint32_t *h = c->host_pinned + kPinnedWords;
    if (owords > kPinnedOffs) {
      oh.resize(owords);
      h = oh.data();
    }
    APO_CUDA_TRY(cudaMemcpyAsync(h, a.offs, owords * 4, cudaMemcpyDeviceToHost, s));
    offs_host = h;
  }
  uint32_t got[kSwWords - 1];  // from kSwCand on
  APO_TRY(read_words(c, words + kSwCand, got, kSwWords - 1, s));
  const uint64_t cnt[3] = {got[0], got[1], got[2]};
  const uint32_t maxlcp = got[kSwMaxLcp - kSwCand];
  uint32_t sigma = got[kSwSigma - kSwCand];
  uint64_t maxtok;
  memcpy(&maxtok, got + (kSwMaxTok - kSwCand), 8);
  // The doubling rounds that the general path counts: its first sort takes h0
  // tokens per key (dense codes when fewer than four plain ones fit), and
  // round r runs iff some LCP is at least h0 * 2^(r-1).
  const int wb = W > 1 ? bits_for(W - 1) : 0;
  const int cb = bits_for(maxtok) <= 32 ? bits_for(maxtok + 1) : 0;
  uint64_t h0 = cb ? (uint64_t)((64 - wb) / cb) : 0;
  if (h0 < 4 && total >= 4096) {
    if (W > 1 && tb == 4) {
      APO_CUDA_TRY(cudaMemsetAsync(set, 0xff, cap * 8, s));
      {
        Launch lp_(c, kKSaDict, total, s);
        k_small_set<<<grid_for(total, 256, c->num_sms), 256, 0, s>>>(static_cast<const uint32_t *>(tokens), total, set,
                                                                     cap - 1, words + kSwSigma);
      }
      APO_CUDA_TRY(cudaGetLastError());
      APO_TRY(read_words(c, words + kSwSigma, &sigma, 1, s));
    }
    if (sigma <= cap / 2) h0 = std::max<uint64_t>(h0, (uint64_t)((64 - wb) / bits_for((uint64_t)sigma + 1)));
  }
  h0 = h0 >= 2 ? std::min<uint64_t>(h0, 32) : 1;
  uint32_t rounds = 0;
  while (maxlcp >= (h0 << rounds)) ++rounds;
  for (int x = 0; x < 3; ++x) out->counts[x] = cnt[x];
  out->counts[3] = rounds;
  uint64_t *const dst[3] = {out->cand_off, out->sel_off, out->trace_off};
  for (int x = 0; x < 3; ++x) {
    if (!dst[x]) continue;
    if (W == 1) {
      dst[x][0] = 0;
      dst[x][1] = cnt[x];
    } else if (offs_host) {
      for (uint32_t w = 0; w <= W; ++w) dst[x][w] = offs_host[(size_t)x * (W + 1) + w];
    }
  }
  const bool cand = out->cand_len || out->cand_id || out->cand_start || out->cand_accepted;
  const bool sel = out->sel_start || out->sel_len || out->sel_trace, tr = out->trace_len || out->trace_start;
  if ((cand && cnt[0] > out->cand_cap) || (sel && cnt[1] > out->sel_cap) || (tr && cnt[2] > out->trace_cap)) {
    set_error("find_repeats: an output capacity is too small (counts written)");
    return APO_ECAPACITY;
  }
  return APO_OK;
}

}  // namespace apo
