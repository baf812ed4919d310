// The optimum of Sec. 3's trace-selection problem for many short windows --
// the yardstick that Alg. 2, a heuristic (Sec. 4.2), is measured against.
//
// Problem (Sec. 3): traces T, sub-strings of S of length >= min_len, each
// with a set of intervals of S that hold it, all intervals disjoint;
// maximise the coverage (summed interval lengths), then the number of
// intervals, then minimise |T|.  As stated, T = {S} covers everything, so
// each trace must match at least two intervals (the traces must repeat).
//
// One thread per window, exhaustive: a depth-first walk over the interval
// sets, positions left to right, each one either uncovered or the start of
// an interval of length min_len, min_len + 1, ...  Per string a counter of
// its intervals in the current set gives "every string at least twice"
// (no counter at 1) and |T| (counters above 0) at every leaf in O(1).
// Cuts that leave the first optimal set in the walk order unchanged:
//   * an interval whose string has no second, disjoint occurrence in the
//     window is never tried, nor one whose string is not in the set yet and
//     does not occur again after it (every set below holds it once);
//   * strings held once need a second interval each: a subtree with fewer
//     positions ahead than those strings are long is skipped;
//   * (coverage, intervals) so far plus the best (coverage, intervals) that
//     repeatable intervals reach from here on, which a recurrence over the
//     positions gives, bounds every set below (lexicographic order is kept by
//     adding to both sides); a subtree whose bound does not beat the best set
//     found before it in the walk, |T| included, is skipped.
// The bound needs a good set early, and the walk order (uncovered first)
// meets poor sets first.  So a first walk in the opposite order (intervals
// before uncovered) finds the optimal value alone, and the second walk, in
// the order that defines the witness, skips what cannot reach that value.
//
// What bounds it: the longest walk of a warp, a serial chain of local-memory
// accesses (65,536 windows of 20 tokens are one wave).  Nodes of the longest
// walk in a warp, on those windows at min_len 2: 98,000 with the coverage of
// the positions ahead as the only bound, 2,900 with the lexicographic bound,
// 1,800 with the value known as well (both walks counted).  Measured on them:
// 175-187 ms before, 5.8-6.4 ms with both walks and one warp per block.
#include <algorithm>
#include <vector>

#include "../../include/apo.h"
#include "apo_internal.cuh"

namespace apo {

namespace {

constexpr int kOptMax = 24;                // longest window
constexpr int kIdStride = kOptMax + 1;     // string id = first start * kIdStride + length
constexpr uint64_t kOptLeaves = 1ull << 24;  // largest admissible enumeration
constexpr uint32_t kOptGuard = 1u << 30;     // node visits after which a walk gives up

template <class T>
__global__ void __launch_bounds__(32)
    k_optimum(const T *__restrict__ tok, const uint32_t *__restrict__ off, uint32_t W, uint32_t m,
              uint32_t *__restrict__ best, uint32_t *__restrict__ wstart, uint32_t *__restrict__ wlen,
              uint32_t *__restrict__ wcount, uint32_t *err) {
  for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w < W; w += gridDim.x * blockDim.x) {
    const uint32_t a0 = off[w];
    const int n = (int)(off[w + 1] - a0);
    T s[kOptMax];
    for (int i = 0; i < n; ++i) s[i] = tok[a0 + i];
    // sid[a][L] = the first start of the length-L string at a
    uint8_t sid[kOptMax][kOptMax + 1];
    for (int a = 0; a < n; ++a) {
      for (int L = 1; L <= n - a; ++L) sid[a][L] = (uint8_t)a;
      for (int b = a - 1; b >= 0; --b) {
        int l = 0;
        while (a + l < n && s[b + l] == s[a + l]) ++l;
        for (int L = 1; L <= l; ++L) sid[a][L] = (uint8_t)b;
      }
    }
    // rep[a] bit L: the length-L string at a occurs again, disjoint from it;
    // later[a] bit L: it does so after position a + L - 1
    uint32_t rep[kOptMax], later[kOptMax];
    for (int a = 0; a < n; ++a) rep[a] = later[a] = 0;
    for (int a = 0; a < n; ++a)
      for (int b = a + 1; b < n; ++b) {
        int l = 0;
        while (b + l < n && s[a + l] == s[b + l]) ++l;
        const int lim = min(l, b - a);  // disjoint: L <= b - a
        const uint32_t lens = (2u << lim) - 2u;
        rep[a] |= lens;
        later[a] |= lens;
        rep[b] |= lens;
      }
    // best (coverage, intervals) of disjoint repeatable intervals at p or
    // after, coverage in the high byte
    const int m1 = m < 1 ? 1 : (int)m;
    uint16_t ahead[kOptMax + 1];
    ahead[n] = 0;
    for (int p = n - 1; p >= 0; --p) {
      int x = ahead[p + 1];
      for (int L = m1; p + L <= n; ++L)
        if (rep[p] >> L & 1u) x = max(x, (int)ahead[p + L] + L * 256 + 1);
      ahead[p] = (uint16_t)x;
    }
    uint8_t cnt[kOptMax * kIdStride];
    for (int i = 0; i < kOptMax * kIdStride; ++i) cnt[i] = 0;
    uint8_t pos[kOptMax + 1], ch[kOptMax + 1];  // ch: 0xff unvisited, 0 uncovered, else interval length
    uint8_t bs[kOptMax], bl[kOptMax];
    // a set's value: coverage * 256 + intervals, then |T|
    int bk = 0, bval = -1, bdist = 1 << 30;
    int vval = -1, vdist = 1 << 30;  // the value the first walk found
    uint32_t guard = 0;
    for (int walk = 0; walk < 2; ++walk) {
      int val = 0, singles = 0, sumlen = 0, distinct = 0;  // sumlen: lengths of the strings held once
      bval = -1;
      bdist = 1 << 30;
      int d = 0;
      pos[0] = 0;
      ch[0] = 0xff;
      while (d >= 0) {
        if (++guard > kOptGuard) {
          atomicExch(err, kDevTimeout);
          break;
        }
        const int p = pos[d];
        int L = ch[d];
        int nx;  // the next choice at p: 0 uncovered, else a length to try from
        if (L == 0xff) {
          if (p == n) {  // a complete interval set
            if (singles == 0 && (val > bval || (val == bval && distinct < bdist))) {
              bval = val;
              bdist = distinct;
              bk = 0;
              for (int k = 0; walk && k < d; ++k)
                if (ch[k]) {
                  bs[bk] = pos[k];
                  bl[bk] = ch[k];
                  ++bk;
                }
            }
            --d;
            continue;
          }
          const int ub = val + ahead[p];
          if (sumlen > n - p || ub < bval || (ub == bval && distinct >= bdist) || ub < vval ||
              (ub == vval && distinct > vdist)) {
            --d;
            continue;
          }
          nx = walk ? 0 : m1;
        } else {
          // back from a child: take the interval of the last choice out
          if (L) {
            const int id = sid[p][L] * kIdStride + L;
            const int c = --cnt[id];
            if (c == 1) {
              ++singles;
              sumlen += L;
            } else if (c == 0) {
              --singles;
              sumlen -= L;
              --distinct;
            }
            val -= L * 256 + 1;
          }
          if (!walk && L == 0) {  // uncovered is the first walk's last choice
            --d;
            continue;
          }
          nx = L ? L + 1 : m1;
        }
        if (nx) {
          // only strings that can repeat: held already, or found again later
          while (p + nx <= n &&
                 !((rep[p] >> nx & 1u) && ((later[p] >> nx & 1u) || cnt[sid[p][nx] * kIdStride + nx])))
            ++nx;
          if (p + nx > n) {
            if (walk) {
              --d;
              continue;
            }
            nx = 0;
          }
        }
        ch[d] = (uint8_t)nx;
        if (nx) {
          const int id = sid[p][nx] * kIdStride + nx;
          const int c = ++cnt[id];
          if (c == 1) {
            ++singles;
            sumlen += nx;
            ++distinct;
          } else if (c == 2) {
            --singles;
            sumlen -= nx;
          }
          val += nx * 256 + 1;
        }
        pos[d + 1] = (uint8_t)(p + (nx ? nx : 1));
        ch[d + 1] = 0xff;
        ++d;
      }
      if (bval == 0) break;  // nothing repeats: the empty set (one window of 24 distinct tokens: 169 -> 152 us)
      vval = bval;
      vdist = bdist;
    }
    const int bcov = bval >> 8, bcnt = bval & 255;
    best[3 * w] = (uint32_t)bcov;
    best[3 * w + 1] = (uint32_t)bcnt;
    best[3 * w + 2] = (uint32_t)bdist;
    for (int k = 0; k < bk; ++k) {
      wstart[a0 + k] = bs[k];
      wlen[a0 + k] = bl[k];
    }
    wcount[w] = (uint32_t)bk;
  }
}

// Interval sets of a length-n window with pieces of at least m: f(n) =
// f(n - 1) + sum_{L >= m} f(n - L), f(0) = 1 (capped).
uint64_t interval_sets(int n, int m) {
  std::vector<uint64_t> f(n + 1, 0);
  f[0] = 1;
  for (int k = 1; k <= n; ++k) {
    uint64_t v = f[k - 1];
    for (int L = std::max(m, 1); L <= k; ++L) v = std::min<uint64_t>(v + f[k - L], 1ull << 62);
    f[k] = v;
  }
  return f[n];
}

}  // namespace

int optimum_batched(apo_ctx *c, const apo_windows *ws, uint32_t min_len, uint32_t *best, uint32_t *wstart,
                    uint32_t *wlen, uint32_t *wcount, cudaStream_t s) {
  const uint64_t W = ws->n_windows;
  min_len = std::min<uint32_t>(min_len, kOptMax + 1);  // longer than any window: no traces
  uint64_t maxn = 0;
  for (uint64_t w = 0; w < W; ++w) maxn = std::max(maxn, ws->win_off[w + 1] - ws->win_off[w]);
  if (maxn > (uint64_t)kOptMax) {
    set_error("apo_optimum_batched: windows of at most 24 tokens");
    return APO_EINVAL;
  }
  if (interval_sets((int)maxn, (int)min_len) > kOptLeaves) {
    set_error("apo_optimum_batched: the exhaustive search is too large (more than 2^24 interval sets "
              "for the longest window at this min_len)");
    return APO_EINVAL;
  }
  APO_TRY(ensure_side(c, (W + 1) * 4, s));
  uint32_t *off = static_cast<uint32_t *>(c->side);
  std::vector<uint32_t> h(W + 1);
  for (uint64_t w = 0; w <= W; ++w) h[w] = (uint32_t)ws->win_off[w];
  APO_CUDA_TRY(cudaMemcpyAsync(off, h.data(), (W + 1) * 4, cudaMemcpyHostToDevice, s));
  const int threads = 32;  // single warps spread evenly: walks differ in length by the window
  const int blocks = (int)std::max<uint64_t>(1, std::min<uint64_t>((W + threads - 1) / threads,
                                                                   (uint64_t)c->num_sms * 64));
  {
    Launch lp_(c, kKOptimum, W, s);
    if (ws->token_bytes == 4)
      k_optimum<<<blocks, threads, 0, s>>>(static_cast<const uint32_t *>(ws->tokens), off, (uint32_t)W, min_len,
                                           best, wstart, wlen, wcount, c->ps.err);
    else
      k_optimum<<<blocks, threads, 0, s>>>(static_cast<const uint64_t *>(ws->tokens), off, (uint32_t)W, min_len,
                                           best, wstart, wlen, wcount, c->ps.err);
  }
  APO_CUDA_TRY(cudaGetLastError());
  return check_device_error(c, s);  // synchronises: the host array h is released on return
}

}  // namespace apo
