// grams.cu -- gram index in front of the exact forward scan (sm_103a).
//
// Pigeonhole principle for edit distance: an alignment of a pattern with at
// most E edits (Eq. 1, Eq. 2; E = K under unit costs) leaves
//   one of E + 1 disjoint pieces of the pattern unedited; with the pieces taken
//   two by two, one of a pair that has at most one edit in all (or the odd
//   last one);
//   one of E / 2 + 1 disjoint pieces with at most one edit.
// The index holds grams: the pieces themselves, or (2-bit text) the strings
// one edit away from longer pieces.  A gram found at a text position allows
// the ends within E edits of its diagonal; the pattern symbols beside it are
// matched with the text beside it, and an end that all of them reach within E
// edits becomes a candidate: the forward scan's own candidates under unit
// costs, a superset of them under edit costs (a distance is at least the
// cheapest cost times the number of edits) or where 2-bit text holds other
// symbols; verification measures them.
//
//   scan   one text position per step of a lane: for each key length, a bit of
//          a table in shared memory; where it is set, the length's directory
//          (open addressing, in L2) and the grams with that key: suspects
//          (position, gram)
//   ends   one thread per suspect: the pattern beside the gram against the
//          text beside it; each (pattern, end) becomes a candidate once (an
//          open-addressing set: an occurrence holds several grams)
//   long   what passed of patterns longer than 32 symbols beside their gram
//
// The cost per text position depends on the number of key lengths and on how
// often grams appear, not on the number of patterns.
#include "end_set.cuh"
#include "kernels.h"

namespace oasm {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kQueue = 64;  // table hits, and suspects, buffered per warp

// ------------------------------------------------------------------- scan
// 2-bit symbols: (byte >> shift) & 3, 16 of them to a word.
__device__ __forceinline__ uint32_t pack2(uint32_t w, uint32_t shift) {
  // the four 2-bit fields meet in the top byte; the partial products are
  // disjoint, so nothing carries into it
  return (((w >> shift) & 0x03030303u) * 0x01041040u) >> 24;
}

// The text at symbol j of the lane's 16: 16 2-bit symbols, or eight bytes.
template <bool kTwoBit>
__device__ __forceinline__ void window(const uint32_t (&t)[6], int j, uint32_t& lo, uint32_t& hi) {
  if (kTwoBit) {
    lo = __funnelshift_r(t[0], t[1], 2 * j);
    hi = 0u;
    return;
  }
  const int q = j >> 2, r = 8 * (j & 3);  // (selects where j is known only here)
  const uint32_t a = q == 0 ? t[0] : q == 1 ? t[1] : q == 2 ? t[2] : t[3];
  const uint32_t b = q == 0 ? t[1] : q == 1 ? t[2] : q == 2 ? t[3] : t[4];
  const uint32_t c = q == 0 ? t[2] : q == 1 ? t[3] : q == 2 ? t[4] : t[5];
  lo = __funnelshift_r(a, b, r);
  hi = __funnelshift_r(b, c, r);
}

// One block per SM; its warps walk 512-symbol tiles of the text arena, 16
// symbols per lane.  A gram is indexed by its first symbols (up to ten 2-bit
// symbols, whose tables are direct: 4^10 bits; three or four bytes, hashed)
// and compared with the text in full where its table bit and directory slot
// are found.  Table hits go through a per-warp queue, so that the directory
// (L2) is read 32 look-ups at a time, and the entries of those look-ups are
// dealt out one per lane.  Bound by the look-ups' latency and issue (ncu, 32 MiB
// of bytes: 61% of the issue slots busy, 31% of the cycles without a warp to
// issue, 21 of 32 lanes active, shared-memory pipe 53%) and, on 2-bit text, by
// the shared-memory pipe (65%, L1 74%; 54% of the issue slots); DRAM 4%.
// (First forms: hashed tables for every gram length, up to 13 symbols, let
// four positions in ten through to the directory, one look-up per lane and
// length at a time: 535 us per 64 MiB of DNA against 1,024 patterns; with the
// queue 430; this form 186.  4,096 byte patterns over 32 MiB: 200, now 126.)
struct GramWarp {
  unsigned long long hit_pos[kQueue];  // arena offset << 4 | key length's number
  unsigned long long susp[kQueue];
  uint32_t hit_lo[kQueue], hit_hi[kQueue];
};

// Ends found from here on would be too few, or not once each.  (Candidates over
// their buffer are counted on, for the next run's.)  Called by whole warps.
__device__ __forceinline__ bool incomplete(const StepCounters* ctr) {
  return __any_sync(kFull, ctr->overflow & (kSetOverflow | kGramOverflow | kGramDense));
}

// Counts a warp's look-ups that have many entries to compare; true once a slice
// has more of them than pay.  A key that many grams share, in a text full of it,
// would have every one of them compared at each of its places (16,384 grams of
// one key, 1 MiB of that key: 32 ms, and 2.5 for the scan).  Called by whole
// warps; a function of its own, for the registers of the scan.  (In the scan it
// costs 1 to 2%, so kCounted is left out where the keys bound it well enough.)
constexpr uint32_t kLookReport = 256;  // entries of 32 look-ups from which they are counted
__device__ __noinline__ bool too_dense(GramCounters* c, StepCounters* ctr, unsigned long long cap,
                                       uint32_t total) {
  unsigned long long all = 0;
  const bool first = (threadIdx.x & 31) == 0;
  if (first) all = atomicAdd(&c->n_look, (unsigned long long)total) + total;
  const bool over = __shfl_sync(kFull, all, 0) > cap;
  if (first && over) atomicOr(&ctr->overflow, kGramDense | 1u);
  return over;
}

template <bool kTwoBit, bool kCounted>
__global__ void __launch_bounds__(kGramThreads, 1) gram_scan_kernel(const GramScan A) {
  extern __shared__ __align__(16) uint32_t bits_s[];
  constexpr int kWarps = kGramThreads / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  GramWarp& Q = reinterpret_cast<GramWarp*>(bits_s + A.n_words)[warp];
  {
    const uint4* src = reinterpret_cast<const uint4*>(A.bits);
    uint4* dst = reinterpret_cast<uint4*>(bits_s);
    for (uint32_t i = threadIdx.x; i < A.n_words / 4; i += kGramThreads) dst[i] = src[i];
  }
  __syncthreads();
  if (blockIdx.x == 0 && warp == 0 && incomplete(A.ctr) && lane == 0)
    atomicAdd(&A.ctr->n_skipped, 1ull);  // no ends of this slice will be looked for
  int hn = 0, qn = 0;  // queued table hits and suspects of this warp
  bool dead = false;   // the suspect buffer is full, or the text is not for the index
  auto flush = [&]() {
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(&A.ctr_slice->n_susp, (unsigned long long)qn);
    base = __shfl_sync(kFull, base, 0);
    for (int i = lane; i < qn; i += 32)
      if (base + i < A.cap_susp) A.susp[base + i] = Q.susp[i];
    if (base + qn > A.cap_susp) {
      dead = true;
      if (lane == 0) atomicOr(&A.ctr->overflow, kGramOverflow | 1u);
    }
    qn = 0;
    __syncwarp();
  };
  // The last 32 (or all) queued table hits: a directory look-up each, then
  // all their entries, one per lane and round, against the text.
  auto look_up = [&]() {
    __syncwarp();
    const int i = max(hn - 32, 0) + lane;
    uint32_t first = 0, left = 0, lo = 0, hi = 0;
    unsigned long long pos = 0;
    // (behind the last item's text lies what an earlier, longer step or another
    // buffer left there)
    if (i < hn && (pos = Q.hit_pos[i]) < A.text_end << 4) {
      lo = Q.hit_lo[i];
      hi = Q.hit_hi[i];
      const GramLen& g = A.len[pos & 15u];
      const uint32_t key = lo & g.mask;
      uint32_t s = (key * kGramDirMul) >> g.dir_shift;
      for (uint32_t pr = 0; pr <= g.max_probe; ++pr) {
        const uint4 sl = __ldg(A.dir + g.dir0 + s);
        if (sl.z == 0) break;
        if (sl.x == key) {
          first = sl.y;
          left = sl.z;
          break;
        }
        s = (s + 1) & g.dir_mask;
      }
      pos >>= 4;
    }
    hn = max(hn - 32, 0);
    uint32_t incl = left;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t x = __shfl_up_sync(kFull, incl, d);
      if (lane >= d) incl += x;
    }
    const uint32_t total = __shfl_sync(kFull, incl, 31);
    if (kCounted && total >= kLookReport)
      dead = too_dense(A.ctr_slice, A.ctr, A.cap_look, total);
    for (uint32_t base = 0; base < total && !dead; base += 32) {
      const uint32_t item = base + unsigned(lane);
      int own = 0;  // the lane whose look-up found the item: lanes with incl <= item
#pragma unroll
      for (int d = 16; d; d >>= 1) {
        const uint32_t x = __shfl_sync(kFull, incl, own + d - 1);
        if (x <= item) own += d;
      }
      own = min(own, 31);
      const uint32_t e = __shfl_sync(kFull, first - (incl - left), own) + item;
      const uint32_t olo = __shfl_sync(kFull, lo, own), ohi = __shfl_sync(kFull, hi, own);
      const unsigned long long opos = __shfl_sync(kFull, pos, own);
      bool ok = false;
      if (item < total) {
        const uint4 en = __ldg(reinterpret_cast<const uint4*>(A.entries + e));
        const uint32_t len = en.y >> 24;
        const uint32_t nb = kTwoBit ? 2 * len : 8 * len;  // bits of the gram
        const uint32_t mlo = nb >= 32 ? ~0u : (1u << nb) - 1u;
        const uint32_t mhi = nb <= 32 ? 0u : nb >= 64 ? ~0u : (1u << (nb - 32)) - 1u;
        ok = (((olo ^ en.z) & mlo) | ((ohi ^ en.w) & mhi)) == 0;
      }
      const unsigned m = __ballot_sync(kFull, ok);
      if (!m) continue;
      if (qn > kQueue - 32) flush();
      if (ok) Q.susp[qn + __popc(m & below)] = (opos << 24) | e;
      qn += __popc(m);
    }
    __syncwarp();
  };
  const uint4* text = reinterpret_cast<const uint4*>(A.arena);
  const unsigned long long stride = (unsigned long long)gridDim.x * kWarps;
  for (unsigned long long tile = A.t_begin + (unsigned long long)blockIdx.x * kWarps + warp;
       tile < A.t_end && !dead; tile += stride) {
    const uint4 v = __ldg(text + tile * 32 + lane);
    uint4 nx = make_uint4(0u, 0u, 0u, 0u);
    if (lane == 31) nx = __ldg(text + tile * 32 + 32);  // inside the arena's end padding at most
    uint32_t t[6];
    if (kTwoBit) {
      t[0] = pack2(v.x, A.shift2) | (pack2(v.y, A.shift2) << 8) | (pack2(v.z, A.shift2) << 16) |
             (pack2(v.w, A.shift2) << 24);
      const uint32_t n = pack2(nx.x, A.shift2) | (pack2(nx.y, A.shift2) << 8) |
                         (pack2(nx.z, A.shift2) << 16) | (pack2(nx.w, A.shift2) << 24);
      t[1] = __shfl_down_sync(kFull, t[0], 1);
      if (lane == 31) t[1] = n;
    } else {
      t[0] = v.x;
      t[1] = v.y;
      t[2] = v.z;
      t[3] = v.w;
      t[4] = __shfl_down_sync(kFull, v.x, 1);
      t[5] = __shfl_down_sync(kFull, v.y, 1);
      if (lane == 31) {
        t[4] = nx.x;
        t[5] = nx.y;
      }
    }
#pragma unroll 1
    for (int l = 0; l < A.n_len; ++l) {
      const GramLen& g = A.len[l];
      // table bit of every position, shifted in from the top: position j of
      // the lane ends at bit 16 + j
      uint32_t acc = 0;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        uint32_t h;
        if (kTwoBit) {
          h = __funnelshift_r(t[0], t[1], 2 * j) & g.mask;
        } else {
          const uint32_t lo = (j & 3) ? __funnelshift_r(t[j >> 2], t[(j >> 2) + 1], 8 * (j & 3))
                                      : t[j >> 2];
          h = ((lo & g.mask) * g.mul) >> g.shift;
        }
        const uint32_t w = bits_s[g.word0 + (h >> 5)];
        acc = __funnelshift_r(acc, __funnelshift_r(w, w, h), 1);
      }
      uint32_t hits = acc >> 16;
      unsigned m;
      while ((m = __ballot_sync(kFull, hits != 0)) != 0) {
        if (hn > kQueue - 32) look_up();
        if (hits) {
          const int j = __ffs(hits) - 1;
          hits &= hits - 1;
          uint32_t lo, hi;
          window<kTwoBit>(t, j, lo, hi);
          const int at = hn + __popc(m & below);
          Q.hit_lo[at] = lo;
          Q.hit_hi[at] = hi;
          Q.hit_pos[at] = ((tile * 512 + unsigned(lane) * 16 + unsigned(j)) << 4) | unsigned(l);
        }
        hn += __popc(m);
      }
    }
  }
  while (hn && !dead) look_up();
  if (qn && !dead) flush();
}

// ------------------------------------------------------------------- ends
// D[e] over the span + 1 ends from lo on, from the symbols before them (text
// is the item's first symbol): bit j of the result is set when D[lo + j] <= E.
// Two to four words.
template <int W>
__device__ uint32_t ends_run(const uint32_t* __restrict__ peq, const uint8_t* __restrict__ text,
                             int64_t lo, int span, int m, int E) {
  uint32_t Pv[W], Mv[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    Pv[w] = 0xffffffffu;
    Mv[w] = 0u;
  }
  int score = m;
  uint32_t hit = 0;
  const int tb = (m - 1) & 31;  // the last row's bit of word W - 1
  const int64_t start = max(lo - (m + E - 1), int64_t(0));
  const int warm = int(lo - start), n = warm + span + 1;
  const uint8_t* t = text + start;
#pragma unroll 4
  for (int i = 0; i < n; ++i) {
    const uint32_t* row = peq + size_t(t[i]) * 4;
    const uint4 q = __ldg(reinterpret_cast<const uint4*>(row));
    const uint32_t eq[4] = {q.x, q.y, q.z, q.w};
    uint32_t php = 0, mhp = 0, carry = 0;
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint32_t x = eq[w] & Pv[w];
      const unsigned long long sum64 = (unsigned long long)x + Pv[w] + carry;
      const uint32_t sum = uint32_t(sum64);
      carry = uint32_t(sum64 >> 32);
      const uint32_t xv = eq[w] | Mv[w];
      const uint32_t xh = (sum ^ Pv[w]) | eq[w];
      const uint32_t ph = Mv[w] | ~(xh | Pv[w]);
      const uint32_t mh = Pv[w] & xh;
      if (w == W - 1) score += int((ph >> tb) & 1u) - int((mh >> tb) & 1u);
      const uint32_t phs = __funnelshift_l(php, ph, 1);
      const uint32_t mhs = __funnelshift_l(mhp, mh, 1);
      php = ph;
      mhp = mh;
      Pv[w] = mhs | ~(xv | phs);
      Mv[w] = phs & xv;
    }
    if (i >= warm && score <= E) hit |= 1u << (i - warm);
  }
  return hit;
}

// A suspect decoded: the pattern, the ends [lo, lo + span] (relative to the
// item's first symbol) that its gram allows (none: span < 0), and where the
// gram lies.
struct Suspect {
  uint32_t wi, pat;
  int m, E, span;
  int before, after, pair, len;   // as in the entry
  int64_t lo, x, n_text;          // x: the gram's first symbol; n_text: symbols of the text
  uint64_t arena0;
};

__device__ __forceinline__ Suspect decode_suspect(const StepParams& P, const GramTables& G,
                                                  unsigned long long key) {
  Suspect s;
  s.span = -1;
  const uint2 en = __ldg(reinterpret_cast<const uint2*>(G.entries + (key & 0xffffffu)));
  const uint64_t x = key >> 24;  // arena offset of the gram
  s.pat = en.x & 0xffffffu;
  s.E = int(en.x >> 28);
  const int K = int((en.x >> 24) & 15u);
  s.before = int(en.y & 255u);
  s.after = int((en.y >> 8) & 255u);
  s.pair = int((en.y >> 16) & 255u);
  s.len = int(en.y >> 24);
  s.m = s.before + s.after + s.len + ((s.pair >> 4) & 3) - 1;
  // the last item that starts at or before the gram
  uint32_t a = 0, b = P.n_items;
  while (a < b) {
    const uint32_t mid = (a + b) >> 1;
    if (P.items[mid].arena_base <= x)
      a = mid + 1;
    else
      b = mid;
  }
  if (a == 0) return s;
  s.wi = a - 1;
  const WorkItem w = P.items[s.wi];
  s.arena0 = w.arena_base;
  s.x = int64_t(x - s.arena0);
  s.n_text = w.e_new - w.base_pos;
  const int64_t last = s.x + s.len - 1;
  if (last >= s.n_text) return s;
  s.lo = max(last + s.after - s.E, max(int64_t(0), w.e_prev - 2 * int64_t(K)) - w.base_pos);
  const int64_t hi = min(last + int64_t(s.after) + s.E, s.n_text - 1);
  if (s.lo <= hi) s.span = int(hi - s.lo);
  return s;
}

// Edits between r (at most 32) pattern symbols beside a found gram and the
// text beside it: the anchored column recurrence (dummy row 0, 1, 2, ...) over
// text symbols t[0], t[d], t[2 d], ..., at most avail, against bits o, o + 1,
// ... of the mask rows.  Returns a value over lim if there are more than lim;
// otherwise
//   kTest  a value of at most lim
//   kLeast the least, over all ends in the text
//   kEnds  the least, and bit j - r + lim of ends for each end j (text
//          symbols matched) within lim
// A cell within lim of a column lies at most lim off the diagonal, so a
// diagonal value over 2 lim ends it.
enum Side { kTest, kLeast, kEnds };
template <Side kMode>
__device__ __forceinline__ int side(const uint32_t* __restrict__ peq, int o,
                                    const uint8_t* __restrict__ t, int d, int r, int avail,
                                    int lim, uint32_t& ends) {
  if (r == 0) {  // nothing to match: every text symbol is an insertion
    if (kMode == kEnds) ends = (0xffffffffu >> (31 - min(lim, avail))) << lim;
    return 0;
  }
  if (kMode == kEnds) ends = r <= lim ? 1u << (lim - r) : 0u;  // no text symbol: r deletions
  if (kMode == kTest && r <= lim) return r;
  int best = r, score = r, diag = 0;
  const int n = min(r + lim, avail), q = o >> 5, sh = o & 31;
  if (n <= 0) return best;
  uint32_t Pv = 0xffffffffu, Mv = 0u;
  // the masks of the next column and the symbol after it are on their way
  // while a column is computed (four columns at a time, symbols from aligned
  // words, read less but measured slower: 300 -> 421 us on DNA)
  const bool two_words = sh + r > 32;
  auto mask = [&](uint32_t c) {
    const uint32_t* row = peq + c * 4 + q;
    return __funnelshift_r(__ldg(row), two_words ? __ldg(row + 1) : 0u, sh);
  };
  uint32_t eq_next = mask(t[0]), c_next = t[min(1, n - 1) * d];
  for (int j = 0; j < n; ++j) {
    const uint32_t eq = eq_next;
    eq_next = mask(c_next);
    c_next = t[min(j + 2, n - 1) * d];
    const uint32_t sum = (eq & Pv) + Pv;
    const uint32_t xv = eq | Mv;
    const uint32_t xh = (sum ^ Pv) | eq;
    const uint32_t ph = Mv | ~(xh | Pv), mh = Pv & xh;
    score += int((ph >> (r - 1)) & 1u) - int((mh >> (r - 1)) & 1u);
    if (kMode == kTest && score <= lim) return score;
    best = min(best, score);
    if (kMode == kEnds && score <= lim) ends |= 1u << (j + 1 - r + lim);
    if (j < r) {
      diag += 1 - int(((xh | Mv) >> j) & 1u);
      if (diag > 2 * lim) return lim + 1;
    }
    const uint32_t phs = (ph << 1) | 1u, mhs = mh << 1;
    Pv = mhs | ~(xv | phs);
    Mv = phs & xv;
  }
  return best;
}

// side() on one side of a suspect's gram, r of the symbols there.
template <Side kMode>
__device__ __forceinline__ int suspect_side(const StepParams& P, const GramTables& G,
                                            const Suspect& s, bool left, int r, int lim,
                                            uint32_t& ends) {
  const size_t p0 = size_t(s.pat) * 256 * 4;
  const uint8_t* text = P.arena + s.arena0 + s.x;
  return side<kMode>(left ? P.peq_rev + p0 : G.peq_fwd + p0, s.m - (left ? s.before : s.after),
                     left ? text - 1 : text + s.len, left ? -1 : 1, r,
                     int(min(left ? s.x : s.n_text - s.x - s.len, int64_t(64))), lim, ends);
}

// The found ends (bit j of hit: lo + j) as candidates, each (pattern, end)
// pair once, one reservation per warp.  Called by whole warps.
__device__ __forceinline__ void put_ends(const StepParams& P, const EndSet& S, const Suspect& s,
                                         uint32_t hit) {
  if (!__any_sync(kFull, hit != 0)) return;
  const unsigned lane = threadIdx.x & 31;
  bool full = false;
  for (uint32_t h = hit; h; h &= h - 1)
    if (!insert_key(S, ((s.arena0 + uint64_t(s.lo + __ffs(h) - 1)) << 24) | s.pat, &full))
      hit &= ~(h & (0u - h));
  if (full) atomicOr(&P.ctr->overflow, kSetOverflow | 1u);
  __syncwarp();
  const int nf = __popc(hit);
  int incl = nf;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int t = __shfl_up_sync(kFull, incl, d);
    if (int(lane) >= d) incl += t;
  }
  const int tot = __shfl_sync(kFull, incl, 31);
  if (!tot) return;
  unsigned long long o = 0;
  if (lane == 0) {
    o = atomicAdd(&P.ctr->n_cand, (unsigned long long)tot);
    const unsigned long long filled =
        atomicAdd(&P.ctr->n_gram, (unsigned long long)tot) + (unsigned long long)tot;
    if (filled > (S.mask + 1) / 4) atomicOr(&P.ctr->overflow, kSetOverflow | 1u);
  }
  o = __shfl_sync(kFull, o, 0) + unsigned(incl - nf);
  bool over = false;
  for (uint32_t h = hit; h; h &= h - 1, ++o) {
    if (o < P.cap_cand) {
      Candidate c;
      c.wi = s.wi;
      c.pat = s.pat;
      c.e_rel = uint64_t(s.lo + __ffs(h) - 1);
      P.cand[o] = c;
    } else {
      over = true;
    }
  }
  if (over) atomicOr(&P.ctr->overflow, 1u);
}

constexpr int kEndThreads = 256;
constexpr int kEndList = 64;

// One thread per suspect, in three rounds so that warps stay full (what stays
// after a round waits in a list per warp):
//   the rest of the gram's pair against the text beside it, within one edit,
//     drops nearly every chance find after a few columns;
//   the pattern symbols on the gram's longer side, then those on the other
//     with the edits that are left;
//   the left side again, and the right side's columns, which are the ends.
// (An occurrence keeps one pair within one edit and one half of it unedited,
// or one gram with its edit; that one's suspect finds its end.)  With more than
// 32 symbols on a side, the 32 next to the gram are matched, and the few
// suspects that pass are left to gram_long_kernel.
// Bound by the latency of the suspects' text and masks (ncu, 3 M suspects: 46% of
// the issue slots busy, half of a warp's cycles wait for a load, 11 of 32 lanes
// active; gram_long_kernel 27%, 25 lanes; DRAM 4%).
// (4,096 byte patterns over 32 MiB, 3 M suspects: the whole pattern for every
// suspect 892 us; its first 32 rows first 576; both sides at once, 9 lanes of a
// warp busy, 965; two rounds, long patterns apart, 375; this form 331; and 85
// in gram_long_kernel.)
__global__ void __launch_bounds__(kEndThreads)
    gram_ends_kernel(const StepParams P, const GramTables G,
                     const unsigned long long* __restrict__ susp, GramCounters* C,
                     unsigned long long cap, unsigned long long* __restrict__ longs,
                     unsigned long long cap_long, const EndSet S) {
  __shared__ unsigned long long list[2][kEndThreads / 32][kEndList];
  const unsigned long long n = min(C->n_susp, cap);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  if (incomplete(P.ctr)) return;
  unsigned long long *pairs = list[0][warp], *passed = list[1][warp];
  int np = 0, nq = 0;  // listed suspects of this warp: whose pair, whose sides matched
  // the ends of the last 32 (or all) suspects that passed
  auto finish = [&]() {
    __syncwarp();
    const int i = max(nq - 32, 0) + lane;
    Suspect s;
    uint32_t hit = 0;
    s.span = -1;
    if (i < nq) s = decode_suspect(P, G, passed[i]);
    nq = max(nq - 32, 0);
    if (s.span >= 0) {
      const int lim = s.E - ((s.pair & kGramEdit) ? 1 : 0);
      uint32_t ends;
      const int left = lim - suspect_side<kLeast>(P, G, s, true, s.before, lim, ends);
      if (left >= 0) {  // edits left for the right side
        suspect_side<kEnds>(P, G, s, false, s.after, left, ends);
        // bit i: the end i + after - left symbols past the gram; hit: from lo on
        const int64_t sh = s.lo - (s.x + s.len - 1 + s.after - left);
        hit = sh >= 0 ? (sh < 32 ? ends >> sh : 0u) : ends << -sh;
        hit &= 0xffffffffu >> (31 - s.span);
      }
    }
    __syncwarp();
    put_ends(P, S, s, hit);
    __syncwarp();
  };
  // both sides of the last 32 (or all) suspects whose pair matched, up to 32
  // symbols each, the longer side first: it ends most of them
  auto sides = [&]() {
    __syncwarp();
    const int i = max(np - 32, 0) + lane;
    const unsigned long long key = i < np ? pairs[i] : 0ull;
    int w = -1;  // 0 .. 2: runs whole (gram_long_kernel); 3: finish
    if (i < np) {
      const Suspect s = decode_suspect(P, G, key);
      const int lim = s.E - ((s.pair & kGramEdit) ? 1 : 0);
      const bool left1 = s.before > s.after;
      uint32_t ends;
      const int k1 = suspect_side<kLeast>(P, G, s, left1, min(left1 ? s.before : s.after, 32), lim,
                                          ends);
      if (k1 <= lim &&
          suspect_side<kTest>(P, G, s, !left1, min(left1 ? s.after : s.before, 32), lim - k1,
                              ends) <= lim - k1)
        w = s.before > 32 || s.after > 32 ? ((s.m - 1) >> 5) - 1 : 3;
    }
    np = max(np - 32, 0);
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      const unsigned b = __ballot_sync(kFull, w == l);
      if (!b) continue;
      unsigned long long at = 0;
      if (lane == 0) at = atomicAdd(&C->n_long[l], (unsigned long long)__popc(b));
      at = __shfl_sync(kFull, at, 0) + __popc(b & below);
      if (w == l) {
        if (at < cap_long) longs[l * cap_long + at] = key;
        else atomicOr(&P.ctr->overflow, kGramOverflow | 1u);
      }
    }
    const unsigned b = __ballot_sync(kFull, w == 3);
    if (w == 3) passed[nq + __popc(b & below)] = key;
    nq += __popc(b);
    if (nq >= 32) finish();
    __syncwarp();
  };
  const unsigned long long stride = (unsigned long long)gridDim.x * kEndThreads;
  const unsigned long long first = (unsigned long long)blockIdx.x * kEndThreads + warp * 32;
  unsigned long long next = first + lane < n ? susp[first + lane] : 0ull;
  for (unsigned long long base = first; base < n; base += stride) {
    const unsigned long long i = base + lane, key = next;
    bool keep = false;
    next = i + stride < n ? susp[i + stride] : 0ull;
    if (i < n) {
      const Suspect s = decode_suspect(P, G, key);
      keep = s.span >= 0;
      const int r = s.pair & 15;
      if (keep && r) {
        uint32_t ends;
        const int lim = min(s.E, 1);
        keep = suspect_side<kTest>(P, G, s, (s.pair & kGramLeft) != 0, r, lim, ends) <= lim;
      }
    }
    const unsigned m = __ballot_sync(kFull, keep);
    if (!m) continue;
    if (keep) pairs[np + __popc(m & below)] = key;
    np += __popc(m);
    if (np >= 32) sides();
  }
  if (np) sides();
  if (nq) finish();
}

// The whole pattern over the ends of the listed suspects, whole warps of one
// word count.
__global__ void __launch_bounds__(kEndThreads)
    gram_long_kernel(const StepParams P, const GramTables G, const GramCounters* C,
                     const unsigned long long* __restrict__ longs, unsigned long long cap_long,
                     const EndSet S) {
  if (incomplete(P.ctr)) return;
  unsigned long long n[3], warps = 0;
#pragma unroll
  for (int l = 0; l < 3; ++l) {
    n[l] = min(C->n_long[l], cap_long);
    warps += (n[l] + 31) / 32;
  }
  const int lane = threadIdx.x & 31;
  const unsigned long long stride = (unsigned long long)gridDim.x * (kEndThreads / 32);
  for (unsigned long long wj = (unsigned long long)blockIdx.x * (kEndThreads / 32) +
                               (threadIdx.x >> 5);
       wj < warps; wj += stride) {
    unsigned long long t = wj;
    int l = 0;
    while (l < 2 && t >= (n[l] + 31) / 32) t -= (n[l++] + 31) / 32;
    const unsigned long long i = t * 32 + lane;
    Suspect s;
    uint32_t hit = 0;
    if (i < n[l]) {
      s = decode_suspect(P, G, longs[l * cap_long + i]);
      const uint32_t* peq = G.peq_fwd + size_t(s.pat) * 256 * 4;
      const uint8_t* text = P.arena + s.arena0;
      if (l == 0) hit = ends_run<2>(peq, text, s.lo, s.span, s.m, s.E);
      else if (l == 1) hit = ends_run<3>(peq, text, s.lo, s.span, s.m, s.E);
      else hit = ends_run<4>(peq, text, s.lo, s.span, s.m, s.E);
    }
    __syncwarp();
    put_ends(P, S, s, hit);
    __syncwarp();
  }
}

// Match masks of every pattern, [pattern][256][4], bit j = symbol j, or
// symbol m - 1 - j (reversed: the verification pass).
__global__ void __launch_bounds__(256)
    peq_kernel(const uint8_t* __restrict__ bytes, const uint8_t* __restrict__ len, uint32_t n_pat,
               uint4* __restrict__ peq, bool reversed) {
  for (uint32_t p = blockIdx.x; p < n_pat; p += gridDim.x) {
    const uint8_t* b = bytes + size_t(p) * OASM_MAX_PATTERN_LEN;
    const int m = len[p];
    uint32_t w[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int q = 0; q < 4; ++q)
      for (int j = 32 * q; j < min(m, 32 * q + 32); ++j)
        if (b[reversed ? m - 1 - j : j] == threadIdx.x) w[q] |= 1u << (j & 31);
    peq[size_t(p) * 256 + threadIdx.x] = make_uint4(w[0], w[1], w[2], w[3]);
  }
}

size_t gram_smem(uint32_t n_words) {
  return size_t(n_words) * 4 + size_t(kGramThreads / 32) * sizeof(GramWarp);
}

}  // namespace

cudaError_t prepare_gram_kernels() {
  const int bytes = int(gram_smem(kGramMaxWords));
  for (auto* kernel : {gram_scan_kernel<false, false>, gram_scan_kernel<false, true>,
                       gram_scan_kernel<true, false>, gram_scan_kernel<true, true>}) {
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t launch_peq(const uint8_t* bytes, const uint8_t* len, uint32_t n_pat, uint32_t* peq,
                       bool reversed, cudaStream_t s) {
  peq_kernel<<<n_pat < 65535u ? n_pat : 65535u, 256, 0, s>>>(
      bytes, len, n_pat, reinterpret_cast<uint4*>(peq), reversed);
  return cudaGetLastError();
}

cudaError_t launch_grams(const StepParams& p, const GramTables& g, const GramScan& a,
                         const EndSet& set, cudaStream_t s) {
  if (a.t_end <= a.t_begin) return cudaSuccess;
  const unsigned long long tiles = a.t_end - a.t_begin;
  const unsigned long long need = (tiles + kGramThreads / 32 - 1) / (kGramThreads / 32);
  const unsigned grid = unsigned(need < (unsigned long long)p.num_sms ? need : p.num_sms);
  auto* scan = a.two_bit ? a.cap_look ? gram_scan_kernel<true, true> : gram_scan_kernel<true, false>
               : a.cap_look ? gram_scan_kernel<false, true> : gram_scan_kernel<false, false>;
  scan<<<grid, kGramThreads, gram_smem(a.n_words), s>>>(a);
  gram_ends_kernel<<<p.num_sms * 4, kEndThreads, 0, s>>>(p, g, a.susp, a.ctr_slice, a.cap_susp,
                                                         a.longs, a.cap_long, set);
  if (g.any_long)
    gram_long_kernel<<<p.num_sms * 6, kEndThreads, 0, s>>>(p, g, a.ctr_slice, a.longs, a.cap_long,
                                                           set);
  return cudaGetLastError();
}

}  // namespace oasm
