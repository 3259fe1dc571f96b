// grams.cu -- gram index in front of the exact forward scan (sm_103a).
//
// Pigeonhole principle for edit distance: an alignment of a pattern with at
// most E edits (Eq. 1, Eq. 2; E = K under unit costs) leaves one of E + 1
// disjoint pieces of the pattern unedited, and one of E / 2 + 1 pieces with
// at most one edit.  The index holds every string such a piece may appear as
// (the piece itself, or every string one edit away from it) as a gram of the
// text, with the pattern symbols that remain after it; a gram found at a text
// position allows the ends within E of that many symbols further on.  Only
// those ends are examined, with the whole pattern's column recurrence, and
// the ones with D[e] <= E become candidates: the forward scan's own
// candidates under unit costs, a superset of them under edit costs (a
// distance is at least the cheapest cost times the number of edits), which
// verification then measures.
//
//   scan   one text position per step of a lane: for each gram length, a bit
//          of a table in shared memory, and where it is set the length's
//          directory (open addressing, in L2): suspects (position, entry)
//   ends   one thread per suspect: the recurrence over the ends the entry
//          allows; each (pattern, end) becomes a candidate once (an
//          open-addressing set: an occurrence holds several grams)
//
// The cost per text position depends on the number of gram lengths and on
// how often grams appear, not on the number of patterns.
#include "kernels.h"

namespace oasm {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr int kQueue = 96;  // suspects buffered per warp

// ------------------------------------------------------------------- scan
// 2-bit symbols: (byte >> shift) & 3, 16 of them to a word.
__device__ __forceinline__ uint32_t pack2(uint32_t w, uint32_t shift) {
  // the four 2-bit fields meet in the top byte; the partial products are
  // disjoint, so nothing carries into it
  return (((w >> shift) & 0x03030303u) * 0x01041040u) >> 24;
}

// Key of the gram of length g.len at symbol j of the lane's 16 (2-bit text:
// the packed symbols; bytes: up to four bytes as they are, more hashed).
template <bool kTwoBit>
__device__ __forceinline__ uint32_t gram_key(const GramLen& g, const uint32_t (&t)[6], int j) {
  if (kTwoBit) return __funnelshift_r(t[0], t[1], 2 * j) & g.mask_lo;
  const int q = j >> 2, r = 8 * (j & 3);
  const uint32_t lo = r ? __funnelshift_r(t[q], t[q + 1], r) : t[q];
  if (g.mask_hi == 0u) return lo & g.mask_lo;
  const uint32_t hi = r ? __funnelshift_r(t[q + 1], t[q + 2], r) : t[q + 1];
  return lo * kGramMixLo + (hi & g.mask_hi) * kGramMixHi;
}

// One block per SM; its warps walk 512-symbol tiles of the text arena, 16
// symbols per lane.  Bound by instruction issue (about nine instructions per
// position and gram length) and by the shared-memory conflicts of the random
// table reads; the directory reads of one warp hide behind the others.
template <bool kTwoBit>
__global__ void __launch_bounds__(kGramThreads, 1) gram_scan_kernel(const GramScan A) {
  extern __shared__ __align__(16) uint32_t bits_s[];
  constexpr int kWarps = kGramThreads / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned long long* queue =
      reinterpret_cast<unsigned long long*>(bits_s + A.n_words) + size_t(warp) * kQueue;
  {
    const uint4* src = reinterpret_cast<const uint4*>(A.bits);
    uint4* dst = reinterpret_cast<uint4*>(bits_s);
    for (uint32_t i = threadIdx.x; i < A.n_words / 4; i += kGramThreads) dst[i] = src[i];
  }
  __syncthreads();
  int qn = 0;         // queued suspects of this warp
  bool dead = false;  // the suspect buffer is full
  auto flush = [&]() {
    __syncwarp();
    unsigned long long base = 0;
    if (lane == 0) base = atomicAdd(A.n_susp, (unsigned long long)qn);
    base = __shfl_sync(kFull, base, 0);
    for (int i = lane; i < qn; i += 32)
      if (base + i < A.cap_susp) A.susp[base + i] = queue[i];
    if (base + qn > A.cap_susp) {
      dead = true;
      if (lane == 0) atomicOr(&A.ctr->overflow, kGramOverflow | 1u);
    }
    qn = 0;
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
      const GramLen g = A.len[l];
      // table bit of every position, shifted in from the top: position j of
      // the lane ends at bit 16 + j
      uint32_t acc = 0;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const uint32_t h = (gram_key<kTwoBit>(g, t, j) * g.mul) >> g.shift;
        const uint32_t w = bits_s[g.word0 + (h >> 5)];
        acc = __funnelshift_r(acc, __funnelshift_r(w, w, h), 1);
      }
      uint32_t hits = acc >> 16;
      // directory look-ups, one per lane and round; then one entry per lane
      // and round into the queue
      uint32_t e = 0, left = 0;
      unsigned long long pos = 0;
      while (__any_sync(kFull, (hits | left) != 0)) {
        if (left == 0 && hits) {
          const int j = __ffs(hits) - 1;
          hits &= hits - 1;
          pos = tile * 512 + unsigned(lane) * 16 + unsigned(j);
          // the key again, at a position known only here
          uint32_t key;
          if (kTwoBit) {
            key = __funnelshift_r(t[0], t[1], 2 * j) & g.mask_lo;
          } else {
            const int q = j >> 2;
            const uint32_t a = q == 0 ? t[0] : q == 1 ? t[1] : q == 2 ? t[2] : t[3];
            const uint32_t b = q == 0 ? t[1] : q == 1 ? t[2] : q == 2 ? t[3] : t[4];
            const uint32_t c = q == 0 ? t[2] : q == 1 ? t[3] : q == 2 ? t[4] : t[5];
            const uint32_t lo = __funnelshift_r(a, b, 8 * (j & 3));
            const uint32_t hi = __funnelshift_r(b, c, 8 * (j & 3));
            key = g.mask_hi == 0u ? (lo & g.mask_lo)
                                  : lo * kGramMixLo + (hi & g.mask_hi) * kGramMixHi;
          }
          uint32_t s = (key * kGramDirMul) >> g.dir_shift;
          for (uint32_t pr = 0; pr <= g.max_probe; ++pr) {
            const uint4 sl = __ldg(A.dir + g.dir0 + s);
            if (sl.z == 0) break;
            if (sl.x == key) {
              e = sl.y;
              left = sl.z;
              break;
            }
            s = (s + 1) & g.dir_mask;
          }
        }
        const unsigned m = __ballot_sync(kFull, left != 0);
        if (!m) continue;
        if (qn > kQueue - 32) flush();
        if (left) {
          queue[qn + __popc(m & ((1u << lane) - 1u))] = (pos << 24) | e;
          ++e;
          --left;
        }
        qn += __popc(m);
        if (dead) break;
      }
      if (dead) break;
    }
  }
  if (qn) flush();
}

// ------------------------------------------------------------------- ends
__device__ __forceinline__ unsigned long long mix_key(unsigned long long k) {
  // a 64-bit finaliser (xor-shift-multiply), spreads keys over the table
  k ^= k >> 33;
  k *= 0xff51afd7ed558ccdull;
  k ^= k >> 33;
  k *= 0xc4ceb9fe1a85ec53ull;
  k ^= k >> 33;
  return k;
}

constexpr int kSetProbes = 64;
__device__ bool insert_key(const EndSet& S, unsigned long long key, bool* full) {
  unsigned long long h = mix_key(key) & S.mask;
  for (int i = 0; i < kSetProbes; ++i) {
    const unsigned long long prev = atomicCAS(&S.slots[h], ~0ull, key);
    if (prev == ~0ull) return true;
    if (prev == key) return false;
    h = (h + 1) & S.mask;
  }
  *full = true;
  return false;
}

// D[e] over the span + 1 ends from lo on, from the symbols before them (text
// is the item's first symbol): bit j of the result is set when D[lo + j] <= E.
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
  for (int i = 0; i < n; ++i) {
    const uint32_t* row = peq + size_t(t[i]) * 4;
    uint32_t eq[W];
    if (W == 1) {
      eq[0] = __ldg(row);
    } else {
      const uint4 q = __ldg(reinterpret_cast<const uint4*>(row));
      const uint32_t q4[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int w = 0; w < W; ++w) eq[w] = q4[w];
    }
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

constexpr int kEndThreads = 256;

__global__ void __launch_bounds__(kEndThreads)
    gram_ends_kernel(const StepParams P, const GramTables G,
                     const unsigned long long* __restrict__ susp, const unsigned long long* n_susp,
                     unsigned long long cap, const EndSet S) {
  if (P.ctr->overflow & 1u) return;
  __shared__ int cnt[4];
  __shared__ unsigned long long order[kEndThreads];
  const unsigned long long n = min(*n_susp, cap);
  const unsigned lane = threadIdx.x & 31;
  const unsigned long long stride = (unsigned long long)gridDim.x * kEndThreads;
  for (unsigned long long base = (unsigned long long)blockIdx.x * kEndThreads; base < n;
       base += stride) {
    // the block's suspects by word count, so that a warp's patterns agree
    if (threadIdx.x < 4) cnt[threadIdx.x] = 0;
    __syncthreads();
    const unsigned long long i = base + threadIdx.x;
    const unsigned long long key = i < n ? susp[i] : 0ull;
    GramEntry en{};
    int W = 3;
    if (i < n) {
      en = G.entries[key & 0xffffffu];
      W = (P.m[en.pat] - 1) >> 5;
    }
    const int rank = atomicAdd(&cnt[W], 1);
    __syncthreads();
    int at = rank;
    for (int w = 0; w < W; ++w) at += cnt[w];
    order[at] = i < n ? key : ~0ull;
    __syncthreads();
    const unsigned long long mine = order[threadIdx.x];
    uint32_t hit = 0;
    uint32_t wi = 0, pat = 0;
    int64_t lo = 0;
    uint64_t arena0 = 0;
    if (mine != ~0ull) {
      en = G.entries[mine & 0xffffffu];
      pat = en.pat;
      const uint64_t x = mine >> 24;  // arena offset of the gram
      const int m = P.m[pat], K = P.K[pat], E = G.edits[pat];
      // the last item that starts at or before the gram
      uint32_t a = 0, b = P.n_items;
      while (a < b) {
        const uint32_t mid = (a + b) >> 1;
        if (P.items[mid].arena_base <= x)
          a = mid + 1;
        else
          b = mid;
      }
      if (a > 0) {
        wi = a - 1;
        const WorkItem w = P.items[wi];
        arena0 = w.arena_base;
        const int64_t last = int64_t(x - arena0) + en.len - 1;  // the gram's last symbol
        const int64_t n_text = w.e_new - w.base_pos;
        lo = max(last + en.rest - E,
                 max(int64_t(0), w.e_prev - 2 * int64_t(K)) - w.base_pos);
        const int64_t hi = min(last + int64_t(en.rest) + E, n_text - 1);
        if (last < n_text && lo <= hi) {
          const uint32_t* peq = G.peq_fwd + size_t(pat) * 256 * 4;
          const uint8_t* text = P.arena + arena0;
          const int span = int(hi - lo);
          if (m <= 32) hit = ends_run<1>(peq, text, lo, span, m, E);
          else if (m <= 64) hit = ends_run<2>(peq, text, lo, span, m, E);
          else if (m <= 96) hit = ends_run<3>(peq, text, lo, span, m, E);
          else hit = ends_run<4>(peq, text, lo, span, m, E);
        }
      }
    }
    __syncwarp();
    // distinct (pattern, end) pairs, one reservation per warp
    bool full = false;
    for (uint32_t h = hit; h; h &= h - 1)
      if (!insert_key(S, ((arena0 + uint64_t(lo + __ffs(h) - 1)) << 24) | pat, &full))
        hit &= ~(h & (0u - h));
    if (full) atomicOr(&P.ctr->overflow, 1u | 32u);
    const int nf = __popc(hit);
    int incl = nf;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(kFull, incl, d);
      if (int(lane) >= d) incl += t;
    }
    const int tot = __shfl_sync(kFull, incl, 31);
    if (tot) {
      unsigned long long o = 0;
      if (lane == 0) {
        o = atomicAdd(&P.ctr->n_cand, (unsigned long long)tot);
        const unsigned long long filled =
            atomicAdd(&P.ctr->n_gram, (unsigned long long)tot) + (unsigned long long)tot;
        if (filled > (S.mask + 1) / 4) atomicOr(&P.ctr->overflow, 1u | 32u);
      }
      o = __shfl_sync(kFull, o, 0) + unsigned(incl - nf);
      bool over = false;
      for (uint32_t h = hit; h; h &= h - 1, ++o) {
        if (o < P.cap_cand) {
          Candidate c;
          c.wi = wi;
          c.pat = pat;
          c.e_rel = uint64_t(lo + __ffs(h) - 1);
          P.cand[o] = c;
        } else {
          over = true;
        }
      }
      if (over) atomicOr(&P.ctr->overflow, 1u);
    }
    __syncthreads();  // cnt and order are reused
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
  return size_t(n_words) * 4 + size_t(kGramThreads / 32) * kQueue * 8;
}

}  // namespace

cudaError_t prepare_gram_kernels() {
  const int bytes = int(gram_smem(kGramMaxWords));
  cudaError_t e = cudaFuncSetAttribute(gram_scan_kernel<true>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(gram_scan_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             bytes);
  return e;
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
  if (a.two_bit)
    gram_scan_kernel<true><<<grid, kGramThreads, gram_smem(a.n_words), s>>>(a);
  else
    gram_scan_kernel<false><<<grid, kGramThreads, gram_smem(a.n_words), s>>>(a);
  gram_ends_kernel<<<p.num_sms * 6, kEndThreads, 0, s>>>(p, g, a.susp, a.n_susp, a.cap_susp, set);
  return cudaGetLastError();
}

}  // namespace oasm
