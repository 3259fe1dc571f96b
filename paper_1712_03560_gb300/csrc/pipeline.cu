// pipeline.cu -- the OASM device path after the forward scan (sm_103a):
//   gather    stream bytes and stored tails -> the step's text arena
//   verify    for each candidate end e: one bit-parallel pass of the reversed
//             pattern over t[e], t[e-1], ... gives lev(p, t[e-l+1..e]) for every
//             length l (Eq. 1 is invariant under reversing both strings), so
//             every hit (i, l, k) of Eq. 2 ending at e is found exactly once
//   sort      stable LSD radix sort of 64-bit hit keys (pair, start, length):
//             the order in which Algorithm 1 meets hits (i ascending, then l)
//   filter    Algorithm 1 in event form over each pair (stream, pattern); a
//             pair's hits are cut at every start that no earlier hit spans,
//             where the filter state is provably empty, and each piece runs
//             on its own thread; the first piece resumes the pair's pending
//             window carried from the previous step
//   finalize  decides carried windows of pairs without hits
//   state     installs the new pending windows and keeps the last T symbols of
//             every stream for the next step
#include <algorithm>
#include <utility>

#include "kernels.h"

namespace oasm {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr uint32_t kInvalid = 0xffffffffu;

// ---------------------------------------------------------------- gather
// 16 bytes at byte offset `mis` of the 32 bytes a | b.
__device__ __forceinline__ uint4 shift_bytes(const uint4& a, const uint4& b, unsigned mis) {
  const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
  const unsigned r = 8 * (mis & 3);
  uint4 o;
  switch (mis >> 2) {  // uniform over a chunk
    case 0:
      o = make_uint4(__funnelshift_r(w[0], w[1], r), __funnelshift_r(w[1], w[2], r),
                     __funnelshift_r(w[2], w[3], r), __funnelshift_r(w[3], w[4], r));
      break;
    case 1:
      o = make_uint4(__funnelshift_r(w[1], w[2], r), __funnelshift_r(w[2], w[3], r),
                     __funnelshift_r(w[3], w[4], r), __funnelshift_r(w[4], w[5], r));
      break;
    case 2:
      o = make_uint4(__funnelshift_r(w[2], w[3], r), __funnelshift_r(w[3], w[4], r),
                     __funnelshift_r(w[4], w[5], r), __funnelshift_r(w[5], w[6], r));
      break;
    default:
      o = make_uint4(__funnelshift_r(w[3], w[4], r), __funnelshift_r(w[4], w[5], r),
                     __funnelshift_r(w[5], w[6], r), __funnelshift_r(w[6], w[7], r));
  }
  return o;
}

// Copies of any alignment, one per block (long chunks) or per warp (short
// ones: packets and tails).  Whole 16-byte vectors at the destination's
// alignment; a source of another alignment is read in its own aligned vectors
// (only those that lie inside the chunk), each once, the other half coming
// from the next lane.  The bytes before and after go one by one.  Bound by
// memory: 64 MiB 122 -> 33 us (byte copies of unaligned texts ran at 70 GB/s).
template <bool kWarp>
__global__ void __launch_bounds__(256)
    gather_kernel(const CopyChunk* __restrict__ chunks, int n, uint8_t* arena) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int me = kWarp ? lane : int(threadIdx.x), team = kWarp ? 32 : 256;
  const int first = kWarp ? int(blockIdx.x) * 8 + warp : int(blockIdx.x);
  const int step = kWarp ? int(gridDim.x) * 8 : int(gridDim.x);
  for (int c = first; c < n; c += step) {
    const CopyChunk ch = chunks[c];
    uint8_t* dst = arena + ch.dst_off;
    const uint8_t* src = ch.src;
    uint32_t head = min(ch.len, uint32_t(-reinterpret_cast<uintptr_t>(dst)) & 15u);
    const unsigned mis = unsigned(reinterpret_cast<uintptr_t>(src + head)) & 15u;
    if (mis > head) head = min(ch.len, head + 16u);  // the first aligned vector starts in the chunk
    const uint32_t body = ch.len - head;
    // vectors whose source (two aligned vectors where it is unaligned) lies
    // inside the chunk
    const uint32_t nv = mis == 0 ? body / 16 : body + mis < 32 ? 0u : (body + mis - 16) / 16;
    const uint4* s4 = reinterpret_cast<const uint4*>(src + head - mis);
    uint4* d4 = reinterpret_cast<uint4*>(dst + head);
    if (mis == 0) {
      uint32_t i = me;
      for (; i + 3 * team < nv; i += 4 * team) {
        const uint4 v0 = s4[i], v1 = s4[i + team], v2 = s4[i + 2 * team], v3 = s4[i + 3 * team];
        d4[i] = v0;
        d4[i + team] = v1;
        d4[i + 2 * team] = v2;
        d4[i + 3 * team] = v3;
      }
      for (; i < nv; i += team) d4[i] = s4[i];
    } else if (nv) {
      // (vector nv is the last one's second half: inside the chunk)
      for (uint32_t i = me; i - lane < nv; i += team) {
        const uint4 a = s4[min(i, nv)];
        uint4 b;
        b.x = __shfl_down_sync(kFull, a.x, 1);
        b.y = __shfl_down_sync(kFull, a.y, 1);
        b.z = __shfl_down_sync(kFull, a.z, 1);
        b.w = __shfl_down_sync(kFull, a.w, 1);
        if (lane == 31) b = s4[min(i + 1, nv)];
        if (i < nv) d4[i] = shift_bytes(a, b, mis);
      }
    }
    for (uint32_t i = me; i < head; i += team) dst[i] = src[i];
    for (uint32_t i = head + 16 * nv + me; i < ch.len; i += team) dst[i] = src[i];
  }
}

// ---------------------------------------------------------------- verify
template <int W>
__device__ __forceinline__ void add_w(const uint32_t* a, const uint32_t* b, uint32_t* s) {
  if (W == 1) {
    s[0] = a[0] + b[0];
  } else if (W == 2) {
    asm("add.cc.u32 %0, %2, %4;\n\taddc.u32 %1, %3, %5;"
        : "=r"(s[0]), "=r"(s[1]) : "r"(a[0]), "r"(a[1]), "r"(b[0]), "r"(b[1]));
  } else if (W == 3) {
    asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(b[0]), "r"(b[1]), "r"(b[2]));
  } else {
    asm("add.cc.u32 %0, %4, %8;\n\taddc.cc.u32 %1, %5, %9;\n\t"
        "addc.cc.u32 %2, %6, %10;\n\taddc.u32 %3, %7, %11;"
        : "=r"(s[0]), "=r"(s[1]), "=r"(s[2]), "=r"(s[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]), "r"(b[2]),
          "r"(b[3]));
  }
}

// Anchored pass: distances of the reversed pattern (bit j = p[m-1-j]) to the
// prefixes of t[e], t[e-1], ...; the dummy row is 0, 1, 2, ... so a +1
// horizontal difference enters the bottom word at every step.  Writes
// dist[l] for l = 1..lmax.
template <int W>
__device__ void anchored_pass(const uint32_t* __restrict__ peq, const uint8_t* __restrict__ tend,
                              int m, int lmax, int8_t* dist) {
  uint32_t Pv[W], Mv[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    Pv[w] = 0xffffffffu;
    Mv[w] = 0u;
  }
  const int tw = (m - 1) >> 5, tb = (m - 1) & 31;
  int score = m;
  for (int l = 1; l <= lmax; ++l) {
    const uint32_t c = tend[-(l - 1)];
    const uint4 q = __ldg(reinterpret_cast<const uint4*>(peq + c * 4));
    const uint32_t eq[4] = {q.x, q.y, q.z, q.w};
    uint32_t x[W], sum[W];
#pragma unroll
    for (int w = 0; w < W; ++w) x[w] = eq[w] & Pv[w];
    add_w<W>(x, Pv, sum);
    uint32_t php = 1u << 31, mhp = 0;  // shift-in: +1 at row 0
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const uint32_t xv = eq[w] | Mv[w];
      const uint32_t xh = (sum[w] ^ Pv[w]) | eq[w];
      const uint32_t ph = Mv[w] | ~(xh | Pv[w]);
      const uint32_t mh = Pv[w] & xh;
      if (w == tw) score += int((ph >> tb) & 1u) - int((mh >> tb) & 1u);
      const uint32_t phs = __funnelshift_l(php, ph, 1);
      const uint32_t mhs = __funnelshift_l(mhp, mh, 1);
      php = ph;
      mhp = mh;
      Pv[w] = mhs | ~(xv | phs);
      Mv[w] = phs & xv;
    }
    dist[l] = int8_t(score > 127 ? 127 : score);
  }
}

// Weighted verification (integer edit costs): the column dynamic program of
// Eq. 1 with costs c_sub, c_ins, c_del, the reversed pattern against t[e],
// t[e-1], ... (an alignment read backwards keeps its operations, so the
// distance is unchanged).  An alignment of cost <= K holds at most
// K / min(c_ins, c_del) insertions and deletions, so it stays within that many
// diagonals of the main one: only those cells are filled, with a bound above
// every distance outside, and every value <= K is exact.  Writes dist[l] for
// l = 1..lmax (127 where the length is too far from l_p to be within K).
// B: half width of the band, whose cells stay in registers (cell d of column l
// is row l + d - B).
// (1,024 DNA patterns of up to 32 symbols over 16 MiB, 178,000 ends: all rows
// in local memory 199 us, this form 31.)
template <int B>
__device__ __noinline__ void weighted_band(const uint8_t* __restrict__ pat,
                                           const uint8_t* __restrict__ tend, int m, int lmax,
                                           int cs, int ci, int cd, int8_t* dist) {
  constexpr int kFar = 1 << 24;
  int x[2 * B + 1];
  uint32_t sym[2 * B + 1];  // symbol of the cell's row (row r: p[m - r])
#pragma unroll
  for (int d = 0; d <= 2 * B; ++d) {
    x[d] = d < B ? kFar : (d - B) * cd;
    const int r = 1 + d - B;
    sym[d] = r >= 1 && r <= m ? pat[m - r] : 256u;
  }
  for (int l = 1; l <= lmax; ++l) {
    const uint32_t c = tend[-(l - 1)];
#pragma unroll
    for (int d = 0; d <= 2 * B; ++d) {
      int v = x[d] + (sym[d] == c ? 0 : cs);
      if (d < 2 * B) v = min(v, x[d + 1] + ci);
      if (d > 0) v = min(v, x[d - 1] + cd);
      if (d < B && d <= B - l) v = d == B - l ? l * ci : kFar;  // row 0 and above
      x[d] = v;
    }
    int at = 127;  // row m
#pragma unroll
    for (int d = 0; d <= 2 * B; ++d)
      if (d == m - l + B) at = x[d];
    dist[l] = int8_t(min(at, 127));
#pragma unroll
    for (int d = 0; d < 2 * B; ++d) sym[d] = sym[d + 1];
    const int r = l + 1 + B;
    sym[2 * B] = r <= m ? pat[m - r] : 256u;
  }
}

// Bands too wide for registers: one column in local memory.
__device__ __noinline__ void weighted_column(const uint8_t* __restrict__ pat,
                                             const uint8_t* __restrict__ tend, int m, int lmax,
                                             int cs, int ci, int cd, int b, int8_t* dist) {
  constexpr int kFar = 1 << 24;
  int col[OASM_MAX_PATTERN_LEN + 1];
  for (int r = 0; r <= m; ++r) col[r] = r <= b ? r * cd : kFar;
  for (int l = 1; l <= lmax; ++l) {
    const uint8_t c = tend[-(l - 1)];
    const int r0 = max(1, l - b), r1 = min(m, l + b);
    int diag = r0 <= r1 ? col[r0 - 1] : 0;
    int up = r0 == 1 ? l * ci : kFar;
    col[r0 - 1 <= m ? r0 - 1 : 0] = up;
    for (int r = r0; r <= r1; ++r) {
      const int left = col[r];
      up = min(min(left + ci, up + cd), diag + (pat[m - r] == c ? 0 : cs));
      diag = left;
      col[r] = up;
    }
    dist[l] = int8_t(r1 == m && r0 <= m ? min(up, 127) : 127);
  }
}

__device__ __forceinline__ void weighted_anchored(const StepParams& P, int p,
                                                  const uint8_t* __restrict__ tend, int m,
                                                  int lmax, int8_t* dist) {
  const uint8_t* pat = P.wpat + size_t(p) * OASM_MAX_PATTERN_LEN;
  const int b = int(P.K[p]) / min(P.c_ins, P.c_del);
  if (b <= 1) weighted_band<1>(pat, tend, m, lmax, P.c_sub, P.c_ins, P.c_del, dist);
  else if (b <= 3) weighted_band<3>(pat, tend, m, lmax, P.c_sub, P.c_ins, P.c_del, dist);
  else weighted_column(pat, tend, m, lmax, P.c_sub, P.c_ins, P.c_del, b, dist);
}

// Distances of every length ending at tend (bit-parallel, or the weighted
// dynamic program: a kernel of its own each, for its registers and stack).
template <bool kWeighted>
__device__ __forceinline__ void lengths_at(const StepParams& P, int p, const uint8_t* tend,
                                           int m, int lmax, int8_t* dist) {
  if (kWeighted) {
    weighted_anchored(P, p, tend, m, lmax, dist);
    return;
  }
  const int W = (m + 31) >> 5;
  const uint32_t* pq = P.peq_rev + size_t(p) * 256 * 4;
  if (W == 1) anchored_pass<1>(pq, tend, m, lmax, dist);
  else if (W == 2) anchored_pass<2>(pq, tend, m, lmax, dist);
  else if (W == 3) anchored_pass<3>(pq, tend, m, lmax, dist);
  else anchored_pass<4>(pq, tend, m, lmax, dist);
}

// Canonical order of emitted records: (work item, pattern, decided_at, k,
// length), packed like the hit keys so it fits the same bit budget.
__device__ __forceinline__ unsigned long long out_key(const StepParams& P, uint64_t pair,
                                                      const WorkItem& w, int64_t decided_at,
                                                      int k, int len, int m, int K) {
  return (pair << (P.start_bits + kLowBits)) | (uint64_t(decided_at - w.base_pos) << kLowBits) |
         (uint64_t(k) << kLenBits) | uint64_t(len - (m - K));
}

__device__ __forceinline__ void put_record(const StepParams& P, unsigned long long o,
                                           const DevHit& h, unsigned long long key) {
  P.out[o] = h;
  P.okeys[o] = key;
  P.ovals[o] = uint32_t(o);
}

template <bool kWeighted>
__device__ void verify_body(const StepParams& P) {
  const unsigned long long n = min(P.ctr->n_cand, P.cap_cand);
  // stop only on an upstream overflow: the hit count must stay exact when this
  // kernel's own output overflows, so the re-run can size the buffer at once
  if (P.ctr->overflow & 1u) return;
  const unsigned lane = threadIdx.x & 31;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long base = (unsigned long long)blockIdx.x * blockDim.x; base < n;
       base += stride) {
    const unsigned long long idx = base + threadIdx.x;
    uint64_t keys[2 * kMaxK + 1];
    DevHit rec;
    unsigned long long rkey = 0;
    int nh = 0;
    if (idx < n) {
      const Candidate c = P.cand[idx];
      if (c.wi != kInvalid) {
        const WorkItem w = P.items[c.wi];
        const int p = int(c.pat);
        const int m = P.m[p], K = P.K[p];
        const int64_t e = w.base_pos + int64_t(c.e_rel);
        const uint8_t* tend = P.arena + w.arena_base + c.e_rel;
        const int64_t lo_start = max(w.base_pos, int64_t(0));
        int8_t dist[kMaxW * 32 + kMaxK + 1];
        if (P.rules.output == OASM_OUT_ENDS) {
          if (e >= w.e_prev && e < w.e_new) {
            const int lmax = int(min(int64_t(m + K), e - lo_start + 1));
            lengths_at<kWeighted>(P, p, tend, m, lmax, dist);
            int best = 127, bl = 0;
            for (int l = 1; l <= lmax; ++l)
              if (dist[l] < best) { best = dist[l]; bl = l; }
            if (best <= K) {
              rec.start = uint64_t(e - bl + 1);
              rec.decided_at = uint64_t(e);
              rec.pattern = uint32_t(p);
              rec.slot = w.slot;
              rec.len = uint32_t(bl);
              rec.k = uint32_t(best);
              rkey = out_key(P, uint64_t(c.wi) * P.n_pat + uint64_t(p), w, e, best, bl, m, K);
              nh = 1;
            }
          }
        } else {
          const int64_t fp = f_prev(w, m, K), fn = f_new(w, m, K);
          const int64_t smin = max(fp + 1, lo_start);
          const int lmax = int(min(int64_t(m + K), e - smin + 1));
          const int lmin = int(max(int64_t(max(1, m - K)), e - fn + 1));
          if (lmin <= lmax) {
            lengths_at<kWeighted>(P, p, tend, m, lmax, dist);
            const uint64_t pair = uint64_t(c.wi) * P.n_pat + uint64_t(p);
            for (int l = lmin; l <= lmax; ++l) {
              const int k = dist[l];
              if (k > K) continue;
              const int64_t st = e - l + 1;
              keys[nh++] = (pair << (P.start_bits + kLowBits)) |
                           (uint64_t(st - w.base_pos) << kLowBits) |
                           (uint64_t(l - (m - K)) << kKBits) | uint64_t(k);
            }
          }
        }
      }
    }
    // warp-aggregated append
    int incl = nh;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const int t = __shfl_up_sync(kFull, incl, d);
      if (int(lane) >= d) incl += t;
    }
    const int tot = __shfl_sync(kFull, incl, 31);
    if (tot == 0) continue;
    const bool raw = P.rules.output != OASM_OUT_FILTERED;
    unsigned long long wbase = 0;
    if (lane == 0) wbase = atomicAdd(raw ? &P.ctr->n_out : &P.ctr->n_hits, (unsigned long long)tot);
    wbase = __shfl_sync(kFull, wbase, 0);
    unsigned long long o = wbase + unsigned(incl - nh);
    bool over = false;
    if (!raw) {
      for (int q = 0; q < nh; ++q, ++o) {
        if (o < P.cap_hits) P.keys[o] = keys[q];
        else over = true;
      }
      if (over) atomicOr(&P.ctr->overflow, 2u);
    } else {
      for (int q = 0; q < nh; ++q, ++o) {
        if (o >= P.cap_out) { over = true; continue; }
        if (P.rules.output == OASM_OUT_ENDS) {
          put_record(P, o, rec, rkey);
        } else {
          const uint64_t key = keys[q];
          const uint32_t pair = uint32_t(key >> (P.start_bits + kLowBits));
          const int p = int(pair % P.n_pat);
          const WorkItem w = P.items[pair / P.n_pat];
          const int m = P.m[p], K = P.K[p];
          const int64_t st = w.base_pos +
                             int64_t((key >> kLowBits) & ((1ull << P.start_bits) - 1));
          const int l = int((key >> kKBits) & 31u) + m - K;
          DevHit h;
          h.start = uint64_t(st);
          h.len = uint32_t(l);
          h.k = uint32_t(key & 15u);
          h.decided_at = uint64_t(st + l - 1);
          h.pattern = uint32_t(p);
          h.slot = w.slot;
          put_record(P, o, h, out_key(P, pair, w, st + l - 1, int(h.k), l, m, K));
        }
      }
      if (over) atomicOr(&P.ctr->overflow, 4u);
    }
  }
}

template <bool kWeighted>
__global__ void __launch_bounds__(256) verify_kernel(const StepParams P) {
  verify_body<kWeighted>(P);
}

// ---------------------------------------------------------------- radix sort
// Stable LSD radix sort, 8-bit digits, every pass in one cooperative launch
// (the element count is on the device; a few launches per pass, most of them
// over few keys, cost more than the passes themselves: 37 us a pass with a
// histogram and a scatter kernel, whose blocks each walked every block's
// histogram; 1 M keys of six digits 266 -> 122 us, up to 2,048 keys of two
// digits 74 -> 8 us).
//   up to kSortTile keys: one block, every pass in shared memory
//   more: each active block owns a contiguous chunk.  Per pass: its digit
//     counts; a scan of each digit's counts over the blocks (one digit per
//     block and turn); the scatter, which ranks a tile of kSortTile keys in
//     shared memory (warp matching per round of 32 keys with a running count
//     per digit, scans over the warps and the digits) and writes the tile out
//     digit run by digit run, consecutive threads on consecutive keys.
// Blocks meet at bounded grid barriers; what other blocks wrote is read past
// L1.
constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kBins = 256;
constexpr int kSortPer = 8;                         // keys per thread and tile
constexpr int kSortTile = kSortThreads * kSortPer;  // 2,048
constexpr uint32_t kGaveUp = 1u << 30;              // over any count of arrivals
// Blocks up to which each walks all blocks' digit counts itself, which saves a
// barrier a pass (14,000 keys of four digits on 8 blocks: 58 -> 43 us).
constexpr unsigned int kSortWalk = 64;

struct SortSmem {
  unsigned long long key[kSortTile];
  uint32_t val[kSortTile];
  unsigned int wcnt[kSortWarps][kBins];
  unsigned int base[kBins];    // global position of the digit's next key
  unsigned int tstart[kBins];  // the digit's first slot in the sorted tile
  unsigned int wsum[kSortWarps];
  int stop;
};

// Exclusive scan of one value per thread, in thread order.
__device__ __forceinline__ unsigned int sort_scan(SortSmem& sm, unsigned int v) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int t = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) sm.wsum[warp] = incl;
  __syncthreads();
  unsigned int pre = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w)
    if (w < warp) pre += sm.wsum[w];
  __syncthreads();  // wsum is reused by the next call
  return pre + incl - v;
}

// Ranks the tile's keys (registers) by one digit: pos[r] = the key's slot in
// the tile sorted by digit; returns this thread's digit's count (digit
// threadIdx.x), its first slot in sm.tstart.
__device__ __forceinline__ unsigned int rank_tile(SortSmem& sm,
                                                  const unsigned long long (&key)[kSortPer],
                                                  int tn, int shift,
                                                  unsigned int (&pos)[kSortPer]) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) sm.wcnt[w][threadIdx.x] = 0;
  __syncthreads();
  unsigned int dig[kSortPer];
#pragma unroll
  for (int r = 0; r < kSortPer; ++r) {
    const int e = warp * (kSortPer * 32) + r * 32 + lane;  // tile index: warp-major
    const bool ok = e < tn;
    const unsigned d = ok ? unsigned((key[r] >> shift) & (kBins - 1u)) : unsigned(kBins);
    dig[r] = d;
    const unsigned peers = __match_any_sync(kFull, d);
    const unsigned below = __popc(peers & lt);
    pos[r] = ok ? sm.wcnt[warp][d & (kBins - 1u)] + below : 0u;
    __syncwarp();
    if (ok && below == 0) sm.wcnt[warp][d] += __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  // per digit: offsets of the warps' keys, then the digit's start in the tile
  unsigned int run = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) {
    const unsigned int c = sm.wcnt[w][threadIdx.x];
    sm.wcnt[w][threadIdx.x] = run;
    run += c;
  }
  sm.tstart[threadIdx.x] = sort_scan(sm, run);
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kSortPer; ++r)
    if (dig[r] < unsigned(kBins)) pos[r] += sm.tstart[dig[r]] + sm.wcnt[warp][dig[r]];
  return run;
}

// All active blocks meet (*bar counts arrivals since the step began); false
// when the bounded wait ran out.  The blocks agree on that: one whose wait runs
// out takes kGaveUp from the count, unless the last block has arrived by then,
// so a barrier that one block gives up is passed by none, and what follows the
// last barrier of a launch runs in all blocks or in none.
__device__ __forceinline__ bool sort_barrier(SortSmem& sm, unsigned int* bar, unsigned int target,
                                             const BarrierBound& bound, StepCounters* ctr) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(bar, 1u);
    target += bound.extra;
    bool met = false;
    for (uint32_t it = 0;; ++it) {
      unsigned int seen;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(bar) : "memory");
      met = int(seen) >= int(target);
      if (met || int(seen) < 0) break;
      if (it < bound.polls) __nanosleep(20);
      // (an exchange fails where another block arrived or gave up meanwhile, as
      // often as there are blocks at most)
      else if (atomicCAS(bar, seen, seen - kGaveUp) == seen) break;
    }
    sm.stop = !met;
    // (bit 0 keeps the filter off the unsorted keys)
    if (!met) atomicOr(&ctr->overflow, kWaitOver | 1u);
    __threadfence();
  }
  __syncthreads();
  return sm.stop == 0;
}

__device__ void sort_body(SortSmem& sm, unsigned long long* keys, unsigned long long* keys_alt,
                          uint32_t* vals, uint32_t* vals_alt, const unsigned long long* count,
                          unsigned long long cap, int lo_bit, int hi_bit, unsigned int* hist,
                          unsigned int* bar, const BarrierBound& bound, StepCounters* ctr) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const unsigned long long n = min(*count, cap);
  // keys per block: an even split, in whole tiles (two or more tiles to a block
  // where one would do measured slower: 1 M keys of six digits 155 -> 179 us)
  const unsigned long long tiles = (n + kSortTile - 1) / kSortTile;
  const unsigned long long chunk = (tiles + gridDim.x - 1) / gridDim.x * kSortTile;
  const unsigned int nb = n ? unsigned((n + chunk - 1) / chunk) : 0u;
  if (blockIdx.x >= nb) return;
  if (n <= kSortTile) {
    const int passes = (hi_bit - lo_bit + 7) / 8;
    unsigned long long key[kSortPer];
    uint32_t val[kSortPer];
#pragma unroll
    for (int r = 0; r < kSortPer; ++r) {
      const int e = warp * (kSortPer * 32) + r * 32 + lane;
      key[r] = e < int(n) ? keys[e] : 0ull;
      val[r] = vals && e < int(n) ? vals[e] : 0u;
    }
    for (int shift = lo_bit; shift < hi_bit; shift += 8) {
      unsigned int pos[kSortPer];
      rank_tile(sm, key, int(n), shift, pos);
#pragma unroll
      for (int r = 0; r < kSortPer; ++r)
        if (warp * (kSortPer * 32) + r * 32 + lane < int(n)) {
          sm.key[pos[r]] = key[r];
          sm.val[pos[r]] = val[r];
        }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < kSortPer; ++r) {
        const int e = warp * (kSortPer * 32) + r * 32 + lane;
        if (e < int(n)) {
          key[r] = sm.key[e];
          val[r] = sm.val[e];
        }
      }
      __syncthreads();
    }
    unsigned long long* ko = (passes & 1) ? keys_alt : keys;
    uint32_t* vo = (passes & 1) ? vals_alt : vals;
#pragma unroll
    for (int r = 0; r < kSortPer; ++r) {
      const int e = warp * (kSortPer * 32) + r * 32 + lane;
      if (e < int(n)) {
        ko[e] = key[r];
        if (vals) vo[e] = val[r];
      }
    }
    return;
  }
  const unsigned long long b0 = chunk * blockIdx.x, b1 = min(n, b0 + chunk);
  unsigned int* total = hist + size_t(kBins) * gridDim.x;  // [kBins] keys of each digit
  unsigned int target = 0, parity = 0;
  for (int shift = lo_bit; shift < hi_bit; shift += 8) {
    // digit counts of the block's chunk
    sm.base[threadIdx.x] = 0;
    __syncthreads();
    unsigned long long i = b0 + threadIdx.x;
    for (; i + 3 * kSortThreads < b1; i += 4 * kSortThreads) {
      unsigned long long k4[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) k4[q] = __ldcg(keys + i + q * kSortThreads);
#pragma unroll
      for (int q = 0; q < 4; ++q) atomicAdd(&sm.base[(k4[q] >> shift) & (kBins - 1u)], 1u);
    }
    for (; i < b1; i += kSortThreads)
      atomicAdd(&sm.base[(__ldcg(keys + i) >> shift) & (kBins - 1u)], 1u);
    __syncthreads();
    unsigned int tot = 0, pre = 0;  // keys of digit threadIdx.x: all, and in earlier blocks
    if (nb <= kSortWalk) {
      // few blocks: each walks the counts of all, hist[block][digit]
      unsigned int* h = hist + size_t(parity) * kSortWalk * kBins;
      parity ^= 1u;  // (the other half may still be read)
      h[size_t(blockIdx.x) * kBins + threadIdx.x] = sm.base[threadIdx.x];
      if (!sort_barrier(sm, bar, target += nb, bound, ctr)) return;
#pragma unroll 8
      for (unsigned int q = 0; q < nb; ++q) {
        const unsigned int v = __ldcg(h + size_t(q) * kBins + threadIdx.x);
        tot += v;
        pre += q < blockIdx.x ? v : 0u;
      }
    } else {
      hist[size_t(threadIdx.x) * gridDim.x + blockIdx.x] = sm.base[threadIdx.x];
      if (!sort_barrier(sm, bar, target += nb, bound, ctr)) return;
      // each digit's counts scanned over the blocks: a digit per block and
      // turn, or, where few blocks would take many turns, per warp (3.7 M keys
      // on 608 blocks: 196 us per block, 226 per warp)
      const bool wide = nb >= kBins / 2;
      for (unsigned int d = wide ? blockIdx.x : blockIdx.x * kSortWarps + warp; d < unsigned(kBins);
           d += wide ? nb : nb * kSortWarps) {
        unsigned int* row = hist + size_t(d) * gridDim.x;
        unsigned int run = 0;
        for (unsigned int c = 0; c < nb; c += wide ? kSortThreads : 32) {
          const unsigned int j = c + (wide ? threadIdx.x : lane);
          const unsigned int v = j < nb ? __ldcg(row + j) : 0u;
          if (wide) {
            const unsigned int excl = sort_scan(sm, v);
            if (j < nb) row[j] = run + excl;
            for (int w = 0; w < kSortWarps; ++w) run += sm.wsum[w];
            __syncthreads();
          } else {
            unsigned int incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const unsigned int t = __shfl_up_sync(kFull, incl, o);
              if (lane >= o) incl += t;
            }
            if (j < nb) row[j] = run + incl - v;
            run += __shfl_sync(kFull, incl, 31);
          }
        }
        if (lane == 0) total[d] = run;
      }
      if (!sort_barrier(sm, bar, target += nb, bound, ctr)) return;
      tot = __ldcg(total + threadIdx.x);
      pre = __ldcg(hist + size_t(threadIdx.x) * gridDim.x + blockIdx.x);
    }
    const unsigned int before = sort_scan(sm, tot);
    sm.base[threadIdx.x] = before + pre;
    for (unsigned long long t0 = b0; t0 < b1; t0 += kSortTile) {
      const int tn = int(min((unsigned long long)kSortTile, b1 - t0));
      unsigned long long key[kSortPer];
      uint32_t val[kSortPer];
      unsigned int pos[kSortPer];
#pragma unroll
      for (int r = 0; r < kSortPer; ++r) {
        const int e = warp * (kSortPer * 32) + r * 32 + lane;
        key[r] = e < tn ? __ldcg(keys + t0 + e) : 0ull;
        val[r] = vals && e < tn ? __ldcg(vals + t0 + e) : 0u;
      }
      const unsigned int cnt = rank_tile(sm, key, tn, shift, pos);
#pragma unroll
      for (int r = 0; r < kSortPer; ++r)
        if (warp * (kSortPer * 32) + r * 32 + lane < tn) {
          sm.key[pos[r]] = key[r];
          sm.val[pos[r]] = val[r];
        }
      __syncthreads();
      for (int e = threadIdx.x; e < tn; e += kSortThreads) {
        const unsigned long long k = sm.key[e];
        const unsigned d = unsigned((k >> shift) & (kBins - 1u));
        const unsigned int g = sm.base[d] + unsigned(e) - sm.tstart[d];
        keys_alt[g] = k;
        if (vals) vals_alt[g] = sm.val[e];
      }
      __syncthreads();
      sm.base[threadIdx.x] += cnt;
    }
    if (shift + 8 < hi_bit && !sort_barrier(sm, bar, target += nb, bound, ctr)) return;
    unsigned long long* tk = keys;
    keys = keys_alt;
    keys_alt = tk;
    uint32_t* tv = vals;
    vals = vals_alt;
    vals_alt = tv;
  }
}

__global__ void __launch_bounds__(kSortThreads, 4)
    sort_kernel(unsigned long long* keys, unsigned long long* keys_alt, uint32_t* vals,
                uint32_t* vals_alt, const unsigned long long* count, unsigned long long cap,
                int lo_bit, int hi_bit, unsigned int* hist, unsigned int* bar,
                const BarrierBound bound, StepCounters* ctr) {
  extern __shared__ __align__(16) unsigned char sort_smem[];
  sort_body(*reinterpret_cast<SortSmem*>(sort_smem), keys, keys_alt, vals, vals_alt, count, cap,
            lo_bit, hi_bit, hist, bar, bound, ctr);
}

__global__ void permute_kernel(const DevHit* __restrict__ src, const uint32_t* __restrict__ idx,
                               DevHit* __restrict__ dst, const StepCounters* ctr,
                               unsigned long long cap) {
  if (ctr->overflow & kWaitOver) return;  // the record sort gave up: idx is incomplete
  const unsigned long long n = min(ctr->n_out, cap);
  for (unsigned long long i = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (unsigned long long)gridDim.x * blockDim.x)
    dst[i] = src[idx[i]];
}

// ---------------------------------------------------------------- filter
// A pair's keys decoded: the hit's start, length and level.
struct PairKeys {
  int64_t base;          // base_pos
  int32_t len0;          // m - K
  uint64_t mask;         // start bits
  __device__ __forceinline__ int64_t start(uint64_t key) const {
    return base + int64_t((key >> kLowBits) & mask);
  }
  __device__ __forceinline__ int len(uint64_t key) const {
    return int(uint32_t(key) >> kKBits & 31u) + len0;
  }
};

// Filter window of one pair.  The level that is pending (idx) is also kept in
// registers, so a hit's rules touch the level rows only to store.
struct Window {
  int pend;
  int idx;
  uint32_t valid;           // levels that hold a row
  int64_t top_start;        // row idx
  int32_t top_len;
  int64_t start[kMaxK + 1];
  int32_t len[kMaxK + 1];
  unsigned long long rpos;  // ordered records: the segment's first position
  uint32_t nrec;            // records the segment wrote so far
};

__device__ __forceinline__ void open_window(Window& W, int K) {
  W.pend = 0;
  W.idx = K;
  W.valid = 0;
  W.nrec = 0;
  W.rpos = 0;
}

__device__ __forceinline__ void load_window(Window& W, const WinHdr& hd, const MemRow* rows,
                                            int K) {
  W.pend = 1;
  W.idx = hd.idx;
  for (int lv = 0; lv <= K; ++lv) {
    const MemRow r = rows[lv];
    W.start[lv] = r.start;
    W.len[lv] = r.len;
    W.valid |= r.valid ? 1u << lv : 0u;
  }
  W.top_start = W.start[W.idx];
  W.top_len = W.len[W.idx];
}

__device__ void emit(const StepParams& P, Window& W, uint32_t pair, int p, int lv, int64_t start,
                     int len, int64_t f, const WorkItem& w) {
  DevHit h;
  h.start = uint64_t(start);
  h.decided_at = uint64_t(f);
  h.pattern = uint32_t(p);
  h.slot = w.slot;
  h.len = uint32_t(len);
  h.k = uint32_t(lv);
  if (P.ordered) {
    const unsigned long long o = W.rpos + W.nrec++;
    if (o < P.cap_rtmp) P.rtmp[o] = h;
    else atomicOr(&P.ctr->overflow, 64u);
    return;
  }
  const unsigned long long o = atomicAdd(&P.ctr->n_out, 1ull);
  if (o >= P.cap_out) {
    atomicOr(&P.ctr->overflow, 4u);
    return;
  }
  put_record(P, o, h, out_key(P, pair, w, f, lv, len, P.m[p], P.K[p]));
}

// A segment's record count, read by the scan (ordered records).
__device__ __forceinline__ void close_segment(const StepParams& P, const Window& W) {
  if (P.ordered && W.nrec) P.seg[W.rpos] = W.nrec;
}

// Validation complete at f (Sec. 4.2): the highest-priority occurrence is
// added, then each lower level j whose counter satisfies Eq. 3 against the
// accumulated length.  r(j) = f - i_j + 1 because a level's counter starts
// at 1 on insertion and grows by one per processed symbol.
__device__ void flush(const StepParams& P, Window& W, uint32_t pair, int p, int K,
                      const WorkItem& w) {
  const int64_t f = W.top_start + W.top_len - 1;
  int64_t acc = 0;
  for (uint32_t left = W.valid & (~0u << W.idx); left; left &= left - 1) {
    const int lv = __ffs(left) - 1;
    const int64_t start = W.start[lv];
    const int len = W.len[lv];
    const int64_t lhs = (f - start + 1) - acc;
    const bool keep = (lv == W.idx) || (P.rules.cmp == OASM_CMP_GT ? lhs > len : lhs >= len);
    if (keep) {
      emit(P, W, pair, p, lv, start, len, f, w);
      acc = (P.rules.acc == OASM_ACC_SUM) ? acc + len : len;
    }
  }
  W.pend = 0;
  W.idx = K;
  W.valid = 0;
}

// A pair's window after this step, for commit_body.
__device__ __forceinline__ void put_window(const StepParams& P, const Window& W, uint32_t pair,
                                           int K) {
  const unsigned long long q = atomicAdd(&P.ctr->n_pool, 1ull);
  if (q >= P.cap_pool) {
    atomicOr(&P.ctr->overflow, 8u);
    return;
  }
  WinHdr hdr;
  hdr.pend = W.pend;
  hdr.idx = W.idx;
  P.pool_hdr[q] = hdr;
  for (int lv = 0; lv <= K; ++lv) {
    const bool v = (W.valid >> lv) & 1u;
    MemRow r;
    r.start = v ? W.start[lv] : 0;
    r.len = v ? W.len[lv] : 0;
    r.valid = v;
    P.pool_mem[q * (kMaxK + 1) + lv] = r;
  }
  P.pool_pair[q] = pair;
  P.pair_pool[pair] = int32_t(q);
}

// R1-R3 applied to one hit met in (i, l) order (event form of Algorithm 1).
__device__ __forceinline__ void apply(const StepParams& P, Window& W, uint32_t pair, int p, int K,
                                      const WorkItem& w, int64_t start, int len, int k) {
  if (W.pend && start > W.top_start + W.top_len - 1) flush(P, W, pair, p, K, w);
  bool put = false;
  if (!W.pend) {  // an empty window opens at the hit's level
    W.pend = 1;
    put = true;
  } else if (k < W.idx) {  // R1
    put = true;
  } else if (k == W.idx) {  // R2 / R3
    const int64_t ce = W.top_start + W.top_len - 1, ne = start + len - 1;
    if (P.rules.replace == OASM_REPLACE_CONTAINED) put = start >= W.top_start && ne <= ce;
    else if (P.rules.replace == OASM_REPLACE_SAME_END) put = ne == ce;
  }
  if (put) {
    W.idx = k;
    W.valid |= 1u << k;
    W.start[k] = W.top_start = start;
    W.len[k] = W.top_len = len;
  }
}

__device__ __forceinline__ uint32_t pair_of(uint64_t key, int sb) {
  return uint32_t(key >> (sb + kLowBits));
}

// One thread per hit; the first hit of a piece runs the piece.  A piece is a
// serial chain, so its latency counts (a planted copy at K = 15 gives some
// hundred hits): its keys are read four at a time ahead of the rules, decoded
// with the pair's constants, and the pending level stays in registers (a
// dozen signatures with K up to 15: 171 -> 72 us; 3.7 M hits of one motif:
// 291 -> 167).
__device__ void filter_body(const StepParams& P, const unsigned long long* S) {
  if (P.ctr->overflow & 3u) return;  // candidates or hits incomplete; keep counting records
  const unsigned long long n = min(P.ctr->n_hits, P.cap_hits);
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  const int sb = P.start_bits;
  for (unsigned long long h = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; h < n;
       h += stride) {
    const uint64_t key0 = S[h], before = h ? S[h - 1] : 0ull;
    const uint32_t pair = pair_of(key0, sb);
    const bool first = h == 0 || pair_of(before, sb) != pair;
    // a piece starts only at the first hit of a start that no earlier hit of
    // the pair (nor the carried window) spans
    if (!first && (before >> kLowBits) == (key0 >> kLowBits)) continue;
    const int p = int(pair % P.n_pat);
    const WorkItem w = P.items[pair / P.n_pat];
    const int m = P.m[p], K = P.K[p];
    const PairKeys D{w.base_pos, m - K, (1ull << sb) - 1};
    const int64_t start0 = D.start(key0);
    if (!first && D.start(before) + D.len(before) - 1 >= start0) continue;
    const size_t hidx = size_t(w.slot) * P.n_pat + p;
    const MemRow* crow = P.mem + size_t(w.slot) * P.mem_stride + P.mem_off[p];
    const WinHdr chdr = P.hdr[hidx];
    int64_t cf = INT64_MIN;  // end of the carried window's top occurrence
    if (chdr.pend) cf = crow[chdr.idx].start + crow[chdr.idx].len - 1;
    if (!first) {
      if (cf >= start0) continue;
      bool spanned = false;
      for (long long j = (long long)h - 2; j >= 0; --j) {
        const uint64_t kj = S[j];
        if (pair_of(kj, sb) != pair) break;
        const int64_t sj = D.start(kj);
        if (sj + m + K <= start0) break;  // ends before start0
        if (sj + D.len(kj) - 1 >= start0) {
          spanned = true;
          break;
        }
      }
      if (spanned) continue;
    }
    Window Wn;
    open_window(Wn, K);
    Wn.rpos = h + (unsigned long long)(first ? pair : pair + 1) * unsigned(P.head);
    int64_t maxend = INT64_MIN;
    if (first && chdr.pend) {
      load_window(Wn, chdr, crow, K);
      maxend = cf;
    }
    const bool per_start_best = P.rules.order == OASM_ORDER_PER_START_BEST;
    // per-start-best: the best hit so far (smallest k, then shortest) of the
    // current start, and the last end of that start's hits
    int64_t bs = 0, bend = 0;
    int bl = 0, bk = 0;
    bool have = false, last = true;
    for (unsigned long long j = h; j < n && last; j += 4) {
      uint64_t k4[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) k4[q] = S[min(j + q, n - 1)];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint64_t key = k4[q];
        if (j + q >= n || pair_of(key, sb) != pair) {  // the pair's last hit is behind
          j = n;
          break;
        }
        const int64_t st = D.start(key);
        const int len = D.len(key), k = int(key & 15u);
        if (!per_start_best) {
          if (j + q != h && st > maxend) {  // next piece
            last = false;
            break;
          }
          apply(P, Wn, pair, p, K, w, st, len, k);
          maxend = max(maxend, st + len - 1);
          continue;
        }
        if (have && st == bs) {
          bend = max(bend, st + len - 1);
          if (k < bk) bl = len, bk = k;
          continue;
        }
        if (have) {
          apply(P, Wn, pair, p, K, w, bs, bl, bk);
          maxend = max(maxend, bend);
          have = false;
          if (st > maxend) {  // next piece
            last = false;
            break;
          }
        }
        have = true;
        bs = st;
        bl = len;
        bk = k;
        bend = st + len - 1;
      }
    }
    if (have) apply(P, Wn, pair, p, K, w, bs, bl, bk);
    if (!last) {
      if (Wn.pend) flush(P, Wn, pair, p, K, w);
    } else {
      if (Wn.pend && (w.eos || Wn.top_start + Wn.top_len - 1 <= f_new(w, m, K)))
        flush(P, Wn, pair, p, K, w);
      put_window(P, Wn, pair, K);
    }
    close_segment(P, Wn);
  }
}

__global__ void __launch_bounds__(128)
    filter_kernel(const StepParams P, const unsigned long long* __restrict__ S) {
  filter_body(P, S);
}

// First index of the sorted hit keys S[0, n) whose pair is >= pr.
__device__ __forceinline__ unsigned long long pair_lower_bound(const unsigned long long* S,
                                                               unsigned long long n,
                                                               unsigned long long pr, int shift) {
  unsigned long long lo = 0, hi = n;
  while (lo < hi) {
    const unsigned long long mid = (lo + hi) >> 1;
    if ((S[mid] >> shift) < pr)
      lo = mid + 1;
    else
      hi = mid;
  }
  return lo;
}

// A pair without hits whose window was carried in: its records, and its entry
// for commit_body, if it can be decided now.
__device__ __noinline__ void decide_window(const StepParams& P, const unsigned long long* S,
                                           uint32_t pair) {
  const int p = int(pair % P.n_pat);
  const WorkItem w = P.items[pair / P.n_pat];
  const int m = P.m[p], K = P.K[p];
  const WinHdr hd = P.hdr[size_t(w.slot) * P.n_pat + p];
  const MemRow* rows = P.mem + size_t(w.slot) * P.mem_stride + P.mem_off[p];
  const MemRow& top = rows[hd.idx];
  if (!w.eos && top.start + top.len - 1 > f_new(w, m, K)) return;
  Window Wn;
  open_window(Wn, K);
  load_window(Wn, hd, rows, K);
  if (P.ordered)  // its segment is the pair's head
    Wn.rpos = pair_lower_bound(S, min(P.ctr->n_hits, P.cap_hits), pair,
                               P.start_bits + kLowBits) +
              (unsigned long long)pair * unsigned(P.head);
  flush(P, Wn, pair, p, K, w);
  close_segment(P, Wn);
  put_window(P, Wn, pair, K);
}

// Emits the records of carried windows that pairs without hits can now decide.
// The stream state changes later, in commit_body, once the records are known to
// fit and, where they are sorted, to be in order (a step that overflows is
// re-run from unchanged state); a decided window leaves an entry for it.
// Nearly every pair of a served step is passed by, so a thread has the 12 bytes
// of four pairs on their way at a time, and the rest of the work is a function
// of its own, for the registers (8 M pairs: one at a time 56 us, this form 28; a
// pass that also cleared the windows 47).
__device__ void finalize_body(const StepParams& P, const unsigned long long* S) {
  if (P.ctr->overflow & ~4u) return;  // (records over their buffer are counted on)
  constexpr int kAhead = 4;
  const unsigned long long npairs = (unsigned long long)P.n_items * P.n_pat;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long pr = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x;
       pr < npairs; pr += kAhead * stride) {
    int32_t q[kAhead], pend[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const uint32_t i = uint32_t(min(pr + j * stride, npairs - 1)), it = i / P.n_pat;
      q[j] = P.pair_pool[i];
      pend[j] = P.hdr[size_t(P.items[it].slot) * P.n_pat + (i - it * P.n_pat)].pend;
    }
#pragma unroll
    for (int j = 0; j < kAhead; ++j)
      if (q[j] < 0 && pend[j] && pr + j * stride < npairs)
        decide_window(P, S, uint32_t(pr + j * stride));
  }
}

__global__ void finalize_kernel(const StepParams P, const unsigned long long* __restrict__ S) {
  finalize_body(P, S);
}

// The step's new windows into the stream state.
__device__ void commit_body(const StepParams& P) {
  if (P.ctr->overflow) return;
  const unsigned long long n = P.ctr->n_pool;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long q = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; q < n;
       q += stride) {
    const uint32_t pair = P.pool_pair[q];
    const uint32_t p = pair % P.n_pat, slot = P.items[pair / P.n_pat].slot;
    MemRow* rows = P.mem + size_t(slot) * P.mem_stride + P.mem_off[p];
    P.hdr[size_t(slot) * P.n_pat + p] = P.pool_hdr[q];
    for (int lv = 0; lv <= P.K[p]; ++lv) rows[lv] = P.pool_mem[q * (kMaxK + 1) + lv];
  }
}

__device__ void tails_body(const StepParams& P) {
  if (P.ctr->overflow) return;
  for (uint32_t i = blockIdx.x; i < P.n_items; i += gridDim.x) {
    const WorkItem w = P.items[i];
    if (w.eos) continue;
    const int64_t nt = min(w.e_new, int64_t(P.T));
    const uint8_t* src = P.arena + w.arena_base + (w.e_new - nt - w.base_pos);
    uint8_t* dst = P.tails + size_t(w.slot) * P.T;
    for (int64_t b = threadIdx.x; b < nt; b += blockDim.x) dst[b] = src[b];
  }
}

__global__ void state_kernel(const StepParams P) {
  commit_body(P);
  tails_body(P);
}

// Run boundaries of the canonically sorted records: the records of work item
// w are [start[w], start[w + 1]), the first index whose key belongs to a pair
// of item w or later (binary search over the sorted keys; pair = item x n_pat
// + pattern sits above bit `shift`).  start[n_items] = the record count.
__global__ void runs_kernel(const unsigned long long* __restrict__ keys,
                            const unsigned long long* count, unsigned long long cap,
                            uint32_t n_items, uint32_t n_pat, int shift,
                            unsigned long long* __restrict__ start) {
  const uint32_t w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w > n_items) return;
  const unsigned long long n = min(*count, cap);
  if (w == n_items) {
    start[w] = n;
    return;
  }
  const unsigned long long first_pair = (unsigned long long)w * n_pat;
  unsigned long long lo = 0, hi = n;  // first index with pair >= first_pair
  while (lo < hi) {
    const unsigned long long mid = (lo + hi) >> 1;
    if ((keys[mid] >> shift) < first_pair)
      lo = mid + 1;
    else
      hi = mid;
  }
  start[w] = lo;
}

// ------------------------------------------------- ordered records
// Exclusive scan of the segment counts seg[0, N] in place, N = hits + pairs
// x head (seg[N] = 0 before: it becomes the record total), as three kernels:
// per-block sums, a scan of those sums, and a per-block rescan from its
// offset.  Each block owns a contiguous chunk of kScanTile-element tiles.
constexpr int kScanThreads = 256;
constexpr int kScanPer = 4;  // elements per thread and tile (one 16-byte load)
constexpr int kScanTile = kScanThreads * kScanPer;
constexpr int kScanMaxBlocks = 1024;

__device__ __forceinline__ unsigned long long seg_count(const StepParams& P) {
  return min(P.ctr->n_hits, P.cap_hits) +
         (unsigned long long)P.n_items * P.n_pat * unsigned(P.head) + 1;
}

__device__ __forceinline__ unsigned long long scan_chunk(unsigned long long n) {
  const unsigned long long tiles = (n + kScanTile - 1) / kScanTile;
  return (tiles + gridDim.x - 1) / gridDim.x * kScanTile;
}

__device__ void seg_reduce_body(const StepParams& P, unsigned long long* part) {
  __shared__ unsigned long long ws[kScanThreads / 32];
  const unsigned long long n = seg_count(P);
  const unsigned long long chunk = scan_chunk(n);
  const unsigned long long b0 = chunk * blockIdx.x, b1 = min(n, b0 + chunk);
  unsigned long long acc = 0;
  // seg is zero-filled to a whole tile past n: whole 16-byte loads
  for (unsigned long long i = b0 + threadIdx.x * kScanPer; i < b1; i += kScanTile) {
    const uint4 v = *reinterpret_cast<const uint4*>(P.seg + i);
    acc += (unsigned long long)v.x + v.y + v.z + v.w;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(kFull, acc, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int w = 0; w < kScanThreads / 32; ++w) t += ws[w];
    part[blockIdx.x] = t;
  }
}

__global__ void __launch_bounds__(kScanThreads)
    seg_reduce_kernel(const StepParams P, unsigned long long* __restrict__ part) {
  seg_reduce_body(P, part);
}

// One block: exclusive offsets of the block sums; the total is the record
// count (checked against the output capacity).
__global__ void __launch_bounds__(kScanMaxBlocks)
    seg_top_kernel(const StepParams P, unsigned long long* __restrict__ part, int nblocks) {
  __shared__ unsigned long long ws[kScanMaxBlocks / 32];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned long long v = t < nblocks ? part[t] : 0ull;
  unsigned long long incl = v;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long u = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += u;
  }
  if (lane == 31) ws[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    unsigned long long x = ws[lane];
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long u = __shfl_up_sync(kFull, x, o);
      if (lane >= o) x += u;
    }
    ws[lane] = x;  // inclusive sums of the warps
  }
  __syncthreads();
  const unsigned long long before = (warp ? ws[warp - 1] : 0ull) + incl - v;
  if (t < nblocks) part[t] = before;
  if (t == kScanMaxBlocks - 1) {
    const unsigned long long total = before + v;
    P.ctr->n_out = total;
    if (total > P.cap_out) atomicOr(&P.ctr->overflow, 4u);
  }
}

__device__ void seg_down_body(const StepParams& P, uint32_t run) {
  __shared__ uint32_t ws[kScanThreads / 32];
  __shared__ uint32_t tile_total;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const unsigned long long n = seg_count(P);
  const unsigned long long chunk = scan_chunk(n);
  const unsigned long long b0 = chunk * blockIdx.x, b1 = min(n, b0 + chunk);
  for (unsigned long long base = b0; base < b1; base += kScanTile) {
    const unsigned long long i = base + unsigned(t) * kScanPer;
    uint4 v = *reinterpret_cast<const uint4*>(P.seg + i);
    const uint32_t s = v.x + v.y + v.z + v.w;
    uint32_t incl = s;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t u = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += u;
    }
    if (lane == 31) ws[warp] = incl;
    __syncthreads();
    if (t == 0) {
      uint32_t acc = 0;
      for (int w = 0; w < kScanThreads / 32; ++w) {
        const uint32_t c = ws[w];
        ws[w] = acc;
        acc += c;
      }
      tile_total = acc;
    }
    __syncthreads();
    uint32_t e = run + ws[warp] + incl - s;
    const uint32_t a = v.x, b = v.y, c = v.z;
    v.x = e;
    v.y = e += a;
    v.z = e += b;
    v.w = e + c;
    if (i < b1) {
      if (i + kScanPer <= b1) {
        *reinterpret_cast<uint4*>(P.seg + i) = v;
      } else {
        const uint32_t o4[4] = {v.x, v.y, v.z, v.w};
        for (int q = 0; q < kScanPer && i + q < b1; ++q) P.seg[i + q] = o4[q];
      }
    }
    run += tile_total;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kScanThreads)
    seg_down_kernel(const StepParams P, const unsigned long long* __restrict__ part) {
  seg_down_body(P, uint32_t(part[blockIdx.x]));  // offsets fit 32 bits (cap_out does)
}

// Segment c holds seg[c + 1] - seg[c] records at rtmp[c ...): they go to
// the output at seg[c].
__device__ void compact_body(const StepParams& P, DevHit* dst) {
  const unsigned long long n = seg_count(P) - 1;
  const unsigned long long stride = (unsigned long long)gridDim.x * blockDim.x;
  for (unsigned long long c = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x; c < n;
       c += stride) {
    const uint32_t a = P.seg[c], b = P.seg[c + 1];
    if (b <= a || b > P.cap_out) continue;
    const uint4* src = reinterpret_cast<const uint4*>(P.rtmp + c);
    uint4* out = reinterpret_cast<uint4*>(dst + a);
    for (uint32_t q = 0; q < 2 * (b - a); ++q) out[q] = src[q];
  }
}

__global__ void compact_kernel(const StepParams P, DevHit* __restrict__ dst) {
  compact_body(P, dst);
}

// start[w] = the first output record of work item w: the offset of the head
// segment of its first pair (w x n_pat); start[n_items] = the record count.
__device__ void runs_ordered_body(const StepParams& P, const unsigned long long* S,
                                  unsigned long long* start) {
  const unsigned long long n = seg_count(P) - 1;
  for (uint32_t w = blockIdx.x * blockDim.x + threadIdx.x; w <= P.n_items;
       w += gridDim.x * blockDim.x) {
    if (w == P.n_items) {
      start[w] = P.seg[n];
      continue;
    }
    const unsigned long long pr = (unsigned long long)w * P.n_pat;
    const unsigned long long h =
        pair_lower_bound(S, min(P.ctr->n_hits, P.cap_hits), pr, P.start_bits + kLowBits);
    start[w] = P.seg[h + pr * unsigned(P.head)];
  }
}

__global__ void runs_ordered_kernel(const StepParams P, const unsigned long long* __restrict__ S,
                                    unsigned long long* __restrict__ start) {
  runs_ordered_body(P, S, start);
}

// ------------------------------------------------- small steps
// Everything after the candidates of a small step (filtered output, ordered
// records) in one cooperative launch: verification, the hit sort, the filter,
// the carried windows, the records' offsets, and the new state, with bounded
// grid barriers between them.  As launches of their own these are a dozen
// kernels of 3 to 14 us and two fills, with a gap after each and 2 us of the
// host before it; small steps are made of that.  The counters, each stream's
// first record and, if there are at most direct_cap, the records go straight
// to pinned host memory.
// A step of one motif over 1,500 bytes: 125 -> 73 us a call.
template <bool kWeighted>
__global__ void __launch_bounds__(kSortThreads, 2)
    small_step_kernel(const StepParams P, const SmallStep A) {
  extern __shared__ __align__(16) unsigned char sort_smem[];
  SortSmem& sm = *reinterpret_cast<SortSmem*>(sort_smem);
  __shared__ unsigned long long before_s, total_s;
  unsigned int target = 0;
  const unsigned long long me = (unsigned long long)blockIdx.x * blockDim.x + threadIdx.x,
                           all = (unsigned long long)gridDim.x * blockDim.x;
  // (after a wait that ran out the host finds no counters, and runs the step
  // again as separate launches: the state is as it was, see sort_barrier)
  auto meet = [&]() { return sort_barrier(sm, A.bar, target += gridDim.x, A.bound, P.ctr); };
  auto leave = [&]() {
    if (me != 0) return;
    StepCounters c = *P.ctr;
    c.overflow |= kSmallLeft;
    *A.counters = c;
  };
  for (unsigned long long i = me; i < (unsigned long long)P.n_items * P.n_pat; i += all)
    P.pair_pool[i] = -1;
  for (unsigned long long i = me; i < A.seg_len / 4; i += all)
    reinterpret_cast<uint4*>(P.seg)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (P.ctr->n_cand > A.max_cand) return leave();
  verify_body<kWeighted>(P);
  if (!meet()) return;
  if (__ldcg(&P.ctr->n_hits) > A.max_hits) return leave();
  sort_body(sm, P.keys, P.keys_alt, nullptr, nullptr, &P.ctr->n_hits, P.cap_hits, A.lo_bit,
            A.hi_bit, A.hist, A.sort_bar, A.bound, P.ctr);
  if (!meet()) return;
  filter_body(P, A.sorted);
  if (!meet()) return;
  finalize_body(P, A.sorted);
  if (!meet()) return;
  seg_reduce_body(P, A.part);
  if (!meet()) return;
  if (threadIdx.x < 32) {  // the sums of the blocks before this one, and of all
    unsigned long long b = 0, t = 0;
    for (unsigned int q = threadIdx.x; q < gridDim.x; q += 32) {
      const unsigned long long v = __ldcg(A.part + q);
      t += v;
      if (q < blockIdx.x) b += v;
    }
    for (int o = 16; o > 0; o >>= 1) {
      b += __shfl_down_sync(kFull, b, o);
      t += __shfl_down_sync(kFull, t, o);
    }
    if (threadIdx.x == 0) {
      before_s = b;
      total_s = t;
    }
  }
  __syncthreads();
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    P.ctr->n_out = total_s;
    if (total_s > P.cap_out) atomicOr(&P.ctr->overflow, 4u);
  }
  seg_down_body(P, uint32_t(before_s));
  if (!meet()) return;
  commit_body(P);
  tails_body(P);
  compact_body(P, total_s <= A.direct_cap ? A.direct : A.dst);
  runs_ordered_body(P, A.sorted, A.run_start);
  if (blockIdx.x == 0 && threadIdx.x == 0) *A.counters = *P.ctr;
}

int grid_for(unsigned long long n, int threads, int cap_blocks) {
  unsigned long long b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > (unsigned long long)cap_blocks) b = cap_blocks;
  return int(b);
}

}  // namespace

cudaError_t launch_gather(const CopyChunk* chunks, int n, bool short_chunks, uint8_t* arena,
                          cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (short_chunks)
    gather_kernel<true><<<min((n + 7) / 8, 65535), 256, 0, s>>>(chunks, n, arena);
  else
    gather_kernel<false><<<min(n, 65535), 256, 0, s>>>(chunks, n, arena);
  return cudaGetLastError();
}

cudaError_t launch_verify(const StepParams& p, cudaStream_t s) {
  // the candidate count lives on the device: size for the capacity, loop inside
  const int grid = grid_for(p.cap_cand, 256, p.num_sms * 16);
  if (p.weighted) verify_kernel<true><<<grid, 256, 0, s>>>(p);
  else verify_kernel<false><<<grid, 256, 0, s>>>(p);
  return cudaGetLastError();
}

int sort_grid(int num_sms) {
  int per_sm = 0;
  if (cudaFuncSetAttribute(sort_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           int(sizeof(SortSmem))) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, sort_kernel, kSortThreads,
                                                    sizeof(SortSmem)) != cudaSuccess)
    return 0;
  return std::min(per_sm, 4) * num_sms;
}

int small_step_grid(int num_sms) {
  for (auto* kernel : {small_step_kernel<false>, small_step_kernel<true>}) {
    int per_sm = 0;
    if (cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             int(sizeof(SortSmem))) != cudaSuccess ||
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kSortThreads,
                                                      sizeof(SortSmem)) != cudaSuccess ||
        per_sm < 1) {
      cudaGetLastError();  // (the next launch reads it otherwise)
      return 0;
    }
  }
  return num_sms;
}

cudaError_t launch_small_step(const StepParams& p, SmallStep a, int nblocks, cudaStream_t s) {
  a.seg_len = ordered_seg_len(p.cap_rtmp);
  a.lo_bit = kKBits;
  a.hi_bit = p.key_bits;
  a.sorted = (((a.hi_bit - a.lo_bit + 7) / 8) & 1) ? p.keys_alt : p.keys;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(nblocks));
  cfg.blockDim = dim3(kSortThreads);
  cfg.dynamicSmemBytes = sizeof(SortSmem);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, p.weighted ? small_step_kernel<true> : small_step_kernel<false>,
                            p, a);
}

size_t sort_hist_len(int nblocks) {
  return size_t(kBins) * std::max(size_t(nblocks) + 1, 2 * size_t(kSortWalk));
}

cudaError_t launch_sort(const SortArgs& a, unsigned long long** keys_out, uint32_t** vals_out,
                        cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(unsigned(a.nblocks));
  cfg.blockDim = dim3(kSortThreads);
  cfg.dynamicSmemBytes = sizeof(SortSmem);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeCooperative;
  at.val.cooperative = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  const cudaError_t e =
      cudaLaunchKernelEx(&cfg, sort_kernel, a.keys, a.keys_alt, a.vals, a.vals_alt, a.count, a.cap,
                         a.lo_bit, a.hi_bit, a.hist, a.bar, a.bound, a.ctr);
  const bool odd = ((a.hi_bit - a.lo_bit + 7) / 8) & 1;
  *keys_out = odd ? a.keys_alt : a.keys;
  if (vals_out) *vals_out = odd ? a.vals_alt : a.vals;
  return e;
}

cudaError_t launch_permute(const DevHit* src, const uint32_t* idx, DevHit* dst,
                           const StepCounters* ctr, unsigned long long cap, int num_sms,
                           cudaStream_t s) {
  permute_kernel<<<grid_for(cap, 256, num_sms * 8), 256, 0, s>>>(src, idx, dst, ctr, cap);
  return cudaGetLastError();
}

cudaError_t launch_filter(const StepParams& p, const unsigned long long* sorted, cudaStream_t s) {
  const int grid = grid_for(p.cap_hits, 128, p.num_sms * 32);
  filter_kernel<<<grid, 128, 0, s>>>(p, sorted);
  return cudaGetLastError();
}

cudaError_t launch_finalize(const StepParams& p, const unsigned long long* sorted,
                            cudaStream_t s) {
  const unsigned long long npairs = (unsigned long long)p.n_items * p.n_pat;
  finalize_kernel<<<grid_for(npairs, 256, p.num_sms * 16), 256, 0, s>>>(p, sorted);
  return cudaGetLastError();
}


int ordered_scan_blocks(int num_sms) { return std::min(kScanMaxBlocks, num_sms * 4); }

size_t ordered_seg_len(size_t cap_rtmp) {
  return (cap_rtmp + 1 + kScanTile - 1) / kScanTile * kScanTile;
}

cudaError_t launch_ordered_scan(const StepParams& p, unsigned long long* part, cudaStream_t s) {
  const int nb = ordered_scan_blocks(p.num_sms);
  seg_reduce_kernel<<<nb, kScanThreads, 0, s>>>(p, part);
  seg_top_kernel<<<1, kScanMaxBlocks, 0, s>>>(p, part, nb);
  seg_down_kernel<<<nb, kScanThreads, 0, s>>>(p, part);
  return cudaGetLastError();
}

cudaError_t launch_ordered_emit(const StepParams& p, const unsigned long long* sorted,
                                DevHit* dst, unsigned long long* run_start, cudaStream_t s) {
  compact_kernel<<<grid_for(p.cap_rtmp, 256, p.num_sms * 8), 256, 0, s>>>(p, dst);
  const uint32_t n = p.n_items + 1;
  runs_ordered_kernel<<<(n + 255) / 256, 256, 0, s>>>(p, sorted, run_start);
  return cudaGetLastError();
}

cudaError_t launch_runs(const unsigned long long* sorted_keys, const StepParams& p,
                        unsigned long long* start, cudaStream_t s) {
  const uint32_t n = p.n_items + 1;
  runs_kernel<<<(n + 255) / 256, 256, 0, s>>>(sorted_keys, &p.ctr->n_out, p.cap_out, p.n_items,
                                              p.n_pat, p.start_bits + kLowBits, start);
  return cudaGetLastError();
}

cudaError_t launch_state(const StepParams& p, cudaStream_t s) {
  if (p.n_items == 0) return cudaSuccess;
  const int windows = p.rules.output == OASM_OUT_FILTERED
                          ? grid_for(p.cap_pool, 128, p.num_sms * 8) : 1;
  state_kernel<<<std::max(int(min(p.n_items, 65535u)), windows), 128, 0, s>>>(p);
  return cudaGetLastError();
}

}  // namespace oasm
