// gram_tables.cu -- which patterns the gram index (grams.cu) takes, their
// grams, and the index's tables.
#include <cmath>

#include "context.h"

namespace oasm {

// Clocks of one SM per text symbol and forward-scan lane group, measured on a
// GB300: 5.3 for a word of Myers/Hyyro (or the cut-off scan, one word) and for
// the K = 2 automaton, 4.5 and 3.5 for the packed automata of K = 1 and K = 0,
// 6.5 for two K = 3 patterns a lane;
// 5.5 for a weighted wave-front group.
double group_cost(int W, int algo) {
  if (algo == kAlgoWeighted) return 5.5;
  if (algo == 1) return 3.5;
  if (algo == 2) return 4.5;
  if (algo == 4) return 6.5;
  return algo == kAlgoCut || algo == 3 ? 5.3 : 5.3 * W;
}

namespace {

double buckets_cost(const std::vector<Bucket>& bs) {
  double c = 0;
  for (const Bucket& b : bs)
    for (const LaneGroup& g : b.groups) c += group_cost(b.W, b.algo) / g.nseg;
  return c;
}
// Clocks of one SM per suspect (the ends kernel's first round, and both), per
// table hit (a directory look-up), and per text symbol and key length.
// (kFilter: the piece filter and the verification of its proposals, per symbol.)
constexpr double kFilter = 15.0;
constexpr double kPair = 6.0, kEnds = 25.0, kLookup = 4.0, kLength = 0.12;

constexpr int kMaxGram2 = 16, kMaxGram = 8;  // symbols of a gram: 2-bit text, bytes
constexpr int kMaxPiece = 12;                // ... of a piece that may hold an edit
constexpr int kMaxKey2 = 10, kMaxKey = 4;    // symbols that are looked up

// Grams of one key length, ordered by key (stable; three passes of 11 bits).
using GramList = std::vector<GramEntry>;

void sort_by_key(GramList& g, uint32_t mask) {
  GramList t(g.size());
  for (int shift = 0; shift < 32; shift += 11) {
    if (shift && (mask >> shift) == 0) break;
    std::vector<uint32_t> at(2049, 0u);
    for (const GramEntry& x : g) at[(((x.lo & mask) >> shift) & 2047u) + 1] += 1;
    for (int i = 0; i < 2048; ++i) at[i + 1] += at[i];
    for (const GramEntry& x : g) t[at[((x.lo & mask) >> shift) & 2047u]++] = x;
    g.swap(t);
  }
}

// The j disjoint pieces of b symbols with the smallest sum of w (w[x] = chance
// that a text position matches symbols x .. x + b - 1).  f: scratch.
double place(const std::vector<double>& w, int m, int j, int b, std::vector<double>& f,
             std::vector<int>* at) {
  // f[t][e]: the best t pieces within the first e symbols (e >= b t)
  const size_t row = size_t(m) + 1;
  f.resize(size_t(j + 1) * row);
  std::fill(f.begin(), f.begin() + row, 0.0);
  for (int t = 1; t <= j; ++t) {
    double* cur = &f[t * row];
    const double* prev = &f[(t - 1) * row];
    double best = 1e30;
    for (int e = b * t; e <= m - b * (j - t); ++e)
      cur[e] = best = std::min(best, prev[e - b] + w[e - b]);
  }
  at->assign(j, 0);
  int e = m;
  for (int t = j; t >= 1; --t) {
    const double* cur = &f[t * row];
    while (e > b * t && cur[e - 1] <= cur[e]) --e;
    e -= b;
    (*at)[t - 1] = e;
  }
  return f[j * row + m];
}

// Grams such that every string within one edit of s contains one of them, as
// (gram, its symbols, the part of s it stands for, edits between the two).  s
// without its last symbol, standing for itself, is contained in s, in s with
// its last symbol changed or missing and in s with an insertion before it; s
// without its first symbol likewise.  The rest, an edit further inside, stands
// for all of s.  (A missing symbol of a run is the run's last one, or its
// first at the start of s: the same string.)
// s: b 2-bit symbols, the first in the low bits.
template <class F>
void one_edit(uint32_t s, int b, F put) {
  auto sym = [&](int i) { return (s >> (2 * i)) & 3u; };
  auto below = [&](int i) { return s & ((1u << (2 * i)) - 1u); };
  put(below(b - 1), b - 1, 0, b - 1, 0);
  put(s >> 2, b - 1, 1, b, 0);
  int head = 0;  // last symbol of the run that s starts with
  while (head + 1 < b && sym(head + 1) == sym(0)) ++head;
  for (int i = head + 1; i + 1 < b; ++i)  // without symbol i
    if (sym(i) != sym(i + 1)) put(below(i) | ((s >> (2 * i + 2)) << (2 * i)), b - 1, 0, b, 1);
  for (int i = 1; i + 1 < b; ++i)
    for (uint32_t c = 0; c < 4; ++c)
      if (c != sym(i)) put((s & ~(3u << (2 * i))) | (c << (2 * i)), b, 0, b, 1);
  for (int i = 2; i + 1 < b; ++i)  // before symbol i
    for (uint32_t c = 0; c < 4; ++c)
      if (c != sym(i))  // (equal: the same string as an insertion after it)
        put(below(i) | (c << (2 * i)) | ((s >> (2 * i)) << (2 * i + 2)), b + 1, 0, b, 1);
}

// Whether piece t of E + 1 is half of a pair.
bool paired(int t, int E) { return t < E || (E & 1); }

}  // namespace

int build_grams(oasm_ctx* ctx, const std::vector<char>& pref, std::vector<char>& served) {
  const uint32_t n = ctx->n_pat;
  served.assign(n, 0);
  Grams& gr = ctx->grams;
  // myers_only and full_words ask for the forward scan's own forms; the keys
  // of the (end, pattern) set hold 24 pattern bits
  if (ctx->cfg.myers_only || ctx->cfg.full_words || n >= (1u << 24)) return OASM_OK;
  std::vector<double> cnt(256, 0.0);
  double tot = 0;
  int n_pref = 0;
  for (uint32_t p = 0; p < n; ++p) {
    n_pref += pref[p] != 0;
    for (uint8_t c : ctx->pats[p]) cnt[c] += 1, tot += 1;
  }
  // clocks of the scan and the filter, and of the scan per pattern
  const double scan_all = buckets_cost(ctx->buckets) + (n_pref ? kFilter : 0.0);
  const double scan_share = buckets_cost(ctx->buckets) / std::max(1, int(n) - n_pref);
  // at most four symbols that two adjacent bits tell apart: 2-bit text (other
  // symbols of the text read as one of the four; the ends run tells)
  int shift2 = -1, distinct = 0;
  for (int c = 0; c < 256; ++c) distinct += cnt[c] > 0;
  for (int s = 0; s <= 6 && distinct <= 4 && shift2 < 0; ++s) {
    int seen = 0;
    bool ok = true;
    for (int c = 0; c < 256; ++c)
      if (cnt[c] > 0) {
        const int bit = 1 << ((c >> s) & 3);
        ok = ok && !(seen & bit);
        seen |= bit;
      }
    if (ok) shift2 = s;
  }
  const bool two = shift2 >= 0;
  std::vector<double> fr(256, 0.0);  // chance of a symbol (2-bit text: of its code)
  for (int c = 0; c < 256; ++c) fr[two ? (c >> shift2) & 3 : c] += cnt[c] / tot;
  if (two)
    for (int c = 0; c < 4; ++c) fr[c] = std::max(fr[c], 1e-3);
  const oasm_costs& co = ctx->costs;
  const int cmin = ctx->weighted ? int(std::min({co.sub, co.ins, co.del})) : 1;
  GramList by_len[kMaxKey2 + 1];
  // The filter's patterns are taken all or none: one that is left keeps the
  // whole filter pass (4,096 patterns over 128 MiB with one filter pattern left
  // by a limit per pattern: 10.4 ms a step, against 3.6 ms with all taken).
  double ends_clk = 0, pref_clk = 0, pref_rate = 0, pref_looks = 0;
  bool pref_left = false;
  std::vector<double> ps, w, scratch;
  std::vector<uint8_t> sym;
  std::vector<int> at, best_at;
  for (uint32_t p = 0; p < n; ++p) {
    const int m = ctx->m[p], E = ctx->K[p] / cmin;
    sym.resize(m);
    ps.resize(m);
    for (int i = 0; i < m; ++i) {
      const uint8_t c = ctx->pats[p][i];
      sym[i] = two ? uint8_t((c >> shift2) & 3) : c;
      ps[i] = fr[sym[i]];
    }
    auto windows = [&](int b) {
      w.resize(m - b + 1);
      for (int x = 0; x + b <= m; ++x) {
        double r = 1;
        for (int i = 0; i < b; ++i) r *= ps[x + i];
        w[x] = r;
      }
    };
    // a byte piece is looked up by its rarest four symbols (and compared from
    // there on); 2-bit pieces from their start
    auto key_at = [&](int x, int b) {
      if (two || b <= kMaxKey) return x;
      int at = x;
      double least = 1e30;
      for (int y = x; y + kMaxKey <= x + b; ++y) {
        double key = 1, all = 1;
        for (int i = 0; i < kMaxKey; ++i) key *= ps[y + i];
        for (int i = y; i < x + b; ++i) all *= ps[i];
        const double cost = key * kLookup + all * kPair;
        if (cost < least) least = cost, at = y;
      }
      return at;
    };
    double best = 1e30, best_q = 0, best_look = 0;
    int best_b = 0, best_h = 0;
    bool best_edit = false;
    // (a) E + 1 pieces of h symbols, two by two: a pair of them holds at most
    // one edit, so one of its halves none, or, for even E, the last piece holds
    // none (E / 2 pairs with two edits or more leave no edit for it)
    {
      const int h = std::min(m / (E + 1), two ? kMaxGram2 : kMaxGram);
      if (h >= (two ? 5 : 3)) {
        windows(h);
        best_q = place(w, m, E + 1, h, scratch, &best_at);
        const int kb = std::min(h, two ? kMaxKey2 : kMaxKey);
        double cost = 0;
        for (int t = 0; t <= E; ++t) {
          const int x = best_at[t], y = key_at(x, h);
          double key = 1;
          for (int i = 0; i < kb; ++i) key *= ps[y + i];
          cost += key * kLookup + w[x] * (paired(t, E) ? kPair : kEnds);
          best_look += key;
        }
        best = cost;
        best_h = h;
      }
    }
    // (b) E / 2 + 1 pieces with at most one edit each (2-bit text)
    if (two && E >= 1) {
      const int j = E / 2 + 1, b = std::min(m / j, kMaxPiece);
      if (b >= 6) {
        windows(b);
        at.clear();
        place(w, m, j, b, scratch, &at);
        // deletions and changes of a uniform text symbol, about 7 b strings
        const double q = j * (b / std::pow(4.0, b - 1) + 3.0 * (b - 2) / std::pow(4.0, b) +
                              3.0 * (b - 3) / std::pow(4.0, b + 1));
        const double look = j * 7.0 * b / std::pow(4.0, std::min(b, kMaxKey2));
        const double cost = q * kEnds + look * kLookup;
        if (cost < best) {
          best = cost;
          best_b = b;
          best_at = at;
          best_edit = true;
          best_q = q;
          best_look = look;
        }
      }
    }
    if (pref[p]) {
      pref_clk += best;
      pref_left = pref_left || pref_clk > 0.7 * kFilter;
      if (pref_left) continue;
    } else if (best > 0.7 * scan_share) {
      continue;
    }
    served[p] = 1;
    gr.n_pat += 1;
    if (!pref[p]) ends_clk += best;
    (pref[p] ? pref_rate : gr.rate) += best_q;
    (pref[p] ? pref_looks : gr.looks) += best_look;
    // a gram for pattern symbols [from, to)
    auto put = [&](uint64_t sym8, int len, int from, int to, int pair) {
      if (from > 32 || m - to > 32) gr.t.any_long = 1;
      by_len[std::min(len, two ? kMaxKey2 : kMaxKey)].push_back(
          GramEntry{p | uint32_t(ctx->K[p]) << 24 | uint32_t(E) << 28, uint8_t(from),
                    uint8_t(m - to), uint8_t(pair | (to - from - len + 1) << 4), uint8_t(len),
                    uint32_t(sym8), uint32_t(sym8 >> 32)});
    };
    auto packed = [&](int x, int len) {
      uint64_t k = 0;
      for (int i = 0; i < len; ++i) k |= uint64_t(sym[x + i]) << ((two ? 2 : 8) * i);
      return k;
    };
    if (best_edit) {
      for (int x : best_at)
        one_edit(uint32_t(packed(x, best_b)), best_b,
                 [&](uint32_t u, int l, int from, int to, int edit) {
                   put(u, l, x + from, x + to, edit ? kGramEdit : 0);
                 });
    }
    // each piece, and how far its pair reaches on the other side (of which
    // kGramPair symbols tell enough: more would only make a warp's lanes wait
    // for the longest)
    for (int t = 0; !best_edit && t <= E; ++t) {
      const int y = key_at(best_at[t], best_h), to = best_at[t] + best_h;
      int pair = 0;
      if (paired(t, E))
        pair = t & 1 ? std::min(kGramPair, y - best_at[t - 1]) | kGramLeft
                     : std::min(kGramPair, best_at[t + 1] + best_h - to);
      put(packed(y, to - y), to - y, y, to, pair);
    }
  }
  if (pref_left) {
    for (GramList& g : by_len)
      g.erase(std::remove_if(g.begin(), g.end(),
                             [&](const GramEntry& e) { return pref[e.pat & 0xffffffu] != 0; }),
              g.end());
    for (uint32_t p = 0; p < n; ++p)
      if (pref[p] && served[p]) {
        served[p] = 0;
        gr.n_pat -= 1;
      }
  } else {
    ends_clk += pref_clk;
    gr.rate += pref_rate;
    gr.looks += pref_looks;
  }
  auto none = [&]() {
    served.assign(n, 0);
    gr.n_pat = 0;
    return OASM_OK;
  };
  if (!gr.n_pat) return OASM_OK;
  // per key length: a table of one bit per key (direct, or hashed to the size
  // that fits), and a directory
  struct Len {
    int len;
    uint32_t mask;
    const GramList* g;
    size_t distinct = 0;
    int bits = 10;  // log2 of the table's bits
  };
  std::vector<Len> lens;
  size_t n_grams = 0;
  for (int len = 1; len <= kMaxKey2; ++len) {
    GramList& g = by_len[len];
    if (g.empty()) continue;
    const int kb = (two ? 2 : 8) * len;
    Len L{len, kb >= 32 ? ~0u : (1u << kb) - 1u, &g};
    sort_by_key(g, L.mask);
    for (size_t i = 0; i < g.size(); ++i)
      L.distinct += i == 0 || ((g[i].lo ^ g[i - 1].lo) & L.mask) != 0;
    n_grams += g.size();
    lens.push_back(L);
  }
  // a suspect holds 24 entry bits
  if (n_grams >= (size_t(1) << 24) || lens.size() > size_t(kGramLens)) return none();
  // 2-bit keys index their table directly (all lengths together fit); a byte
  // length's table is doubled, the fullest first, while the budget lasts (256
  // bits per gram are plenty)
  auto most = [&](const Len& L) { return (size_t(1) << L.bits) >= 256 * L.distinct; };
  for (Len& L : lens)
    if (two) L.bits = 2 * L.len;
  while (!two) {
    size_t words = 0;
    Len* pick = nullptr;
    for (Len& L : lens) {
      words += std::max<size_t>(4, (size_t(1) << L.bits) / 32);
      if (!most(L) && (!pick || double(L.distinct) / double(size_t(1) << L.bits) >
                                    double(pick->distinct) / double(size_t(1) << pick->bits)))
        pick = &L;
    }
    if (!pick || words + (size_t(1) << pick->bits) / 32 > kGramMaxWords) break;
    pick->bits += 1;
  }
  std::vector<uint32_t> bits;
  std::vector<uint4> dir;
  std::vector<GramEntry> entries;
  entries.reserve(n_grams);
  double false_bits = 0;
  GramScan& a = gr.scan;
  a.n_len = int(lens.size());
  a.two_bit = two ? 1 : 0;
  a.shift2 = two ? uint32_t(shift2) : 0u;
  for (size_t li = 0; li < lens.size(); ++li) {
    const Len& L = lens[li];
    const GramList& list = *L.g;
    GramLen& g = a.len[li];
    g.mask = L.mask;
    g.mul = two ? 1u : kGramBitMul;
    g.shift = two ? 0u : uint32_t(32 - L.bits);
    g.word0 = uint32_t(bits.size());
    bits.resize(bits.size() + std::max<size_t>(4, (size_t(1) << L.bits) / 32), 0u);
    int db = 4;
    while ((size_t(1) << db) < 2 * L.distinct) ++db;
    g.dir0 = uint32_t(dir.size());
    g.dir_shift = uint32_t(32 - db);
    g.dir_mask = (1u << db) - 1u;
    g.max_probe = 0;
    dir.resize(dir.size() + (size_t(1) << db), make_uint4(0u, 0u, 0u, 0u));
    uint32_t of_key = 0;  // entries of one key, at most
    for (size_t i = 0; i < list.size();) {
      const uint32_t key = list[i].lo & L.mask, h = (key * g.mul) >> g.shift;
      const uint32_t first = uint32_t(entries.size());
      for (; i < list.size() && (list[i].lo & L.mask) == key; ++i) entries.push_back(list[i]);
      bits[g.word0 + (h >> 5)] |= 1u << (h & 31);
      uint32_t s = (key * kGramDirMul) >> g.dir_shift, pr = 0;
      while (dir[g.dir0 + s].z != 0) {
        s = (s + 1) & g.dir_mask;
        ++pr;
      }
      dir[g.dir0 + s] = make_uint4(key, first, uint32_t(entries.size()) - first, 0u);
      g.max_probe = std::max(g.max_probe, pr);
      of_key = std::max(of_key, uint32_t(entries.size()) - first);
    }
    gr.most_looks += of_key;
    if (!two) false_bits += double(L.distinct) / double(size_t(1) << L.bits);
  }
  a.n_words = uint32_t((bits.size() + 3) & ~size_t(3));
  bits.resize(a.n_words, 0u);
  gr.clk = ends_clk + kLength * double(lens.size()) + kLookup * false_bits;
  if (gr.clk > 0.7 * scan_all) return none();  // not enough to gain
  gr.all_pref = true;
  for (uint32_t p = 0; p < n; ++p) gr.all_pref = gr.all_pref && (!pref[p] || served[p]);
  auto up = [&](auto** dst, const auto& v) -> cudaError_t {
    using T = typename std::decay<decltype(v[0])>::type;
    T* d = nullptr;
    cudaError_t e = dev_alloc(&d, v.size() * sizeof(T));
    if (e != cudaSuccess) return e;
    *dst = d;
    return cudaMemcpy(d, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  };
  uint32_t* peq = nullptr;
  cudaError_t e = up(&a.bits, bits);
  if (e == cudaSuccess) e = up(&a.dir, dir);
  if (e == cudaSuccess) e = up(&gr.t.entries, entries);
  if (e == cudaSuccess) e = dev_alloc(&peq, size_t(n) * 256 * 4 * sizeof(uint32_t));
  CK(e);
  gr.t.peq_fwd = peq;
  a.entries = gr.t.entries;
  CK(launch_peq(ctx->d_bytes, ctx->d_m, n, peq, false, ctx->stream));
  return OASM_OK;
}

// Clocks per text symbol that the index saves, for the step rule.
void finish_grams(oasm_ctx* ctx) {
  Grams& gr = ctx->grams;
  gr.saved_clk = buckets_cost(ctx->buckets) - buckets_cost(gr.rest) - gr.clk +
                 (ctx->n_pref_pat && gr.all_pref ? kFilter : 0.0);
  if (gr.saved_clk <= 0) gr.n_pat = 0;
}

}  // namespace oasm
