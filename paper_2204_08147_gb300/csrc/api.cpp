// Host side of the C ABI: contexts, Hamiltonian descriptors, workspace planning and
// the orchestration of the estimator (Algorithm 1 twice, the small dense step in
// between, the Gram at the end).
#include <sched.h>

#include <algorithm>
#include <array>
#include <chrono>
#include <atomic>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <deque>
#include <functional>
#include <condition_variable>
#include <map>
#include <memory>
#include <mutex>
#include <string>
#include <thread>
#include <vector>

#include "rdm_api_internal.h"

namespace rdm {

static thread_local std::string g_last_error;

void set_error(const char* fmt, ...) {
  char buf[1024];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_last_error = buf;
}

bool sym_eig(int n, const double* a, double* w, double* vt);
bool tdense_fT(int n, int p, const double* t, int n_beta, const double* betas, double* t_min,
               double* c_out);

#define CK(call)                                                                     \
  do {                                                                               \
    cudaError_t e_ = (call);                                                         \
    if (e_ != cudaSuccess) {                                                         \
      set_error("%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
      return RDM_ECUDA;                                                              \
    }                                                                                \
  } while (0)

// ---------------------------------------------------------------- descriptors

static uint32_t site_bit(int n, int q) { return 1u << (n - 1 - q); }

rdm_status compile_model(const rdm_model* m, HostModel* out) {
  if (!m) {
    set_error("model is NULL");
    return RDM_EINVAL;
  }
  const int n = m->n_sites;
  if (n < 1 || n > 30 || m->n_sys < 0 || m->n_sys > 2 || m->n_sys >= n) {
    set_error("unsupported sizes: n_sites=%d n_sys=%d (need 1<=n_sites<=30, 0<=n_sys<=2, n_sys<n_sites)",
              n, m->n_sys);
    return RDM_EINVAL;
  }
  if (!std::isfinite(m->lambda_sb)) {
    set_error("lambda_sb is not finite");
    return RDM_EINVAL;
  }
  HostModel h;
  h.n = n;
  h.ns = m->n_sys;
  h.lambda = m->lambda_sb;
  auto at = [&](const double* t, int a, int b) { return t ? t[(size_t)a * n + b] : 0.0; };
  double bound = 0.0;
  for (int a = 0; a < n; ++a)
    for (int b = a + 1; b < n; ++b) {
      const bool sb = (a < h.ns) != (b < h.ns);
      const double s = sb ? m->lambda_sb : 1.0;
      const double jx = at(m->jx, a, b), jy = at(m->jy, a, b), jz = at(m->jz, a, b);
      if (!std::isfinite(jx) || !std::isfinite(jy) || !std::isfinite(jz)) {
        set_error("non-finite coupling at (%d,%d)", a, b);
        return RDM_EINVAL;
      }
      bound += std::fabs(s * jx) + std::fabs(s * jy) + std::fabs(s * jz);
      const uint32_t mask = site_bit(n, a) | site_bit(n, b);
      if (jx != 0.0 || jy != 0.0) {
        FlipTerm t{mask, 0u, s * (jx + jy), s * (jx - jy)};
        if (t.c_odd != 0.0 || t.c_even != 0.0) h.flips.push_back(t);
      }
      if (jz != 0.0 && s != 0.0) h.diags.push_back(DiagTerm{mask, 0u, s * jz});
    }
  for (int q = 0; q < n; ++q) {
    const double hz = m->hz ? m->hz[q] : 0.0, gx = m->gx ? m->gx[q] : 0.0;
    if (!std::isfinite(hz) || !std::isfinite(gx)) {
      set_error("non-finite field at site %d", q);
      return RDM_EINVAL;
    }
    bound += std::fabs(hz) + std::fabs(gx);
    if (gx != 0.0) h.flips.push_back(FlipTerm{site_bit(n, q), 0u, gx, gx});
    if (hz != 0.0) h.diags.push_back(DiagTerm{site_bit(n, q), 0u, hz});
  }
  h.hnorm = bound;
  *out = std::move(h);
  return RDM_OK;
}

double partner_tiles(const HostModel& h) {
  struct G {
    int n = 0;
    bool low_free = true;
    bool parity_only = false;
  };
  std::map<uint32_t, G> groups;
  const uint32_t low = (1u << kTileBits) - 1u;
  for (const FlipTerm& f : h.flips) {
    const uint32_t hi = f.mask >> kTileBits;
    if (!hi) continue;
    G& g = groups[hi];
    g.n++;
    g.low_free = g.low_free && (f.mask & low) == 0;
    g.parity_only = (f.c_odd == 0.0) != (f.c_even == 0.0);
  }
  double t = 0.0;
  for (const auto& kv : groups) t += (kv.second.low_free && kv.second.n == 1 && kv.second.parity_only) ? 0.5 : 1.0;
  return t;
}

// Masks of h with the bath bits moved: internal bath bit i takes old bit src[i].
static HostModel permute_bath(const HostModel& h, const std::vector<uint8_t>& src) {
  const int nb = h.n - h.ns;
  HostModel o = h;
  auto map = [&](uint32_t m) {
    uint32_t r = m & ~((1u << nb) - 1u);  // system bits stay
    for (int i = 0; i < nb; ++i) r |= ((m >> src[i]) & 1u) << i;
    return r;
  };
  for (FlipTerm& f : o.flips) f.mask = map(f.mask);
  for (DiagTerm& d : o.diags) d.mask = map(d.mask);
  o.bath_src = src;
  return o;
}

// Partner-tile count of flip masks `m` (parity-only flags `po`) after moving bath bit
// src[i] to bit i: the same count as partner_tiles, on bare masks (the search's inner
// loop).
static double partner_tiles_of(const std::vector<uint32_t>& m, const std::vector<char>& po,
                               const std::vector<uint8_t>& src, int nb, std::vector<std::pair<uint32_t, uint32_t>>& w) {
  w.clear();
  const uint32_t low = (1u << kTileBits) - 1u, sys = ~((1u << nb) - 1u);
  for (size_t t = 0; t < m.size(); ++t) {
    uint32_t r = m[t] & sys;
    for (int i = 0; i < nb; ++i) r |= ((m[t] >> src[i]) & 1u) << i;
    if (r >> kTileBits) w.emplace_back(r >> kTileBits, (r & low) ? 2u : (po[t] ? 0u : 1u));
  }
  std::sort(w.begin(), w.end());
  double c = 0.0;
  for (size_t i = 0; i < w.size();) {
    size_t j = i;
    while (j < w.size() && w[j].first == w[i].first) ++j;
    c += (j - i == 1 && w[i].second == 0u) ? 0.5 : 1.0;
    i = j;
  }
  return c;
}

// Local search over transpositions of bath bits, restarted from shuffled orders (a
// fixed pseudo-random sequence, so a model always gets the same order); kept only if it
// lowers the partner-tile count.
void order_bath_bits(HostModel* h) {
  const int nb = h->n - h->ns;
  if (h->n <= kTileBits || nb < 2 || nb > 30) return;
  std::vector<uint32_t> m;
  std::vector<char> po;
  for (const FlipTerm& f : h->flips) {
    m.push_back(f.mask);
    po.push_back((f.c_odd == 0.0) != (f.c_even == 0.0));
  }
  std::vector<uint8_t> cur(nb);
  for (int i = 0; i < nb; ++i) cur[i] = (uint8_t)i;
  std::vector<std::pair<uint32_t, uint32_t>> w;
  const double c0 = partner_tiles_of(m, po, cur, nb, w);
  if (c0 == 0.0 || m.empty()) return;
  // If every transposition of neighbouring bath bits maps the set of (mask, parity-only)
  // pairs onto itself, so does every permutation (they generate the symmetric group),
  // and every order has the same count: nothing to search (a field on every site, or
  // all-to-all couplings).
  {
    std::vector<std::pair<uint32_t, char>> base(m.size()), sw(m.size());
    for (size_t t = 0; t < m.size(); ++t) base[t] = {m[t], po[t]};
    std::sort(base.begin(), base.end());
    bool symmetric = true;
    for (int i = 0; i + 1 < nb && symmetric; ++i) {
      for (size_t t = 0; t < m.size(); ++t) {
        const uint32_t x = m[t], bi = (x >> i) & 1u, bj = (x >> (i + 1)) & 1u;
        sw[t] = {bi == bj ? x : x ^ ((1u << i) | (1u << (i + 1))), po[t]};
      }
      std::sort(sw.begin(), sw.end());
      symmetric = sw == base;
    }
    if (symmetric) return;
  }
  // The search below depends only on the bath size and the multiset of (mask,
  // parity-only) pairs: a structure seen before (a serving stream's chains of one length
  // with other couplings) takes the order found then.
  static std::mutex cache_mu;
  static std::map<std::vector<uint64_t>, std::vector<uint8_t>> cache;  // empty: keep the order
  std::vector<uint64_t> key{(uint64_t)nb | ((uint64_t)h->n << 8)};
  for (size_t t = 0; t < m.size(); ++t) key.push_back((uint64_t)m[t] | ((uint64_t)po[t] << 32));
  std::sort(key.begin() + 1, key.end());
  {
    std::lock_guard<std::mutex> lk(cache_mu);
    auto f = cache.find(key);
    if (f != cache.end()) {
      if (!f->second.empty()) *h = permute_bath(*h, f->second);
      return;
    }
  }
  double best = c0;
  uint64_t x = 0x9E3779B97F4A7C15ull;
  auto next = [&]() {
    x ^= x << 13;
    x ^= x >> 7;
    x ^= x << 17;
    return x;
  };
  // 8 descents (from the caller's order, then from shuffled orders), the best kept
  const int iters = (int)std::min<size_t>(20000, 4000000 / (m.size() * (size_t)nb + 1) + 200);
  std::vector<uint8_t> best_order = cur;
  for (int start = 0; start < 8; ++start) {
    if (start > 0)
      for (int i = nb - 1; i > 0; --i) std::swap(cur[i], cur[(int)(next() % (uint64_t)(i + 1))]);
    double c_run = partner_tiles_of(m, po, cur, nb, w);
    for (int it = 0; it < iters; ++it) {
      const int a = (int)(next() % (uint64_t)nb), b = (int)(next() % (uint64_t)nb);
      if (a == b) continue;
      std::swap(cur[a], cur[b]);
      const double c = partner_tiles_of(m, po, cur, nb, w);
      if (c <= c_run)
        c_run = c;
      else
        std::swap(cur[a], cur[b]);
    }
    if (c_run < best) {
      best = c_run;
      best_order = cur;
    }
  }
  {
    std::lock_guard<std::mutex> lk(cache_mu);
    if (cache.size() >= 256) cache.clear();
    cache[key] = best < c0 ? best_order : std::vector<uint8_t>{};
  }
  if (best < c0) *h = permute_bath(*h, best_order);
}

// Sorted distinct m_lo of the diagonal terms with both a high and a low part (TileDiag).
static std::vector<uint32_t> tile_diag_mlo(const HostModel& h) {
  std::vector<uint32_t> lo;
  for (const DiagTerm& d : h.diags)
    if ((d.mask >> kTileBits) != 0 && (d.mask & (uint32_t)(kTileRows - 1)) != 0)
      lo.push_back(d.mask & (uint32_t)(kTileRows - 1));
  std::sort(lo.begin(), lo.end());
  lo.erase(std::unique(lo.begin(), lo.end()), lo.end());
  return lo;
}

// Row layout of the A table (TileDiag) for the sorted groups mlo: A_q takes one entry
// per row group when its sign depends on the row group, else one entry. Returns the
// entries per tile.
static int tile_diag_layout(const std::vector<uint32_t>& mlo, uint32_t* dep, int off[8]) {
  constexpr uint32_t kRG = 1u << kTileRegShift;
  *dep = 0;
  for (uint32_t m : mlo)
    if (m & (kRG - 1)) *dep |= 1u << (m >> kTileRegShift);
  int n = 0;
  for (int q = 0; q < 8; ++q) {
    off[q] = n;
    if (q < (1 << kTileRegBits)) n += ((*dep >> q) & 1u) ? (int)kRG : 1;
  }
  return n;
}

// The order in which the tiled SpMM walks the 2^b tiles of a slice: by the number of
// set tile bits, and within one count by the ascending list of set bits in
// lexicographic order (the simplicial order of the b-cube, whose prefixes have the
// smallest vertex boundary of all sets of their size; Harper 1966). A tile's partners
// across single and paired high bits then lie in the same or a neighbouring count
// class, so the W_j tiles a slice still needs stay few enough to be kept in L2; in
// tile-index order the partner across the top bit comes half a slice later.
std::vector<uint32_t> tile_walk_order(int b) {
  std::vector<uint32_t> out;
  out.reserve((size_t)1 << b);
  for (int w = 0; w <= b; ++w) {
    std::vector<int> c(w);  // the set bits, ascending; first subset {0, .., w-1}
    for (int i = 0; i < w; ++i) c[i] = i;
    while (true) {
      uint32_t t = 0;
      for (int i = 0; i < w; ++i) t |= 1u << c[i];
      out.push_back(t);
      int i = w - 1;  // the last position that can still move right
      while (i >= 0 && c[i] == b - w + i) --i;
      if (i < 0) break;
      ++c[i];
      for (int q = i + 1; q < w; ++q) c[q] = c[q - 1] + 1;
    }
  }
  return out;
}

// Sorts the flip terms into the tiled SpMM's tables (TiledTerms). Every mask has one bit (a
// field) or two (a hop), so a term is placed by where its spins sit.
void make_term_image(const HostModel& h, TermImage* img) {
  constexpr uint32_t kRG = (1u << kTileRegShift) - 1u;  // row-group bits
  struct Coef {
    uint32_t flags = 0;
    double c[7] = {};  // cf, co[3], ce[3]
    void field(double v) {
      flags |= kPatField;
      c[0] += v;
    }
    void reg(uint32_t bit, double o, double e) {
      const int a = __builtin_ctz(bit);
      flags |= kPatReg << a;
      c[1 + a] = o;
      c[4 + a] = e;
    }
  };
  struct Lane {
    uint32_t low;
    double o, e;
  };
  struct Pattern {
    uint32_t high = 0;
    Coef k;
    std::vector<Lane> lanes;
  };
  std::map<uint32_t, Pattern> parts;  // by m_high != 0
  std::map<uint32_t, Coef> groups;    // in-tile hops of a row-group spin with register spins
  std::vector<Lane> own;
  std::vector<double> reg_coef(16, 0.0);
  img->reg_flags = 0;
  img->all_uniform = 1;
  for (const FlipTerm& f : h.flips) {
    if (f.c_odd != f.c_even) img->all_uniform = 0;
    const uint32_t high = f.mask >> kTileBits, low = f.mask & (uint32_t)(kTileRows - 1);
    const uint32_t rg = low & kRG, reg = low >> kTileRegShift;
    if (high) {
      Pattern& P = parts[high];
      P.high = high;
      if (low == 0u) {
        if (__builtin_popcount(high) == 1) {
          P.k.field(f.c_odd);
        } else {  // flat, two high spins
          P.k.c[1] = f.c_odd;
          P.k.c[4] = f.c_even;
        }
      } else if (reg) {
        P.k.reg(reg, f.c_odd, f.c_even);
      } else {
        P.lanes.push_back(Lane{low, f.c_odd, f.c_even});
      }
    } else if (rg == 0u) {
      img->reg_flags |= 1u << reg;
      reg_coef[reg] = f.c_odd;
      reg_coef[8 + reg] = f.c_even;
    } else if (reg) {
      groups[rg].reg(reg, f.c_odd, f.c_even);
    } else {
      own.push_back(Lane{low, f.c_odd, f.c_even});
    }
  }
  // the field of a row-group spin joins the spin's group (the same loads)
  for (size_t t = 0; t < own.size();) {
    auto g = groups.find(own[t].low);
    if (g != groups.end()) {
      g->second.field(own[t].o);
      own.erase(own.begin() + t);
    } else {
      ++t;
    }
  }
  // Pairable patterns: one high spin without a field, hops that are all parity-only (c_even
  // = 0: XX + YY with J^x = J^y), the same in-tile partners in every such pattern. For a
  // given tile, a pattern whose spin is down acts on the rows whose in-tile spin is up and
  // one whose spin is up on the others, so the SpMM consumes one of each together and every
  // row takes exactly one of the two loads (no idle lanes).
  auto partners_of = [&](const Pattern& P, std::vector<uint32_t>* out) -> bool {
    out->clear();
    if (__builtin_popcount(P.high) != 1 || (P.k.flags & kPatField)) return false;
    for (int a = 0; a < 3; ++a)
      if (P.k.flags & (kPatReg << a)) {
        if (P.k.c[4 + a] != 0.0 || P.k.c[1 + a] == 0.0) return false;
        out->push_back(1u << (kTileRegShift + a));
      }
    for (const Lane& t : P.lanes) {
      if (t.e != 0.0 || t.o == 0.0) return false;
      out->push_back(t.low);
    }
    std::sort(out->begin(), out->end());
    return !out->empty();
  };
  std::vector<Pattern*> pairs, singles, flats;
  std::vector<uint32_t> first, cur;
  // From the farthest partner tile (largest m_high, the likeliest L2 miss) to the nearest,
  // so the slow copies enter the SpMM's copy ring early.
  for (auto it = parts.rbegin(); it != parts.rend(); ++it) {
    Pattern& P = it->second;
    std::sort(P.lanes.begin(), P.lanes.end(), [](const Lane& x, const Lane& y) { return x.low < y.low; });
    if (P.lanes.empty() && !(P.k.flags & (kPatReg * 7u))) {
      if (P.k.flags & kPatField) {  // a field alone
        P.k.c[1] = P.k.c[4] = P.k.c[0];
        P.k.flags = 0;
      }
      flats.push_back(&P);
      continue;
    }
    const bool ok = partners_of(P, &cur);
    if (ok && first.empty()) first = cur;
    (ok && cur == first ? pairs : singles).push_back(&P);
  }
  if (pairs.size() < 2) {
    singles.insert(singles.begin(), pairs.begin(), pairs.end());
    pairs.clear();
  }
  std::vector<uint32_t> pat_high, pat_flags, lane_low, grp_low, grp_flags;
  std::vector<int> pat_start;
  std::vector<double> pat_coef, lane_coef, grp_coef;
  auto put_lane = [&](const Lane& t) {
    lane_low.push_back(t.low);
    lane_coef.push_back(t.o);
    lane_coef.push_back(t.e);
  };
  for (const Lane& t : own) put_lane(t);
  for (const auto* list : {&pairs, &singles, &flats})
    for (const Pattern* P : *list) {
      pat_high.push_back(P->high);
      pat_flags.push_back(P->k.flags);
      pat_start.push_back((int)lane_low.size());
      pat_coef.insert(pat_coef.end(), P->k.c, P->k.c + 7);
      for (const Lane& t : P->lanes) put_lane(t);
    }
  pat_start.push_back((int)lane_low.size());
  for (const auto& kv : groups) {
    grp_low.push_back(kv.first);
    grp_flags.push_back(kv.second.flags);
    grp_coef.insert(grp_coef.end(), kv.second.c, kv.second.c + 7);
  }
  // The diagonal split of the tiled SpMM: low table, K_0 terms, mixed groups by m_lo
  // (std::map keeps them in ascending m_lo, hence ascending m_lo >> kTileRegShift).
  std::vector<double> dg_low(kTileRows, 0.0);
  std::vector<uint32_t> dg_thi, dg_mlo;
  std::vector<double> dg_tc;
  std::vector<int> dg_slot{0}, dg_hstart(9, 0);
  {
    std::map<uint32_t, std::vector<const DiagTerm*>> mixed;
    std::vector<const DiagTerm*> k0;
    for (const DiagTerm& d : h.diags) {
      const uint32_t hi = d.mask >> kTileBits, lo = d.mask & (uint32_t)(kTileRows - 1);
      if (hi == 0) {
        for (uint32_t r = 0; r < (uint32_t)kTileRows; ++r)
          dg_low[r] += (__builtin_popcount(r & lo) & 1) ? -d.c : d.c;
      } else if (lo == 0) {
        k0.push_back(&d);
      } else {
        mixed[lo].push_back(&d);
      }
    }
    for (const DiagTerm* d : k0) {
      dg_thi.push_back(d->mask >> kTileBits);
      dg_tc.push_back(d->c);
    }
    dg_slot.push_back((int)dg_thi.size());
    for (auto& kv : mixed) {
      dg_mlo.push_back(kv.first);
      for (const DiagTerm* d : kv.second) {
        dg_thi.push_back(d->mask >> kTileBits);
        dg_tc.push_back(d->c);
      }
      dg_slot.push_back((int)dg_thi.size());
    }
    for (int hh = 0; hh <= 8; ++hh) {
      int g = 0;
      while (g < (int)dg_mlo.size() && (int)(dg_mlo[g] >> kTileRegShift) < hh) ++g;
      dg_hstart[hh] = g;
    }
  }
  img->dg_entries = tile_diag_layout(dg_mlo, &img->dg_dep, img->dg_off);
  const bool tiled = h.n >= kTileBits;
  img->tiled = tiled ? 1 : 0;
  img->n_part = (int)pat_high.size();
  img->n_pair = (int)pairs.size();
  img->n_single = (int)singles.size();
  img->n_lane = (int)lane_low.size();
  img->n_own = (int)own.size();
  img->n_grp = (int)grp_low.size();
  auto& b = img->bytes;
  b.clear();
  auto put = [&](const void* src, size_t n) -> size_t {
    const size_t off = (b.size() + 15) / 16 * 16;
    b.resize(off + std::max<size_t>(n, 16), 0);
    if (n) std::memcpy(b.data() + off, src, n);
    return off;
  };
  img->off_flips = put(h.flips.data(), h.flips.size() * sizeof(FlipTerm));
  img->off_diags = put(h.diags.data(), h.diags.size() * sizeof(DiagTerm));
  img->off_pat_high = put(pat_high.data(), pat_high.size() * 4);
  img->off_pat_start = put(pat_start.data(), pat_start.size() * 4);
  img->off_pat_flags = put(pat_flags.data(), pat_flags.size() * 4);
  img->off_pat_coef = put(pat_coef.data(), pat_coef.size() * 8);
  img->off_lane_low = put(lane_low.data(), lane_low.size() * 4);
  img->off_lane_coef = put(lane_coef.data(), lane_coef.size() * 8);
  img->off_grp_low = put(grp_low.data(), grp_low.size() * 4);
  img->off_grp_flags = put(grp_flags.data(), grp_flags.size() * 4);
  img->off_grp_coef = put(grp_coef.data(), grp_coef.size() * 8);
  img->off_reg_coef = put(reg_coef.data(), reg_coef.size() * 8);
  img->n_dg_groups = (int)dg_mlo.size();
  img->n_dg_terms = (int)dg_thi.size();
  img->off_dg_low = put(dg_low.data(), dg_low.size() * 8);
  img->off_dg_mlo = put(dg_mlo.data(), dg_mlo.size() * 4);
  img->off_dg_hstart = put(dg_hstart.data(), dg_hstart.size() * 4);
  img->off_dg_thi = put(dg_thi.data(), dg_thi.size() * 4);
  img->off_dg_tc = put(dg_tc.data(), dg_tc.size() * 8);
  img->off_dg_slot = put(dg_slot.data(), dg_slot.size() * 4);
  const std::vector<uint32_t> walk = tile_walk_order(tiled ? h.n - kTileBits : 0);
  img->off_tile_order = put(walk.data(), walk.size() * 4);
}

void bind_terms(const TermImage& img, char* dev, rdm_ham* ham) {
  ham->d_flips = reinterpret_cast<FlipTerm*>(dev + img.off_flips);
  ham->d_diags = reinterpret_cast<DiagTerm*>(dev + img.off_diags);
  TiledTerms& t = ham->tiled;
  t.ready = img.tiled;
  t.n_part = img.n_part;
  t.n_pair = img.n_pair;
  t.n_single = img.n_single;
  t.n_lane = img.n_lane;
  t.n_own = img.n_own;
  t.n_grp = img.n_grp;
  t.all_uniform = img.all_uniform;
  t.reg_flags = img.reg_flags;
  t.pat_high = reinterpret_cast<const uint32_t*>(dev + img.off_pat_high);
  t.pat_start = reinterpret_cast<const int*>(dev + img.off_pat_start);
  t.pat_flags = reinterpret_cast<const uint32_t*>(dev + img.off_pat_flags);
  t.pat_coef = reinterpret_cast<const double*>(dev + img.off_pat_coef);
  t.lane_low = reinterpret_cast<const uint32_t*>(dev + img.off_lane_low);
  t.lane_coef = reinterpret_cast<const double*>(dev + img.off_lane_coef);
  t.grp_low = reinterpret_cast<const uint32_t*>(dev + img.off_grp_low);
  t.grp_flags = reinterpret_cast<const uint32_t*>(dev + img.off_grp_flags);
  t.grp_coef = reinterpret_cast<const double*>(dev + img.off_grp_coef);
  t.reg_coef = reinterpret_cast<const double*>(dev + img.off_reg_coef);
  t.tile_order = reinterpret_cast<const uint32_t*>(dev + img.off_tile_order);
  TileDiag& d = t.dg;
  d.n_groups = img.n_dg_groups;
  d.n_terms = img.n_dg_terms;
  d.dep = img.dg_dep;
  for (int q = 0; q < 8; ++q) d.off[q] = img.dg_off[q];
  d.n_entries = img.dg_entries;
  d.low = reinterpret_cast<const double*>(dev + img.off_dg_low);
  d.mlo = reinterpret_cast<const uint32_t*>(dev + img.off_dg_mlo);
  d.hstart = reinterpret_cast<const int*>(dev + img.off_dg_hstart);
  d.thi = reinterpret_cast<const uint32_t*>(dev + img.off_dg_thi);
  d.tc = reinterpret_cast<const double*>(dev + img.off_dg_tc);
  d.slot_start = reinterpret_cast<const int*>(dev + img.off_dg_slot);
}

// ---------------------------------------------------------------- layout

static int ilog2_exact(int64_t x) {
  int r = 0;
  while ((int64_t(1) << r) < x) ++r;
  return (int64_t(1) << r) == x ? r : -1;
}

// Blocks per slice of the plain (untiled) kernels: enough to cover the rows once with
// kThreads / TPR rows per block, at most 1216 blocks over all slices.
static int untiled_gridx(const Layout& L) {
  const int rpb = kThreads / L.TPR;
  const int64_t gx = (L.D + rpb - 1) / rpb;
  const int64_t cap = std::max<int64_t>(1, 1216 / L.n_slices);
  return (int)std::min(gx, cap);
}

// Chooses the slice geometry for n_v bath vectors of block size d_s.
rdm_status plan_layout(const HostModel& h, int n_v, int precision, Layout* L, int* n_v_pad, int rec_ds) {
  if (precision != RDM_FP32 && precision != RDM_FP64) {
    set_error("precision must be RDM_FP32 or RDM_FP64");
    return RDM_EINVAL;
  }
  Layout l{};
  l.n_bits = h.n;
  l.n_bath_bits = h.n - h.ns;
  l.D = int64_t(1) << h.n;
  l.DS = rec_ds > 0 ? rec_ds : 1 << h.ns;  // block size of one recurrence
  l.precision = precision;
  l.elem = precision == RDM_FP32 ? 4 : 8;
  l.VW = precision == RDM_FP32 ? 4 : (l.DS == 4 ? 4 : 2);
  int cols = (1 << h.ns) * n_v;
  int bcols;
  if ((16 * kTiledLanes / l.elem) % l.DS == 0 && h.n >= kTileBits) {
    // tiled layout: narrow slices of kTiledLanes 16-byte vectors per row (32 bytes)
    const int sc = 16 * kTiledLanes / l.elem;
    bcols = (cols + sc - 1) / sc * sc;
    l.Bs = sc;
  } else if (cols >= 128 / l.elem) {
    const int slice_cols = 128 / l.elem;  // 128-byte rows per slice
    bcols = (cols + slice_cols - 1) / slice_cols * slice_cols;
    l.Bs = slice_cols;
  } else {
    bcols = l.VW;
    while (bcols < cols) bcols *= 2;
    l.Bs = bcols;
  }
  l.B = bcols;
  l.n_slices = l.B / l.Bs;
  l.TPR = l.Bs / l.VW;
  l.gridx = untiled_gridx(l);
  if (layout_tiled(l)) l.gridx = spmm_tiled_grid(l);  // the tiled SpMM's blocks per slice
  *L = l;
  *n_v_pad = l.B / l.DS;
  return RDM_OK;
}

// Layout of a caller's single-slice block of n_cols columns (apply / starting block).
static rdm_status plan_single(const HostModel& h, int n_cols, int precision, int ds, Layout* L) {
  if (precision != RDM_FP32 && precision != RDM_FP64) {
    set_error("bad precision %d (RDM_FP64 or RDM_FP32)", precision);
    return RDM_EINVAL;
  }
  Layout l{};
  l.n_bits = h.n;
  l.n_bath_bits = h.n - h.ns;
  l.D = int64_t(1) << h.n;
  l.DS = ds;
  l.precision = precision;
  l.elem = precision == RDM_FP32 ? 4 : 8;
  l.VW = precision == RDM_FP32 ? 4 : (ds == 4 ? 4 : 2);
  const int maxc = 128 / l.elem;
  if (n_cols < l.VW || n_cols > maxc || ilog2_exact(n_cols / l.VW) < 0 || n_cols % l.VW) {
    set_error("n_cols=%d unsupported: need %d * 2^m columns, at most %d", n_cols, l.VW, maxc);
    return RDM_EINVAL;
  }
  l.B = l.Bs = n_cols;
  l.n_slices = 1;
  l.TPR = n_cols / l.VW;
  const int rpb = kThreads / l.TPR;
  l.gridx = (int)std::min<int64_t>((l.D + rpb - 1) / rpb, 1216);
  *L = l;
  return RDM_OK;
}

// ---------------------------------------------------------------- workspace

struct Arena {
  char* base = nullptr;
  size_t cap = 0, off = 0;
  template <typename T>
  T* take(size_t count) {
    const size_t a = 256;
    off = (off + a - 1) / a * a;
    T* p = reinterpret_cast<T*>(base + off);
    off += count * sizeof(T);
    return p;
  }
};

struct Plan {
  Layout L;   // the recurrences' layout (block size d_s, or 1 per column when single)
  Layout Lg;  // the same memory grouped by d_s columns: the Gram view
  bool single;                        // one block-size-1 recurrence per column
  int n_v, n_v_pad, k, n_beta, nbc;  // nbc: betas per pass-2 sweep
  int nsc = 0;                        // pass 2: slices per sweep (0: all of them)
  bool gauss;                         // Gaussian bath vectors are generated once into a buffer
  bool store;                         // keep all k+1 Krylov blocks (no second pass)
  size_t tk_bytes;                    // K table of the tiled diagonal (0 if untiled)
  bool dev_dense;                     // the small dense step can run on the device
  int vstride;                        // its Chebyshev degree bound + 1
};

// Float64 counts of the arrays whose size depends on the grouping: reduction partials (the
// recurrences' kernels take one grid's at a time, the Gram kernels gram1 for each beta of a
// launch, as many betas as there is room for), the E coefficients of a beta chunk and the
// Gram results of a chunk, each large enough for the recurrences' layout and for the Gram
// view.
struct PlanSizes {
  size_t partials, gram1, e, gram;
};
static PlanSizes plan_sizes(const Plan& p) {
  const Layout& L = p.L;
  const Layout& G = p.Lg;
  const size_t rec = (size_t)L.n_groups() * L.DS * L.DS, view = (size_t)G.n_groups() * G.DS * G.DS;
  // (the packed first pass runs the untiled grid on a tiled layout: room for both)
  const size_t prec = (size_t)L.n_slices * std::max(L.gridx, untiled_gridx(L)) * L.groups_per_slice() * L.DS * L.DS;
  const size_t per_block = (size_t)G.n_slices * G.groups_per_slice() * G.DS * G.DS;
  const size_t gram1 = per_block * gram_gridx(G);
  return PlanSizes{std::max(gram1, 8 * std::max(prec, per_block * G.gridx)), gram1,
                   (size_t)p.k * p.nbc * std::max(rec, view), (size_t)p.nbc * std::max(rec, view)};
}

static size_t plan_bytes(const Plan& p) {
  Arena a;  // dry run: only offsets
  const Layout& L = p.L;
  const size_t ng = L.n_groups(), nv = (size_t)L.DS * L.DS;
  const PlanSizes z = plan_sizes(p);
  a.take<char>(L.block_bytes() * (p.store ? (size_t)p.k + 1 : 3));
  if (!p.store) a.take<char>(L.block_bytes() / (size_t)L.n_slices * (size_t)(p.nsc ? p.nsc : L.n_slices) * p.nbc);
  a.take<double>(z.partials);
  a.take<double>((size_t)(p.k + 2) * ng * nv * 3);
  a.take<double>((size_t)p.k * ng * nv * 2);
  a.take<double>(z.e);
  a.take<double>(z.gram);
  a.take<double>((size_t)p.n_v_pad * 65);
  a.take<uint32_t>(4);
  a.take<char>(p.tk_bytes);
  if (p.gauss) a.take<char>((size_t)p.n_v * ((size_t)1 << L.n_bath_bits) * L.elem);
  if (p.gauss) a.take<double>((size_t)p.n_v * ((size_t)1 << L.n_bath_bits));  // raw Gaussians
  if (p.dev_dense) {  // device small dense step: bounds, Chebyshev vectors, results, betas
    const size_t ne = (size_t)p.k * L.DS * L.DS;
    a.take<double>(2 * ng);
    a.take<double>(ng * (size_t)p.vstride * ne);
    a.take<double>(ng * (size_t)p.n_beta * ne);
    a.take<double>((size_t)p.n_beta);
    a.take<char>(dense_jobs_bytes(1));
  }
  return a.off + 256;
}

// beta_max: the largest beta of the grid (< 0: unknown, plan for the largest degree).
// dense: plan room for the device small dense step if it fits the recurrences.
static rdm_status make_plan_impl(const HostModel& hm, int n_beta, int n_v, int k, const rdm_opts* o,
                                 size_t avail, Plan* out, double beta_max, bool dense) {
  if (n_beta < 1 || n_v < 1 || n_v > 4096 || k < 1 || k > kMaxSteps) {
    set_error("need n_beta >= 1, 1 <= n_v <= 4096, 1 <= k <= %d (got %d, %d, %d)", kMaxSteps, n_beta, n_v, k);
    return RDM_EINVAL;
  }
  if (o->recurrence != RDM_BLOCK && o->recurrence != RDM_SINGLE) {
    set_error("recurrence must be RDM_BLOCK or RDM_SINGLE");
    return RDM_EINVAL;
  }
  Plan p{};
  p.single = o->recurrence == RDM_SINGLE && hm.ns > 0;
  rdm_status st = plan_layout(hm, n_v, o->precision, &p.L, &p.n_v_pad, p.single ? 1 : -1);
  if (st != RDM_OK) return st;
  p.Lg = p.L;
  if (p.single) {
    p.Lg.DS = 1 << hm.ns;
    if (p.L.VW % p.Lg.DS != 0) {
      set_error("RDM_SINGLE needs whole d_s-column groups per 16-byte vector (float32, or "
                "float64 with d_s <= 2)");
      return RDM_EINVAL;
    }
  }
  p.n_v = n_v;
  p.k = k;
  p.n_beta = n_beta;
  p.nbc = 1;
  p.gauss = o->vec_dist == RDM_GAUSS;
  p.store = false;
  p.dev_dense = dense && dense_device_fits(k, p.L.DS);
  // (rounded up to a multiple of 32, so Hamiltonians with nearby norm bounds plan the
  // same workspace)
  p.vstride = std::min(kChebMaxDegree + 1,
                       ((beta_max < 0 ? kChebMaxDegree : dense_device_max_degree(beta_max, hm.hnorm)) + 32) / 32 * 32);
  if (layout_tiled(p.L)) {
    uint32_t dep;
    int off[8];
    const int n_entries = tile_diag_layout(tile_diag_mlo(hm), &dep, off);
    p.tk_bytes = (size_t)(p.L.D >> kTileBits) * (size_t)tile_diag_stride(n_entries, p.L.elem) *
                 (size_t)p.L.elem;
  } else {
    p.tk_bytes = 0;
  }
  if (o->passes != RDM_PASSES_RECOMPUTE) {
    Plan q = p;
    q.store = true;
    q.nbc = n_beta;
    if (gram_stored_max_betas(q.Lg, k) >= 1 && plan_bytes(q) <= avail) {
      *out = q;
      return RDM_OK;
    }
    if (o->passes == RDM_PASSES_STORE) {
      set_error("storing %d Krylov blocks needs %zu bytes of device memory, %zu available", k + 1,
                plan_bytes(q), avail);
      return RDM_ENOMEM;
    }
  }
  if (plan_bytes(p) > avail) {
    set_error("estimate needs %zu bytes of device memory, %zu available", plan_bytes(p), avail);
    return RDM_ENOMEM;
  }
  while (p.nbc < n_beta) {
    Plan q = p;
    q.nbc = p.nbc + 1;
    if (plan_bytes(q) > avail) break;
    p = q;
  }
  // Fewer betas per sweep than the grid: every sweep repeats the whole recurrence for
  // every bath vector. Sweeps over groups of slices (of bath vectors) with all betas
  // repeat none of it, and the same memory holds psi for all betas of fewer slices.
  if (p.nbc < n_beta && !p.single && p.L.n_slices > 1) {
    Plan q = p;
    q.nbc = n_beta;
    int best = 0;
    for (int ns = 1; ns < p.L.n_slices; ++ns) {
      q.nsc = ns;
      if (plan_bytes(q) > avail) break;
      best = ns;
    }
    if (best > 0) {
      q.nsc = best;
      p = q;
    }
  }
  *out = p;
  return RDM_OK;
}

// The plan with the device small dense step when its arrays fit beside the rest, else
// the plan without it (the host step needs no device memory).
static rdm_status make_plan(const HostModel& hm, int n_beta, int n_v, int k, const rdm_opts* o,
                            size_t avail, Plan* out, double beta_max = -1.0) {
  rdm_status st = make_plan_impl(hm, n_beta, n_v, k, o, avail, out, beta_max, true);
  if (st == RDM_ENOMEM || (st == RDM_OK && out->dev_dense && o->passes == RDM_PASSES_AUTO && !out->store)) {
    Plan q;
    const rdm_status s2 = make_plan_impl(hm, n_beta, n_v, k, o, avail, &q, beta_max, false);
    // keep the stored basis (or any plan at all) rather than the device step
    if (s2 == RDM_OK && (st != RDM_OK || q.store)) {
      *out = q;
      return RDM_OK;
    }
  }
  return st;
}

size_t estimate_bytes(const HostModel& h, int n_beta, int n_v, int k, const rdm_opts* o, size_t avail,
                      rdm_status* status, double beta_max) {
  Plan p;
  const rdm_status st = make_plan(h, n_beta, n_v, k, o, avail, &p, beta_max);
  if (status) *status = st;
  if (st != RDM_OK) return 0;
  return plan_bytes(p);
}

size_t estimate_footprint(const HostModel& h, int n_beta, int n_v, int k, int precision, int dist,
                          int passes, int nbc, int recurrence, double beta_max) {
  rdm_opts o{precision, dist, RDM_GRAM,
             passes == RDM_PASSES_STORE ? RDM_PASSES_STORE : RDM_PASSES_RECOMPUTE, 0, recurrence};
  Plan p;
  if (make_plan(h, n_beta, n_v, k, &o, SIZE_MAX, &p, beta_max) != RDM_OK) return 0;
  if (!p.store) p.nbc = std::max(1, std::min(nbc, n_beta));
  return plan_bytes(p);
}

}  // namespace rdm

using namespace rdm;

// ---------------------------------------------------------------- ABI: context

extern "C" const char* rdm_last_error(void) { return g_last_error.c_str(); }

extern "C" rdm_status rdm_create(rdm_ctx** out, int device, void* stream) {
  if (!out) {
    set_error("rdm_create: out is NULL");
    return RDM_EINVAL;
  }
  *out = nullptr;
  int ndev = 0;
  CK(cudaGetDeviceCount(&ndev));
  if (device < 0 || device >= ndev) {
    set_error("rdm_create: device %d out of range (%d devices)", device, ndev);
    return RDM_EINVAL;
  }
  CK(cudaSetDevice(device));
  std::unique_ptr<rdm_ctx> c(new rdm_ctx());
  c->device = device;
  if (stream) {
    c->stream = reinterpret_cast<cudaStream_t>(stream);
    c->owns_stream = false;
  } else {
    CK(cudaStreamCreateWithFlags(&c->stream, cudaStreamNonBlocking));
    c->owns_stream = true;
  }
  *out = c.release();
  return RDM_OK;
}

extern "C" void rdm_destroy(rdm_ctx* ctx) {
  if (!ctx) return;
  rdm_serve_stop(ctx);
  cudaSetDevice(ctx->device);
  cudaStreamSynchronize(ctx->stream);
  if (ctx->own_ws) cudaFree(ctx->own_ws);
  if (ctx->owns_stream) cudaStreamDestroy(ctx->stream);
  delete ctx;
}

extern "C" rdm_status rdm_set_workspace(rdm_ctx* ctx, void* ptr, size_t bytes) {
  if (!ctx) {
    set_error("rdm_set_workspace: ctx is NULL");
    return RDM_EINVAL;
  }
  if (ptr && (reinterpret_cast<uintptr_t>(ptr) % 256 != 0)) {
    set_error("rdm_set_workspace: pointer must be 256-byte aligned");
    return RDM_EINVAL;
  }
  ctx->ws = ptr ? reinterpret_cast<char*>(ptr) : nullptr;
  ctx->ws_bytes = ptr ? bytes : 0;
  return RDM_OK;
}

extern "C" rdm_status rdm_synchronize(rdm_ctx* ctx) {
  if (!ctx) {
    set_error("rdm_synchronize: ctx is NULL");
    return RDM_EINVAL;
  }
  CK(cudaSetDevice(ctx->device));
  CK(cudaStreamSynchronize(ctx->stream));
  return RDM_OK;
}

// ---------------------------------------------------------------- ABI: model

extern "C" rdm_status rdm_build_hamiltonian(rdm_ctx* ctx, const rdm_model* model, rdm_ham** out) {
  if (!ctx || !out) {
    set_error("rdm_build_hamiltonian: ctx and out must be non-NULL");
    return RDM_EINVAL;
  }
  *out = nullptr;
  HostModel hm;
  rdm_status st = compile_model(model, &hm);
  if (st != RDM_OK) return st;
  HostModel caller_order;
  if (ctx->bath_order) {
    caller_order = hm;
    order_bath_bits(&hm);
  }
  CK(cudaSetDevice(ctx->device));
  auto upload = [&](HostModel&& m, rdm_ham** o) -> rdm_status {
    std::unique_ptr<rdm_ham> h(new rdm_ham());
    h->ctx = ctx;
    h->device = ctx->device;
    h->model = std::move(m);
    TermImage img;
    make_term_image(h->model, &img);
    CK(cudaMalloc(&h->d_terms, img.bytes.size()));
    bind_terms(img, reinterpret_cast<char*>(h->d_terms), h.get());
    CK(cudaMemcpyAsync(h->d_terms, img.bytes.data(), img.bytes.size(), cudaMemcpyHostToDevice,
                       ctx->stream));
    CK(cudaStreamSynchronize(ctx->stream));
    *o = h.release();
    return RDM_OK;
  };
  const bool reordered = !hm.bath_src.empty();
  rdm_ham* h = nullptr;
  st = upload(std::move(hm), &h);
  if (st != RDM_OK) return st;
  if (reordered) {
    st = upload(std::move(caller_order), &h->caller);
    if (st != RDM_OK) {
      rdm_destroy_hamiltonian(h);
      return st;
    }
  }
  *out = h;
  return RDM_OK;
}

extern "C" rdm_status rdm_set_spmm_form(rdm_ctx* ctx, int form) {
  if (!ctx) {
    set_error("rdm_set_spmm_form: NULL context");
    return RDM_EINVAL;
  }
  if (form < 0 || form > 2) {
    set_error("rdm_set_spmm_form: form must be 0, 1 or 2");
    return RDM_EINVAL;
  }
  ctx->spmm_form = form;
  return RDM_OK;
}

extern "C" rdm_status rdm_set_packed_form(rdm_ctx* ctx, int form) {
  if (!ctx) {
    set_error("rdm_set_packed_form: NULL context");
    return RDM_EINVAL;
  }
  if (form < 0 || form > 2) {
    set_error("rdm_set_packed_form: form must be 0, 1 or 2");
    return RDM_EINVAL;
  }
  std::lock_guard<std::mutex> lk(ctx->tuning.mu);
  ctx->packed_form = form;
  ctx->tuning.blocks_per_sm.clear();
  return RDM_OK;
}

extern "C" rdm_status rdm_set_device_dense(rdm_ctx* ctx, int enable) {
  if (!ctx) {
    set_error("rdm_set_device_dense: NULL context");
    return RDM_EINVAL;
  }
  if (enable < 0 || enable > 2) {
    set_error("rdm_set_device_dense: mode must be 0, 1 or 2");
    return RDM_EINVAL;
  }
  ctx->device_dense = enable;
  return RDM_OK;
}

extern "C" rdm_status rdm_set_bath_order(rdm_ctx* ctx, int enable) {
  if (!ctx) {
    set_error("rdm_set_bath_order: NULL context");
    return RDM_EINVAL;
  }
  ctx->bath_order = enable != 0;
  return RDM_OK;
}

extern "C" rdm_status rdm_bath_order(const rdm_model* model, int* order_out, double* tiles_caller,
                                     double* tiles_chosen) {
  HostModel hm;
  rdm_status st = compile_model(model, &hm);
  if (st != RDM_OK) return st;
  const double c0 = partner_tiles(hm);
  order_bath_bits(&hm);
  if (tiles_caller) *tiles_caller = c0;
  if (tiles_chosen) *tiles_chosen = partner_tiles(hm);
  if (order_out) {
    const int n = hm.n;
    for (int q = 0; q < n; ++q) order_out[q] = q;
    // internal site q is bit n-1-q; a bath bit i carries the caller's bit bath_src[i]
    for (int i = 0; i < (int)hm.bath_src.size(); ++i) order_out[n - 1 - i] = n - 1 - hm.bath_src[i];
  }
  return RDM_OK;
}

// The model restricted to sites [first, first + count), renumbered from 0, with no
// system sites: the bath part (first = n_sys) or the system part (first = 0).
namespace {
struct PartModel {
  std::vector<double> jx, jy, jz, hz, gx;
  rdm_model m{};
};
rdm_status part_model(const rdm_model* model, int first, int count, PartModel* pm) {
  const int n = model->n_sites;
  pm->jx.assign((size_t)count * count, 0.0);
  pm->jy = pm->jx;
  pm->jz = pm->jx;
  pm->hz.assign(count, 0.0);
  pm->gx.assign(count, 0.0);
  for (int a = 0; a < count; ++a) {
    for (int b = a + 1; b < count; ++b) {
      const size_t src = (size_t)(first + a) * n + (first + b), dst = (size_t)a * count + b;
      if (model->jx) pm->jx[dst] = model->jx[src];
      if (model->jy) pm->jy[dst] = model->jy[src];
      if (model->jz) pm->jz[dst] = model->jz[src];
    }
    if (model->hz) pm->hz[a] = model->hz[first + a];
    if (model->gx) pm->gx[a] = model->gx[first + a];
  }
  pm->m = rdm_model{count, 0, pm->jx.data(), pm->jy.data(), pm->jz.data(), pm->hz.data(), pm->gx.data(), 1.0};
  return RDM_OK;
}
}  // namespace

extern "C" rdm_status rdm_build_bath_hamiltonian(rdm_ctx* ctx, const rdm_model* model, rdm_ham** out) {
  if (!ctx || !model || !out) {
    set_error("rdm_build_bath_hamiltonian: NULL argument");
    return RDM_EINVAL;
  }
  HostModel check;
  rdm_status st = compile_model(model, &check);  // validates sizes and values
  if (st != RDM_OK) return st;
  PartModel pm;
  part_model(model, model->n_sys, model->n_sites - model->n_sys, &pm);
  return rdm_build_hamiltonian(ctx, &pm.m, out);
}

extern "C" rdm_status rdm_system_hamiltonian(const rdm_model* model, double* hs_out) {
  if (!model || !hs_out) {
    set_error("rdm_system_hamiltonian: NULL argument");
    return RDM_EINVAL;
  }
  HostModel check;
  rdm_status st = compile_model(model, &check);
  if (st != RDM_OK) return st;
  const int ns = model->n_sys, ds = 1 << ns;
  std::fill(hs_out, hs_out + (size_t)ds * ds, 0.0);
  if (ns == 0) return RDM_OK;
  PartModel pm;
  part_model(model, 0, ns, &pm);
  HostModel hs;
  st = compile_model(&pm.m, &hs);
  if (st != RDM_OK) return st;
  // the term convention of the SpMM (FlipTerm, DiagTerm), written out densely
  for (uint32_t s = 0; s < (uint32_t)ds; ++s) {
    for (const FlipTerm& f : hs.flips)
      hs_out[(size_t)(s ^ f.mask) * ds + s] += (__builtin_popcount(s & f.mask) & 1) ? f.c_odd : f.c_even;
    for (const DiagTerm& d : hs.diags)
      hs_out[(size_t)s * ds + s] += (__builtin_popcount(s & d.mask) & 1) ? -d.c : d.c;
  }
  return RDM_OK;
}

void rdm::Pass1Graph::reset() {
  if (exec) cudaGraphExecDestroy(exec);
  exec = nullptr;
  key.clear();
}

// Touches only the handle's own resources (not its context, which a caller may have
// destroyed first). cudaFree waits for the device, so no launch of the recorded graph
// is still running when it is destroyed.
extern "C" void rdm_destroy_hamiltonian(rdm_ham* ham) {
  if (!ham) return;
  if (ham->caller) rdm_destroy_hamiltonian(ham->caller);
  cudaSetDevice(ham->device);
  if (ham->d_terms) cudaFree(ham->d_terms);
  for (void* p : ham->d_apply_aux)
    if (p) cudaFree(p);
  ham->graph.reset();
  if (ham->graph.capture) cudaStreamDestroy(ham->graph.capture);
  ham->graph.capture = nullptr;
  delete ham;
}

extern "C" rdm_status rdm_hamiltonian_info(const rdm_ham* ham, int* n_sites, int* n_sys,
                                           int* n_flip, int* n_diag, double* norm_bound) {
  if (!ham) {
    set_error("rdm_hamiltonian_info: ham is NULL");
    return RDM_EINVAL;
  }
  if (n_sites) *n_sites = ham->model.n;
  if (n_sys) *n_sys = ham->model.ns;
  if (n_flip) *n_flip = (int)ham->model.flips.size();
  if (n_diag) *n_diag = (int)ham->model.diags.size();
  if (norm_bound) *norm_bound = ham->model.hnorm;
  return RDM_OK;
}

// ---------------------------------------------------------------- ABI: kernels

extern "C" rdm_status rdm_apply_hamiltonian(rdm_ham* ham, int precision, const void* x, void* y,
                                            int n_cols) {
  if (!ham || !x || !y) {
    set_error("rdm_apply_hamiltonian: NULL argument");
    return RDM_EINVAL;
  }
  if (precision != RDM_FP32 && precision != RDM_FP64) {
    set_error("rdm_apply_hamiltonian: bad precision %d", precision);
    return RDM_EINVAL;
  }
  ham = ham->caller_view();  // x and y are in the caller's state order
  Layout L;
  rdm_status st = plan_single(ham->model, n_cols, precision, 1, &L);
  if (st != RDM_OK) return st;
  const size_t bytes = L.block_bytes();
  const char* xb = reinterpret_cast<const char*>(x);
  const char* yb = reinterpret_cast<const char*>(y);
  if (xb < yb + bytes && yb < xb + bytes) {
    set_error("rdm_apply_hamiltonian: x and y overlap");
    return RDM_EINVAL;
  }
  if ((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(y)) % 16) {
    set_error("rdm_apply_hamiltonian: x and y must be 16-byte aligned");
    return RDM_EINVAL;
  }
  CK(cudaSetDevice(ham->ctx->device));
  SpmmArgs a{};
  a.flips = ham->d_flips;
  a.n_flip = (int)ham->model.flips.size();
  a.diags = ham->d_diags;
  a.n_diag = (int)ham->model.diags.size();
  a.w = x;
  a.z = y;
  cudaStream_t s = ham->ctx->stream;
  const bool tiled = layout_tiled(L) && ham->tiled.ready;
  uint32_t* err = nullptr;
  if (tiled) {
    // The tiled SpMM reads the K table of the diagonal and reports copy-ring
    // failures in an error word; both are kept per Hamiltonian and precision.
    const int pi = precision == RDM_FP32 ? 1 : 0;
    if (!ham->d_apply_aux[pi]) {
      const size_t tk = (size_t)(L.D >> kTileBits) *
                        (size_t)tile_diag_stride(ham->tiled.dg.n_entries, L.elem) * (size_t)L.elem;
      void* p = nullptr;
      CK(cudaMalloc(&p, 256 + tk));
      ham->d_apply_aux[pi] = p;
      CK(launch_tile_diag(L, ham->tiled.dg, static_cast<char*>(p) + 256, s));
    }
    err = static_cast<uint32_t*>(ham->d_apply_aux[pi]);
    a.tiled = ham->tiled;
    a.tile_k = static_cast<char*>(ham->d_apply_aux[pi]) + 256;
    a.err = err;
    CK(cudaMemsetAsync(err, 0, sizeof(uint32_t), s));
  }
  Profiler& pr = ham->ctx->prof;
  const int ev = pr.begin(kKApply, s, true);
  CK(launch_spmm(L, kModeApply, a, s));
  pr.end(kKApply, ev, s, 2.0 * (double)bytes);
  if (tiled) {
    uint32_t h_err = 0;
    CK(cudaMemcpyAsync(&h_err, err, sizeof(uint32_t), cudaMemcpyDeviceToHost, s));
    CK(cudaStreamSynchronize(s));
    if (h_err) {
      set_error("rdm_apply_hamiltonian: a bulk-copy wait in the SpMM kernel gave up (device error)");
      return RDM_ECUDA;
    }
  }
  return RDM_OK;
}

extern "C" rdm_status rdm_starting_block(rdm_ham* ham, int precision, int n_v, uint64_t seed,
                                         int dist, void* x) {
  if (!ham || !x || n_v < 1) {
    set_error("rdm_starting_block: NULL argument or n_v < 1");
    return RDM_EINVAL;
  }
  if (dist != RDM_RADEMACHER && dist != RDM_GAUSS && dist != RDM_BASIS) {
    set_error("rdm_starting_block: bad distribution %d", dist);
    return RDM_EINVAL;
  }
  ham = ham->caller_view();  // x is in the caller's state order
  const int ds = 1 << ham->model.ns;
  if (dist == RDM_BASIS && (int64_t)n_v > (int64_t(1) << (ham->model.n - ham->model.ns))) {
    set_error("rdm_starting_block: RDM_BASIS needs n_v <= d_b");
    return RDM_EINVAL;
  }
  Layout L;
  rdm_status st = plan_single(ham->model, ds * n_v, precision, ds, &L);
  if (st != RDM_OK) return st;
  CK(cudaSetDevice(ham->ctx->device));
  cudaStream_t s = ham->ctx->stream;
  double* norms = nullptr;
  if (dist == RDM_GAUSS) {
    CK(cudaMallocAsync(&norms, sizeof(double) * (size_t)n_v * 65, s));
    CK(launch_gauss_norms(int64_t(1) << L.n_bath_bits, n_v, seed, 0, norms + n_v, norms, s));
  }
  CK(launch_init_block(L, dist, seed, 0, n_v, norms, nullptr, x, s));
  if (norms) CK(cudaFreeAsync(norms, s));
  return RDM_OK;
}

// ---------------------------------------------------------------- ABI: estimate

extern "C" rdm_status rdm_workspace_size(const rdm_ham* ham, int n_beta, int n_v, int k,
                                         const rdm_opts* opts, size_t* bytes) {
  if (!ham || !opts || !bytes) {
    set_error("rdm_workspace_size: NULL argument");
    return RDM_EINVAL;
  }
  Plan p;
  rdm_opts o = *opts;
  if (o.passes == RDM_PASSES_AUTO) o.passes = RDM_PASSES_RECOMPUTE;  // the smaller of the two
  rdm_status st = make_plan(ham->model, n_beta, n_v, k, &o, SIZE_MAX, &p);
  if (st != RDM_OK) return st;
  if (!p.store) p.nbc = 1;
  *bytes = plan_bytes(p);
  return RDM_OK;
}

namespace rdm {

static void build_t(int ds, int k, int ng, int l, const std::vector<double>& ta,
                    const std::vector<double>& tb, std::vector<double>& t) {
  const int n = k * ds, nv = ds * ds;
  t.assign((size_t)n * n, 0.0);
  for (int j = 0; j < k; ++j) {
    const double* A = &ta[((size_t)j * ng + l) * nv];
    for (int a = 0; a < ds; ++a)
      for (int b = 0; b < ds; ++b) t[(size_t)(j * ds + a) * n + j * ds + b] = A[a * ds + b];
    if (j + 1 < k) {
      const double* Bm = &tb[((size_t)j * ng + l) * nv];
      for (int a = 0; a < ds; ++a)
        for (int b = 0; b < ds; ++b) {
          t[(size_t)((j + 1) * ds + a) * n + j * ds + b] = Bm[a * ds + b];
          t[(size_t)(j * ds + b) * n + (j + 1) * ds + a] = Bm[a * ds + b];
        }
    }
  }
}

// Host threads for the small dense step: the CPUs this process may run on (its
// affinity mask, which a container's cpuset narrows), or RDM_HOST_THREADS if set.
static int host_threads() {
  static const int n = [] {
    if (const char* e = std::getenv("RDM_HOST_THREADS")) {
      const int v = std::atoi(e);
      if (v > 0) return v;
    }
    cpu_set_t set;
    CPU_ZERO(&set);
    if (sched_getaffinity(0, sizeof set, &set) == 0) {
      const int c = CPU_COUNT(&set);
      if (c > 0) return c;
    }
    return std::max(1, (int)std::thread::hardware_concurrency());
  }();
  return n;
}

// Persistent host worker threads for the small dense step (started on first use, one
// fewer than the usable cores: the calling thread works too). Several callers (the
// serving loop's workers) may run jobs at once; idle workers help the oldest job.
class HostPool {
 public:
  static HostPool& get() {
    static HostPool pool(host_threads() - 1);
    return pool;
  }
  // f(0) .. f(n-1), each exactly once, spread over the workers and the caller.
  void run(int n, const std::function<void(int)>& f) {
    if (n <= 0) return;
    if (th_.empty() || n == 1) {
      for (int i = 0; i < n; ++i) f(i);
      return;
    }
    Job j;
    j.f = &f;
    j.n = n;
    {
      std::lock_guard<std::mutex> lk(mu_);
      jobs_.push_back(&j);
    }
    cv_.notify_all();
    work(j);
    std::unique_lock<std::mutex> lk(mu_);
    drop(&j);
    done_.wait(lk, [&] { return j.done == j.n && j.refs == 0; });
  }
  ~HostPool() {
    {
      std::lock_guard<std::mutex> lk(mu_);
      stop_ = true;
    }
    cv_.notify_all();
    for (auto& t : th_) t.join();
  }

 private:
  struct Job {
    const std::function<void(int)>* f = nullptr;
    int n = 0;
    std::atomic<int> next{0};
    int done = 0;  // guarded by mu_
    int refs = 0;  // workers inside work(); guarded by mu_
  };
  explicit HostPool(int workers) {
    for (int t = 0; t < workers; ++t) th_.emplace_back([this] { loop(); });
  }
  void work(Job& j) {
    int mine = 0;
    for (int i; (i = j.next.fetch_add(1)) < j.n; ++mine) (*j.f)(i);
    if (mine) {
      std::lock_guard<std::mutex> lk(mu_);
      j.done += mine;
    }
  }
  void drop(Job* j) {  // with mu_ held
    for (auto it = jobs_.begin(); it != jobs_.end(); ++it)
      if (*it == j) {
        jobs_.erase(it);
        return;
      }
  }
  void loop() {
    std::unique_lock<std::mutex> lk(mu_);
    for (;;) {
      cv_.wait(lk, [&] { return stop_ || !jobs_.empty(); });
      if (stop_) return;
      Job* j = jobs_.front();
      if (j->next.load() >= j->n) {  // every index taken: nothing left to help with
        drop(j);
        continue;
      }
      ++j->refs;
      lk.unlock();
      work(*j);
      lk.lock();
      if (--j->refs == 0) done_.notify_all();
      else if (j->done == j->n) done_.notify_all();
    }
  }
  std::mutex mu_;
  std::condition_variable cv_, done_;
  std::deque<Job*> jobs_;
  std::vector<std::thread> th_;
  bool stop_ = false;
};

template <typename F>
static void parallel_for(int n, F&& f) {
  const std::function<void(int)> fn = std::forward<F>(f);
  HostPool::get().run(n, fn);
}

extern "C" rdm_status rdm_function_of_t_batch(int n_mat, int n, int p, const double* t, int n_beta,
                                              const double* betas, double* t_min, double* c) {
  if (n_mat < 1 || n < 1 || n > 8192 || p < 1 || p > n || n_beta < 1 || !t || !betas || !t_min || !c) {
    set_error("rdm_function_of_t_batch: need n_mat >= 1, 1 <= p <= n <= 8192, n_beta >= 1, non-NULL arrays");
    return RDM_EINVAL;
  }
  for (int b = 0; b < n_beta; ++b)
    if (!(betas[b] >= 0.0) || !std::isfinite(betas[b])) {
      set_error("rdm_function_of_t_batch: beta[%d] must be finite and >= 0", b);
      return RDM_EINVAL;
    }
  const size_t nn = (size_t)n * n;
  for (size_t i = 0; i < nn * (size_t)n_mat; ++i)
    if (!std::isfinite(t[i])) {
      set_error("rdm_function_of_t_batch: T has a non-finite entry");
      return RDM_EINVAL;
    }
  std::vector<char> ok(n_mat, 1);
  const size_t cstride = (size_t)n_beta * n * p;
  parallel_for(n_mat, [&](int r) {
    ok[r] = tdense_fT(n, p, t + r * nn, n_beta, betas, &t_min[r], c + r * cstride) ? 1 : 0;
  });
  for (int r = 0; r < n_mat; ++r)
    if (!ok[r]) {
      set_error("rdm_function_of_t_batch: QR iteration did not converge on matrix %d", r);
      return RDM_ENUMERIC;
    }
  return RDM_OK;
}

// One rdm_estimate call in three stages: prepare() plans the workspace and issues the
// per-estimate set-up (tables, bath vectors, starting block); pass1() runs Algorithm 1's
// k steps (plain launches, or a graph replay), unless the caller runs them in a packed
// launch with other estimates (packed_item()); finish() does the small dense step, the
// Gram form and the normalisation, and fills `out`.
class EstimateRun {
 public:
  EstimateRun(rdm_ham* ham_, cudaStream_t s_, const double* betas_, int n_beta_, int n_v_, int k_,
              uint64_t seed_, const rdm_opts* o_, rdm_result* out_, Profiler* prof_)
      : ham(ham_), hm(ham_->model), s(s_), betas(betas_), n_beta(n_beta_), n_v(n_v_), k(k_), seed(seed_),
        o(o_), out(out_), prof(prof_) {}
  rdm_status prepare(char* ws, size_t ws_bytes);
  // on: the stream of the launches (s, or one forked from it); graph: a recording may be
  // replayed or made
  rdm_status pass1(cudaStream_t on, bool graph);
  rdm_status finish();  // fetch_t, every dense_task, finish_rest
  // finish() in stages, so a batch can run the dense steps of all its items in one
  // parallel pass: fetch_t copies T back; dense_task(r) is recurrence r's small dense step
  // (thread-safe across r); finish_rest does the Gram form and the normalisation.
  rdm_status fetch_t();
  int n_dense_tasks() const { return dense_on_device || wants_device ? 0 : n_rec; }
  void dense_task(int r);
  // The device path of the dense step (fetch_t decides wants_device): the job's
  // descriptor for launch_dense_jobs, its betas on the device, and the results back.
  bool wants_device = false;
  DenseJob dense_job();
  rdm_status upload_betas();
  rdm_status fetch_dense();
  int rec_ds() const { return ds; }
  rdm_status finish_rest();
  double host_ms_dense = 0.0;
  // Whether the packed launch can take this estimate's first pass (stored basis, one
  // recurrence of block size d_s per bath vector, a block of at most kPackedMaxBlock
  // bytes), and its description for that launch.
  bool packable() const;
  PackedItem packed_item() const;
  const Plan& plan() const { return p; }
  bool packed_done = false;  // the first pass ran in a launch shared with other items
  // Before prepare(): the first pass may run in clusters (k_pass1_cluster); after it,
  // whether it does.
  bool in_clusters = false;
  // float32 blocks of the tiled SpMM (from 32 tiles): their own launches, side by side with
  // other items', are faster than the packed launch's untiled units at every size measured,
  // least so for many items of one slice: 40 of 32 tiles (N = 15) 15.9 against 22.6 ms for
  // d_s = 2 and 24.2 against 32.2 for d_s = 4; 16 of 128 tiles 11.3 against 26.7.
  bool tiled_launches() const { return sa.tile_k != nullptr && !in_clusters && L.precision == RDM_FP32; }

 private:
  rdm_ham* ham;
  const HostModel& hm;
  cudaStream_t s;
  const double* betas;
  int n_beta, n_v, k;
  uint64_t seed;
  const rdm_opts* o;
  rdm_result* out;
  Profiler* prof;

  Plan p;
  Layout L, Lg;
  Layout Lgr;   // Lg on the Gram kernels' grid (gram_gridx)
  Layout Lrow;  // L on the row-parallel kernels' own grid (untiled_gridx)
  int ds = 0, nv = 0, ng = 0, dso = 0, nvo = 0, ngo = 0, sub = 1, n_rec = 0;
  int64_t d_b = 0;
  bool store = false;
  int nblk = 0;
  std::vector<char*> blk;
  char* psi = nullptr;
  PlanSizes psz{};
  size_t pstride_g = 0, cstride = 0;
  double* partials = nullptr;
  double* coef = nullptr;
  double* d_ta = nullptr;
  double* d_tb = nullptr;
  double* d_e = nullptr;
  double* d_gram = nullptr;
  double* d_norm = nullptr;
  uint32_t* d_flags = nullptr;
  char* d_tk = nullptr;
  char* d_vbuf = nullptr;
  double* d_graw = nullptr;
  double* d_lohi = nullptr;  // device small dense step (dense.cu)
  double* d_cheb = nullptr;
  double* d_c = nullptr;
  double* d_betas = nullptr;
  char* d_jobs = nullptr;
  bool dense_on_device = false;
  bool coef_on_device = false;  // the Gram coefficients too (nothing of c, M, T comes back)
  double thr_abs_sq = 0, thr_rel_sq = 0;
  SpmmArgs sa{};
  double blk_b = 0;
  uint64_t h2d = 0, d2h = 0;
  // bytes of f, quad, jlast and kb (device_coefficients), each rounded up to 8
  size_t coef_scratch() const {
    return (size_t)n_beta * n_v * (sizeof(double) * (1 + (size_t)nv) + sizeof(int)) + (size_t)n_beta * sizeof(int) + 16;
  }
  double gram_tau() const {
    return 1e-3 * (o->precision == RDM_FP32 ? 1.1920928955078125e-07 : 2.220446049250313e-16);
  }
  rdm_status device_coefficients(double e0, std::vector<double>& quad, std::vector<int>& kbeta);
  int cur = 0, prv = -1, nxt = 1;
  std::vector<double> ta, tb, mz, cstore, tmin;
  std::vector<char> okv;

  double* MZ(int j) const { return coef + (size_t)j * cstride; }  // j = 1..k+1
  double* CP(int j) const { return coef + (size_t)(k + 2) * cstride + (size_t)j * cstride; }
  double* CW(int j) const { return coef + (size_t)2 * (k + 2) * cstride + (size_t)j * cstride; }
  // Launch wrappers: count every launch; time the block-sized kernels with events.
  template <typename F>
  cudaError_t timed(int kind, double bytes, F&& launch) {
    const int ev = prof ? prof->begin(kind, s, true) : -1;
    const cudaError_t e = launch();
    if (prof) prof->end(kind, ev, s, bytes);
    return e;
  }
  template <typename F>
  cudaError_t counted(F&& launch) {
    if (prof) prof->begin(kKSmall, s, false);
    return launch();
  }
  rdm_status init_block(char* w) {
    const BathPerm bp = hm.perm();  // bath vectors drawn in the caller's bath order
    CK(timed(kKInit, blk_b, [&] {
      return launch_init_block(Lrow, o->vec_dist, seed, o->first_vector, n_v, nullptr, d_vbuf, w, s, sub, &bp);
    }));
    return RDM_OK;
  }
};

constexpr size_t kPackedMaxBlock = size_t(64) << 20;

// A stream beside another: fork makes it wait for what `s` holds, join makes `s` wait for it.
struct SideStream {
  cudaStream_t stream = nullptr;
  cudaEvent_t ev = nullptr;
  bool open = false;
  cudaError_t fork(cudaStream_t s) {
    cudaError_t e = cudaStreamCreateWithFlags(&stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventRecord(ev, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(stream, ev, 0);
    open = e == cudaSuccess;
    return e;
  }
  cudaError_t join(cudaStream_t s) {
    cudaError_t e = cudaEventRecord(ev, stream);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(s, ev, 0);
    if (e == cudaSuccess) open = false;
    return e;
  }
  ~SideStream() {
    if (stream && open) cudaStreamSynchronize(stream);  // fork without join: a failed launch
    if (ev) cudaEventDestroy(ev);
    if (stream) cudaStreamDestroy(stream);  // (its work completes first)
  }
};
using SideStreams = std::array<SideStream, 7>;

// The first n of `side` forked from s, and joined to it again.
static rdm_status fork_all(SideStreams& side, int n, cudaStream_t s) {
  for (int w = 0; w < n; ++w)
    if (side[w].fork(s) != cudaSuccess) {
      set_error("batch: no side stream: %s", cudaGetErrorString(cudaGetLastError()));
      return RDM_ECUDA;
    }
  return RDM_OK;
}
static rdm_status join_all(SideStreams& side, int n, cudaStream_t s) {
  rdm_status st = RDM_OK;
  for (int w = 0; w < n; ++w) {
    if (!side[w].open) continue;  // (its fork failed)
    const cudaError_t e = side[w].join(s);
    if (e != cudaSuccess && st == RDM_OK) {
      set_error("batch: %s", cudaGetErrorString(e));
      st = RDM_ECUDA;
    }
  }
  return st;
}
// Estimates whose blocks have fewer 1024-state tiles (all slices together) run the plain
// SpMM (rdm_set_spmm_form).
constexpr int64_t kTiledMinTiles = 32;
// Below this many betas the host's eigendecomposition path is faster than the device
// small dense step for a single estimate (its per-beta rotations are what the device
// step saves; its float64 multisection is latency-bound on few recurrences).
constexpr int kDeviceDenseMinBetas = 8;

size_t packed_store_footprint(const HostModel& h, int n_beta, int n_v, int k, const rdm_opts* o, double beta_max) {
  if (o->recurrence != RDM_BLOCK) return 0;
  rdm_opts q = *o;
  q.passes = RDM_PASSES_STORE;
  Plan p;
  if (make_plan(h, n_beta, n_v, k, &q, SIZE_MAX, &p, beta_max) != RDM_OK) return 0;
  if (!p.store || p.single || p.L.block_bytes() > kPackedMaxBlock) return 0;
  return (plan_bytes(p) + 255) / 256 * 256;
}

static double max_beta(const double* b, int n) {
  double m = 0.0;
  for (int i = 0; i < n; ++i) m = std::max(m, b[i]);
  return m;
}

rdm_status EstimateRun::prepare(char* ws, size_t ws_bytes) {
  rdm_status st = make_plan(hm, n_beta, n_v, k, o, ws_bytes, &p, max_beta(betas, n_beta));
  if (st != RDM_OK) return st;
  L = p.L;    // the recurrences (block size ds)
  Lg = p.Lg;  // the Gram view (groups of dso columns)
  // The orthogonalisation and the starting block are bound by HBM and need about 8
  // resident blocks per SM over all slices, whatever the tiled SpMM's one persistent block
  // per SM and slice. On that grid a block of one slice (N = 24, 4 bath vectors) had 152
  // blocks, and one of 200 slices (N = 16, 400 bath vectors) 30 400 of 3 rows a thread.
  Lrow = L;
  Lrow.gridx = untiled_gridx(L);
  Lgr = Lg;
  Lgr.gridx = gram_gridx(Lg);
  ds = L.DS, nv = ds * ds, ng = L.n_groups();
  dso = 1 << hm.ns, nvo = dso * dso, ngo = Lg.n_groups();
  sub = p.single ? dso : 1;  // recurrences per bath vector
  n_rec = n_v * sub;         // real recurrences
  d_b = int64_t(1) << L.n_bath_bits;
  if (o->vec_dist == RDM_BASIS && o->first_vector + (int64_t)n_v > d_b) {
    set_error("RDM_BASIS needs first_vector + n_v <= d_b = %lld", (long long)d_b);
    return RDM_EINVAL;
  }
  if (!ws) {
    set_error("internal: estimator called without a workspace");
    return RDM_EINVAL;
  }
  Arena ar;
  ar.base = ws;
  ar.cap = ws_bytes;
  store = p.store;
  nblk = store ? k + 1 : 3;
  blk.assign(nblk, nullptr);
  {
    char* base = ar.take<char>(L.block_bytes() * nblk);
    for (int i = 0; i < nblk; ++i) blk[i] = base + (size_t)i * L.block_bytes();
  }
  psi = store ? nullptr
              : ar.take<char>(L.block_bytes() / (size_t)L.n_slices * (size_t)(p.nsc ? p.nsc : L.n_slices) * p.nbc);
  psz = plan_sizes(p);
  pstride_g = psz.gram1;
  partials = ar.take<double>(psz.partials);
  coef = ar.take<double>((size_t)(k + 2) * ng * nv * 3);
  d_ta = ar.take<double>((size_t)k * ng * nv);
  d_tb = ar.take<double>((size_t)k * ng * nv);
  d_e = ar.take<double>(psz.e);
  d_gram = ar.take<double>(psz.gram);
  d_norm = ar.take<double>((size_t)p.n_v_pad * 65);
  d_flags = ar.take<uint32_t>(4);
  d_tk = ar.take<char>(p.tk_bytes);
  d_vbuf = p.gauss ? ar.take<char>((size_t)n_v * (size_t)d_b * L.elem) : nullptr;
  d_graw = p.gauss ? ar.take<double>((size_t)n_v * (size_t)d_b) : nullptr;
  if (p.dev_dense) {
    const size_t ne = (size_t)k * ds * ds;
    d_lohi = ar.take<double>(2 * (size_t)ng);
    d_cheb = ar.take<double>((size_t)ng * p.vstride * ne);
    d_c = ar.take<double>((size_t)ng * n_beta * ne);
    d_betas = ar.take<double>((size_t)n_beta);
    d_jobs = ar.take<char>(dense_jobs_bytes(1));
  }
  cstride = (size_t)ng * nv;

  CK(cudaMemsetAsync(d_flags, 0, 4 * sizeof(uint32_t), s));
  const double tau_abs = o->precision == RDM_FP64 ? 1e-12 : 1e-6;
  const double tau_rel = o->precision == RDM_FP64 ? 1e-7 : 1e-5;
  thr_abs_sq = (tau_abs * hm.hnorm) * (tau_abs * hm.hnorm);
  thr_rel_sq = tau_rel * tau_rel;

  sa = SpmmArgs{};
  sa.flips = ham->d_flips;
  sa.n_flip = (int)hm.flips.size();
  sa.diags = ham->d_diags;
  sa.n_diag = (int)hm.diags.size();
  sa.tiled = ham->tiled;
  {
    // The tiled SpMM's persistent blocks walk the tiles of all slices; with only a few
    // tiles most of them idle and its fixed cost per launch (about 25 us: tables into
    // shared memory, the first copies, the partial sums) dominates, and the plain kernel
    // (a block per row range and slice) is faster. Measured on GB300: plain faster at
    // 8 tiles (c1: 12 vs 31 us per launch), tiled faster from 64 tiles on.
    const int64_t tiles = p.tk_bytes ? ((int64_t)L.n_slices << (L.n_bits - kTileBits)) : 0;
    const int form = ham->ctx ? ham->ctx->spmm_form : 0;  // (the serving loop's own Hamiltonians have none)
    in_clusters = in_clusters && form != 2 && packable() && pass1_cluster_fits(L, ham->tiled);
    sa.tile_k = p.tk_bytes && (in_clusters || form == 1 || (form == 0 && tiles >= kTiledMinTiles)) ? d_tk : nullptr;
  }
  sa.err = d_flags + 1;

  blk_b = (double)L.block_bytes();
  h2d = d2h = 0;

  // Once per estimate: the per-tile diagonal table and (Gaussian case) the bath vectors.
  if (sa.tile_k) CK(counted([&] { return launch_tile_diag(L, ham->tiled.dg, d_tk, s); }));
  if (p.gauss) {
    CK(counted([&] {
      return launch_gauss_norms(d_b, n_v, seed, o->first_vector, d_norm + p.n_v_pad, d_norm, s, d_graw);
    }));
    if (prof) prof->begin(kKSmall, s, false);  // the norm kernel is two launches
    CK(counted([&] { return launch_gauss_fill(L, n_v, seed, o->first_vector, d_norm, d_vbuf, s, d_graw); }));
  }
  // ---- pass 1 starts from the starting block and M_1 = I, Cp_1 = 0.
  st = init_block(blk[0]);
  if (st != RDM_OK) return st;
  CK(counted([&] { return launch_coef_init(L, StepCoefs{MZ(1), CP(1), nullptr}, s); }));
  cur = 0, prv = -1, nxt = 1;
  return RDM_OK;
}

bool EstimateRun::packable() const {
  return store && !p.single && L.block_bytes() <= kPackedMaxBlock && L.n_slices * L.gridx <= (1 << 20);
}

PackedItem EstimateRun::packed_item() const {
  PackedItem it{};
  it.L = L;
  // the untiled grid of the plain kernels (the tiled SpMM's own grid is not used here);
  // the partials buffer is sized for the larger of the two (plan_sizes)
  it.L.gridx = untiled_gridx(L);
  it.sa = sa;
  it.sa.partials = partials;
  it.blk = blk[0];
  it.coef = coef;
  it.ta = d_ta;
  it.tb = d_tb;
  it.flags = d_flags;
  it.thr_abs_sq = thr_abs_sq;
  it.thr_rel_sq = thr_rel_sq;
  it.k = k;
  it.n_rec = n_rec;
  return it;
}

rdm_status EstimateRun::pass1(cudaStream_t on, bool graph) {
  rdm_status st = RDM_OK;
  // k steps; `launch` false only walks the buffer rotation (the launches are replayed
  // from a graph).
  auto pass1 = [&](cudaStream_t ls, bool launch) -> rdm_status {
    for (int j = 1; j <= k; ++j) {
      if (launch) {
        sa.w = blk[cur];
        sa.w_prev = prv >= 0 ? blk[prv] : nullptr;
        sa.z = blk[nxt];
        sa.mz = MZ(j);
        sa.cp = CP(j);
        sa.partials = partials;
        CK(timed(kKSpmm1, blk_b * (prv >= 0 ? 3 : 2), [&] { return launch_spmm(L, kModePass1, sa, ls); }));
        CK(counted([&] {
          return launch_small_a(L, partials, MZ(j), d_ta + (size_t)(j - 1) * cstride, CW(j), d_flags, ls);
        }));
        CK(timed(kKOrth1, blk_b * 3, [&] { return launch_orth(Lrow, blk[cur], blk[nxt], CW(j), partials, ls); }));
        CK(counted([&] {
          return launch_small_b(Lrow, partials, MZ(j), d_tb + (size_t)(j - 1) * cstride, MZ(j + 1), CP(j + 1),
                                thr_abs_sq, thr_rel_sq, n_rec, d_flags, ls);
        }));
      }
      const int old_prev = prv;
      prv = cur;
      cur = nxt;
      if (store)
        nxt = cur + 1;
      else
        nxt = old_prev >= 0 ? old_prev : 3 - prv - cur;
    }
    return RDM_OK;
  };
  // Graph path: not while kernels are being timed one by one or several items' launches are
  // in flight (a handle's recording may be replaced), and only for handles of a context (the
  // serving loop's per-request handles are used once).
  bool replayed = false;
  Pass1Graph& pg = ham->graph;
  std::unique_lock<std::mutex> glk(pg.mu, std::defer_lock);
  if (graph && ham->ctx && ham->ctx->graphs && !(prof && prof->on) && glk.try_lock()) {
    auto bits = [](double x) {
      uint64_t u;
      std::memcpy(&u, &x, sizeof u);
      return u;
    };
    const std::vector<uint64_t> key = {
        (uint64_t)(uintptr_t)s, (uint64_t)(uintptr_t)blk[0], (uint64_t)(uintptr_t)blk[1],
        (uint64_t)(uintptr_t)(nblk > 2 ? blk[2] : nullptr), (uint64_t)nblk, (uint64_t)(uintptr_t)partials,
        (uint64_t)(uintptr_t)coef, (uint64_t)(uintptr_t)d_ta, (uint64_t)(uintptr_t)d_tb,
        (uint64_t)(uintptr_t)d_flags, (uint64_t)(uintptr_t)sa.tile_k, (uint64_t)k, (uint64_t)n_rec,
        (uint64_t)store, bits(thr_abs_sq), bits(thr_rel_sq), (uint64_t)L.n_bits, (uint64_t)L.n_bath_bits,
        (uint64_t)L.D, (uint64_t)L.DS, (uint64_t)L.B, (uint64_t)L.Bs, (uint64_t)L.n_slices, (uint64_t)L.VW,
        (uint64_t)L.TPR, (uint64_t)L.gridx, (uint64_t)L.precision, (uint64_t)L.elem};
    if (pg.exec && pg.key == key) {
      CK(cudaGraphLaunch(pg.exec, on));
      replayed = true;
    } else if (pg.seen == key) {
      // second call with this configuration: record it (on a private stream, since the
      // legacy default stream cannot be captured), then run the recording
      pg.reset();
      if (!pg.capture) CK(cudaStreamCreateWithFlags(&pg.capture, cudaStreamNonBlocking));
      CK(cudaStreamBeginCapture(pg.capture, cudaStreamCaptureModeRelaxed));
      const int c0 = cur, p0 = prv, n0 = nxt;
      const rdm_status rs = pass1(pg.capture, true);
      cudaGraph_t g = nullptr;
      const cudaError_t ce = cudaStreamEndCapture(pg.capture, &g);
      cudaGraphExec_t ex = nullptr;
      if (rs == RDM_OK && ce == cudaSuccess && g && cudaGraphInstantiate(&ex, g, 0) == cudaSuccess) {
        pg.exec = ex;
        pg.key = key;
        CK(cudaGraphLaunch(pg.exec, on));
        replayed = true;
      } else {
        cudaGetLastError();  // fall back to direct launches below
      }
      cur = c0, prv = p0, nxt = n0;  // the walk below advances the rotation once
      if (g) cudaGraphDestroy(g);
    } else {
      pg.seen = key;
    }
  }
  st = pass1(on, !replayed);
  return st;
}

rdm_status EstimateRun::fetch_t() {
  const int mode = ham->ctx ? ham->ctx->device_dense : 1;
  wants_device = p.dev_dense && (mode == 2 || (mode == 1 && n_beta >= kDeviceDenseMinBetas));
  // With the basis stored and block recurrences, the coefficients are formed where c is.
  // On the host they took the copies of c and E (52 MB each way for 64 vectors, 64 betas and
  // 100 steps of d_s = 4) and about 1 ms per solve of the small batch. Their scratch is the
  // Chebyshev vectors' (dead once c is formed).
  coef_on_device = wants_device && store && !p.single && n_beta <= 65535 &&
                   coef_scratch() <= (size_t)ng * p.vstride * k * nv * sizeof(double);
  const bool t_back = !wants_device || out->t_a || out->t_b;
  uint32_t flags[4];
  d2h += sizeof flags;
  if (t_back) {
    ta.assign((size_t)k * cstride, 0.0);
    tb.assign((size_t)k * cstride, 0.0);
    CK(cudaMemcpyAsync(ta.data(), d_ta, ta.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    CK(cudaMemcpyAsync(tb.data(), d_tb, tb.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    d2h += (ta.size() + tb.size()) * sizeof(double);
  }
  if (!coef_on_device) {
    mz.assign((size_t)(k + 1) * cstride, 0.0);
    CK(cudaMemcpyAsync(mz.data(), MZ(1), mz.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
    d2h += mz.size() * sizeof(double);
  }
  CK(cudaMemcpyAsync(flags, d_flags, sizeof flags, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  if (flags[1]) {
    set_error("a bulk-copy wait in the SpMM kernel gave up (device error)");
    return RDM_ECUDA;
  }
  if (flags[0] & kFlagNonFinite) {
    set_error("non-finite Lanczos coefficient (overflow or invalid model)");
    return RDM_ENUMERIC;
  }
  // ---- small dense step (host float64): f(T_r) E1 for every beta (eq. fT) with the
  // per-recurrence shift t_min(r); E0 = min_r t_min(r) (Sec. 3.2), then rescaling. A
  // recurrence r is bath vector r (block) or column r = l dso + i (single).
  const int n = k * ds;
  if (!coef_on_device) cstore.assign((size_t)n_rec * n_beta * n * ds, 0.0);
  tmin.assign(n_rec, 0.0);
  okv.assign(n_rec, 1);
  dense_on_device = false;
  return RDM_OK;
}

DenseJob EstimateRun::dense_job() {
  DenseJob j{};
  j.k = k;
  j.ng = ng;
  j.n_rec = n_rec;
  j.n_beta = n_beta;
  j.vstride = p.vstride;
  j.hnorm = hm.hnorm;
  j.beta_max = max_beta(betas, n_beta);
  j.ta = d_ta;
  j.tb = d_tb;
  j.betas = d_betas;
  j.lohi = d_lohi;
  j.V = d_cheb;
  j.cout = d_c;
  return j;
}

rdm_status EstimateRun::upload_betas() {
  CK(cudaMemcpyAsync(d_betas, betas, sizeof(double) * n_beta, cudaMemcpyHostToDevice, s));
  h2d += sizeof(double) * n_beta;
  return RDM_OK;
}

rdm_status EstimateRun::fetch_dense() {
  std::vector<double> lohi(2 * (size_t)n_rec);
  if (!coef_on_device)
    CK(cudaMemcpyAsync(cstore.data(), d_c, cstore.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
  CK(cudaMemcpyAsync(lohi.data(), d_lohi, lohi.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  d2h += (cstore.size() + lohi.size()) * sizeof(double);
  for (int r = 0; r < n_rec; ++r) {
    tmin[r] = lohi[2 * (size_t)r];
    okv[r] = std::isfinite(tmin[r]) ? 1 : 0;
  }
  for (double x : cstore)
    if (!std::isfinite(x)) {
      set_error("the device small dense step gave a non-finite coefficient");
      return RDM_ENUMERIC;
    }
  dense_on_device = true;
  return RDM_OK;
}

void EstimateRun::dense_task(int r) {
  const int n = k * ds;
  std::vector<double> t;
  build_t(ds, k, ng, r, ta, tb, t);
  okv[r] = tdense_fT(n, ds, t.data(), n_beta, betas, &tmin[r], &cstore[(size_t)r * n_beta * n * ds]);
}

rdm_status EstimateRun::finish() {
  rdm_status st = fetch_t();
  if (st != RDM_OK) return st;
  if (wants_device) {
    const auto t0 = std::chrono::steady_clock::now();
    st = upload_betas();
    if (st != RDM_OK) return st;
    const DenseJob j = dense_job();
    const int ev = prof ? prof->begin(kKDense, s, true) : -1;
    const cudaError_t e = launch_dense_jobs(ds, &j, 1, d_jobs, s);
    if (prof) prof->end(kKDense, ev, s, 0.0);
    CK(e);
    st = fetch_dense();
    if (st != RDM_OK) return st;
    host_ms_dense = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  } else {
    const auto t0 = std::chrono::steady_clock::now();
    parallel_for(n_rec, [&](int r) { dense_task(r); });
    host_ms_dense = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  }
  return finish_rest();
}

// eq. rho_est and ln Z_t from per-vector Grams g[beta][l][i][j] relative to the shift
// e0: rho*(beta) = the symmetric part of sum_l G_l over its trace, ln Z_t = ln(d_b tr /
// n_v) - beta e0. False when a trace is not a positive finite number.
static bool normalise_grams(const std::vector<double>& g, int n_beta, int n_v, int dso, double d_b,
                            const double* betas, double e0, double* rho, double* lnz) {
  const int nvo = dso * dso;
  bool ok = true;
  for (int bi = 0; bi < n_beta; ++bi) {
    std::vector<double> sum(nvo, 0.0);
    for (int l = 0; l < n_v; ++l)
      for (int v = 0; v < nvo; ++v) sum[v] += g[((size_t)bi * n_v + l) * nvo + v];
    double tr = 0.0;
    for (int i = 0; i < dso; ++i) tr += sum[i * dso + i];
    ok = ok && std::isfinite(tr) && tr > 0;
    for (int i = 0; i < dso; ++i)
      for (int jj = 0; jj < dso; ++jj)
        rho[(size_t)bi * nvo + i * dso + jj] = 0.5 * (sum[i * dso + jj] + sum[jj * dso + i]) / tr;
    if (lnz) lnz[bi] = std::log(d_b * tr / n_v) - betas[bi] * e0;
  }
  return ok;
}

// The Gram coefficients on the device: E in d_e, quad and the steps each beta needs back.
rdm_status EstimateRun::device_coefficients(double e0, std::vector<double>& quad, std::vector<int>& kbeta) {
  const size_t nq = (size_t)n_beta * n_v;
  std::vector<double> f(nq);
  for (int l = 0; l < n_v; ++l)
    for (int bi = 0; bi < n_beta; ++bi) f[(size_t)l * n_beta + bi] = std::exp(-0.5 * betas[bi] * (tmin[l] - e0));
  const double tau = gram_tau();
  CoefJob j{};
  j.k = k;
  j.ng = ng;
  j.n_v = n_v;
  j.n_beta = n_beta;
  j.tau2 = tau * tau;
  j.c = d_c;
  j.f = d_cheb;
  j.mz = MZ(1);
  j.e = d_e;
  j.quad = d_cheb + nq;
  j.kb = reinterpret_cast<int*>(j.quad + nq * nv);
  j.jlast = j.kb + (n_beta + 1) / 2 * 2;
  CK(cudaMemcpyAsync(d_cheb, f.data(), nq * sizeof(double), cudaMemcpyHostToDevice, s));
  h2d += nq * sizeof(double);
  CK(counted([&] { return launch_gram_coef(ds, j, s); }));
  if (prof) prof->begin(kKSmall, s, false);  // (two launches)
  std::vector<double> back(nq * nv + (size_t)(n_beta + 1) / 2);
  CK(cudaMemcpyAsync(back.data(), j.quad, back.size() * sizeof(double), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  d2h += back.size() * sizeof(double);
  std::copy_n(back.data(), nq * nv, quad.data());
  std::memcpy(kbeta.data(), back.data() + nq * nv, (size_t)n_beta * sizeof(int));
  for (double x : quad)
    if (!std::isfinite(x)) {
      set_error("the device small dense step gave a non-finite coefficient");
      return RDM_ENUMERIC;
    }
  return RDM_OK;
}

rdm_status EstimateRun::finish_rest() {
  rdm_status st = RDM_OK;
  const int n = k * ds;
  uint32_t flags[4];
  double host_ms = host_ms_dense;
  const auto host_t0 = std::chrono::steady_clock::now();
  auto host_lap = [&]() {
    const auto t1 = std::chrono::steady_clock::now();
    return std::chrono::duration<double, std::milli>(t1 - host_t0).count();
  };
  double e0 = INFINITY;
  for (int r = 0; r < n_rec; ++r) {
    if (!okv[r]) {
      set_error("eigensolver did not converge on T_%d", r);
      return RDM_ENUMERIC;
    }
    e0 = std::min(e0, tmin[r]);
  }
  host_ms += host_lap();
  // c[beta][r] = exp(-beta (t_min(r) - E0)/2) * (the t_min(r)-shifted c)
  auto coef_c = [&](int r, int bi, std::vector<double>& c) {
    const double* src = &cstore[((size_t)r * n_beta + bi) * n * ds];
    const double f = std::exp(-0.5 * betas[bi] * (tmin[r] - e0));
    c.resize((size_t)n * ds);
    for (size_t i = 0; i < c.size(); ++i) c[i] = f * src[i];
  };
  // Per bath vector and beta: quad = c^T c (its diagonal only for single recurrences)
  // and E_{j,beta} = M_j c_{j,beta}; E goes to the recurrences' layout for pass 2 and
  // to the Gram view (diagonal d_s x d_s blocks for single recurrences) for the
  // stored-basis Gram.
  const size_t cstride_g = (size_t)ngo * nvo;
  const bool e_view = store;
  std::vector<double> quad((size_t)n_beta * n_v * nvo, 0.0), gram((size_t)n_beta * n_v * nvo, 0.0);
  std::vector<double> hE(coef_on_device ? 0 : psz.e);
  std::vector<double> hg(psz.gram);
  // Trailing Krylov steps whose coefficient blocks are below the working precision
  // relative to the whole coefficient vector (|c_j| <= 1e-3 eps |c| for every vector, at
  // one beta) cannot change psi = sum_j Q_j c_j at that precision. Their E_j are set to
  // zero for that beta (so the result does not depend on how betas are chunked), and the
  // Gram pass (stored basis) or the recurrence of pass 2 stops after the last step any
  // beta of the chunk needs.
  const double tau = gram_tau();
  auto last_significant = [&](const std::vector<double>& c, int width) -> int {
    double tot = 0.0;
    for (double x : c) tot = std::fma(x, x, tot);
    int last = 0;
    for (int j = 0; j < k; ++j) {
      double sj = 0.0;
      for (int t = 0; t < ds * width; ++t) {
        const double x = c[(size_t)j * ds * width + t];
        sj = std::fma(x, x, sj);
      }
      if (sj > tau * tau * tot) last = j + 1;
    }
    return last;
  };
  std::vector<int> jlast((size_t)p.nbc * n_v, 1), kbeta(p.nbc, 1);
  // betas of one Gram launch: their partials fit the buffer (one beta's do: plan_sizes; a
  // group of slices takes less than the whole), the launches are even
  auto gram_betas = [&](size_t stride, int nb) {
    const int slots = (int)std::min<size_t>(kGramLaunchBetas, psz.partials / stride);
    const int launches = (nb + slots - 1) / slots;
    return (nb + launches - 1) / launches;
  };
  for (int b0 = 0; b0 < n_beta; b0 += p.nbc) {
    const int nb = std::min(p.nbc, n_beta - b0);
    if (coef_on_device) {  // (the whole grid: a stored basis has one chunk)
      st = device_coefficients(e0, quad, kbeta);
      if (st != RDM_OK) return st;
    } else {
      std::fill(hE.begin(), hE.end(), 0.0);
      std::fill(jlast.begin(), jlast.end(), 1);
      const auto coef_t0 = std::chrono::steady_clock::now();
      parallel_for(n_v, [&](int l) {
        std::vector<double> c;
        for (int bi = 0; bi < nb; ++bi) {
          double* q = &quad[((size_t)(b0 + bi) * n_v + l) * nvo];
          if (!p.single) {
            coef_c(l, b0 + bi, c);
            jlast[(size_t)bi * n_v + l] = last_significant(c, ds);
            for (int a = 0; a < ds; ++a)
              for (int b = 0; b < ds; ++b) {
                double sacc = 0.0;
                for (int r = 0; r < n; ++r) sacc = std::fma(c[(size_t)r * ds + a], c[(size_t)r * ds + b], sacc);
                q[a * ds + b] = sacc;
              }
            for (int j = 0; j < k; ++j) {
              const double* M = &mz[(size_t)j * cstride + (size_t)l * nv];
              double* Ej = &hE[(((size_t)j * p.nbc + bi) * ng + l) * nv];
              for (int a = 0; a < ds; ++a)
                for (int b = 0; b < ds; ++b) {
                  double sacc = 0.0;
                  for (int m = 0; m < ds; ++m) sacc = std::fma(M[a * ds + m], c[(size_t)(j * ds + m) * ds + b], sacc);
                  Ej[a * ds + b] = sacc;
                }
            }
            continue;
          }
          for (int i = 0; i < dso; ++i) {  // single recurrences: column r = l dso + i
            const int r = l * dso + i;
            coef_c(r, b0 + bi, c);
            int& jl = jlast[(size_t)bi * n_v + l];
            jl = std::max(i == 0 ? 1 : jl, last_significant(c, 1));
            double sacc = 0.0;
            for (int m = 0; m < n; ++m) sacc += c[m] * c[m];
            q[i * dso + i] = sacc;
            for (int j = 0; j < k; ++j) {
              const double e = mz[(size_t)j * cstride + r] * c[j];
              if (e_view)
                hE[(((size_t)j * p.nbc + bi) * ngo + l) * nvo + i * dso + i] = e;
              else
                hE[((size_t)j * p.nbc + bi) * ng + r] = e;
            }
          }
        }
      });
      host_ms += std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - coef_t0).count();
      for (int bi = 0; bi < nb; ++bi) {
        const int kb =
            std::max(1, *std::max_element(jlast.begin() + (size_t)bi * n_v, jlast.begin() + (size_t)(bi + 1) * n_v));
        kbeta[bi] = kb;
        for (int j = kb; j < k; ++j) {  // E_j of this beta beyond its last needed step
          double* e0p = &hE[((size_t)j * p.nbc + bi) * (e_view ? ngo * nvo : ng * nv)];
          std::fill(e0p, e0p + (size_t)(e_view ? ngo * nvo : ng * nv), 0.0);
        }
      }
      CK(cudaMemcpyAsync(d_e, hE.data(), hE.size() * sizeof(double), cudaMemcpyHostToDevice, s));
      h2d += hE.size() * sizeof(double);
    }
    if (store) {
      // ---- psi = sum_j W_j E_j over the stored blocks, Gram fused (Gram view).
      const int gmax = gram_betas(pstride_g, nb);
      for (int q = 0; q < nb; q += gmax) {
        const int nq = std::min(gmax, nb - q);
        CK(timed(kKGram, blk_b * *std::max_element(kbeta.begin() + q, kbeta.begin() + q + nq), [&] {
          return launch_gram_stored(Lgr, blk[0], &kbeta[q], d_e, p.nbc, q, nq, partials, pstride_g, s);
        }));
        CK(counted([&] {
          return launch_reduce_gram(Lgr, partials, pstride_g, nq, d_gram + (size_t)q * cstride_g, s);
        }));
      }
    } else {
      // ---- pass 2: recompute W_j (bit-identical) and accumulate psi, one sweep per
      // group of nsc slices (the whole block unless the plan splits it).
      const int nsc = p.nsc > 0 ? p.nsc : L.n_slices;
      const size_t slice_b = L.block_bytes() / (size_t)L.n_slices;
      // betas by their last needed step, longest first, so step j updates only the psi
      // of the betas still active there
      std::vector<int> ord(nb), kb(nb);
      std::vector<double> hEc;
      for (int s0 = 0; s0 < L.n_slices; s0 += nsc) {
        const int nsl = std::min(nsc, L.n_slices - s0);
        Layout Ls = L, Lgs = Lgr;  // (the whole block's Gram grid: the same sums)
        Ls.n_slices = Lgs.n_slices = nsl;
        Ls.B = nsl * L.Bs;
        Lgs.B = nsl * Lg.Bs;
        Layout Lsr = Ls;
        Lsr.gridx = untiled_gridx(Ls);  // the row-parallel kernels' grid, as Lrow
        const int g0 = s0 * L.groups_per_slice(), ngs = Ls.n_groups();
        const int g0o = s0 * Lg.groups_per_slice(), ngso = Lgs.n_groups();
        const size_t off = (size_t)s0 * slice_b, cs = (size_t)ngs * nv, cso = (size_t)ngso * nvo;
        const double bs = (double)Ls.block_bytes();
        int ke = 1;
        for (int bi = 0; bi < nb; ++bi) {
          kb[bi] = 1;
          for (int l = g0o; l < std::min(n_v, g0o + ngso); ++l) kb[bi] = std::max(kb[bi], jlast[(size_t)bi * n_v + l]);
          ke = std::max(ke, kb[bi]);
          ord[bi] = bi;
        }
        std::stable_sort(ord.begin(), ord.end(), [&](int x, int y) { return kb[x] > kb[y]; });
        hEc.assign((size_t)k * p.nbc * cs, 0.0);
        for (int j = 0; j < k; ++j)
          for (int r = 0; r < nb; ++r)
            std::copy_n(&hE[(((size_t)j * p.nbc + ord[r]) * ng + g0) * nv], cs, &hEc[((size_t)j * p.nbc + r) * cs]);
        CK(cudaMemcpyAsync(d_e, hEc.data(), hEc.size() * sizeof(double), cudaMemcpyHostToDevice, s));
        h2d += hEc.size() * sizeof(double);
        // Basis blocks of the sweep: W_i (i = 1, 2, ..) in a ring. With a slice group
        // smaller than the block, the three full-width blocks of pass 1 (dead by now) hold
        // more than three blocks of the group: the last mb blocks are kept and psi is
        // updated from them together every mb steps (the same fma sequence per element),
        // reading and writing psi once per mb steps.
        const size_t cb = Ls.block_bytes();
        const size_t e_smem = (size_t)nb * Ls.groups_per_slice() * nv * L.elem;
        int mb = (int)std::min<size_t>(kPsiBatchMax, 3 * L.block_bytes() / cb - 2);
        while (mb > 1 && (size_t)mb * e_smem > ((size_t)160 << 10)) --mb;
        if (mb < 2) mb = 1;
        const int ring = mb > 1 ? mb + 2 : 3;
        auto wblk = [&](int i) -> char* {
          return mb > 1 ? blk[0] + (size_t)((i - 1) % ring) * cb : blk[(i - 1) % 3] + off;
        };
        auto active = [&](int j) {  // betas still active at step j
          int na = 0;
          while (na < nb && kb[ord[na]] > j) ++na;
          return na;
        };
        {
          const BathPerm bp = hm.perm();
          const char* vb = d_vbuf ? d_vbuf + (size_t)(g0 / sub) * (size_t)d_b * L.elem : nullptr;
          CK(timed(kKInit, bs, [&] {
            return launch_init_block(Lsr, o->vec_dist, seed, o->first_vector + g0 / sub, n_v - g0 / sub, nullptr, vb,
                                     wblk(1), s, sub, &bp);
          }));
        }
        CK(timed(kKPsiInit, bs * (1 + nb), [&] { return launch_psi_init(Lsr, wblk(1), psi, d_e, nb, s); }));
        int j0 = 1;  // first step whose psi update is pending
        for (int j = 1; j < ke; ++j) {
          const int na = active(j);
          sa.w = wblk(j);
          sa.w_prev = j >= 2 ? wblk(j - 1) : nullptr;
          sa.z = wblk(j + 1);
          sa.mz = MZ(j) + (size_t)g0 * nv;
          sa.cp = CP(j) + (size_t)g0 * nv;
          sa.partials = nullptr;
          CK(timed(kKSpmm2, bs * (j >= 2 ? 3 : 2), [&] { return launch_spmm(Ls, kModePass2, sa, s); }));
          const int nf = mb > 1 ? 0 : na;  // betas updated by the orthogonalisation itself
          CK(timed(kKOrth2, bs * (3 + 2 * nf), [&] {
            return launch_orth_psi(Lsr, wblk(j), wblk(j + 1), CW(j) + (size_t)g0 * nv, psi,
                                   d_e + (size_t)j * p.nbc * cs, nf, s);
          }));
          if (mb > 1 && (j - j0 + 1 == mb || j == ke - 1)) {
            const int m = j - j0 + 1, n0 = active(j0);
            PsiBatch wb{};
            for (int a = 0; a < m; ++a) wb.w[a] = wblk(j0 + a + 1);
            CK(timed(kKPsiBatch, bs * (m + 2 * n0), [&] {
              return launch_psi_batch(Lsr, wb, m, psi, d_e + (size_t)j0 * p.nbc * cs, (size_t)p.nbc * cs, n0, s);
            }));
            j0 = j + 1;
          }
        }
        const size_t ps = (size_t)Lgs.n_slices * Lgs.gridx * Lgs.groups_per_slice() * nvo;
        const int gmax = gram_betas(ps, nb);
        for (int r = 0; r < nb; r += gmax) {
          const int nq = std::min(gmax, nb - r);
          CK(timed(kKGram, bs * nq, [&] {
            return launch_final_gram(Lgs, psi + (size_t)r * Ls.block_bytes(), nq, partials, ps, s);
          }));
          CK(counted([&] { return launch_reduce_gram(Lgs, partials, ps, nq, d_gram + (size_t)r * cso, s); }));
        }
        CK(cudaMemcpyAsync(hg.data(), d_gram, (size_t)nb * cso * sizeof(double), cudaMemcpyDeviceToHost, s));
        d2h += (size_t)nb * cso * sizeof(double);
        CK(cudaStreamSynchronize(s));
        for (int r = 0; r < nb; ++r)
          for (int l = g0o; l < std::min(n_v, g0o + ngso); ++l)
            for (int v = 0; v < nvo; ++v)
              gram[((size_t)(b0 + ord[r]) * n_v + l) * nvo + v] = hg[((size_t)r * ngso + (l - g0o)) * nvo + v];
      }
      continue;
    }
    CK(cudaMemcpyAsync(hg.data(), d_gram, (size_t)nb * cstride_g * sizeof(double),
                       cudaMemcpyDeviceToHost, s));
    d2h += (size_t)nb * cstride_g * sizeof(double);
    CK(cudaStreamSynchronize(s));
    for (int bi = 0; bi < nb; ++bi)
      for (int l = 0; l < n_v; ++l)
        for (int v = 0; v < nvo; ++v)
          gram[((size_t)(b0 + bi) * n_v + l) * nvo + v] = hg[((size_t)bi * ngo + l) * nvo + v];
  }
  CK(cudaMemcpyAsync(flags, d_flags, sizeof flags, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  d2h += sizeof flags;
  if (prof) {
    prof->collect();
    if (prof->on) {
      prof->launches[kKHostDense]++;
      prof->ms[kKHostDense] += host_ms;
    }
  }

  // ---- normalisation (eq. rho_est) and ln Z_t.
  auto finish = [&](const std::vector<double>& g, double* rho, double* lnz) -> bool {
    return normalise_grams(g, n_beta, n_v, dso, (double)d_b, betas, e0, rho, lnz);
  };
  const bool gram_main = o->form == RDM_GRAM;
  bool ok = finish(gram_main ? gram : quad, out->rho, out->ln_z);
  if (out->rho_other) finish(gram_main ? quad : gram, out->rho_other, nullptr);
  if (out->gram_l) std::copy(gram.begin(), gram.end(), out->gram_l);
  if (out->quad_l) std::copy(quad.begin(), quad.end(), out->quad_l);
  if (out->t_a || out->t_b)
    for (int l = 0; l < n_v; ++l)
      for (int j = 0; j < k; ++j)
        for (int v = 0; v < nvo; ++v) {
          double a = 0.0, b = 0.0;
          if (!p.single) {
            a = ta[((size_t)j * ng + l) * nv + v];
            b = tb[((size_t)j * ng + l) * nv + v];
          } else if (v % (dso + 1) == 0) {  // diagonal: column l dso + v / dso
            a = ta[(size_t)j * ng + (size_t)l * dso + v / dso];
            b = tb[(size_t)j * ng + (size_t)l * dso + v / dso];
          }
          if (out->t_a) out->t_a[((size_t)l * k + j) * nvo + v] = a;
          if (out->t_b) out->t_b[((size_t)l * k + j) * nvo + v] = b;
        }
  out->e0 = e0;
  out->h2d_bytes = h2d;
  out->d2h_bytes = d2h;
  out->flags = (flags[0] & RDM_FLAG_DEFLATED) | (p.n_v_pad != n_rec ? RDM_FLAG_PADDED : 0u);
  if (!ok) {
    set_error("the estimated tr(sum_l G_l) is not a positive finite number (underflow or breakdown)");
    return RDM_ENUMERIC;
  }
  return RDM_OK;
}

// Bath vectors per shard when an estimate's vectors run in consecutive shards that each
// keep their whole Krylov basis: the estimator is a sum over bath vectors (eq.
// trace_est), so shards of whole slices run one after another in the same workspace,
// each with one pass of the recurrence and the stored-basis Gram, instead of two passes
// over all of them. Chosen when the whole basis does not fit in `avail` but a shard's
// does (the largest such shard); 0 otherwise.
static int store_shard_vectors(const HostModel& h, int n_beta, int n_v, int k, const rdm_opts* o, size_t avail,
                               double beta_max, Plan* shard_plan) {
  if (o->passes != RDM_PASSES_AUTO || o->recurrence != RDM_BLOCK) return 0;
  const std::string saved = rdm_last_error();  // the trial plans below may fail quietly
  rdm_opts q = *o;
  q.passes = RDM_PASSES_STORE;
  Plan p;
  int n_found = 0;
  Layout L;
  int pad = 0;
  if (make_plan(h, n_beta, n_v, k, &q, avail, &p, beta_max) != RDM_OK &&
      plan_layout(h, n_v, o->precision, &L, &pad) == RDM_OK) {
    const int vps = L.groups_per_slice();  // bath vectors per slice
    for (int ns = L.n_slices - 1; ns >= 1 && n_found == 0; --ns) {
      const int n_sh = ns * vps;
      if (n_sh >= n_v) continue;
      if (make_plan(h, n_beta, n_sh, k, &q, avail, &p, beta_max) == RDM_OK) {
        if (shard_plan) *shard_plan = p;
        n_found = n_sh;
      }
    }
  }
  set_error("%s", saved.c_str());
  return n_found;
}

// The shards of store_shard_vectors, folded as the whole run: shard r's Gram sums are
// relative to its own shift E0_r, so each is scaled by exp(-beta (E0_r - E0)) with E0
// the smallest of them (Sec. 3.2), then normalised as eq. rho_est.
static rdm_status estimate_shards(rdm_ham* ham, cudaStream_t s, char* ws, size_t ws_bytes, const double* betas,
                                  int n_beta, int n_v, int k, uint64_t seed, const rdm_opts* o, rdm_result* out,
                                  Profiler* prof, int n_sh) {
  const HostModel& hm = ham->model;
  const int dso = 1 << hm.ns, nvo = dso * dso;
  const double d_b = std::ldexp(1.0, hm.n - hm.ns);
  std::vector<double> gram((size_t)n_beta * n_v * nvo), quad(gram.size()), e0s;
  std::vector<int> offs;
  rdm_opts q = *o;
  q.passes = RDM_PASSES_STORE;
  uint32_t flags = 0;
  uint64_t h2d = 0, d2h = 0;
  for (int off = 0; off < n_v; off += n_sh) {
    const int cnt = std::min(n_sh, n_v - off);
    q.first_vector = o->first_vector + off;
    std::vector<double> rho((size_t)n_beta * nvo), lnz(n_beta), g((size_t)n_beta * cnt * nvo), qd(g.size());
    rdm_result r{};
    r.rho = rho.data();
    r.ln_z = lnz.data();
    r.gram_l = g.data();
    r.quad_l = qd.data();
    r.t_a = out->t_a ? out->t_a + (size_t)off * k * nvo : nullptr;
    r.t_b = out->t_b ? out->t_b + (size_t)off * k * nvo : nullptr;
    EstimateRun run(ham, s, betas, n_beta, cnt, k, seed, &q, &r, prof);
    rdm_status st = run.prepare(ws, ws_bytes);
    if (st == RDM_OK) st = run.pass1(s, true);
    if (st == RDM_OK) st = run.finish();
    if (st != RDM_OK) return st;
    e0s.push_back(r.e0);
    offs.push_back(off);
    flags |= r.flags;
    h2d += r.h2d_bytes;
    d2h += r.d2h_bytes;
    for (int bi = 0; bi < n_beta; ++bi)
      for (int l = 0; l < cnt; ++l)
        for (int v = 0; v < nvo; ++v) {
          gram[((size_t)bi * n_v + off + l) * nvo + v] = g[((size_t)bi * cnt + l) * nvo + v];
          quad[((size_t)bi * n_v + off + l) * nvo + v] = qd[((size_t)bi * cnt + l) * nvo + v];
        }
  }
  const double e0 = *std::min_element(e0s.begin(), e0s.end());
  for (size_t r = 0; r < offs.size(); ++r) {
    const int cnt = std::min(n_sh, n_v - offs[r]);
    for (int bi = 0; bi < n_beta; ++bi) {
      const double f = std::exp(-betas[bi] * (e0s[r] - e0));
      for (int l = 0; l < cnt; ++l)
        for (int v = 0; v < nvo; ++v) {
          gram[((size_t)bi * n_v + offs[r] + l) * nvo + v] *= f;
          quad[((size_t)bi * n_v + offs[r] + l) * nvo + v] *= f;
        }
    }
  }
  auto finish = [&](const std::vector<double>& g, double* rho, double* lnz) -> bool {
    return normalise_grams(g, n_beta, n_v, dso, d_b, betas, e0, rho, lnz);
  };
  const bool gram_main = o->form == RDM_GRAM;
  const bool ok = finish(gram_main ? gram : quad, out->rho, out->ln_z);
  if (out->rho_other) finish(gram_main ? quad : gram, out->rho_other, nullptr);
  if (out->gram_l) std::copy(gram.begin(), gram.end(), out->gram_l);
  if (out->quad_l) std::copy(quad.begin(), quad.end(), out->quad_l);
  out->e0 = e0;
  out->flags = flags;
  out->h2d_bytes = h2d;
  out->d2h_bytes = d2h;
  if (!ok) {
    set_error("the estimated tr(sum_l G_l) is not a positive finite number (underflow or breakdown)");
    return RDM_ENUMERIC;
  }
  return RDM_OK;
}

rdm_status estimate_impl(rdm_ham* ham, cudaStream_t s, char* ws, size_t ws_bytes,
                         const double* betas, int n_beta, int n_v, int k, uint64_t seed,
                         const rdm_opts* o, rdm_result* out, Profiler* prof) {
  const int n_sh =
      store_shard_vectors(ham->model, n_beta, n_v, k, o, ws_bytes, max_beta(betas, n_beta), nullptr);
  if (n_sh > 0) return estimate_shards(ham, s, ws, ws_bytes, betas, n_beta, n_v, k, seed, o, out, prof, n_sh);
  EstimateRun run(ham, s, betas, n_beta, n_v, k, seed, o, out, prof);
  rdm_status st = run.prepare(ws, ws_bytes);
  if (st == RDM_OK) st = run.pass1(s, true);
  if (st == RDM_OK) st = run.finish();
  return st;
}

// ---------------------------------------------------------------- batches

// Bytes of one launch's descriptors (items, step and prefix tables, barrier words).
static constexpr size_t packed_meta_bytes(int n_items, int k_max) {
  return ((sizeof(PackedItem) * (size_t)n_items + sizeof(int) * ((size_t)k_max + 2 + 3 * ((size_t)n_items + 1)) +
           64 + 255) / 256) * 256;
}

// Bytes at the front of a batch workspace for the descriptors of all its launches: at most
// kBatchLaunches (a cluster launch per d_s and tiles per slice, a packed launch per precision
// and d_s), which part the items but have a table of steps each.
constexpr int kBatchLaunches = 3 * (kClusterMaxLog + 1) + 6;
static constexpr size_t batch_meta_bytes(int n_items, int k_max) { return 6 * packed_meta_bytes(n_items, k_max); }
// The largest sum of the launches' descriptors: every launch with the largest k and its size
// rounded up by all it can be.
static constexpr bool batch_meta_holds() {
  for (int n = 1; n <= 4 * kBatchLaunches; ++n)  // beyond, six times an item's bytes outgrow one item's
    for (int k = 1; k <= kMaxSteps; ++k) {
      const size_t launches = n < kBatchLaunches ? n : kBatchLaunches;
      const size_t sum = (size_t)n * (sizeof(PackedItem) + 3 * sizeof(int)) + launches * (packed_meta_bytes(0, k) + 255);
      if (sum > batch_meta_bytes(n, k)) return false;
    }
  return true;
}
static_assert(batch_meta_holds(), "descriptors of a batch's launches");

// One packed launch for the items `idx` of `runs` (same precision and d_s), with the
// grid chosen by the autotuner. meta: device scratch of packed_meta_bytes.
static rdm_status run_packed(rdm_ctx* ctx, cudaStream_t s, std::vector<EstimateRun*>& runs, int precision,
                             int ds, char* meta, Profiler* prof) {
  std::stable_sort(runs.begin(), runs.end(),
                   [](const EstimateRun* a, const EstimateRun* b) { return a->plan().k > b->plan().k; });
  const int n = (int)runs.size();
  const int k_max = runs[0]->plan().k;
  std::vector<PackedItem> items(n);
  std::vector<int> pre_rows(n + 1, 0), pre_groups(n + 1, 0), pre_slices(n + 1, 0), active(k_max + 1, 0);
  size_t smem = 16;
  double bytes = 0.0;
  for (int i = 0; i < n; ++i) {
    items[i] = runs[i]->packed_item();
    const Layout& L = items[i].L;
    pre_rows[i + 1] = pre_rows[i] + L.gridx * L.n_slices;
    pre_groups[i + 1] = pre_groups[i] + L.n_groups();
    pre_slices[i + 1] = pre_slices[i] + L.n_slices;
    smem = std::max(smem, spmm_terms_smem(precision, items[i].sa.n_flip, items[i].sa.n_diag));
    bytes += 6.0 * (double)L.block_bytes() * items[i].k;  // SpMM 3 blocks + orth 3 blocks per step
  }
  for (int j = 1; j <= k_max; ++j) {
    int na = 0;
    while (na < n && items[na].k >= j) ++na;
    active[j] = na;
  }
  // host image of the descriptors, one copy
  const size_t o_items = 0, o_active = sizeof(PackedItem) * n;
  const size_t o_rows = o_active + sizeof(int) * (k_max + 1), o_groups = o_rows + sizeof(int) * (n + 1);
  const size_t o_slices = o_groups + sizeof(int) * (n + 1);
  const size_t o_bar = (o_slices + sizeof(int) * (n + 1) + 15) / 16 * 16;
  std::vector<char> img(o_bar);
  std::memcpy(img.data() + o_items, items.data(), sizeof(PackedItem) * n);
  std::memcpy(img.data() + o_active, active.data(), sizeof(int) * (k_max + 1));
  std::memcpy(img.data() + o_rows, pre_rows.data(), sizeof(int) * (n + 1));
  std::memcpy(img.data() + o_groups, pre_groups.data(), sizeof(int) * (n + 1));
  std::memcpy(img.data() + o_slices, pre_slices.data(), sizeof(int) * (n + 1));
  CK(cudaMemcpyAsync(meta, img.data(), img.size(), cudaMemcpyHostToDevice, s));
  PackedPlan pp{};
  pp.items = reinterpret_cast<const PackedItem*>(meta + o_items);
  pp.n_items = n;
  pp.k_max = k_max;
  pp.active = reinterpret_cast<const int*>(meta + o_active);
  pp.pre_rows = reinterpret_cast<const int*>(meta + o_rows);
  pp.pre_groups = reinterpret_cast<const int*>(meta + o_groups);
  pp.pre_slices = reinterpret_cast<const int*>(meta + o_slices);
  pp.bar = reinterpret_cast<uint32_t*>(meta + o_bar);
  // the pageable host image must outlive its copy
  CK(cudaStreamSynchronize(s));

  int sms = 0;
  CK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, ctx->device));
  const int max_bpsm = packed_max_blocks_per_sm(precision, ds, smem);
  if (max_bpsm < 1) {
    set_error("packed first pass: no block fits an SM (%zu bytes of term tables)", smem);
    return RDM_EINVAL;
  }
  const int units = std::max(pre_rows[n], pre_groups[n]);
  auto grid_for = [&](int bpsm) { return std::max(1, std::min(bpsm * sms, units)); };
  // bpsm > 0: the cooperative launch on bpsm blocks per SM; kLocal: one block per slice
  constexpr int kLocal = -1;
  auto launch = [&](int bpsm) -> cudaError_t {
    cudaError_t e = cudaMemsetAsync(pp.bar, 0, 3 * sizeof(uint32_t), s);
    if (e != cudaSuccess) return e;
    if (bpsm == kLocal) return launch_pass1_local(precision, ds, pp, pre_slices[n], smem, s);
    return launch_pass1_packed(precision, ds, pp, grid_for(bpsm), smem, s);
  };
  // Autotuner: key = (precision, d_s, size class = log2 of the block-sized units of the
  // batch, in steps of 3 (a factor 8)).
  int lg = 0;
  while ((1 << lg) < pre_rows[n]) ++lg;
  lg /= 3;
  const uint64_t key = (uint64_t)precision | ((uint64_t)ds << 4) | ((uint64_t)lg << 8);
  int bpsm = 0;
  {
    std::lock_guard<std::mutex> lk(ctx->tuning.mu);
    auto f = ctx->tuning.blocks_per_sm.find(key);
    if (f != ctx->tuning.blocks_per_sm.end()) bpsm = f->second == kLocal ? kLocal : std::min(f->second, max_bpsm);
  }
  if (bpsm == 0) {
    // Time each candidate once on this batch (the first pass is idempotent: it only
    // reads the starting block and M_1, Cp_1), keep the fastest for the key. Both
    // launch forms run the same units with the same arithmetic: the choice does not
    // change a result.
    std::vector<int> cand;
    int form = 0;
    {
      std::lock_guard<std::mutex> lk(ctx->tuning.mu);
      form = ctx->packed_form;
    }
    if (form != 2)
      for (int c : {1, 2, 4, 8})
        if (c <= max_bpsm && (cand.empty() || grid_for(c) > grid_for(cand.back()))) cand.push_back(c);
    if (form != 1) cand.push_back(kLocal);
    cudaEvent_t e0, e1;
    CK(cudaEventCreate(&e0));
    CK(cudaEventCreate(&e1));
    float best = 0.0f;
    for (int c : cand) {
      CK(cudaEventRecord(e0, s));
      CK(launch(c));
      CK(cudaEventRecord(e1, s));
      CK(cudaEventSynchronize(e1));
      float ms = 0.0f;
      CK(cudaEventElapsedTime(&ms, e0, e1));
      if (bpsm == 0 || ms < best) {
        best = ms;
        bpsm = c;
      }
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    std::lock_guard<std::mutex> lk(ctx->tuning.mu);
    ctx->tuning.blocks_per_sm[key] = bpsm;
    ctx->tuning.tuning_runs += cand.size();
  }
  const int ev = prof ? prof->begin(kKPacked, s, true) : -1;
  const cudaError_t le = launch(bpsm);
  if (prof) prof->end(kKPacked, ev, s, bytes);
  CK(le);
  uint32_t bar_err = 0;
  CK(cudaMemcpyAsync(&bar_err, pp.bar + 2, sizeof bar_err, cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  if (bar_err) {
    set_error("packed first pass: a grid-barrier wait gave up (device error)");
    return RDM_ECUDA;
  }
  return RDM_OK;
}

// The first passes of `runs` in clusters: one launch per (d_s, tiles per slice), the
// launches side by side on a few streams (on s alone while launches are timed), joined
// before return. meta: device scratch for the descriptors (packed_meta_bytes of each group);
// *used: bytes of it taken. keep: the descriptors' host images, which must outlive the work.
static rdm_status run_clusters(cudaStream_t s, const std::vector<EstimateRun*>& runs, char* meta, size_t* used,
                               std::vector<std::vector<char>>* keep, Profiler* prof) {
  struct Group {
    int ds, c_log, n_slices = 0, k = 0;
    size_t smem = 0;
    double bytes = 0.0;
    std::vector<PackedItem> items;
    std::vector<int> pre{0};
  };
  std::map<std::pair<int, int>, Group> groups;
  for (const EstimateRun* r : runs) {
    const PackedItem it = r->packed_item();
    const std::pair<int, int> key(it.L.DS, it.L.n_bits - kTileBits);
    Group& g = groups[key];
    g.ds = key.first;
    g.c_log = key.second;
    g.items.push_back(it);
    g.n_slices += it.L.n_slices;
    g.pre.push_back(g.n_slices);
    g.k = std::max(g.k, it.k);
    g.smem = std::max(g.smem, pass1_cluster_smem(it.sa.tiled));
    g.bytes += 6.0 * (double)it.L.block_bytes() * it.k;
  }
  // the longest launches first (steps times blocks)
  std::vector<Group*> order;
  for (auto& kv : groups) order.push_back(&kv.second);
  std::stable_sort(order.begin(), order.end(), [](const Group* x, const Group* y) {
    return ((int64_t)x->k * x->n_slices << x->c_log) > ((int64_t)y->k * y->n_slices << y->c_log);
  });
  // Forked before the first launch: the side streams wait for what s holds now (the items'
  // starting blocks), not for that launch.
  SideStreams side;
  const int n_side = prof && prof->on ? 0 : (int)std::min(side.size(), order.size() - 1);
  rdm_status st = fork_all(side, n_side, s);
  for (size_t q = 0; q < order.size() && st == RDM_OK; ++q) {
    Group& g = *order[q];
    // (launches of items with different k do not need the k-sorted order of the packed grid)
    const size_t o_pre = sizeof(PackedItem) * g.items.size();
    std::vector<char> img(o_pre + sizeof(int) * g.pre.size());
    std::memcpy(img.data(), g.items.data(), o_pre);
    std::memcpy(img.data() + o_pre, g.pre.data(), sizeof(int) * g.pre.size());
    char* dev = meta + *used;
    *used += packed_meta_bytes((int)g.items.size(), g.k);
    cudaStream_t ls = n_side && q > 0 ? side[(q - 1) % n_side].stream : s;
    PackedPlan pp{};
    pp.items = reinterpret_cast<const PackedItem*>(dev);
    pp.n_items = (int)g.items.size();
    pp.k_max = g.k;
    pp.pre_slices = reinterpret_cast<const int*>(dev + o_pre);
    cudaError_t e = cudaMemcpyAsync(dev, img.data(), img.size(), cudaMemcpyHostToDevice, ls);
    keep->push_back(std::move(img));
    const int ev = prof ? prof->begin(kKPacked, ls, true) : -1;
    if (e == cudaSuccess) e = launch_pass1_cluster(g.ds, pp, g.c_log, g.n_slices, g.smem, ls);
    if (prof) prof->end(kKPacked, ev, ls, g.bytes);
    if (e != cudaSuccess) {
      set_error("first pass in clusters: %s", cudaGetErrorString(e));
      st = RDM_ECUDA;
    }
  }
  const rdm_status sj = join_all(side, n_side, s);
  return st != RDM_OK ? st : sj;
}

rdm_status estimate_batch_impl(rdm_ctx* ctx, cudaStream_t s, char* ws, size_t ws_bytes,
                               rdm_batch_item* items, int n, const size_t* need, Profiler* prof) {
  std::vector<std::unique_ptr<EstimateRun>> runs(n);
  size_t off = 0;
  // the launches' descriptors go first, then those of the device small dense step
  int k_max = 1;
  for (int i = 0; i < n; ++i) k_max = std::max(k_max, items[i].k);
  const size_t meta_b = batch_meta_bytes(n, k_max);
  char* meta = ws;
  off = meta_b + dense_jobs_bytes(n);
  rdm_status first_bad = RDM_OK;
  bool clusters = true;  // (a packed_form other than 0 asks for the untiled units)
  if (ctx) {
    std::lock_guard<std::mutex> lk(ctx->tuning.mu);
    clusters = ctx->packed_form == 0;
  }
  for (int i = 0; i < n; ++i) {
    rdm_batch_item& it = items[i];
    runs[i] = std::make_unique<EstimateRun>(it.ham, s, it.betas, it.n_beta, it.n_v, it.k, it.seed, &it.opts,
                                            it.out, prof);
    runs[i]->in_clusters = clusters;
    it.status = runs[i]->prepare(ws + off, need[i]);
    off += need[i];
    if (it.status != RDM_OK && first_bad == RDM_OK) first_bad = it.status;
  }
  // First passes in clusters, and the others packed, one launch per (precision, d_s); their
  // descriptors follow one another in meta (batch_meta_holds).
  size_t meta_off = 0;
  std::vector<std::vector<char>> keep;
  {
    std::vector<EstimateRun*> group;
    std::vector<int> idx;
    for (int i = 0; i < n; ++i)
      if (items[i].status == RDM_OK && runs[i]->in_clusters) {
        group.push_back(runs[i].get());
        idx.push_back(i);
      }
    if (!group.empty()) {
      const rdm_status st = run_clusters(s, group, meta, &meta_off, &keep, prof);
      for (int i : idx) {
        if (st != RDM_OK) items[i].status = st;
        runs[i]->packed_done = true;
      }
      if (st != RDM_OK && first_bad == RDM_OK) first_bad = st;
    }
  }
  for (int prec : {RDM_FP32, RDM_FP64})
    for (int ds : {1, 2, 4}) {
      std::vector<EstimateRun*> group;
      std::vector<int> idx;
      for (int i = 0; i < n; ++i)
        if (items[i].status == RDM_OK && runs[i]->packable() && !runs[i]->in_clusters &&
            !(clusters && runs[i]->tiled_launches()) &&
            runs[i]->plan().L.precision == prec && runs[i]->plan().L.DS == ds) {
          group.push_back(runs[i].get());
          idx.push_back(i);
        }
      if (group.empty()) continue;
      int group_k = 1;
      for (int i : idx) group_k = std::max(group_k, items[i].k);
      const rdm_status st = run_packed(ctx, s, group, prec, ds, meta + meta_off, prof);
      meta_off += packed_meta_bytes((int)group.size(), group_k);
      if (st != RDM_OK)
        for (int i : idx) {
          items[i].status = st;
          if (first_bad == RDM_OK) first_bad = st;
        }
      for (int i : idx) items[i].status = items[i].status == RDM_OK ? RDM_OK : items[i].status;
      for (int i : idx) runs[i]->packed_done = true;
    }
  // First passes of the other items, side by side on a few streams: an item of few tiles
  // fills a part of the GPU and is bound by its launches' latency. One after another, with a
  // host wait each, 40 items of one slice (N = 15, d_s = 4) took 91 ms where the packed launch
  // took 32; on 4 streams 34.8, on 6 28.0, on 8 24.2. Then every item's T back to the host.
  {
    std::vector<int> own;
    for (int i = 0; i < n; ++i)
      if (items[i].status == RDM_OK && !runs[i]->packed_done) own.push_back(i);
    SideStreams side;
    const int n_side = prof && prof->on ? 0 : (int)std::min(side.size(), own.empty() ? 0 : own.size() - 1);
    rdm_status st = fork_all(side, n_side, s);
    for (size_t q = 0; q < own.size(); ++q) {
      const size_t w = n_side ? q % (n_side + 1) : 0;
      if (st == RDM_OK) items[own[q]].status = runs[own[q]]->pass1(w ? side[w - 1].stream : s, own.size() == 1);
    }
    const rdm_status sj = join_all(side, n_side, s);
    if (st == RDM_OK) st = sj;
    for (int i : own) {
      if (st != RDM_OK) items[i].status = st;
      if (items[i].status != RDM_OK && first_bad == RDM_OK) first_bad = items[i].status;
    }
  }
  for (int i = 0; i < n; ++i) {
    if (items[i].status != RDM_OK) continue;
    const rdm_status st = runs[i]->fetch_t();
    items[i].status = st;
    if (st != RDM_OK && first_bad == RDM_OK) first_bad = st;
  }
  // the device small dense steps of all items that take it: one launch per d_s over all
  // their recurrences
  char* dense_meta = ws + meta_b;
  for (int ds : {1, 2, 4}) {
    std::vector<DenseJob> jobs;
    std::vector<int> idx;
    for (int i = 0; i < n; ++i)
      if (items[i].status == RDM_OK && runs[i]->wants_device && runs[i]->rec_ds() == ds) {
        const rdm_status st = runs[i]->upload_betas();
        if (st != RDM_OK) {
          items[i].status = st;
          continue;
        }
        jobs.push_back(runs[i]->dense_job());
        idx.push_back(i);
      }
    if (jobs.empty()) continue;
    const int ev = prof ? prof->begin(kKDense, s, true) : -1;
    const cudaError_t e = launch_dense_jobs(ds, jobs.data(), (int)jobs.size(), dense_meta, s);
    if (prof) prof->end(kKDense, ev, s, 0.0);
    for (int i : idx) {
      rdm_status st = RDM_OK;
      if (e != cudaSuccess) {
        set_error("device small dense step: %s", cudaGetErrorString(e));
        st = RDM_ECUDA;
      } else {
        st = runs[i]->fetch_dense();
      }
      items[i].status = st;
      if (st != RDM_OK && first_bad == RDM_OK) first_bad = st;
    }
  }
  // the small dense steps of all items in one pass over the host worker pool
  std::vector<std::pair<int, int>> tasks;
  for (int i = 0; i < n; ++i)
    if (items[i].status == RDM_OK)
      for (int r = 0; r < runs[i]->n_dense_tasks(); ++r) tasks.emplace_back(i, r);
  const auto t0 = std::chrono::steady_clock::now();
  parallel_for((int)tasks.size(), [&](int t) { runs[tasks[t].first]->dense_task(tasks[t].second); });
  const double dense_ms = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  for (int i = 0; i < n; ++i) {
    if (items[i].status != RDM_OK) continue;
    // the pass's wall time, shared out by the items' task counts (items whose step ran on
    // the device keep their own time)
    if (runs[i]->n_dense_tasks() > 0)
      runs[i]->host_ms_dense = dense_ms * runs[i]->n_dense_tasks() / (double)tasks.size();
    const rdm_status st = runs[i]->finish_rest();
    items[i].status = st;
    if (st != RDM_OK && first_bad == RDM_OK) first_bad = st;
  }
  return first_bad;
}

size_t batch_workspace_bytes(const rdm_batch_item* items, int n, const size_t* avail, size_t* need) {
  int k_max = 1;
  for (int i = 0; i < n; ++i) k_max = std::max(k_max, items[i].k);
  size_t tot = batch_meta_bytes(n, k_max) + dense_jobs_bytes(n);
  for (int i = 0; i < n; ++i) {
    rdm_status st = RDM_OK;
    need[i] = estimate_bytes(items[i].ham->model, items[i].n_beta, items[i].n_v, items[i].k, &items[i].opts,
                             avail[i], &st, max_beta(items[i].betas, items[i].n_beta));
    if (need[i] == 0) return 0;
    need[i] = (need[i] + 255) / 256 * 256;
    tot += need[i];
  }
  return tot;
}

}  // namespace rdm

static bool valid_opts(const rdm_opts* o);

// Grows the context-owned workspace to at least `need` bytes. A grown workspace gets
// 1/8 of headroom (within `usable`), so calls whose plans differ slightly (another
// Hamiltonian's Chebyshev bound, another k) reuse it instead of freeing and
// reallocating it -- which would also invalidate the first-pass graphs keyed on its
// addresses.
static rdm_status grow_own_workspace(rdm_ctx* ctx, size_t need, size_t usable) {
  if (ctx->own_bytes >= need) return RDM_OK;
  CK(cudaStreamSynchronize(ctx->stream));
  if (ctx->own_ws) CK(cudaFree(ctx->own_ws));
  ctx->own_ws = nullptr;
  ctx->own_bytes = 0;
  size_t want = need + need / 8;
  want = (want + (size_t(1) << 21) - 1) / (size_t(1) << 21) * (size_t(1) << 21);
  if (want > usable) want = need;
  if (cudaMalloc(reinterpret_cast<void**>(&ctx->own_ws), want) != cudaSuccess) {
    cudaGetLastError();
    want = need;
    CK(cudaMalloc(reinterpret_cast<void**>(&ctx->own_ws), want));
  }
  ctx->own_bytes = want;
  return RDM_OK;
}

extern "C" rdm_status rdm_estimate_batch(rdm_ctx* ctx, rdm_batch_item* items, int n_items) {
  if (!ctx || !items || n_items < 1) {
    set_error("rdm_estimate_batch: NULL context or items, or n_items < 1");
    return RDM_EINVAL;
  }
  for (int i = 0; i < n_items; ++i) {
    items[i].status = RDM_EINVAL;
    if (!items[i].ham || items[i].ham->ctx != ctx) {
      set_error("rdm_estimate_batch: item %d has no Hamiltonian of this context", i);
      return RDM_EINVAL;
    }
    rdm_status st = check_estimate_args(items[i].ham, items[i].betas, items[i].n_beta, &items[i].opts,
                                        items[i].out);
    if (st != RDM_OK) return st;
  }
  CK(cudaSetDevice(ctx->device));
  size_t free_b = 0, total_b = 0;
  CK(cudaMemGetInfo(&free_b, &total_b));
  const size_t usable = ctx->ws ? ctx->ws_bytes : (size_t)(0.85 * (double)(free_b + ctx->own_bytes));
  // Items run in consecutive sub-batches whose workspaces fit together; an item whose
  // sizes are invalid or that does not fit on its own fails alone.
  rdm_status first_bad = RDM_OK;
  std::vector<rdm_batch_item*> ok_items;
  for (int i = 0; i < n_items; ++i) {
    rdm_status st = RDM_OK;
    const size_t need = estimate_bytes(items[i].ham->model, items[i].n_beta, items[i].n_v, items[i].k,
                                       &items[i].opts, usable, &st, max_beta(items[i].betas, items[i].n_beta));
    if (need == 0) {
      items[i].status = st != RDM_OK ? st : RDM_ENOMEM;
      if (first_bad == RDM_OK) first_bad = items[i].status;
      continue;
    }
    ok_items.push_back(&items[i]);
  }
  size_t i0 = 0;
  while (i0 < ok_items.size()) {
    // greedy: as many consecutive items as fit (at least one)
    std::vector<rdm_batch_item> sub;
    std::vector<size_t> need;
    size_t tot = 0;
    size_t i1 = i0;
    std::vector<size_t> avail;
    while (i1 < ok_items.size()) {
      sub.push_back(*ok_items[i1]);
      need.assign(sub.size(), 0);
      avail.assign(sub.size(), usable);
      const size_t t2 = batch_workspace_bytes(sub.data(), (int)sub.size(), avail.data(), need.data());
      if (t2 == 0 || (t2 > usable && i1 > i0)) {
        sub.pop_back();
        break;
      }
      tot = t2;
      ++i1;
    }
    need.assign(sub.size(), 0);
    avail.assign(sub.size(), usable);
    tot = batch_workspace_bytes(sub.data(), (int)sub.size(), avail.data(), need.data());
    char* ws = ctx->ws;
    rdm_status st = RDM_OK;
    if (tot > usable) {
      set_error("rdm_estimate_batch: an item needs %zu bytes of device memory, %zu usable", tot, usable);
      st = RDM_ENOMEM;
    } else if (!ws) {
      st = grow_own_workspace(ctx, tot, usable);
      ws = ctx->own_ws;
    }
    if (st == RDM_OK)
      st = estimate_batch_impl(ctx, ctx->stream, ws, tot, sub.data(), (int)sub.size(), need.data(), &ctx->prof);
    for (size_t q = 0; q < sub.size(); ++q) ok_items[i0 + q]->status = st == RDM_ENOMEM && tot > usable ? st
                                                                                                       : sub[q].status;
    if (st != RDM_OK && first_bad == RDM_OK) first_bad = st;
    i0 = i1;
  }
  return first_bad;
}

extern "C" rdm_status rdm_packed_tuning(rdm_ctx* ctx, int* n_keys, uint64_t* tuning_runs) {
  if (!ctx) {
    set_error("rdm_packed_tuning: NULL context");
    return RDM_EINVAL;
  }
  std::lock_guard<std::mutex> lk(ctx->tuning.mu);
  if (n_keys) *n_keys = (int)ctx->tuning.blocks_per_sm.size();
  if (tuning_runs) *tuning_runs = ctx->tuning.tuning_runs;
  return RDM_OK;
}

static bool valid_opts(const rdm_opts* o) {
  return o && (o->precision == RDM_FP32 || o->precision == RDM_FP64) &&
         (o->vec_dist == RDM_RADEMACHER || o->vec_dist == RDM_GAUSS || o->vec_dist == RDM_BASIS) &&
         (o->form == RDM_GRAM || o->form == RDM_QUADRATURE) &&
         (o->passes == RDM_PASSES_AUTO || o->passes == RDM_PASSES_STORE ||
          o->passes == RDM_PASSES_RECOMPUTE) &&
         o->first_vector >= 0 && o->first_vector < (int64_t(1) << 23);
}

rdm_status rdm::check_estimate_args(const rdm_ham* ham, const double* betas, int n_beta,
                                    const rdm_opts* opts, const rdm_result* out) {
  if (!ham || !betas || !out || !out->rho) {
    set_error("rdm_estimate: ham, betas, out and out->rho must be non-NULL");
    return RDM_EINVAL;
  }
  if (!valid_opts(opts)) {
    set_error("rdm_estimate: invalid opts");
    return RDM_EINVAL;
  }
  for (int i = 0; i < n_beta; ++i)
    if (!(betas[i] >= 0) || !std::isfinite(betas[i])) {
      set_error("rdm_estimate: beta[%d] must be finite and >= 0", i);
      return RDM_EINVAL;
    }
  return RDM_OK;
}

extern "C" rdm_status rdm_estimate(rdm_ham* ham, const double* betas, int n_beta, int n_v, int k,
                                   uint64_t seed, const rdm_opts* opts, rdm_result* out) {
  rdm_status st = check_estimate_args(ham, betas, n_beta, opts, out);
  if (st != RDM_OK) return st;
  rdm_ctx* ctx = ham->ctx;
  CK(cudaSetDevice(ctx->device));
  if (ctx->ws)
    return estimate_impl(ham, ctx->stream, ctx->ws, ctx->ws_bytes, betas, n_beta, n_v, k, seed, opts,
                         out, &ctx->prof);
  // Context-owned workspace: sized by what the plan needs given the device memory
  // this context may use (85% of what is free plus what it already holds), kept
  // for later calls.
  size_t free_b = 0, total_b = 0;
  CK(cudaMemGetInfo(&free_b, &total_b));
  const size_t usable = (size_t)(0.85 * (double)(free_b + ctx->own_bytes));
  rdm_status pst = RDM_OK;
  size_t need = estimate_bytes(ham->model, n_beta, n_v, k, opts, usable, &pst, max_beta(betas, n_beta));
  if (need == 0) return pst != RDM_OK ? pst : RDM_ENOMEM;  // make_plan set the message
  {
    Plan sp;  // shards that keep their basis take the workspace of one shard's plan
    if (store_shard_vectors(ham->model, n_beta, n_v, k, opts, usable, max_beta(betas, n_beta), &sp) > 0)
      need = plan_bytes(sp);
  }
  const rdm_status gst = grow_own_workspace(ctx, need, usable);
  if (gst != RDM_OK) return gst;
  return estimate_impl(ham, ctx->stream, ctx->own_ws, ctx->own_bytes, betas, n_beta, n_v, k, seed,
                       opts, out, &ctx->prof);
}
