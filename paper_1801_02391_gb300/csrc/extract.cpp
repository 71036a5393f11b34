// Host steps of the single-pulse extraction (Sec. 2.4): grouping of candidate signals
// across windows (step b), MBD consistency (step c), window count and best member
// (step d), the DM merge of the coarse DM search (Sec. 5.3) and cross-matching of
// baselines.  Sequential and O(events x window length): each insertion asks "which
// is the first group (in creation order) holding a member whose [k0, k0 + l) overlaps
// mine", answered from a per-AP array of the smallest group id covering that AP.  Steps b to d of
// one (series, DM trial) depend on its own events only, so event lists are split there
// across host threads, and the DM merge between series; cross-matching sees the merged pulses of all.
#include <algorithm>
#include <climits>
#include <cmath>
#include <thread>

#include "frbx_internal.h"

namespace frbx {

namespace {

constexpr double kTwoPi = 6.283185307179586;  // same double as 2 * pi

struct Grouper {
  std::vector<int> min_gid;   // per AP
  std::vector<int> touched;
  int n_groups = 0;

  explicit Grouper(int T) : min_gid((size_t)std::max(T, 1), INT_MAX) {}

  void reset() {
    for (int t : touched) min_gid[(size_t)t] = INT_MAX;
    touched.clear();
    n_groups = 0;
  }
  // Returns the group the range [k0, k0 + l) joins (a new one if none overlaps).
  int insert(int k0, int l) {
    const int T = (int)min_gid.size();
    const int lo = std::max(0, k0), hi = std::min(T, k0 + l);
    int g = INT_MAX;
    for (int t = lo; t < hi; ++t) g = std::min(g, min_gid[(size_t)t]);
    if (g == INT_MAX) g = n_groups++;
    for (int t = lo; t < hi; ++t) {
      if (min_gid[(size_t)t] == INT_MAX) touched.push_back(t);
      min_gid[(size_t)t] = std::min(min_gid[(size_t)t], g);
    }
    return g;
  }
};

// cos and sin of 2 pi q / Lm for every MBD cell, evaluated as for a single one
struct CircleTable {
  std::vector<double> th, c, s;
  explicit CircleTable(int Lm) : th((size_t)std::max(Lm, 0)), c(th.size()), s(th.size()) {
    for (size_t q = 0; q < th.size(); ++q) {
      th[q] = (kTwoPi * (double)q) / (double)Lm;
      c[q] = std::cos(th[q]);
      s[q] = std::sin(th[q]);
    }
  }
};

// Step c: circular mean of the MBD over the group (period t_ambig; angle 2 pi q / Lm) and
// removal of members at or beyond a quarter period from it.
void mbd_filter(std::vector<const frbx_event *> *grp, const CircleTable &t) {
  double sc = 0.0, ss = 0.0;
  for (const frbx_event *e : *grp) {
    sc += t.c[e->mbd_idx];
    ss += t.s[e->mbd_idx];
  }
  const double mu = std::atan2(ss, sc);
  size_t n = 0;
  for (const frbx_event *e : *grp) {
    // remainder(x, 2 pi) of x in [-pi, 3 pi): x or x - 2 pi, which is exact from pi on (Sterbenz)
    const double x = t.th[e->mbd_idx] - mu, r = x > M_PI ? x - kTwoPi : x;
    if (std::fabs(r) < M_PI / 2) (*grp)[n++] = e;
  }
  grp->resize(n);
}

// Steps b to d of the (series, DM trial)s whose events are ev[0, n_ev), sorted by series, DM trial,
// window and k0: their pulses, in that order and, within one, in discovery order.
void extract_events(const ExtractConfig &cfg, const CircleTable &circle, const frbx_event *ev, int64_t n_ev, bool use_mbd,
                    std::vector<Pulse> *out) {
  // window visiting order: longest first (step b)
  std::vector<int> order(cfg.n_win);
  for (int w = 0; w < cfg.n_win; ++w) order[w] = w;
  std::stable_sort(order.begin(), order.end(),
                   [&](int x, int y) { return cfg.win_len[x] > cfg.win_len[y]; });
  Grouper gp(cfg.T);
  std::vector<std::vector<const frbx_event *>> groups;  // the first n_groups are in use
  std::vector<std::pair<int64_t, int64_t>> wr(cfg.n_win);
  for (int64_t pos = 0; pos < n_ev;) {
    const int s = ev[pos].series, d = ev[pos].dm_idx;
    for (int w = 0; w < cfg.n_win; ++w) wr[w] = {0, 0};
    while (pos < n_ev && ev[pos].series == s && ev[pos].dm_idx == d) {
      const int w = ev[pos].win_idx;
      int64_t e = pos;
      while (e < n_ev && ev[e].series == s && ev[e].dm_idx == d && ev[e].win_idx == w) ++e;
      wr[w] = {pos, e};
      pos = e;
    }
    gp.reset();
    size_t n_groups = 0;
    for (int w : order) {
      for (int64_t i = wr[w].first; i < wr[w].second; ++i) {
        const size_t g = (size_t)gp.insert(ev[i].k0, cfg.win_len[w]);
        if (g == n_groups) {
          if (n_groups == groups.size()) groups.emplace_back();
          groups[n_groups++].clear();
        }
        groups[g].push_back(&ev[i]);
      }
    }
    for (size_t gi = 0; gi < n_groups; ++gi) {
      auto &grp = groups[gi];
      if ((int)grp.size() < cfg.nwin_min) continue;  // fewer members than windows asked for
      if (use_mbd) mbd_filter(&grp, circle);
      if (grp.empty()) continue;
      // step d: distinct windows (their lengths are distinct), best member (first inserted on ties)
      unsigned seen = 0u;
      const frbx_event *best = grp[0];
      for (const frbx_event *e : grp) {
        seen |= 1u << e->win_idx;
        if (e->pnorm > best->pnorm) best = e;
      }
      const int nw = __builtin_popcount(seen);
      if (nw < cfg.nwin_min) continue;
      Pulse p;
      p.series = s;
      p.d = d;
      p.w = best->win_idx;
      p.l = cfg.win_len[best->win_idx];
      p.k0 = best->k0;
      p.m = best->sbd_idx;
      p.q = best->mbd_idx;
      p.n_win = nw;
      p.group = -1;
      p.amp = best->amp;
      p.p = best->pnorm;
      out->push_back(p);
    }
  }
}

// Sec. 5.3: per series, one pulse per overlap group across DM trials, the one of highest power.
// p[0, n): sorted by series, DM trials ascending.
void merge_dm(const ExtractConfig &cfg, const Pulse *p, size_t n, std::vector<Pulse> *merged) {
  Grouper gm(cfg.T);
  std::vector<size_t> best_of;
  for (size_t i = 0; i < n;) {
    const int s = p[i].series;
    gm.reset();
    best_of.clear();
    for (; i < n && p[i].series == s; ++i) {
      const size_t g = (size_t)gm.insert(p[i].k0, p[i].l);
      if (g == best_of.size()) best_of.push_back(i);
      else if (p[i].p > p[best_of[g]].p) best_of[g] = i;
    }
    for (size_t k : best_of) merged->push_back(p[k]);
  }
}

// Events (pulses, in the DM merge) per host thread: a thread costs about 20 us to start, an event about 50 ns.
constexpr int64_t kEventsPerThread = 2000;

// Cuts [0, n) into contiguous parts of about equal length, at most one per kEventsPerThread items and per host
// thread, none between items i - 1 and i that belong together(i), calls parts(their number) and runs
// run(part, begin, end) for each, the last one on the calling thread.
template <class Together, class Parts, class Run>
void on_threads(int64_t n, Together together, Parts parts, Run run) {
  const int hw = (int)std::max(1u, std::thread::hardware_concurrency());
  const int n_th = (int)std::max<int64_t>(1, std::min<int64_t>({n / kEventsPerThread, (int64_t)hw, (int64_t)32}));
  parts((size_t)n_th);
  std::vector<int64_t> cut((size_t)n_th + 1, n);
  cut[0] = 0;
  for (int t = 1; t < n_th; ++t) {
    int64_t i = std::max(cut[(size_t)t - 1], n * t / n_th);
    while (i > 0 && i < n && together(i)) ++i;
    cut[(size_t)t] = i;
  }
  auto part = [&](int t) {
    if (cut[(size_t)t] < cut[(size_t)t + 1]) run((size_t)t, cut[(size_t)t], cut[(size_t)t + 1]);
  };
  std::vector<std::thread> th;
  th.reserve((size_t)n_th);
  for (int t = 0; t + 1 < n_th; ++t) {
    try {
      th.emplace_back(part, t);
    } catch (...) {  // no thread to be had: this part runs here (no exception crosses the C ABI)
      part(t);
    }
  }
  part(n_th - 1);
  for (auto &x : th) x.join();
}

void append(const std::vector<std::vector<Pulse>> &parts, std::vector<Pulse> *out) {
  size_t n = out->size();
  for (const auto &p : parts) n += p.size();
  out->reserve(n);
  for (const auto &p : parts) out->insert(out->end(), p.begin(), p.end());
}

}  // namespace

// Runs of (series, DM trial)s go to host threads, then, for the DM merge of their pulses, runs of series; the
// parts' pulses are concatenated in order: the same output as one pass.  Where one window is enough, nearly
// every event is a pulse: 64 series x 16 DM trials with 464000 of them 34.6 -> 8.4 ms on 16 cores against the
// merge on one thread, 15.6 ms with both steps split by series.
void extract_pulses(const ExtractConfig &cfg, const frbx_event *ev, int64_t n_ev, int n_series,
                    bool use_mbd, std::vector<Pulse> *pre_merge, std::vector<Pulse> *merged) {
  (void)n_series;
  const CircleTable circle(use_mbd ? cfg.Lm : 0);
  std::vector<std::vector<Pulse>> part;
  on_threads(
      n_ev, [&](int64_t i) { return ev[i].series == ev[i - 1].series && ev[i].dm_idx == ev[i - 1].dm_idx; },
      [&](size_t n) { part.resize(n); },
      [&](size_t t, int64_t e0, int64_t e1) { extract_events(cfg, circle, ev + e0, e1 - e0, use_mbd, &part[t]); });
  std::vector<Pulse> all = std::move(part[0]);
  part[0].clear();
  append(part, &all);
  on_threads(
      (int64_t)all.size(), [&](int64_t i) { return all[(size_t)i].series == all[(size_t)i - 1].series; },
      [&](size_t n) { part.assign(n, {}); },
      [&](size_t t, int64_t i0, int64_t i1) { merge_dm(cfg, all.data() + i0, (size_t)(i1 - i0), &part[t]); });
  append(part, merged);
  if (pre_merge) *pre_merge = std::move(all);
}

void cross_match(int T, std::vector<Pulse> *merged, int n_bl, std::vector<GroupOut> *groups) {
  // baselines ascending, then pulses by ascending start (stable)
  std::vector<int> idx(merged->size());
  for (size_t i = 0; i < idx.size(); ++i) idx[i] = (int)i;
  std::stable_sort(idx.begin(), idx.end(), [&](int x, int y) {
    const Pulse &a = (*merged)[(size_t)x], &b = (*merged)[(size_t)y];
    if (a.series != b.series) return a.series < b.series;
    return a.k0 < b.k0;
  });
  (void)n_bl;
  Grouper gp(T);
  groups->clear();
  for (int i : idx) {
    Pulse &p = (*merged)[(size_t)i];
    const int g = gp.insert(p.k0, p.l);
    if (g == (int)groups->size()) groups->push_back(GroupOut{0ull, 0, 0});
    GroupOut &go = (*groups)[(size_t)g];
    go.mask |= 1ull << p.series;
    go.n_pulses += 1;
    p.group = g;
  }
  for (GroupOut &go : *groups) go.n_baselines = __builtin_popcountll(go.mask);
}

}  // namespace frbx
