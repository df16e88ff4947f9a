// Host-only check of the FP32 work list (no device work), built and run by
// tests/test_list_host.py like plan_check.cu: the closed form that the window kernel writes
// it from (main_unit, UnitOrder, band_columns) against the list that build_plan makes for
// the same call, entry by entry: single, batched and several-settings calls, half tiles and
// several tiles a unit, column chunks, strips side by side from one to all. And the
// tensor-core path's rules around its list: the pairs' units against the single CTAs', the
// shapes that the autotuner times, and the unit lengths of the option.
#include "../paper_2603_02059_gb300/csrc/traknn_api.cu"

#include <cstdio>

namespace {

int g_fail = 0;

bool same(const WorkUnit& a, const WorkUnit& b) {
  return a.series == b.series && a.strip == b.strip && a.jlo == b.jlo && a.jhi == b.jhi &&
         a.slot == b.slot && a.pad[0] == b.pad[0];
}

// Every write of write_units (kernels_aux.cu), by one thread.
void written(const TcPlan& p, std::vector<WorkUnit>& units, std::vector<long long>& off,
             std::vector<int>& slot) {
  const UnitList& ul = p.list;
  for (int gs = 0; gs < ul.strips; ++gs) {
    int b = 0;
    while (b + 1 < p.table.n && p.table.s[b + 1].strip_base <= gs) ++b;
    const SeriesInfo& si = p.table.s[b];
    const int s = gs - si.strip_base, R = si.rows_out;
    off[gs] = (long long)s * si.M - (long long)R * ((long long)s * (s + 1) / 2);
    slot[gs] = (int)((long long)s * R / si.cols) * ul.egroups;
    if (ul.nser > 1 && b > 0) continue;
    WorkUnit u{b, s, 0, 0, 0, {ul.nser, 0, 0}};
    band_columns(si.M, R, s, ul.bw, ul.nser > 1 ? ul.emax : si.e, &u.jlo, &u.jhi);
    units.at(ul.nmain + gs) = u;
    const UnitOrder o = unit_order(si, ul.group);
    const int g = s / o.group;
    int base = si.unit_base + s - g * o.group;
    for (int lane = 0; lane < 32; ++lane) base += o.after(g, lane, 32);
    for (int c = (int)((long long)s * R / si.cols); c < o.ranges(); ++c)
      units.at(base + o.before(g, c)) = main_unit(si, b, s, c, ul.nser);
  }
}

void check(int64_t N, int64_t D, int L, int e, int B, bool shared, int group, int chunks) {
  std::vector<HostSeries> sd(B);
  for (int b = 0; b < B; ++b)
    sd[b] = HostSeries{nullptr, shared ? N : std::max<int64_t>(30, N - 131 * b), L + b % 3, 5, e,
                       nullptr, nullptr, nullptr};
  if (shared)
    std::stable_sort(sd.begin(), sd.end(),
                     [](const HostSeries& x, const HostSeries& y) { return x.L < y.L; });
  static traknn_ctx h;
  h.sm_count = 152;
  h.group_strips = group;
  h.col_chunks = chunks;
  static TcPlan p, q;
  fp32_plan(&h, sd.data(), B, D, shared, p);
  std::vector<WorkUnit> units(p.nunits + p.nband, WorkUnit{-1, -1, -1, -1, -1, {0, 0, 0}});
  std::vector<long long> off(p.strips, -1);
  std::vector<int> slot(p.strips, -1);
  written(p, units, off, slot);
  // the same call's list, from the columns of a range
  const int cols = p.table.s[0].cols;
  bool ok = true;
  for (int b = 0; b < B; ++b) {  // (ranges differ by series unless they share)
    if (shared && b > 0) break;
    const SeriesInfo& si = p.table.s[b];
    std::vector<HostSeries> one(sd.begin() + b, shared ? sd.end() : sd.begin() + b + 1);
    if (shared && si.step != kTileCols - (sd[B - 1].L - 1)) continue;  // half tiles: no such plan
    build_plan(one.data(), (int)one.size(), D, 1, si.cols, 1, p.list.group, shared, 0, INT_MAX, {},
               p.egroups, D <= 64 ? 2 : 1, q);
    const int n0 = si.unit_base, n1 = shared || b + 1 == B ? p.nunits : p.table.s[b + 1].unit_base;
    ok = ok && n1 - n0 == q.nunits;
    for (int i = 0; ok && i < q.nunits; ++i) {
      WorkUnit u = units[n0 + i];
      u.series -= b;
      ok = same(u, q.units[i]);
    }
    // band units: one per strip here; build_plan leaves empty ones out
    for (int s = 0, i = q.nunits; ok && s < (si.M + si.rows_out - 1) / si.rows_out; ++s) {
      WorkUnit u = units[p.list.nmain + si.strip_base + s];
      u.series -= b;
      if (u.jlo < u.jhi) ok = i < q.nunits + q.nband && same(u, q.units[i++]);
    }
    for (size_t s = 0; ok && s < q.col_off.size(); ++s)
      ok = off[si.strip_base + s] == q.col_off[s] && slot[si.strip_base + s] == q.slot_lo[s];
    ok = ok && q.table.s[0].slots == si.slots && q.table.s[0].rows_out == si.rows_out;
  }
  for (const WorkUnit& u : units) ok = ok && u.strip >= 0;  // every entry written
  if (!ok) {
    std::printf("FAIL N=%lld D=%lld L=%d e=%d B=%d shared=%d group=%d chunks=%d (cols %d)\n",
                (long long)N, (long long)D, L, e, B, (int)shared, group, chunks, cols);
    ++g_fail;
  }
}

void check_pairs(int64_t N, int L, int part_lo, int part_hi, const std::vector<int>& pstrip) {
  const HostSeries sd{nullptr, N, L, 5, L - 1, nullptr, nullptr, nullptr};
  static TcPlan p;
  build_plan(&sd, 1, 100, 1, 0, 1, 19, false, part_lo, part_hi, pstrip, 1, 2, p);
  p.part_lo = part_lo;
  p.part_hi = part_hi;
  pair_units(p);
  const int K = (int)p.pu.size() - 1, R = p.table.s[0].rows_out;
  bool ok = (int)p.pp.size() == K + 1;
  for (int q = 0; ok && q < K; ++q) {
    // (strip, range) of a phase's pairs, both members, against the single units
    std::vector<std::pair<int, int>> want, got;
    for (int u = p.pu[q]; u < p.pu[q + 1]; ++u) want.emplace_back(p.units[u].strip, p.units[u].slot);
    for (int u = p.pp[q]; u < p.pp[q + 1]; ++u)
      for (int r = 0; r <= p.units[u].pad[1]; ++r) {
        const WorkUnit& w = p.units[u];  // (the second strip may start beyond the range)
        if (r == 0 || std::max(w.jlo, (w.strip + r) * R) < w.jhi)
          got.emplace_back(w.strip + r, w.slot);
      }
    std::sort(want.begin(), want.end());
    std::sort(got.begin(), got.end());
    ok = ok && want == got;
  }
  if (!ok) {
    std::printf("FAIL pairs N=%lld L=%d part %d %d\n", (long long)N, L, part_lo, part_hi);
    ++g_fail;
  }
}

void check_unit_cols(int64_t N, int k, int cols) {
  const HostSeries sd{nullptr, N, 5, k, 4, nullptr, nullptr, nullptr};
  const int got = fit_cols(&sd, 1, cols);
  const double M = (double)(N - 4);
  auto bytes = [&](double c) { return 2.0 * M * std::ceil(M / c) * ((k + 3) / 4 * 4 + 44) * 8.0; };
  // the option's length where its lists fit, else the first doubling that makes them
  if (bytes(got) > 16e9 || (got > cols && bytes(got / 2) <= 16e9)) {
    std::printf("FAIL unit_cols N=%lld k=%d %d -> %d\n", (long long)N, k, cols, got);
    ++g_fail;
  }
}

void check_tuning(int64_t N, int64_t D, int k, int group_opt) {
  static traknn_ctx h;
  h.sm_count = 152;
  h.group_strips = group_opt;
  const HostSeries sd{nullptr, N, 5, k, 4, nullptr, nullptr, nullptr};
  int tiles = 8, group = 0;
  default_shape(&h, &sd, 1, D, 1, 0, INT_MAX, &tiles, &group);
  tiles = unit_tiles(&sd, 1, D, 1, tiles);
  const auto v = tune_shapes(&h, &sd, 1, D);
  const bool one_tile = D > 756 || k > 32;  // the default's units, which the others exceed
  bool ok = !one_tile || v[0] == std::make_pair(tiles, group);
  for (const auto& s : v) {
    const double lists = (double)(N - 4) * std::ceil((N - 4) / (s.first * 256.0 - 4));
    ok = ok && 2.0 * lists * ((k + 3) / 4 * 4 + 44) * 8.0 <= 16e9;
  }
  ok = ok && (N > 100000 || v.size() == (group_opt ? 3u : 9u) + one_tile);
  if (!ok) {
    std::printf("FAIL tuning N=%lld D=%lld k=%d\n", (long long)N, (long long)D, k);
    ++g_fail;
  }
}

}  // namespace

int main() {
  for (int64_t N : {130, 300, 1100, 5000, 27394})
    for (int L : {1, 5, 17}) {
      const int R = kTileRows - (L - 1), strips = (int)((N - L + R) / R);
      check_pairs(N, L, 0, INT_MAX, {});
      check_pairs(N, L, strips / 3, strips / 2 + 1, {});
      const std::vector<int> ps = phase_plan(strips, R, N);
      if (!ps.empty()) check_pairs(N, L, 0, INT_MAX, ps);
    }
  for (int64_t N : {500, 27394, 200000, 1000000})
    for (int cols : {1, 256, 5000}) check_unit_cols(N, 20, cols), check_unit_cols(N, 64, cols);
  for (int64_t N : {500, 10957, 27394, 300000})
    for (int64_t D : {32, 3726})
      for (int k : {10, 64})
        for (int g : {0, 12}) check_tuning(N, D, k, g);

  for (int64_t N : {20, 129, 300, 1100, 2501, 5000, 27394})
    for (int64_t D : {16, 200, 3726})
      for (int L : {1, 5, 15})
        for (int e : {0, 4, 3000}) {
          for (int group : {0, 1, 7, 4096}) check(N, D, L, e, 1, false, group, 0);
          check(N, D, L, e, 1, false, 0, 3);
          check(N, D, L, e, 7, false, 0, 0);
          check(N, D, L, e, 7, false, 5, 32);
          check(N, D, L, e, 5, true, 0, 0);
        }
  std::printf("%s\n", g_fail ? "list check failed" : "list check ok");
  return g_fail ? 1 : 0;
}
