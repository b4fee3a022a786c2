// Autotuner (pg_autotune, pg_batch_tune): coordinate descent over the
// schedule options that leave the counts unchanged — PROPAGATE-S's pass
// schedule, push or pull sparse rounds, words a lane gathers per arc, lanes
// per work piece, the dense-round threshold, the changed-bit test.
// Every candidate runs the real propagation twice (the faster run is kept, so
// one-time costs such as a new piece list or a graph capture do not count);
// its counts must hash to the same value as the first run's.
#include <chrono>
#include <cstring>
#include <vector>

#include "host.cuh"

namespace pg {

// FNV-1a over 8-byte words (then the tail bytes): a cheap fingerprint for
// comparing two runs' counts.
uint64_t fnv1a(uint64_t h, const void *data, size_t bytes) {
  const unsigned char *p = static_cast<const unsigned char *>(data);
  size_t i = 0;
  for (; i + 8 <= bytes; i += 8) {
    uint64_t w;
    std::memcpy(&w, p + i, 8);
    h ^= w;
    h *= 1099511628211ULL;
  }
  for (; i < bytes; ++i) {
    h ^= p[i];
    h *= 1099511628211ULL;
  }
  return h;
}

pg_status tune_options(const TuneRun &run, int32_t s_bits, int32_t max_trials, pg_options *inout,
                       pg_tune_report *rep, bool s_mode) {
  pg_tune_report r{};
  pg_options cur = *inout;
  double best = 0.0;
  uint64_t want = 0;
  auto measure = [&](const pg_options &o, double *ms) -> pg_status {
    double t_min = 0.0;
    for (int k = 0; k < 3; ++k) {  // the best of three: the first may build a CUDA graph
      uint64_t h = 0;
      double t = 0.0;
      pg_status rc = run(o, &t, &h);
      if (rc) return rc;
      if (r.trials == 0 && k == 0) want = h;
      if (h != want) return PG_EDEVICE;  // a schedule changed the counts
      t_min = k == 0 ? t : std::min(t_min, t);
    }
    r.trials += 1;
    *ms = t_min;
    return PG_OK;
  };
  pg_status rc = measure(cur, &best);
  if (rc) return rc;
  r.default_ms = best;
  auto try_value = [&](pg_options cand) -> pg_status {
    if (r.trials >= max_trials) return PG_OK;
    double t = 0.0;
    pg_status e = measure(cand, &t);
    if (e) return e;
    if (t < 0.98 * best) {
      best = t;
      cur = cand;
      r.improved += 1;
    }
    return PG_OK;
  };
  const int npasses = (s_bits + 63) / 64;
  if (s_mode && npasses > 1) {
    // PROPAGATE-S, first the pass schedule: (copies, words) = one pass at a
    // time, passes on copies of the graph, or passes as signature words
    const int pairs[][2] = {{1, 1}, {2, 1}, {4, 1}, {0, 2}, {0, 4}, {0, 8}};
    for (const auto &pr : pairs) {
      if (pr[1] > 2 * npasses) continue;
      if (pr[0] == cur.passes_together && pr[1] == cur.pass_words) continue;
      pg_options o = cur;
      o.passes_together = pr[0];
      o.pass_words = pr[1];
      if ((rc = try_value(o))) return rc;
    }
  }
  // words per node of the runs that follow (PROPAGATE-S: one, or its passes
  // as words when they may be)
  int W = (s_bits + 63) / 64;
  if (s_mode)
    W = cur.pass_words > 1 ? std::min(cur.pass_words, npasses)
        : cur.pass_words == 0 && cur.passes_together <= 1 ? std::min(8, npasses)
                                                           : 1;
  const int cw_class = W <= 1 ? 1 : W <= 2 ? 2 : W <= 4 ? 4 : 8;
  std::vector<int> wpt;
  for (int c : {0, 1, 2, 4, 8})
    if (c <= cw_class && cw_class > 1) wpt.push_back(c);
  const int lanes[] = {0, 1, 2, 4, 8, 16, 32};
  const float dens[] = {0.01f, 0.02f, 0.05f, 0.1f, 0.2f, 0.5f};
  const int tests[] = {0, 1, 2, 3};
  if (W > 8) {  // a warp per row piece, or lanes over 8-word chunks
    pg_options o = cur;
    o.wide_rows = cur.wide_rows == 2 ? 0 : 2;
    if ((rc = try_value(o))) return rc;
  }
  // sparse rounds pulled instead of pushed from the frontier (push rounds
  // apply to rows of up to 8 words)
  if (W <= 8) {
    pg_options o = cur;
    o.sparse_push = cur.sparse_push == 1 ? 0 : 1;
    if ((rc = try_value(o))) return rc;
  }
  const bool wide = W > 8 && cur.wide_rows != 2;  // lanes and chunk width then fixed
  for (int c : wpt) {
    if (wide || c == cur.words_per_thread) continue;
    pg_options o = cur;
    o.words_per_thread = c;
    if ((rc = try_value(o))) return rc;
  }
  // the resident round loop reads no group_lanes: those runs would differ by
  // their noise only
  const bool resident = W <= 8 && resident_schedule(cur) &&
                        (cur.words_per_thread == 0 || cur.words_per_thread >= cw_class);
  for (int g : lanes) {
    if (wide || resident || g == cur.group_lanes) continue;
    pg_options o = cur;
    o.group_lanes = g;
    if ((rc = try_value(o))) return rc;
  }
  if (cur.direction == PG_DIR_AUTO)
    for (float d : dens) {
      if (d == cur.dense_threshold || (!resident && !cur.dense_threshold && d == 0.05f)) continue;
      pg_options o = cur;
      o.dense_threshold = d;
      if ((rc = try_value(o))) return rc;
    }
  for (int tc : tests) {
    if (tc == cur.test_changed) continue;
    pg_options o = cur;
    o.test_changed = tc;
    if ((rc = try_value(o))) return rc;
  }
  r.best_ms = best;
  *inout = cur;
  if (rep) *rep = r;
  return PG_OK;
}

}  // namespace pg

using namespace pg;

#ifdef PG_DEBUG_BOUNDS
// For tests: the tuner's search, with the time of each schedule from ms.
extern "C" pg_status pg_debug_tune(int32_t s_bits, int32_t s_mode, int32_t max_trials,
                                   double (*ms)(const pg_options *), pg_options *inout,
                                   pg_tune_report *report) {
  TuneRun run = [&](const pg_options &o, double *t, uint64_t *hash) -> pg_status {
    *t = ms(&o);
    *hash = 1;
    return PG_OK;
  };
  return tune_options(run, s_bits, max_trials, inout, report, s_mode != 0);
}
#endif

extern "C" pg_status pg_autotune(pg_graph *g, const int32_t *seeds, int32_t s, int32_t algorithm,
                                 int32_t max_trials, pg_options *inout, pg_tune_report *report,
                                 void *stream) {
  if (!g || !seeds || s < 1 || !inout || max_trials < 1 || algorithm < 0 || algorithm > 1)
    return PG_EINVAL;
  const bool s_mode = algorithm == PG_ALG_S;
  auto call = [&](pg_counts *c, const pg_options *o) {
    return s_mode ? pg_propagate_s(g, seeds, s, c, o, stream)
                  : pg_propagate_p(g, seeds, s, c, o, stream);
  };
  int32_t cap = 0;
  pg_status rc = pg_query_rounds_bound(g, &cap);
  if (rc) return rc;
  // a first run finds T, so that later runs write only rows 0..T
  std::vector<uint32_t> counts;
  int32_t rows = std::min(cap, 4096);
  pg_counts c{};
  for (;;) {
    counts.assign((size_t)(rows + 1) * s, 0u);
    c = pg_counts{s, rows, 0, 0, counts.data(), nullptr};
    rc = call(&c, inout);
    if (rc == PG_ERANGE && rows < cap) {
      rows = cap;
      continue;
    }
    if (rc) return rc;
    break;
  }
  rows = c.rounds;
  TuneRun run = [&](const pg_options &o, double *ms, uint64_t *hash) -> pg_status {
    pg_counts cc{s, rows, 0, 0, counts.data(), nullptr};
    const auto t0 = std::chrono::steady_clock::now();
    pg_status e = call(&cc, &o);
    const auto t1 = std::chrono::steady_clock::now();
    if (e) return e;
    *ms = std::chrono::duration<double, std::milli>(t1 - t0).count();
    uint64_t h = fnv1a(1469598103934665603ULL, &cc.rounds, sizeof(cc.rounds));
    *hash = fnv1a(h, counts.data(), sizeof(uint32_t) * (size_t)(cc.rounds + 1) * s);
    return PG_OK;
  };
  return tune_options(run, s, max_trials, inout, report, s_mode);
}
