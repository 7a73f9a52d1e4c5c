// Host build of a thread's walk over a leaf (leaf_walk.cuh) and of its
// membership test (leaf_thread.cuh) for the CPU tests.
#include "../paper_2305_05055_gb300/csrc/leaf_thread.cuh"

extern "C" uint64_t lw_sum(const uint8_t* leaf, uint32_t u, uint32_t m, int form,
                           uint64_t span) {
  uint64_t s = 0;
  if (form == 0) return leafwalk::leaf_sum(leaf, u, m, span);
  if (form == 1) return leafwalk::sum_walked(leaf, u);
  return (form == 2 ? leafwalk::sum_few<4>(leaf, u, m, s) : leafwalk::sum_many(leaf, u, m, s)) ? s : ~0ull;
}

extern "C" uint32_t lw_visit(const uint8_t* leaf, uint32_t u, uint64_t* out) {
  uint32_t n = 0;
  leafwalk::leaf_visit(leaf, u, [&](uint64_t v) { out[n++] = v; });
  return n;
}

extern "C" void lw_range(const uint8_t* leaf, uint32_t u, uint64_t lo, uint64_t hi, uint64_t* out) {
  out[0] = out[1] = 0;
  leafwalk::leaf_range_sum(leaf, u, lo, hi, out[0], out[1]);
}

extern "C" void lw_take(const uint8_t* leaf, uint32_t u, uint64_t lo, uint64_t most,
                        uint64_t* out) {
  uint32_t below, taken;
  leafwalk::leaf_take_sum(leaf, u, lo, most, below, taken, out[2]);
  out[0] = below;
  out[1] = taken;
}

extern "C" uint32_t lw_below(const uint8_t* leaf, uint32_t u, uint64_t x) {
  leafwalk::Mark at;
  return leafwalk::leaf_below(leaf, u, x, at);
}

extern "C" int lw_has(const uint8_t* leaf, uint32_t u, uint64_t x) {
  return leafthr::leaf_has(leaf, u, x) ? 1 : 0;
}

// Elements < x and their sum, from the last mark below x.
extern "C" void lw_marked(const uint8_t* leaf, uint32_t u, uint64_t x, uint64_t* out) {
  leafwalk::Mark m[2048 / leafwalk::kMark];
  uint32_t n = 0, at = 0;
  leafwalk::leaf_marks(leaf, u, out[2], n, [&](uint32_t i, const leafwalk::Mark& v) { m[i] = v; });
  out[0] = out[1] = 0;
  out[3] = n;
  leafwalk::Walk k;
  k.val = leafwalk::leaf_head(leaf);
  if (k.val >= x) return;
  for (uint32_t i = 1; i * leafwalk::kMark < u; i++)
    if (m[i].val < x) at = i;
  out[0] = at ? m[at].sum : k.val;
  out[1] = at ? m[at].cnt : 1;
  if (at) k = leafwalk::walk_at(m[at]);
  leafwalk::below_sum(leaf, u, at * leafwalk::kMark, k, x, out[0], out[1]);
}

extern "C" uint32_t lw_between(const uint8_t* leaf, uint32_t u, uint64_t lo, uint64_t hi,
                               uint64_t* out) {
  uint32_t n = 0;
  leafwalk::leaf_range_visit(leaf, u, lo, hi, [&](uint64_t v) { out[n++] = v; });
  return n;
}

extern "C" void lw_masked(const uint8_t* leaf, uint32_t u, uint32_t mask, uint32_t value,
                          uint64_t* out) {
  out[0] = out[1] = 0;
  leafwalk::leaf_masked_sum(leaf, u, mask, value, out[0], out[1]);
}

// The elements from lo on, starting where the search for it ended; returns
// how many (0 when it did not end at a code).
extern "C" uint32_t lw_from(const uint8_t* leaf, uint32_t u, uint64_t lo, uint64_t* out) {
  leafwalk::Mark at;
  const uint32_t r = leafwalk::leaf_below(leaf, u, lo, at);
  uint32_t n = 0, idx = at.cnt;
  if (at.sum)
    leafwalk::visit_from(leaf, u, (uint32_t)at.sum, leafwalk::walk_at(at),
                         [&](uint64_t v) { if (idx++ >= r) out[n++] = v; }, [] { return false; });
  return n;
}

// A team's runs one after another: the elements in order, and whether each
// run's own count and sum of deltas say the same.
extern "C" uint32_t lw_team(const uint8_t* leaf, uint32_t u, uint64_t* out) {
  uint32_t n = 0;
  uint64_t v = out[n++] = leafwalk::leaf_head(leaf);
  for (uint32_t tl = 0; tl < leafwalk::kTeam; tl++) {
    leafwalk::Run r = leafwalk::team_run(leaf, u, tl);
    const uint32_t n0 = n;
    r.k.val = v;
    leafwalk::run_visit(leaf, u, r, [&](uint64_t x) { out[n++] = x; });
    v += r.delta;
    if (n - n0 != r.codes || out[n - 1] != v) return 0;
  }
  return n;
}
