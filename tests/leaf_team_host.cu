// Host build of a leaf's walk by 8, 16 or 32 lanes (leaf_walk.cuh) for the CPU tests.
#include "../paper_2305_05055_gb300/csrc/leaf_walk.cuh"

// The lanes' runs one after another: the elements in order, and whether each
// run's own count, deltas and (SUM) sum say the same.  Returns how many elements.
template <uint32_t N, bool SUM>
static uint32_t team(const uint8_t* leaf, uint32_t u, uint64_t* out) {
  uint32_t n = 0;
  uint64_t v = out[n++] = leafwalk::leaf_head(leaf);
  for (uint32_t tl = 0; tl < N; tl++) {
    leafwalk::Run r = leafwalk::team_run<N, SUM>(leaf, u, tl);
    const uint32_t n0 = n;
    uint64_t s = 0;
    r.k.val = v;
    leafwalk::run_visit(leaf, u, r, [&](uint64_t x) { out[n++] = x; s += x; });
    if (SUM && s != r.codes * v + r.sum) return 0;
    v += r.delta;
    if (n - n0 != r.codes || out[n - 1] != v) return 0;
  }
  return n;
}

extern "C" uint32_t lt_team(const uint8_t* leaf, uint32_t u, int lanes, int sum, uint64_t* out) {
  if (lanes == 8) return sum ? team<8, true>(leaf, u, out) : team<8, false>(leaf, u, out);
  if (lanes == 16) return sum ? team<16, true>(leaf, u, out) : team<16, false>(leaf, u, out);
  return sum ? team<32, true>(leaf, u, out) : team<32, false>(leaf, u, out);
}
