// Host build of the thread-granular leaf insert and delete for codes of any
// length (leaf_thread.cuh with 64-bit code records) for the CPU tests.
#include "../paper_2305_05055_gb300/csrc/leaf_thread.cuh"

extern "C" int lt_long(uint8_t* leaf, uint32_t LB, uint32_t uold, uint32_t m, const uint64_t* keys,
                       uint32_t s, uint32_t* out, int del) {
  uint64_t y[leafthr::kKeys] = {0, 0, 0, 0};
  for (uint32_t i = 0; i < s && i < leafthr::kKeys; i++) y[i] = keys[i];
  uint32_t rpos[leafthr::kKeys], epos[leafthr::kKeys], ekey[leafthr::kKeys];
  uint64_t rval[leafthr::kKeys], rcode[leafthr::kKeys];
  int32_t esa[leafthr::kKeys];
  const leafthr::ScratchLong S{rpos, rval, rcode, epos, esa, ekey, 1};
  leafthr::Result R{};
  const uint32_t st = del ? leafthr::delete_leaf(leaf, LB, uold, m, y, s, S, R)
                          : leafthr::insert_leaf(leaf, LB, uold, m, y, s, S, R);
  out[0] = R.nb;
  out[1] = R.newc;
  out[2] = R.added;
  out[3] = (uint32_t)R.newhead;
  out[4] = (uint32_t)(R.newhead >> 32);
  return (int)st;
}
