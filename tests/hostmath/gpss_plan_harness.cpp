// Host build of the rules by which a call is laid out (gpss_plan.h), for the
// CPU tests.  Compiled by tests/test_host_plan.py with g++.
#include "gpss_plan.h"

using namespace gpss;

extern "C" {

int ph_grad_segments(int product, int comb_prec, int D, int max_chunk, int ck, int n_vch, int n_sm,
                     int64_t steps) {
  return grad_segments(
      {product != 0, comb_prec, D, D * (D + 1) / 2, max_chunk, ck, n_vch, steps, n_sm});
}

int ph_prod_scalars(int grad, int plain_term, int max_chunk, int n_vch, int n_sm) {
  return prod_scalars_at_once(grad != 0, plain_term != 0, max_chunk, n_vch, n_sm);
}

int ph_upload_groups(const int64_t *ev_off, const int32_t *ch_first, int n_series,
                     int64_t block_chunks, int *cut) {
  const std::vector<int> c = upload_groups(ev_off, ch_first, n_series, block_chunks);
  for (size_t i = 0; i < c.size(); ++i) cut[i] = c[i];
  return (int)c.size() - 1;
}

// take_first and take_rest against an allocator of `limit` bytes.  n[4], bytes:
// the lists (first, fast, and the rest of the fast and of the plain way); held: bytes taken
// in the end; got[i]: buffer i is in hand; begun: the way after the first step.
// Returns 0 none, 1 plain, 2 fast.
int ph_take_scratch(size_t limit, const int *n, const size_t *bytes, size_t *held, int *got,
                    int *begun) {
  std::vector<void *> addr(n[0] + n[1] + n[2] + n[3], (void *)8);
  std::vector<Buffer> list[4];
  for (int l = 0, i = 0; l < 4; ++l)
    for (int k = 0; k < n[l]; ++k, ++i) list[l].push_back({&addr[i], bytes[i]});
  std::vector<size_t> taken;
  *held = 0;
  auto take = [&](void **p, size_t b) {
    *p = (void *)8;  // a failed allocation may leave anything
    if (*held + b > limit) return false;
    *held += b;
    taken.push_back(b);
    return true;
  };
  auto give = [&] {
    *held -= taken.back();
    taken.pop_back();
  };
  Scratch way = take_first(list[0], list[1], take, give);
  *begun = way == Scratch::none ? 0 : way == Scratch::plain ? 1 : 2;
  if (way != Scratch::none) way = take_rest(way, list[1], list[2], list[3], take, give);
  for (size_t i = 0; i < addr.size(); ++i) got[i] = addr[i] != nullptr;
  return way == Scratch::none ? 0 : way == Scratch::plain ? 1 : 2;
}

}  // extern "C"
