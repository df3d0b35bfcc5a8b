// Host build of the rules by which a call is laid out (gpss_plan.h), for the
// CPU tests.  Compiled by tests/test_host_plan.py with g++.
#include "gpss_plan.h"

using namespace gpss;

extern "C" {

int ph_grad_segments(int product, int comb_prec, int D, int max_chunk, int ck, int n_vch,
                     int n_sm) {
  return grad_segments({product != 0, comb_prec, D, D * (D + 1) / 2, max_chunk, ck, n_vch, n_sm});
}

}  // extern "C"
