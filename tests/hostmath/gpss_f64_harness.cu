// Host build of FP64 parts of the CUDA path's device arithmetic, for CPU
// tests.  Compiled by tests/test_host_f64.py with nvcc into a shared library.
#include "gpss_kernels.cuh"
#include "gpss_prod.cuh"

using namespace gpss;

extern "C" {

// out2: an event's share of the sums (prod_tally)
void hf_prod_tally(double S, double dS, double e, double de, double *out2) {
  out2[0] = out2[1] = 0.0;
  prod_tally(S, dS, e, de, 1.0f / (float)S, out2[0], out2[1]);
}

}  // extern "C"
