// Runs the certified exact scan on the caller's own scratch, so that a test can read the
// screen's scores out of it.  Linked against libchamfer.so.
#include "../../paper_2307_03043_gb300/csrc/common.cuh"

extern "C" {

long long scores_workspace(long long T, long long nB, int d, int dtype, int sm_count) {
  return static_cast<long long>(chx::exact_tc_workspace(T, nB, d, dtype, sm_count, 0));
}

int scores_run(void* A, void* B, int dtype, long long nA, long long nB, int d, const int64_t* idx, long long T,
               float* norms, void* work, float* min_d, int64_t* argmin, int sm_count) {
  try {
    ch_set a, b;
    a.data = A;
    a.n = nA;
    b.data = B;
    b.n = nB;
    a.d = b.d = d;
    a.dtype = b.dtype = dtype;
    chx::launch_norms(&b, norms, nullptr, nullptr);
    chx::launch_exact_tc(&a, idx, T, &b, norms, work, min_d, argmin, sm_count, 0, nullptr, 0);
    return static_cast<int>(cudaStreamSynchronize(nullptr));
  } catch (const chx::Err& e) {
    return -1;
  }
}

}  // extern "C"
