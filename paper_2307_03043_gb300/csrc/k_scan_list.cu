// k_scan_list.cu -- the exact scan's list form (scan_exact.cuh): the samples that the
// certified and chained scans leave over.
#include "scan_exact.cuh"

namespace chx {

// Most samples of a call whose minima the kernel's last block writes out itself, which
// saves the usual call (nothing listed) a launch; a block would be slow with more.
constexpr int64_t kListOwnOut = int64_t(1) << 16;

__global__ void k_scan_list_out(ScanList sl) {
  pdl_entry();
  const int64_t n = *sl.count;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x)
    list_out(sl, i);
}

void launch_scan_list(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, int metric, const int32_t* list,
                      uint32_t* ctl, unsigned long long* best, float* min_d, int64_t* argmin, int sm_count,
                      cudaStream_t s) {
  const ScanPart grid{nullptr, nullptr, sm_count, nullptr};  // its grid: sm_count x resident blocks
  ScanList sl{list, ctl, ctl + 2, best, T <= kListOwnOut ? min_d : nullptr, argmin};
  scan_form<true>(A, qidx, T, B, metric, grid, s, sl);
  launch_check("scan_list");
  if (sl.min_d) return;
  sl.min_d = min_d;
  launch_k(k_scan_list_out, 2 * sm_count, 256, 0, s, sl);
  launch_check("scan_list_out");
}

}  // namespace chx
