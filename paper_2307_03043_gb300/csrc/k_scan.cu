// k_scan.cu -- the exact scan's plain form (scan_exact.cuh): launch and merge.
#include "scan_exact.cuh"

namespace chx {

__global__ void k_scan_merge(const float* part_val, const int64_t* part_idx, int chunks, int64_t T,
                             const int64_t* qidx, float* min_d, int64_t* argmin) {
  pdl_entry();
  const int64_t l = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (l >= T) return;
  float bv = part_val[l];
  int64_t bi = part_idx[l];
  for (int c = 1; c < chunks; ++c) {
    const float v = part_val[int64_t(c) * T + l];
    const int64_t i = part_idx[int64_t(c) * T + l];
    if (v < bv || (v == bv && i < bi)) {
      bv = v;
      bi = i;
    }
  }
  const bool none = qidx && qidx[l] < 0;
  min_d[l] = none ? 0.0f : bv;
  if (argmin) argmin[l] = none ? -1 : bi;
}

bool scan_list_fits(int64_t T, int d) { return T < (int64_t(1) << 31) && scan_fits(d); }

int scan_exact_chunks(int64_t T, int64_t nB, int d, int dtype, int sm_count) {
  if (d <= kScanSmallMaxD) return scan_small_chunks(T, nB, sm_count);
  // B is cut into equal chunks, one block per (sample tile, chunk).  The count
  // minimises (waves of resident blocks) x (B tiles per block), the kernel's time
  // when every wave runs at the same rate; ties go to fewer chunks (less merging).
  const TileShape t = tile_for(d);
  const int64_t qtiles = ceil_div(std::max<int64_t>(T, 1), t.QT);
  const int64_t resident = int64_t(sm_count) * scan_blocks_per_sm(d, scan_double_buffered(dtype, d));
  const int64_t btiles = ceil_div(std::max<int64_t>(nB, 1), int64_t(t.BT) * t.SUB);  // stages
  const int64_t max_chunks = std::max<int64_t>(1, std::min<int64_t>(ceil_div(btiles, 4), 4 * resident));
  int64_t best = 1, best_cost = INT64_MAX;
  for (int64_t c = 1; c <= max_chunks; ++c) {
    const int64_t cost = ceil_div(qtiles * c, resident) * ceil_div(btiles, c);
    if (cost < best_cost) {
      best_cost = cost;
      best = c;
    }
    if (qtiles * c >= 8 * resident) break;  // past eight waves the cost only flattens
  }
  return static_cast<int>(best);
}

void launch_scan_exact(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, int metric, ScanPart part,
                       int sm_count, cudaStream_t s) {
  (void)sm_count;
  if (T == 0) return;
  if (A->d <= kScanSmallMaxD) return launch_scan_small(A, qidx, T, B, metric, part, s);
  CHX_CHECK(scan_fits(A->d), CH_ENOTSUP, "dimension too large for the exact scan");
  scan_form<false>(A, qidx, T, B, metric, part, s, ScanList{});
  launch_check("scan_exact");
}

void launch_scan_merge(ScanPart part, int64_t T, int64_t nB, const int64_t* qidx, float* min_d, int64_t* argmin,
                       cudaStream_t s) {
  if (T == 0) return;
  if (part.best) return launch_scan_small_out(part, T, nB, qidx, min_d, argmin, s);
  launch_k(k_scan_merge, static_cast<int>(ceil_div(T, 256)), 256, 0, s, part.val, part.idx, part.chunks, T, qidx, min_d,
                                                                  argmin);
  launch_check("scan_merge");
}

}  // namespace chx
