// k_rerank.cu -- the canonical rerank after the tensor-core screen (Fig. 1,
// step 3): for each sample, the R best screened entries by screen score, the
// canonical binary32 distance of every column they stand for, and the minimum.
#include "common.cuh"

namespace chx {

namespace {

constexpr int kRerankWarps = 8;  // samples per block; each warp's candidate list in dynamic shared memory

// One warp per sample: the R best screened entries over all chunks (by s, then
// index), the canonical binary32 distance of each of an entry's occ columns
// (first column + o * stride, o < occ, columns < nB), and their minimum (ties:
// smaller index).
template <int DT, int METRIC>
__global__ void __launch_bounds__(32 * kRerankWarps) k_rerank(const void* A, const float* scA, int64_t nA, const void* B,
                                                const float* scB, int64_t nB, int d, const int64_t* idx, int64_t T,
                                                const float* part_s, const int32_t* part_i, int parts, int per,
                                                int occ, int stride, int R, float* min_d, int64_t* argmin) {
  pdl_entry();
  extern __shared__ float s_dyn[];  // [kRerankWarps][parts * per] scores, then as many indices
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nc = parts * per;
  float* s_s = s_dyn + wib * nc;
  int32_t* s_i = reinterpret_cast<int32_t*>(s_dyn + kRerankWarps * nc) + wib * nc;
  const int64_t l = int64_t(blockIdx.x) * kRerankWarps + wib;
  if (l >= T) return;
  const int64_t a = idx ? idx[l] : l;
  if (a < 0 || a >= nA) {
    if (lane == 0) {
      min_d[l] = 0.0f;
      if (argmin) argmin[l] = -1;
    }
    return;
  }
  for (int p = lane; p < nc; p += 32) {
    const int c = p / per, k = p % per;
    const size_t off = (size_t(c) * T + l) * per + k;
    s_s[p] = part_s[off];
    s_i[p] = part_i[off];
  }
  __syncwarp();
  float best = __int_as_float(0x7F800000);
  int64_t bidx = INT64_MAX;
  for (int round = 0; round < R; ++round) {
    float ms = __int_as_float(0x7F800000);
    int32_t mi = INT32_MAX;
    int mp = -1;
    for (int p = lane; p < nc; p += 32) {
      const float v = s_s[p];
      const int32_t i = s_i[p];
      if (i >= 0 && (v < ms || (v == ms && i < mi))) {
        ms = v;
        mi = i;
        mp = p;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float os = __shfl_xor_sync(0xFFFFFFFFu, ms, o);
      const int32_t oi = __shfl_xor_sync(0xFFFFFFFFu, mi, o);
      const int op = __shfl_xor_sync(0xFFFFFFFFu, mp, o);
      if (os < ms || (os == ms && oi < mi)) {
        ms = os;
        mi = oi;
        mp = op;
      }
    }
    if (mi == INT32_MAX || mi < 0) break;  // fewer than R entries
    if (lane == (mp & 31)) s_i[mp] = -1;  // taken
    __syncwarp();
    // canonical distances to the entry's columns, all at once (lane r sums
    // coordinates j = r mod 32 of each; the reduction trees run side by side)
    int64_t bo[kRerankMaxOcc];
    bool vo[kRerankMaxOcc];
    float part[kRerankMaxOcc];
#pragma unroll
    for (int o = 0; o < kRerankMaxOcc; ++o) {
      bo[o] = int64_t(mi) + int64_t(o) * stride;
      vo[o] = o < occ && bo[o] < nB;
      part[o] = 0.0f;
    }
#pragma unroll 4
    for (int j = lane; j < d; j += 32) {
      const float x = load_elem<DT>(A, a, d, j, scA);
#pragma unroll
      for (int o = 0; o < kRerankMaxOcc; ++o) {
        if (vo[o]) {
          const float t = __fsub_rn(x, load_elem<DT>(B, bo[o], d, j, scB));
          part[o] = (METRIC == CH_L1) ? __fadd_rn(part[o], fabsf(t)) : __fmaf_rn(t, t, part[o]);
        }
      }
    }
#pragma unroll
    for (int sh = 16; sh >= 1; sh >>= 1) {
#pragma unroll
      for (int o = 0; o < kRerankMaxOcc; ++o) part[o] = __fadd_rn(part[o], __shfl_down_sync(0xFFFFFFFFu, part[o], sh));
    }
#pragma unroll
    for (int o = 0; o < kRerankMaxOcc; ++o) {
      const float dist = __shfl_sync(0xFFFFFFFFu, (METRIC == CH_L1) ? part[o] : __fsqrt_rn(part[o]), 0);
      if (vo[o] && (dist < best || (dist == best && bo[o] < bidx))) {
        best = dist;
        bidx = bo[o];
      }
    }
  }
  if (lane == 0) {
    min_d[l] = best;
    if (argmin) argmin[l] = bidx;
  }
}

}  // namespace

void launch_rerank(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, const float* part_s,
                   const int32_t* part_i, int parts, int per, int occ, int stride, int R, float* min_d,
                   int64_t* argmin, cudaStream_t s) {
  CHX_CHECK(parts * per <= kRerankMaxCand && occ <= kRerankMaxOcc, CH_EINVAL, "rerank candidate list too long");
  const int blocks = static_cast<int>(ceil_div(T, kRerankWarps));
  const size_t smem = size_t(kRerankWarps) * parts * per * 8;
#define CHX_RERANK(DT)                                                                                        \
  do {                                                                                                        \
    CHX_CUDA(cudaFuncSetAttribute(k_rerank<DT, CH_L2>, cudaFuncAttributeMaxDynamicSharedMemorySize,             \
                                  static_cast<int>(size_t(kRerankWarps) * kRerankMaxCand * 8)));               \
    launch_k(k_rerank<DT, CH_L2>, blocks, 32 * kRerankWarps, smem, s, A->data, A->scales, A->n, B->data,        \
             B->scales, B->n, A->d, qidx, T, part_s, part_i, parts, per, occ, stride, R, min_d, argmin);       \
  } while (0)
  if (A->dtype == CH_F32) CHX_RERANK(CH_F32);
  else if (A->dtype == CH_BF16) CHX_RERANK(CH_BF16);
  else CHX_RERANK(CH_FP8E4M3);
#undef CHX_RERANK
  launch_check("rerank");
}

// ------------------------------------------------------------------ certified scan
namespace {

// 16 bytes of a row (4 binary32 or 8 bf16 coordinates) as binary32
template <int DT>
__device__ __forceinline__ void cert_vec(const void* row, int m, float (&v)[DT == CH_F32 ? 4 : 8]) {
  const uint4 w = __ldg(static_cast<const uint4*>(row) + m);
  if constexpr (DT == CH_F32) {
    v[0] = __uint_as_float(w.x);
    v[1] = __uint_as_float(w.y);
    v[2] = __uint_as_float(w.z);
    v[3] = __uint_as_float(w.w);
  } else {
    const uint32_t q[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      v[2 * e] = __uint_as_float(q[e] << 16);
      v[2 * e + 1] = __uint_as_float(q[e] & 0xFFFF0000u);
    }
  }
}

// canonical squared l2 distance of two rows by one thread: the 32 partials in
// registers, then the halving tree
template <int DT>
__device__ __forceinline__ float cert_dist(const void* q, const void* b, int d) {
  constexpr int PER = DT == CH_F32 ? 4 : 8;
  const int words = d / PER;
  float p[32];
#pragma unroll
  for (int r = 0; r < 32; ++r) p[r] = 0.0f;
#pragma unroll 1
  for (int m0 = 0; m0 < words; m0 += 32 / PER) {
#pragma unroll
    for (int m = 0; m < 32 / PER; ++m)
      if (m0 + m < words) {
        float x[PER], y[PER];
        cert_vec<DT>(q, m0 + m, x);
        cert_vec<DT>(b, m0 + m, y);
#pragma unroll
        for (int e = 0; e < PER; ++e) {
          const float t = __fsub_rn(x[e], y[e]);
          p[m * PER + e] = __fmaf_rn(t, t, p[m * PER + e]);
        }
      }
  }
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1)
#pragma unroll
    for (int r = 0; r < s; ++r) p[r] = __fadd_rn(p[r], p[r + s]);
  return p[0];
}

// One warp per sample.  The best screened entry gives a first canonical P; then
// every column that the bound (k_screen.cu, certified exact scan) does not exclude
// is evaluated: the four columns of each class entry at or below the threshold and,
// where a class's second-smallest tile minimum is at or below it too, all of the
// class's columns in the chunk.  The entries collect in a queue, eight at a time
// give a column to every lane, and a lane computes its column's distance alone (no
// shuffles, 32 rows in flight); the threshold tightens after each such batch.  A
// sample with more than c.limit columns, with values outside the bound's range, or
// whose screen gave up is listed instead.
constexpr int kCertQueue = 8 + 32;  // a batch and the entries one part can add

template <int DT>
__global__ void __launch_bounds__(32 * kRerankWarps, 2) k_certify(const void* A, int64_t nA, const int64_t* qidx,
                                                               const void* B, CertArgs c, float* min_d,
                                                               int64_t* argmin) {
  pdl_entry();
  __shared__ int32_t s_queue[kRerankWarps][kCertQueue];
  const int lane = threadIdx.x & 31;
  int32_t* queue = s_queue[threadIdx.x >> 5];
  const int64_t l = int64_t(blockIdx.x) * kRerankWarps + (threadIdx.x >> 5);
  if (l >= c.T) return;
  const int64_t g = c.l0 + l;
  const int64_t a = qidx ? qidx[g] : g;
  if (a < 0) {
    if (lane == 0) {
      min_d[g] = 0.0f;
      if (argmin) argmin[g] = -1;
    }
    return;
  }
  auto give_up = [&] {
    if (lane == 0) {
      const uint32_t at = atomicAdd(&c.ctl[0], 1u);
      c.list[at] = static_cast<int32_t>(g);
      c.best[at] = ~0ull;
    }
  };
  if (a >= nA || *reinterpret_cast<volatile const uint32_t*>(&c.ctl[1])) {
    give_up();
    return;
  }
  const size_t row_bytes = size_t(c.d) * (DT == CH_F32 ? 4 : 2);
  const char* qrow = static_cast<const char*>(A) + size_t(a) * row_bytes;
  const size_t stride = size_t(c.T) * 32;  // entries of one part
  const size_t at = size_t(l) * 32 + lane;
  // |q|^2, and the best entry over all parts (lane = class)
  float qn = 0.0f;
  for (int j = lane; j < c.d; j += 32) {
    const float x = load_elem<DT>(qrow, 0, c.d, j, nullptr);
    qn = __fmaf_rn(x, x, qn);
  }
  float ms = __int_as_float(0x7F800000);
  int32_t mi = INT32_MAX;
#pragma unroll 4
  for (int p = 0; p < c.parts; ++p) {
    const float v = __ldg(&c.part_s[p * stride + at]);
    const int32_t i = __ldg(&c.part_i[p * stride + at]);
    if (i >= 0 && v < ms) {
      ms = v;
      mi = i;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    qn = __fadd_rn(qn, __shfl_xor_sync(0xFFFFFFFFu, qn, o));
    const float os = __shfl_xor_sync(0xFFFFFFFFu, ms, o);
    const int32_t oi = __shfl_xor_sync(0xFFFFFFFFu, mi, o);
    if (os < ms || (os == ms && oi < mi)) {
      ms = os;
      mi = oi;
    }
  }
  if (mi == INT32_MAX || !(qn < 1e37f)) {
    give_up();
    return;
  }
  float best = __int_as_float(0x7F800000);  // this lane's minimum and its column
  uint32_t bidx = 0xFFFFFFFFu;
  float bestP = best, thr = best;           // the warp's smallest squared distance, and its threshold
  // queue[0 .. cnt - 1], cnt <= 8: lane 4 e + o takes column queue[e] + 32 o
  auto batch = [&](int cnt) {
    const int64_t b = lane < 4 * cnt ? int64_t(queue[lane >> 2]) + 32 * (lane & 3) : c.nB;
    float P = __int_as_float(0x7F800000);
    if (b < c.nB) {
      P = cert_dist<DT>(qrow, static_cast<const char*>(B) + size_t(b) * row_bytes, c.d);
      const float dist = __fsqrt_rn(P);
      if (dist < best || (dist == best && static_cast<uint32_t>(b) < bidx)) {
        best = dist;
        bidx = static_cast<uint32_t>(b);
      }
    }
    // distances are >= 0 (or NaN, above every number): their bits order like integers
    bestP = fminf(bestP, __uint_as_float(__reduce_min_sync(0xFFFFFFFFu, __float_as_uint(P))));
    thr = __double2float_ru(static_cast<double>(bestP) * c.p_scale - static_cast<double>(qn) * c.q_scale + 0x1p-100);
  };
  if (lane == 0) queue[0] = mi;
  __syncwarp();
  batch(1);
  if (!(bestP < 1e37f)) {
    give_up();
    return;
  }
  // columns to evaluate under this threshold
  const int64_t tiles = c.chunk_len / c.tile;
  int64_t cols = 0;
#pragma unroll 4
  for (int p = 0; p < c.parts; ++p) {
    const bool e = __ldg(&c.part_s[p * stride + at]) <= thr;
    const bool all = __ldg(&c.part_2[p * stride + at]) <= thr;
    cols += 4 * __popc(__ballot_sync(0xFFFFFFFFu, e && !all)) + 4 * tiles * __popc(__ballot_sync(0xFFFFFFFFu, all));
  }
  if (cols > c.limit) {
    give_up();
    return;
  }
  int n = 0;  // queued entries
  auto drain = [&](int keep) {  // batches of eight until at most keep entries are left
    __syncwarp();
    while (n > keep) {
      const int cnt = min(n, 8);
      batch(cnt);
      n -= cnt;
      const int32_t v = lane < n ? queue[lane + cnt] : 0;  // n <= 32 after a full batch
      __syncwarp();
      if (lane < n) queue[lane] = v;
      __syncwarp();
    }
  };
  for (int p = 0; p < c.parts; ++p) {
    const float s1 = __ldg(&c.part_s[p * stride + at]);
    const float s2 = __ldg(&c.part_2[p * stride + at]);
    const int32_t i = __ldg(&c.part_i[p * stride + at]);
    const unsigned all = __ballot_sync(0xFFFFFFFFu, s2 <= thr);
    const bool mine = s1 <= thr && i >= 0 && i != mi && !(all >> lane & 1u);
    const unsigned one = __ballot_sync(0xFFFFFFFFu, mine);
    if (mine) queue[n + __popc(one & ((1u << lane) - 1u))] = i;
    n += __popc(one);
    drain(7);
    for (unsigned rest = all; rest; rest &= rest - 1) {
      const int64_t c0 = int64_t(p / c.slices) * c.chunk_len + (p % c.slices) * 128 + (__ffs(rest) - 1);
      const int64_t end = min(c.nB, (int64_t(p / c.slices) + 1) * c.chunk_len);
      for (int64_t b = c0; b < end; b += 32 * int64_t(c.tile)) {  // 32 tiles of the class at a time
        const int64_t mb = b + int64_t(lane) * c.tile;
        if (mb < end) queue[n + lane] = static_cast<int32_t>(mb);
        n += static_cast<int>(min(int64_t(32), (end - b + c.tile - 1) / c.tile));
        drain(7);
      }
    }
  }
  drain(0);
  const uint32_t least = __reduce_min_sync(0xFFFFFFFFu, __float_as_uint(best));
  bidx = __reduce_min_sync(0xFFFFFFFFu, __float_as_uint(best) == least ? bidx : 0xFFFFFFFFu);
  if (lane == 0) {
    min_d[g] = __uint_as_float(least);
    if (argmin) argmin[g] = static_cast<int64_t>(bidx);
  }
}

}  // namespace

void launch_certify(const ch_set* A, const int64_t* qidx, const ch_set* B, const CertArgs& c, float* min_d,
                    int64_t* argmin, cudaStream_t s) {
  const int blocks = static_cast<int>(ceil_div(c.T, kRerankWarps));
  if (A->dtype == CH_F32)
    launch_k(k_certify<CH_F32>, blocks, 32 * kRerankWarps, 0, s, A->data, A->n, qidx, B->data, c, min_d, argmin);
  else
    launch_k(k_certify<CH_BF16>, blocks, 32 * kRerankWarps, 0, s, A->data, A->n, qidx, B->data, c, min_d, argmin);
  launch_check("certify");
}

}  // namespace chx
