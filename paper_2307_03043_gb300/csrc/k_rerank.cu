// k_rerank.cu -- the canonical rerank after the tensor-core screen (Fig. 1,
// step 3): for each sample, the R best screened entries by screen score, the
// canonical binary32 distance of every column they stand for, and the minimum.
#include "common.cuh"

namespace chx {

namespace {

constexpr int kRerankWarps = 8;  // samples per block, a warp each

// 16 bytes of a row as binary32 (FP8: times the row's scale)
template <int DT>
constexpr int kRowPer = DT == CH_F32 ? 4 : DT == CH_BF16 ? 8 : 16;
template <int DT>
__device__ __forceinline__ void row_vec(const void* row, int m, float sc, float (&v)[kRowPer<DT>]) {
  const uint4 w = __ldg(static_cast<const uint4*>(row) + m);
  const uint32_t q[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int e = 0; e < kRowPer<DT>; ++e) {
    if constexpr (DT == CH_F32) v[e] = __uint_as_float(q[e]);
    else if constexpr (DT == CH_BF16) v[e] = __uint_as_float(e & 1 ? q[e / 2] & 0xFFFF0000u : q[e / 2] << 16);
    else v[e] = __fmul_rn(e4m3_to_f32(static_cast<uint8_t>(q[e / 4] >> (8 * (e % 4)))), sc);
  }
}

// row a of a set, widened, into the warp's shared-memory row q [d]
template <int DT>
__device__ __forceinline__ void stage_query(float* q, const char* row, float sc, int d, int lane) {
  for (int m = lane; m < d / kRowPer<DT>; m += 32) {
    float v[kRowPer<DT>];
    row_vec<DT>(row, m, sc, v);
#pragma unroll
    for (int e = 0; e < kRowPer<DT>; e += 4)
      *reinterpret_cast<float4*>(q + m * kRowPer<DT> + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
  }
  __syncwarp();
}

// p += |x - y| (l1) or (x - y)^2 (l2), rounded as the canonical distance rounds
template <int METRIC>
__device__ __forceinline__ void add_term(float& p, float x, float y) {
  const float t = __fsub_rn(x, y);
  p = METRIC == CH_L1 ? __fadd_rn(p, fabsf(t)) : __fmaf_rn(t, t, p);
}

// Canonical l1 sums or squared l2 distances of the staged row q to up to 32 rows of B.
// Two forms for rows of a multiple of 16 bytes, the same sums in the same order:
//  * lane_dist, rows below 512 bytes: a row per lane, the 32 partials in its registers,
//    no shuffles; a warp keeps 32 rows in flight.  Its loads touch a sector per lane, so
//    wide rows outgrow L1 between them;
//  * group_dist, wider rows: 32 / C lanes per row (C coordinates per 16-byte word), each
//    owning C partials, so a row is read in whole 64- or 128-byte pieces; NR rows per
//    lane group side by side.
// Kernel time of the rerank of 8 entries x 4 columns, this form / the earlier four rows per
// warp with a shuffle tree each, caches as the call leaves them (cold in brackets): f32
// d = 128, 4.6k samples of 100k 25 / 27 us (31 / 29), bf16 d = 384, 300k 49 / 58 (49 / 57),
// bf16 d = 768, 200k 89 / 93 (87 / 93), fp8 d = 384, 300k 50 / 100 (51 / 107).  The
// line lies between the rows measured in both forms, cold: 384 bytes (fp8 d = 384) has the
// lane form at half the earlier time; at 512 (f32 d = 128), 768 and 1536 bytes the lane
// form took 37, 122 and 256 us, the group form 31, 67 and 97.
constexpr int kWideRow = 512;

template <int DT, int METRIC>
__device__ __forceinline__ float lane_dist(const float* __restrict__ q, const void* __restrict__ b, float sb, int d) {
  constexpr int PER = kRowPer<DT>;
  const int words = d / PER;
  float p[32];
#pragma unroll
  for (int r = 0; r < 32; ++r) p[r] = 0.0f;
#pragma unroll 1
  for (int m0 = 0; m0 < words; m0 += 32 / PER) {
#pragma unroll
    for (int m = 0; m < 32 / PER; ++m)
      if (m0 + m < words) {
        float y[PER];
        row_vec<DT>(b, m0 + m, sb, y);
#pragma unroll
        for (int e = 0; e < PER; e += 4) {
          const float4 x = *reinterpret_cast<const float4*>(q + (m0 + m) * PER + e);
          const float xx[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
          for (int k = 0; k < 4; ++k) add_term<METRIC>(p[m * PER + e + k], xx[k], y[e + k]);
        }
      }
  }
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1)
#pragma unroll
    for (int r = 0; r < s; ++r) p[r] = __fadd_rn(p[r], p[r + s]);
  return p[0];
}

// cols [32] in shared memory (entries from ncols on are ignored): the distance of row
// cols[lane] on every lane < ncols
template <int DT, int METRIC>
__device__ __forceinline__ float group_dist(const float* __restrict__ q, const char* __restrict__ B, size_t row_bytes,
                                            const float* __restrict__ scB, const int32_t* cols, int ncols, int d) {
  constexpr int C = kRowPer<DT>, LPR = 32 / C, G = 32 / LPR, NR = DT == CH_F32 ? 4 : DT == CH_BF16 ? 2 : 1;
  const int lane = threadIdx.x & 31, sub = lane % LPR, grp = lane / LPR;
  const int chunks = d / C;
  float mine = 0.0f;
  for (int base = 0; base < ncols; base += G * NR) {
    const void* row[NR];
    float sb[NR], p[NR][C];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
      const int at = base + k * G + grp;
      const int64_t b = cols[at < ncols ? at : 0];
      row[k] = B + size_t(b) * row_bytes;
      sb[k] = DT == CH_FP8E4M3 ? scB[b] : 1.0f;
#pragma unroll
      for (int i = 0; i < C; ++i) p[k][i] = 0.0f;
    }
#pragma unroll 4
    for (int m = sub; m < chunks; m += LPR) {
      float x[C];
#pragma unroll
      for (int e = 0; e < C; e += 4) {
        const float4 t = *reinterpret_cast<const float4*>(q + m * C + e);
        x[e] = t.x;
        x[e + 1] = t.y;
        x[e + 2] = t.z;
        x[e + 3] = t.w;
      }
#pragma unroll
      for (int k = 0; k < NR; ++k) {
        float y[C];
        row_vec<DT>(row[k], m, sb[k], y);
#pragma unroll
        for (int i = 0; i < C; ++i) add_term<METRIC>(p[k][i], x[i], y[i]);
      }
    }
#pragma unroll
    for (int k = 0; k < NR; ++k) {
#pragma unroll
      for (int s = 16; s >= C; s >>= 1)
#pragma unroll
        for (int i = 0; i < C; ++i) p[k][i] = __fadd_rn(p[k][i], __shfl_down_sync(0xFFFFFFFFu, p[k][i], s / C, LPR));
#pragma unroll
      for (int s = C / 2; s >= 1; s >>= 1)
#pragma unroll
        for (int i = 0; i < s; ++i) p[k][i] = __fadd_rn(p[k][i], p[k][i + s]);
      // group g's sum sits on its first lane and belongs to column base + k G + g
      const int g = lane - base - k * G;
      const float v = __shfl_sync(0xFFFFFFFFu, p[k][0], (g >= 0 && g < G ? g : 0) * LPR);
      if (g >= 0 && g < G) mine = v;
    }
  }
  return mine;
}

// One warp per sample: the R best screened entries over all chunks (by s, then
// index), the canonical binary32 distance of each of an entry's occ columns
// (first column + o * stride, o < occ <= 4, columns < nB), and their minimum (ties:
// smaller index).  Lane k holds the entries k, k + 32, ... and its smallest one; a
// round takes the smallest of those by two integer minima and only the lane that
// gave it looks its entries over again.  Eight entries then give every lane one column.
template <int DT, bool WIDE>
__global__ void __launch_bounds__(32 * kRerankWarps) k_rerank(const void* A, const float* scA, int64_t nA, const void* B,
                                                const float* scB, int64_t nB, int d, const int64_t* idx, int64_t T,
                                                const float* part_s, const int32_t* part_i, int parts, int per,
                                                int occ, int stride, int R, float* min_d, int64_t* argmin) {
  pdl_entry();
  extern __shared__ __align__(16) float s_dyn[];  // per warp: the query [d], scores and columns [parts * per]
  __shared__ int32_t s_first[kRerankWarps][8], s_cols[WIDE ? kRerankWarps : 1][32];
  const int wib = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nc = parts * per;
  float* q = s_dyn + size_t(wib) * ((d + 3) / 4 * 4 + 2 * nc);
  uint32_t* s_s = reinterpret_cast<uint32_t*>(q + (d + 3) / 4 * 4);
  int32_t* s_i = reinterpret_cast<int32_t*>(s_s + nc);
  int32_t* first = s_first[wib];
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
  const size_t row_bytes = size_t(d) * (DT == CH_F32 ? 4 : DT == CH_BF16 ? 2 : 1);
  stage_query<DT>(q, static_cast<const char*>(A) + size_t(a) * row_bytes, DT == CH_FP8E4M3 ? scA[a] : 1.0f, d, lane);
  // entries in integer order (-0 as +0; NaN scores and empty entries last), this lane's smallest
  constexpr uint32_t kNone = 0xFFFFFFFFu;
  uint32_t ms = kNone;
  int32_t mi = INT32_MAX;
  int mp = -1;
  auto smaller = [&](uint32_t v, int32_t i, int p) {
    if (v != kNone && (v < ms || (v == ms && i < mi))) {
      ms = v;
      mi = i;
      mp = p;
    }
  };
#pragma unroll 4
  for (int p = lane; p < nc; p += 32) {
    const int c = p / per, k = p % per;
    const size_t off = (size_t(c) * T + l) * per + k;
    const float v = part_s[off];
    const int32_t i = part_i[off];
    const uint32_t e = i >= 0 && v == v ? ord_enc(v + 0.0f) : kNone;
    s_s[p] = e;
    s_i[p] = i;
    smaller(e, i, p);
  }
  float best = __int_as_float(0x7F800000);  // this lane's minimum and its column
  uint32_t bcol = kNone;
  for (int r0 = 0; r0 < R; r0 += 8) {
    int n = 0;
    for (; n < min(8, R - r0); ++n) {
      const uint32_t least = __reduce_min_sync(0xFFFFFFFFu, ms);
      if (least == kNone) break;  // fewer than R entries
      const int32_t col = __reduce_min_sync(0xFFFFFFFFu, ms == least ? mi : INT32_MAX);
      if (lane == 0) first[n] = col;
      if (ms == least && mi == col) {  // taken; columns are distinct, so one lane
        s_s[mp] = kNone;
        ms = kNone;
        mi = INT32_MAX;
        for (int p = lane; p < nc; p += 32) smaller(s_s[p], s_i[p], p);
      }
    }
    __syncwarp();
    int32_t col = -1;  // this lane's column
    if ((lane >> 2) < n && (lane & 3) < occ) {
      const int64_t b = int64_t(first[lane >> 2]) + int64_t(lane & 3) * stride;
      if (b < nB) col = static_cast<int32_t>(b);
    }
    float P = 0.0f;
    if constexpr (WIDE) {
      if (n > 0) {
        int32_t* cols = s_cols[wib];
        cols[lane] = col >= 0 ? col : 0;  // idle lanes read row 0 (an entry's own column may be past the end)
        __syncwarp();
        P = group_dist<DT, CH_L2>(q, static_cast<const char*>(B), row_bytes, scB, cols, 4 * n, d);
      }
    } else if (col >= 0) {
      P = lane_dist<DT, CH_L2>(q, static_cast<const char*>(B) + size_t(col) * row_bytes, DT == CH_FP8E4M3 ? scB[col] : 1.0f, d);
    }
    if (col >= 0) {
      const float dist = __fsqrt_rn(P);
      if (dist < best || (dist == best && static_cast<uint32_t>(col) < bcol)) {
        best = dist;
        bcol = static_cast<uint32_t>(col);
      }
    }
    __syncwarp();
    if (n < 8) break;
  }
  const uint32_t least = __reduce_min_sync(0xFFFFFFFFu, __float_as_uint(best));
  bcol = __reduce_min_sync(0xFFFFFFFFu, __float_as_uint(best) == least ? bcol : kNone);
  if (lane == 0) {
    min_d[l] = __uint_as_float(least);
    if (argmin) argmin[l] = bcol == kNone ? INT64_MAX : static_cast<int64_t>(bcol);
  }
}

}  // namespace

void launch_rerank(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, const float* part_s,
                   const int32_t* part_i, int parts, int per, int occ, int stride, int R, float* min_d,
                   int64_t* argmin, cudaStream_t s) {
  CHX_CHECK(parts * per <= kRerankMaxCand && occ <= kRerankMaxOcc, CH_EINVAL, "rerank candidate list too long");
  const int blocks = static_cast<int>(ceil_div(T, kRerankWarps));
  const size_t smem = size_t(kRerankWarps) * ((size_t(A->d) + 3) / 4 * 4 + 2 * size_t(parts) * per) * 4;
  auto run = [&](auto kern) {
    // a constant value, so concurrent callers on other threads never race on it
    CHX_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  static_cast<int>(size_t(kRerankWarps) * (kMaxDim + 2 * kRerankMaxCand) * 4)));
    launch_k(kern, blocks, 32 * kRerankWarps, smem, s, A->data, A->scales, A->n, B->data, B->scales, B->n, A->d, qidx, T,
             part_s, part_i, parts, per, occ, stride, R, min_d, argmin);
  };
  const bool wide = size_t(A->d) * elem_size(A->dtype) >= kWideRow;
  if (A->dtype == CH_F32) wide ? run(k_rerank<CH_F32, true>) : run(k_rerank<CH_F32, false>);
  else if (A->dtype == CH_BF16) wide ? run(k_rerank<CH_BF16, true>) : run(k_rerank<CH_BF16, false>);
  else wide ? run(k_rerank<CH_FP8E4M3, true>) : run(k_rerank<CH_FP8E4M3, false>);
  launch_check("rerank");
}

// ------------------------------------------------------------------ certified scan
namespace {

// One warp per sample.  The best screened entry gives a first canonical P; then
// every column that the bound (k_screen.cu, certified exact scan) does not exclude
// is evaluated: the four columns of each class entry at or below the threshold and,
// where a class's second-smallest tile minimum is at or below it too, all of the
// class's columns in the chunk.  The entries collect in a queue, eight at a time
// give a column to every lane, and the warp computes the 32 distances in the form its
// rows allow (FORM below); the threshold tightens after each such batch.  A point
// at distance 0 leaves only smaller indices to look at: however often a query is
// repeated in B, its first copy answers it.  A sample with more than c.limit columns,
// with values outside the bound's range, or whose screen gave up is listed instead.
constexpr int kCertQueue = 8 + 32;  // a batch and the entries one part can add

// FORM: how a batch's distances are formed.  Rows of a multiple of 16 bytes on aligned
// bases: a row per lane (lane_dist) or, from kWideRow bytes on, per lane group
// (group_dist); any others: CF_ROWS.
enum : int { CF_LANE = 0, CF_GROUP = 1, CF_ROWS = 2 };

// CF_ROWS, for rows of any length: four rows at a time, lane r summing coordinates
// j = r mod 32 of each, the tree by shuffles; cols as for group_dist
template <int DT, int METRIC>
__device__ __forceinline__ float rows_dist(const float* __restrict__ q, const void* __restrict__ B,
                                           const float* __restrict__ scB, const int32_t* cols, int ncols, int d) {
  const int lane = threadIdx.x & 31;
  float mine = 0.0f;
  for (int base = 0; base < ncols; base += 4) {
    int64_t b[4];
    float p[4];
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      b[o] = cols[base + o < ncols ? base + o : 0];
      p[o] = 0.0f;
    }
#pragma unroll 4
    for (int j = lane; j < d; j += 32) {
      const float x = q[j];
#pragma unroll
      for (int o = 0; o < 4; ++o) add_term<METRIC>(p[o], x, load_elem<DT>(B, b[o], d, j, scB));
    }
#pragma unroll
    for (int sh = 16; sh >= 1; sh >>= 1)
#pragma unroll
      for (int o = 0; o < 4; ++o) p[o] = __fadd_rn(p[o], __shfl_down_sync(0xFFFFFFFFu, p[o], sh));
#pragma unroll
    for (int o = 0; o < 4; ++o) {
      const float v = __shfl_sync(0xFFFFFFFFu, p[o], 0);
      if (lane == base + o) mine = v;
    }
  }
  return mine;
}

template <int DT, int METRIC, int FORM>
__global__ void __launch_bounds__(32 * kRerankWarps, 2) k_certify(const void* A, const float* scA, int64_t nA,
                                                                  const int64_t* qidx, const void* B, const float* scB,
                                                                  CertArgs c, float* min_d, int64_t* argmin) {
  pdl_entry();
  extern __shared__ __align__(16) float s_dyn[];  // the queries [warps][d]
  __shared__ int32_t s_queue[kRerankWarps][kCertQueue], s_cols[FORM != CF_LANE ? kRerankWarps : 1][32];
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
  const size_t row_bytes = size_t(c.d) * (DT == CH_F32 ? 4 : DT == CH_BF16 ? 2 : 1);
  const size_t stride = size_t(c.T) * 32;  // entries of one part
  const size_t at = size_t(l) * 32 + lane;
  float* q = s_dyn + size_t(threadIdx.x >> 5) * ((c.d + 3) / 4 * 4);
  if constexpr (FORM == CF_ROWS) {
    for (int j = lane; j < c.d; j += 32) q[j] = load_elem<DT>(A, a, c.d, j, scA);
    __syncwarp();
  } else {
    stage_query<DT>(q, static_cast<const char*>(A) + size_t(a) * row_bytes, DT == CH_FP8E4M3 ? scA[a] : 1.0f, c.d, lane);
  }
  // |q|^2 where the threshold has a share of it, and the best entry over all parts (lane = class)
  float qn = 0.0f;
  if (c.q_scale != 0.0)
    for (int j = lane; j < c.d; j += 32) qn = __fmaf_rn(q[j], q[j], qn);
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
  // queue[0 .. cnt - 1], cnt <= 8: lane 4 e + o takes column queue[e] + o occ_cols
  auto batch = [&](int cnt) {
    const int64_t b = lane < 4 * cnt ? int64_t(queue[lane >> 2]) + c.occ_cols * (lane & 3) : c.nB;
    float P = __int_as_float(0x7F800000);
    if constexpr (FORM != CF_LANE) {
      int32_t* cols = s_cols[threadIdx.x >> 5];
      __syncwarp();
      cols[lane] = static_cast<int32_t>(b < c.nB ? b : 0);
      __syncwarp();
      const float v = FORM == CF_GROUP
                          ? group_dist<DT, METRIC>(q, static_cast<const char*>(B), row_bytes, scB, cols, 4 * cnt, c.d)
                          : rows_dist<DT, METRIC>(q, B, scB, cols, 4 * cnt, c.d);
      if (b < c.nB) P = v;
    } else if (b < c.nB) {
      P = lane_dist<DT, METRIC>(q, static_cast<const char*>(B) + size_t(b) * row_bytes,
                                DT == CH_FP8E4M3 ? scB[b] : 1.0f, c.d);
    }
    if (b < c.nB) {
      const float dist = METRIC == CH_L1 ? P : __fsqrt_rn(P);
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
  // a point at distance 0 (its index): none from it on matters
  const uint32_t stop = bestP == 0.0f ? __reduce_min_sync(0xFFFFFFFFu, best == 0.0f ? bidx : 0xFFFFFFFFu) : 0xFFFFFFFFu;
  // columns to evaluate under this threshold
  const int64_t tiles = c.chunk_len / c.tile;
  int64_t cols = 0;
  if (stop == 0xFFFFFFFFu) {
#pragma unroll 4
    for (int p = 0; p < c.parts; ++p) {
      const bool e = __ldg(&c.part_s[p * stride + at]) <= thr;
      const bool all = __ldg(&c.part_2[p * stride + at]) <= thr;
      cols += 4 * __popc(__ballot_sync(0xFFFFFFFFu, e && !all)) + 4 * tiles * __popc(__ballot_sync(0xFFFFFFFFu, all));
    }
  } else {  // entries and tiles before it
    for (int p = 0; p < c.parts; ++p) {
      const int64_t c0 = int64_t(p / c.slices) * c.chunk_len + (p % c.slices) * c.slice_cols + lane * c.class_cols;
      const int64_t n = (int64_t(stop) - c0 + c.tile - 1) / c.tile;
      const int64_t mine = __ldg(&c.part_2[p * stride + at]) <= thr ? max(int64_t(0), min(tiles, n))
                           : __ldg(&c.part_s[p * stride + at]) <= thr &&
                                 static_cast<uint32_t>(__ldg(&c.part_i[p * stride + at])) < stop;
      cols += 4 * int64_t(__reduce_add_sync(0xFFFFFFFFu, static_cast<uint32_t>(mine)));
    }
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
    const bool mine = s1 <= thr && i != mi && static_cast<uint32_t>(i) < stop && !(all >> lane & 1u);
    const unsigned one = __ballot_sync(0xFFFFFFFFu, mine);
    if (mine) queue[n + __popc(one & ((1u << lane) - 1u))] = i;
    n += __popc(one);
    drain(7);
    for (unsigned rest = all; rest; rest &= rest - 1) {
      const int64_t c0 =
          int64_t(p / c.slices) * c.chunk_len + (p % c.slices) * c.slice_cols + (__ffs(rest) - 1) * c.class_cols;
      const int64_t end = min(min(c.nB, int64_t(stop)), (int64_t(p / c.slices) + 1) * c.chunk_len);
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

void launch_certify(const ch_set* A, const int64_t* qidx, const ch_set* B, int metric, const CertArgs& c, float* min_d,
                    int64_t* argmin, cudaStream_t s) {
  const int blocks = static_cast<int>(ceil_div(c.T, kRerankWarps));
  const size_t row = size_t(c.d) * elem_size(A->dtype);
  const bool aligned = row % 16 == 0 && !((reinterpret_cast<uintptr_t>(A->data) | reinterpret_cast<uintptr_t>(B->data)) & 15);
  auto run = [&](auto kern) {
    CHX_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kRerankWarps * kMaxDim * 4));
    launch_k(kern, blocks, 32 * kRerankWarps, size_t(kRerankWarps) * ((c.d + 3) / 4 * 4) * 4, s, A->data, A->scales, A->n,
             qidx, B->data, B->scales, c, min_d, argmin);
  };
  auto form = [&](auto dt, auto m) {
    constexpr int DT = decltype(dt)::value, METRIC = decltype(m)::value;
    if (!aligned) run(k_certify<DT, METRIC, CF_ROWS>);
    else if (row >= kWideRow) run(k_certify<DT, METRIC, CF_GROUP>);
    else run(k_certify<DT, METRIC, CF_LANE>);
  };
  auto go = [&](auto dt) {
    metric == CH_L1 ? form(dt, std::integral_constant<int, CH_L1>{}) : form(dt, std::integral_constant<int, CH_L2>{});
  };
  if (A->dtype == CH_F32) go(std::integral_constant<int, CH_F32>{});
  else if (A->dtype == CH_BF16) go(std::integral_constant<int, CH_BF16>{});
  else go(std::integral_constant<int, CH_FP8E4M3>{});
  launch_check("certify");
}

}  // namespace chx
