// k_scan.cu -- exact sampled nearest-neighbour scan (Fig. 1, step 3) and the
// exact brute force (Section 1) on CUDA cores.
//
// Every (q, b) pair is evaluated with the canonical binary32 distance: 32
// strided partials p_r = sum_{j = r mod 32} term_j in increasing j, combined
// by the halving tree p_r += p_{r+s}, s = 16, 8, 4, 2, 1.  A thread holds a
// PQ x PB block of pairs and walks the tree depth first (leaves in bit-reversed
// order), so each pair needs ~6 live registers instead of 32; subtrees whose
// leaves are all beyond d are +0 and skipped (adding +0 to a non-negative
// partial is exact).  The result is bit-identical to the definition, for both
// the minimum and the smallest-index argmin.
#include <type_traits>

#include "common.cuh"

namespace chx {

// Resident blocks per SM of k_scan_exact: the register cap (80 per thread,
// no spills) lets three 256-thread blocks share an SM, so one block's tile
// copy overlaps the others' arithmetic.
constexpr int kScanBlocksPerSM = 3;

// NJ > 0: d lies in (32 (NJ - 1), 32 NJ], so every partial holds NJ - 1 or NJ
// terms and the loops unroll; NJ = 0: any d, runtime loops.
template <int METRIC, int PQ, int PB, int QS, int BS, int NJ>
struct Tree {
  // the term of coordinate j for every pair; FIRST starts the partial with it
  // (|t| or t*t alone, bit-identical to adding it to +0)
  template <bool FIRST>
  static __device__ __forceinline__ void term(float (&acc)[PQ][PB], const float* __restrict__ Qt,
                                              const float* __restrict__ Bt, int j) {
    float qv[PQ], bv[PB];
    if constexpr (PQ == 2) {
      const float2 t = *reinterpret_cast<const float2*>(Qt + j * QS);
      qv[0] = t.x;
      qv[1] = t.y;
    } else {
#pragma unroll
      for (int p = 0; p < PQ; ++p) qv[p] = Qt[j * QS + p];
    }
    if constexpr (PB == 4) {
      const float4 t = *reinterpret_cast<const float4*>(Bt + j * BS);
      bv[0] = t.x;
      bv[1] = t.y;
      bv[2] = t.z;
      bv[3] = t.w;
    } else if constexpr (PB == 2) {
      const float2 t = *reinterpret_cast<const float2*>(Bt + j * BS);
      bv[0] = t.x;
      bv[1] = t.y;
    } else {
#pragma unroll
      for (int b = 0; b < PB; ++b) bv[b] = Bt[j * BS + b];
    }
#pragma unroll
    for (int p = 0; p < PQ; ++p)
#pragma unroll
      for (int b = 0; b < PB; ++b) {
        const float t = __fsub_rn(qv[p], bv[b]);
        if constexpr (METRIC == CH_L1)
          acc[p][b] = FIRST ? fabsf(t) : __fadd_rn(acc[p][b], fabsf(t));
        else
          acc[p][b] = FIRST ? __fmul_rn(t, t) : __fmaf_rn(t, t, acc[p][b]);
      }
  }

  // leaf R (R < d): sum over j = R, R+32, ... of |q_j - b_j| or (q_j - b_j)^2
  template <int R>
  static __device__ __forceinline__ void leaf(float (&acc)[PQ][PB], const float* __restrict__ Qt,
                                              const float* __restrict__ Bt, int d) {
    term<true>(acc, Qt, Bt, R);
    if constexpr (NJ > 0) {
#pragma unroll
      for (int t = 1; t < NJ; ++t)
        if (t < NJ - 1 || R + 32 * t < d) term<false>(acc, Qt, Bt, R + 32 * t);
    } else {
      for (int j = R + 32; j < d; j += 32) term<false>(acc, Qt, Bt, j);
    }
  }

  // value of partial R after tree steps 16 .. S  (S = 32: the leaf itself)
  template <int R, int S>
  static __device__ __forceinline__ void node(float (&out)[PQ][PB], const float* __restrict__ Qt,
                                              const float* __restrict__ Bt, int d) {
    if constexpr (S == 32) {
      leaf<R>(out, Qt, Bt, d);
    } else {
      node<R, 2 * S>(out, Qt, Bt, d);
      if (NJ >= 2 || R + S < d) {  // d > 32: no partial is empty
        float tmp[PQ][PB];
        node<R + S, 2 * S>(tmp, Qt, Bt, d);
#pragma unroll
        for (int p = 0; p < PQ; ++p)
#pragma unroll
          for (int b = 0; b < PB; ++b) out[p][b] = __fadd_rn(out[p][b], tmp[p][b]);
      }
    }
  }
};

// Copies coordinates jl, jl + 8, ... of source row `row` (-1: zeros) into column
// r of a coordinate-major tile (Ts[j * S + r]).  Lane (rl, jl) = (lane & 3,
// lane >> 2) of a warp takes row 4g + rl of row group g: one warp instruction
// reads 8 consecutive coordinates of 4 rows and, with S = 4 mod 8, stores to
// 32 distinct banks.
template <int DT, int S, int NJ>
__device__ __forceinline__ void stage_row(float* __restrict__ Ts, int r, const void* __restrict__ base,
                                          const float* __restrict__ scales, int64_t row, int d, int jl) {
  static_assert(S % 8 == 4, "conflict-free staging needs S = 4 mod 8");
  if constexpr (NJ > 0) {
#pragma unroll
    for (int k = 0; k < 4 * NJ; ++k) {
      const int j = jl + 8 * k;
      if (k < 4 * (NJ - 1) || j < d) Ts[j * S + r] = row >= 0 ? load_elem<DT>(base, row, d, j, scales) : 0.0f;
    }
  } else {
    for (int j = jl; j < d; j += 8) Ts[j * S + r] = row >= 0 ? load_elem<DT>(base, row, d, j, scales) : 0.0f;
  }
}

// The binary32 form of stage_row as asynchronous 4-byte copies (cp.async, no
// register round trip): row < 0 fills zeros (source size 0).  The copies land
// after cp.async.wait_group.
template <int S, int NJ>
__device__ __forceinline__ void stage_row_async(float* __restrict__ Ts, int r, const float* __restrict__ base,
                                                int64_t row, int d, int jl) {
  static_assert(S % 8 == 4, "conflict-free staging needs S = 4 mod 8");
  const float* src = base + (row >= 0 ? row : 0) * int64_t(d);
  const uint32_t n = row >= 0 ? 4u : 0u;
  auto one = [&](int j) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(static_cast<uint32_t>(
                     __cvta_generic_to_shared(Ts + j * S + r))),
                 "l"(src + j), "r"(n)
                 : "memory");
  };
  if constexpr (NJ > 0) {
#pragma unroll
    for (int k = 0; k < 4 * NJ; ++k) {
      const int j = jl + 8 * k;
      if (k < 4 * (NJ - 1) || j < d) one(j);
    }
  } else {
    for (int j = jl; j < d; j += 8) one(j);
  }
}

// One block: QT samples against a chunk of B, staged SUB x BT rows at a time
// (one pair of barriers per stage); each thread owns PQ samples x PB rows of
// every BT-row sub-tile.
// LIST (what the certified scan leaves over): the samples are the *count listed
// ones, known only on the device, so a persistent grid cuts B into as many chunks
// as keep its blocks busy for that count (none listed: every block returns), and
// the minima fold into best[] as (distance bits, index) words by atomicMin.
struct ScanList {
  const int32_t* list;
  const uint32_t* count;
  unsigned long long* best;
};

template <int DT, int METRIC, int QT, int BT, int PQ, int PB, int NJ, int SUB, bool DB, bool LIST>
__global__ void __launch_bounds__(256, kScanBlocksPerSM)
    k_scan_exact(const void* __restrict__ A, const float* __restrict__ scA, const int64_t* __restrict__ qidx, int64_t T,
                 int64_t nA, const void* __restrict__ B, const float* __restrict__ scB, int64_t nB, int d,
                 int64_t chunk_len, float* part_val, int64_t* part_idx, ScanList sl) {
  pdl_entry();
  int64_t qtiles = 1, items = 1;
  if constexpr (LIST) {
    T = *sl.count;
    if (T == 0) return;
    qtiles = (T + QT - 1) / QT;
    const int64_t stages = (nB + BT * SUB - 1) / (BT * SUB);
    const int64_t want = max(int64_t(1), min((stages + 3) / 4, (4 * int64_t(gridDim.x) + qtiles - 1) / qtiles));
    chunk_len = (stages + want - 1) / want * (BT * SUB);
    items = qtiles * ((nB + chunk_len - 1) / chunk_len);
  }
  constexpr int NTQ = QT / PQ, NTB = BT / PB;
  static_assert(NTQ * NTB == 256, "256 threads");
  static_assert(NTB == 16, "16 thread rows (the occupancy estimate assumes it)");
  constexpr int ST = BT * SUB;  // rows per stage
  constexpr int QS = QT + 4, BS = ST + 4;
  extern __shared__ __align__(16) float smem[];
  float* Qs = smem;
  float* Bs = smem + size_t(d) * QS;  // DB: two stages, the next one in flight during this one's arithmetic
  __shared__ float r_val[NTB][QT];
  __shared__ int64_t r_idx[NTB][QT];

  const int tid = threadIdx.x;
  const int tq = tid % NTQ, tb = tid / NTQ;
  for (int64_t item = LIST ? int64_t(blockIdx.x) : 0; item < items; item += gridDim.x) {
  const int64_t q0 = (LIST ? item % qtiles : int64_t(blockIdx.x)) * QT;
  const int64_t b_begin = (LIST ? item / qtiles : int64_t(blockIdx.y)) * chunk_len;
  const int64_t b_end = min(nB, b_begin + chunk_len);

  // tiles are staged transposed (coordinate-major), four rows per warp instruction
  const int warp = tid >> 5, rl = (tid & 31) & 3, jl = (tid & 31) >> 2;
  for (int g = warp; g < QT / 4; g += 8) {
    const int q = 4 * g + rl;
    int64_t l = q0 + q;
    if constexpr (LIST) l = l < T ? int64_t(sl.list[l]) : INT64_MAX;
    int64_t a = (LIST ? l != INT64_MAX : l < T) ? (qidx ? qidx[l] : l) : -1;
    if (a >= nA) a = -1;
    stage_row<DT, QS, NJ>(Qs, q, A, scA, a, d, jl);
  }

  float best_val[PQ], best_p0[PQ];
  int64_t best_idx[PQ];
#pragma unroll
  for (int p = 0; p < PQ; ++p) {
    best_val[p] = __int_as_float(0x7F800000);
    best_p0[p] = __int_as_float(0x7F800000);
    best_idx[p] = INT64_MAX;
  }
  const float* Qt = Qs + tq * PQ;
  // stage `st` (rows b0 .. b0 + ST - 1 of the chunk) into buffer `buf`
  auto stage_async = [&](int64_t b0, int buf) {
    const int64_t rows = min(static_cast<int64_t>(ST), b_end - b0);
    float* dst = Bs + size_t(buf) * d * BS;
    for (int g = warp; g < ST / 4; g += 8) {
      const int r = 4 * g + rl;
      stage_row_async<BS, NJ>(dst, r, static_cast<const float*>(B), r < rows ? b0 + r : int64_t(-1), d, jl);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  if constexpr (DB) {
    if (b_begin < b_end) stage_async(b_begin, 0);
  }
  int buf = 0;
  for (int64_t b0 = b_begin; b0 < b_end; b0 += ST, buf ^= 1) {
    __syncthreads();
    const int64_t rows = min(static_cast<int64_t>(ST), b_end - b0);
    if constexpr (DB) {
      // the next stage goes into the other buffer (its last readers passed the
      // barrier above); then this stage's copies are waited for
      if (b0 + ST < b_end) {
        stage_async(b0 + ST, buf ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
    } else {
      for (int g = warp; g < ST / 4; g += 8) {
        const int r = 4 * g + rl;
        stage_row<DT, BS, NJ>(Bs, r, B, scB, r < rows ? b0 + r : int64_t(-1), d, jl);
      }
    }
    __syncthreads();
    const float* Bt = Bs + (DB ? size_t(buf) * d * BS : 0) + tb * PB;
    // distances of this thread's pairs in sub-tile `sub`, folded into its minima
    auto scan_sub = [&](int sub) {
      float out[PQ][PB];
      Tree<METRIC, PQ, PB, QS, BS, NJ>::template node<0, 1>(out, Qt, Bt + sub * BT, d);
#pragma unroll
      for (int p = 0; p < PQ; ++p)
#pragma unroll
        for (int b = 0; b < PB; ++b) {
          const int r = sub * BT + tb * PB + b;
          if (r < rows) {
            const float v = out[p][b];
            if constexpr (METRIC == CH_L1) {
              if (v < best_val[p]) {
                best_val[p] = v;
                best_idx[p] = b0 + r;
              }
            } else if (v < best_p0[p]) {
              best_p0[p] = v;
              const float sv = __fsqrt_rn(v);
              if (sv < best_val[p]) {
                best_val[p] = sv;
                best_idx[p] = b0 + r;
              }
            }
          }
        }
    };
    if constexpr (SUB == 1) {
      scan_sub(0);
    } else {
#pragma unroll 1
      for (int sub = 0; sub < SUB && sub * BT < rows; ++sub) scan_sub(sub);
    }
  }
#pragma unroll
  for (int p = 0; p < PQ; ++p) {
    r_val[tb][tq * PQ + p] = best_val[p];
    r_idx[tb][tq * PQ + p] = best_idx[p];
  }
  __syncthreads();
  if (tid < QT) {
    float bv = r_val[0][tid];
    int64_t bi = r_idx[0][tid];
    for (int k = 1; k < NTB; ++k) {
      const float v = r_val[k][tid];
      const int64_t i = r_idx[k][tid];
      if (v < bv || (v == bv && i < bi)) {
        bv = v;
        bi = i;
      }
    }
    const int64_t l = q0 + tid;
    if constexpr (LIST) {
      if (l < T && bi != INT64_MAX)
        atomicMin(&sl.best[l], (static_cast<unsigned long long>(__float_as_uint(bv)) << 32) | static_cast<uint32_t>(bi));
    } else if (l < T) {
      part_val[int64_t(blockIdx.y) * T + l] = bv;
      part_idx[int64_t(blockIdx.y) * T + l] = bi;
    }
  }
  if constexpr (LIST) __syncthreads();  // the tiles and minima are rewritten by the next item
  }
}

// the listed samples' minima to their places
__global__ void k_scan_list_out(ScanList sl, float* min_d, int64_t* argmin) {
  pdl_entry();
  const int64_t n = *sl.count;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const unsigned long long v = sl.best[i];
    const int64_t l = sl.list[i];
    min_d[l] = v == ~0ull ? __int_as_float(0x7F800000) : __uint_as_float(static_cast<uint32_t>(v >> 32));
    if (argmin) argmin[l] = v == ~0ull ? INT64_MAX : static_cast<int64_t>(v & 0xFFFFFFFFull);
  }
}

// Small dimensions (d <= 4, known at compile time): every partial p_r of the
// canonical distance holds the single term of coordinate r, so the halving tree
// reduces to a fixed expression, folded here at compile time.
constexpr int kSmallMaxD = 4;
constexpr int64_t kSmallSegment = int64_t(1) << 31;  // rows whose index fits best[]'s low word
constexpr int kSmallBT = 1024;   // rows of B per shared-memory stage
constexpr int kSmallSub = 32;    // rows per sub-tile: the unit the minima are tracked and evaluated in
constexpr int kSmallPQ = 4;      // samples per thread of a lone scan
constexpr int kSmallQ = 256 * kSmallPQ;
constexpr int kBatchPQ = 8;      // most samples per thread of a batched scan

// partial R after tree steps 16 .. S (S = 32: the leaf) for d = D <= 32 terms
template <int D, int R, int S>
__device__ __forceinline__ float small_node(const float (&leaf)[D]) {
  if constexpr (S == 32) {
    return leaf[R];
  } else if constexpr (R + S < D) {
    return __fadd_rn(small_node<D, R, 2 * S>(leaf), small_node<D, R + S, 2 * S>(leaf));
  } else {
    return small_node<D, R, 2 * S>(leaf);
  }
}

// canonical l1 sum or squared l2 sum of q and b
template <int METRIC, int D>
__device__ __forceinline__ float small_canon(const float (&q)[D], const float (&b)[D]) {
  float leaf[D];
#pragma unroll
  for (int j = 0; j < D; ++j) {
    const float t = __fsub_rn(q[j], b[j]);
    leaf[j] = (METRIC == CH_L1) ? fabsf(t) : __fmul_rn(t, t);
  }
  return small_node<D, 0, 1>(leaf);
}

// element j of row r, the storage type known at run time (the scans of d <= 4 spend
// their time past the loads, and one instantiation serves every type)
__device__ __forceinline__ float elem_of(int dtype, const void* base, int64_t r, int d, int j, const float* scales) {
  return dtype == CH_F32    ? load_elem<CH_F32>(base, r, d, j, scales)
         : dtype == CH_BF16 ? load_elem<CH_BF16>(base, r, d, j, scales)
                            : load_elem<CH_FP8E4M3>(base, r, d, j, scales);
}

// 256 x PQ samples (l0 + thread + 256 p) against rows b_begin .. b_end - 1 of B; the
// minimum (distance bits, index) of each folds into best[] by atomicMin.
//
// A thread keeps PQ samples in registers and walks a shared-memory stage of B two
// rows at a time in packed f32x2 instructions (broadcast 16-byte reads), keeping only
// each sample's smallest value per 32-row sub-tile and the sub-tiles that hold its
// smallest ones; a warp then evaluates the canonical distance of the rows of the
// sub-tiles that matter, a row per lane.
//   l1: the value is the canonical sum itself (3 packed subtractions, 4 additions of
//       |t| and one three-input minimum for two rows at d = 3); the first sub-tile
//       with the smallest value holds the answer.
//   l2: the value is L = |b|^2 shrink - 2 q.b (d packed fused multiply-adds for two
//       rows, the norms staged with the rows) instead of the canonical 3 d - 1
//       operations per row.  With u = 2^-24: the norm's chain is within d u |b|^2, the
//       d fmas within 1.01 d u (|b|^2 + 2 |q||b|) and 2 |q||b| <= |q|^2 + |b|^2, so with
//       shrink = 1 - 4 d u every row has |q - b|^2 >= L + |q|^2 (1 - 1.01 d u).  A row
//       that ties with or beats a canonical squared distance P (itself within 10 u, and
//       equal square roots within 2^-22) therefore has
//         L <= P (1 + 2^-19) - |q|^2 (1 - (2.1 d + 2) u) + 2^-100.
//       The best sub-tile gives P; the second is evaluated where it meets this, the
//       whole chunk where the third does (or where magnitudes leave the bound's range).
// 512 pairs of d = 3 (2.1e10 distances): see launch_scan_small_batch.
template <int METRIC, int D, int PQ>
__device__ __forceinline__ void small_item(int dtype, const void* __restrict__ A, const float* __restrict__ scA,
                                           int64_t nA, const int64_t* __restrict__ qidx, int64_t T,
                                           const void* __restrict__ B, const float* __restrict__ scB, int64_t b_begin,
                                           int64_t b_end, int64_t l0, unsigned long long* __restrict__ best,
                                           uint64_t* __restrict__ Bs) {
  constexpr bool kL2 = METRIC == CH_L2;
  constexpr int W = (kL2 ? D + 1 : D) + ((kL2 ? D + 1 : D) & 1);  // 64-bit words per row pair, even
  const float kInf = __int_as_float(0x7F800000);
  const int lane = threadIdx.x & 31;
  const float u = 0x1p-24f;
  auto load_q = [&](int p, float (&q)[D]) {
    const int64_t l = l0 + 256 * p;
    const int64_t a = l < T ? (qidx ? qidx[l] : l) : -1;
#pragma unroll
    for (int j = 0; j < D; ++j) q[j] = (a >= 0 && a < nA) ? elem_of(dtype, A, a, D, j, scA) : 0.0f;
  };
  uint64_t q2[PQ][D];
  float b1[PQ], b2[PQ], b3[PQ];
  int i1[PQ], i2[PQ];
#pragma unroll
  for (int p = 0; p < PQ; ++p) {
    float q[D];
    load_q(p, q);
#pragma unroll
    for (int j = 0; j < D; ++j) q2[p][j] = kL2 ? f2_pack(-2.0f * q[j], -2.0f * q[j]) : f2_pack(q[j], q[j]);
    b1[p] = b2[p] = b3[p] = kInf;
    i1[p] = i2[p] = -1;
  }
  for (int64_t s0 = b_begin; s0 < b_end; s0 += kSmallBT) {
    const int rows = static_cast<int>(min(static_cast<int64_t>(kSmallBT), b_end - s0));
    const int subs = (rows + kSmallSub - 1) / kSmallSub;
    __syncthreads();
    for (int f = threadIdx.x; f < subs * (kSmallSub / 2); f += 256) {
      float v[2][D], n[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool ok = 2 * f + h < rows;
        n[h] = ok ? 0.0f : kInf;
#pragma unroll
        for (int j = 0; j < D; ++j) {
          // past the end: +inf values for either metric
          v[h][j] = ok ? elem_of(dtype, B, s0 + 2 * f + h, D, j, scB) : (kL2 ? 0.0f : kInf);
          if (kL2 && ok) n[h] = __fmaf_rn(v[h][j], v[h][j], n[h]);
        }
        if (kL2) n[h] = __fmul_rd(n[h], 1.0f - 4 * D * u);
      }
      uint64_t* dst = Bs + size_t(f) * W;
#pragma unroll
      for (int j = 0; j < D; ++j) dst[j] = kL2 ? f2_pack(v[0][j], v[1][j]) : f2_pack(-v[0][j], -v[1][j]);
      if (kL2) dst[D] = f2_pack(n[0], n[1]);
    }
    __syncthreads();
    const int sub0 = static_cast<int>((s0 - b_begin) / kSmallSub);
#pragma unroll 1
    for (int sub = 0; sub < subs; ++sub) {
      const ulonglong2* src = reinterpret_cast<const ulonglong2*>(Bs + size_t(sub) * (kSmallSub / 2) * W);
      float m[PQ];
#pragma unroll
      for (int p = 0; p < PQ; ++p) m[p] = kInf;
#pragma unroll 4
      for (int r = 0; r < kSmallSub / 2; ++r) {
        uint64_t w[W];
#pragma unroll
        for (int k = 0; k < W / 2; ++k) {
          const ulonglong2 t = src[r * (W / 2) + k];
          w[2 * k] = t.x;
          w[2 * k + 1] = t.y;
        }
#pragma unroll
        for (int p = 0; p < PQ; ++p) {
          float2 v;
          if constexpr (kL2) {
            uint64_t acc = w[D];
#pragma unroll
            for (int j = 0; j < D; ++j) f2_fma(acc, q2[p][j], w[j]);
            v = f2_unpack(acc);
          } else {
            float lo[D], hi[D];
#pragma unroll
            for (int j = 0; j < D; ++j) {
              const float2 t = f2_unpack(f2_add(q2[p][j], w[j]));
              lo[j] = fabsf(t.x);
              hi[j] = fabsf(t.y);
            }
            v = make_float2(small_node<D, 0, 1>(lo), small_node<D, 0, 1>(hi));
          }
          m[p] = fmin3(m[p], v.x, v.y);
        }
      }
#pragma unroll
      for (int p = 0; p < PQ; ++p) {
        const bool c1 = m[p] < b1[p];
        if constexpr (kL2) {
          b3[p] = fminf(b3[p], fmaxf(b2[p], m[p]));
          i2[p] = c1 ? i1[p] : m[p] < b2[p] ? sub0 + sub : i2[p];
          b2[p] = fminf(b2[p], fmaxf(b1[p], m[p]));
        }
        i1[p] = c1 ? sub0 + sub : i1[p];
        b1[p] = fminf(b1[p], m[p]);
      }
    }
  }
  // the rows of sub-tile `sub`, one per lane (+inf past the end)
  auto row_of = [&](int sub, float (&b)[D]) {
    const int64_t r = b_begin + int64_t(sub) * kSmallSub + lane;
    const bool ok = sub >= 0 && r < b_end;
#pragma unroll
    for (int j = 0; j < D; ++j) b[j] = ok ? elem_of(dtype, B, r, D, j, scB) : kInf;
    return static_cast<uint32_t>(ok ? r : 0xFFFFFFFFll);
  };
#pragma unroll 1
  for (int p = 0; p < PQ; ++p) {
    if (l0 - threadIdx.x + 256 * p >= T) break;
    // (p varies at run time: pick this group's trackers without indexing registers)
    float t2 = kInf, t3 = kInf;
    int e1 = -1, e2 = -1;
#pragma unroll
    for (int k = 0; k < PQ; ++k)
      if (k == p) {
        t2 = b2[k];
        t3 = b3[k];
        e1 = i1[k];
        e2 = i2[k];
      }
    float q[D];
    load_q(p, q);
    uint32_t dmin = 0xFFFFFFFFu, imin = 0xFFFFFFFFu;  // this lane's sample: distance bits and index
    float P = kInf;
    // folds the warp's rows b (index r) into sample s
    auto fold = [&](int s, const float (&qs)[D], const float (&b)[D], uint32_t r) {
      const float v = small_canon<METRIC, D>(qs, b);
      const uint32_t bits = r != 0xFFFFFFFFu ? __float_as_uint(kL2 ? __fsqrt_rn(v) : v) : 0xFFFFFFFFu;
      const uint32_t least = __reduce_min_sync(0xFFFFFFFFu, bits);
      const uint32_t at = __reduce_min_sync(0xFFFFFFFFu, bits == least ? r : 0xFFFFFFFFu);
      float least_p = 0.0f;
      if constexpr (kL2) least_p = __uint_as_float(__reduce_min_sync(0xFFFFFFFFu, r != 0xFFFFFFFFu ? __float_as_uint(v) : 0x7F800000u));
      if (lane == s) {
        if (least < dmin || (least == dmin && at < imin)) {
          dmin = least;
          imin = at;
        }
        P = fminf(P, least_p);
      }
    };
#pragma unroll 1
    for (int s = 0; s < 32; s += 4) {
      float b[4][D];
      uint32_t r[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) r[k] = row_of(__shfl_sync(0xFFFFFFFFu, e1, s + k), b[k]);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        float qs[D];
#pragma unroll
        for (int j = 0; j < D; ++j) qs[j] = __shfl_sync(0xFFFFFFFFu, q[j], s + k);
        fold(s + k, qs, b[k], r[k]);
      }
    }
    if constexpr (kL2) {
      float qn = 0.0f;
#pragma unroll
      for (int j = 0; j < D; ++j) qn = __fmaf_rn(q[j], q[j], qn);
      const float thr = __fadd_ru(__fsub_ru(__fmul_ru(P, 1.0f + 0x1p-19f), __fmul_rd(qn, 1.0f - (2.125f * D + 2) * u)),
                                  0x1p-100f);
      const bool far = !(qn < 1e37f) || !(P < 1e37f) || t3 <= thr;  // the whole chunk
      for (unsigned rest = __ballot_sync(0xFFFFFFFFu, !far && t2 <= thr); rest; rest &= rest - 1) {
        const int s = __ffs(rest) - 1;
        float qs[D], b[D];
#pragma unroll
        for (int j = 0; j < D; ++j) qs[j] = __shfl_sync(0xFFFFFFFFu, q[j], s);
        const uint32_t r = row_of(__shfl_sync(0xFFFFFFFFu, e2, s), b);
        fold(s, qs, b, r);
      }
      for (unsigned rest = __ballot_sync(0xFFFFFFFFu, far); rest; rest &= rest - 1) {
        const int s = __ffs(rest) - 1;
        float qs[D];
#pragma unroll
        for (int j = 0; j < D; ++j) qs[j] = __shfl_sync(0xFFFFFFFFu, q[j], s);
        // a row per lane, folded once at the end
        unsigned long long mine = ~0ull;
#pragma unroll 4
        for (int64_t r = b_begin + lane; r < b_end; r += 32) {
          float b[D];
#pragma unroll
          for (int j = 0; j < D; ++j) b[j] = elem_of(dtype, B, r, D, j, scB);
          const float v = __fsqrt_rn(small_canon<METRIC, D>(qs, b));
          mine = min(mine, (static_cast<unsigned long long>(__float_as_uint(v)) << 32) | static_cast<uint32_t>(r));
        }
        const uint32_t least = __reduce_min_sync(0xFFFFFFFFu, static_cast<uint32_t>(mine >> 32));
        const uint32_t at = __reduce_min_sync(0xFFFFFFFFu, (mine >> 32) == least ? static_cast<uint32_t>(mine) : 0xFFFFFFFFu);
        if (lane == s) {
          dmin = least;
          imin = at;
        }
      }
    }
    const int64_t l = l0 + 256 * p;
    // +inf and NaN (bits from 0x7F800000 on) are no minimum, as for the other scans
    if (dmin >= 0x7F800000u) {
      dmin = 0x7F800000u;
      imin = 0xFFFFFFFFu;
    }
    if (l < T) atomicMin(&best[l], (static_cast<unsigned long long>(dmin) << 32) | imin);
  }
}

// one pair: blockIdx.x = block of samples, blockIdx.y = chunk of B
template <int METRIC, int D>
__global__ void __launch_bounds__(256, 3) k_scan_small(int dtype, const void* __restrict__ A,
                                                       const float* __restrict__ scA, const int64_t* __restrict__ qidx,
                                                       int64_t T, int64_t nA, const void* __restrict__ B,
                                                       const float* __restrict__ scB, int64_t nB, int64_t chunk_len,
                                                       unsigned long long* best) {
  pdl_entry();
  __shared__ __align__(16) uint64_t Bs[kSmallBT / 2 * (D + 2)];
  const int64_t b_begin = int64_t(blockIdx.y) * chunk_len;
  small_item<METRIC, D, kSmallPQ>(dtype, A, scA, nA, qidx, T, B, scB, b_begin, min(nB, b_begin + chunk_len),
                                  int64_t(blockIdx.x) * kSmallQ + threadIdx.x, best, Bs);
}

// The batched form: one persistent launch over items (pair, groups of 256 samples,
// chunk of B) of many pairs of one storage type, metric and dimension, largest
// first, each block taking the next one from a counter.
template <int METRIC, int D>
__global__ void __launch_bounds__(256, 2) k_scan_small_batch(int dtype, const SmallScanPair* __restrict__ pairs,
                                                             const SmallScanItem* __restrict__ items, int64_t n_items,
                                                             int64_t chunk_len, unsigned int* next) {
  pdl_entry();
  __shared__ __align__(16) uint64_t Bs[kSmallBT / 2 * (D + 2)];
  __shared__ unsigned int s_w;
  for (;;) {
    __syncthreads();  // Bs and s_w are free again
    if (threadIdx.x == 0) s_w = atomicAdd(next, 1u);
    __syncthreads();
    const int64_t w = s_w;
    if (w >= n_items) return;
    const SmallScanItem it = items[w];
    const SmallScanPair pr = pairs[it.pair];
    const int64_t l0 = int64_t(it.group) * 256 + threadIdx.x, b_end = min(pr.nB, it.b0 + chunk_len);
    const auto run = [&](auto pq) {
      small_item<METRIC, D, decltype(pq)::value>(dtype, pr.A, pr.scA, pr.nA, pr.qidx, pr.T, pr.B, pr.scB, it.b0, b_end,
                                                 l0, pr.best, Bs);
    };
    switch (it.groups) {
      case 1: case 2: run(std::integral_constant<int, 2>{}); break;
      case 3: case 4: run(std::integral_constant<int, 4>{}); break;
      case 5: run(std::integral_constant<int, 5>{}); break;
      case 6: run(std::integral_constant<int, 6>{}); break;
      case 7: run(std::integral_constant<int, 7>{}); break;
      default: run(std::integral_constant<int, 8>{}); break;
    }
  }
}

// the lone small scan's minima to its outputs; best [segs][T], segment s holding the
// rows from s * 2^31 on
__global__ void k_scan_best_out(const unsigned long long* best, int segs, int64_t T, const int64_t* qidx, float* min_d,
                                int64_t* argmin) {
  pdl_entry();
  const int64_t l = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (l >= T) return;
  uint32_t bits = 0x7F800000u;
  int64_t at = INT64_MAX;
  for (int s = 0; s < segs; ++s) {
    const unsigned long long v = best[s * T + l];
    if (static_cast<uint32_t>(v >> 32) < bits) {
      bits = static_cast<uint32_t>(v >> 32);
      at = int64_t(s) * kSmallSegment + static_cast<int64_t>(v & 0xFFFFFFFFull);
    }
  }
  const bool none = qidx && qidx[l] < 0;
  min_d[l] = none ? 0.0f : __uint_as_float(bits);
  if (argmin) argmin[l] = none ? -1 : at;
}

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

struct TileShape {
  int QT, BT, SUB;  // samples, rows per sub-tile, sub-tiles per stage
};

// small d stages more rows per barrier pair, so the copy of a stage is not
// short next to its latency
static TileShape tile_for(int d) {
  if (d <= 32) return {32, 64, 4};
  if (d <= 192) return {32, 64, 1};
  if (d <= 768) return {32, 32, 1};
  return {16, 16, 1};
}

// Binary32 rows of d <= 64 stage B through two buffers with asynchronous copies,
// the next stage in flight during this one's arithmetic (100k x 100k, T = 4606:
// d = 8 l1 0.82 -> 0.74 ms, d = 16 l1 1.22 -> 1.06 ms, d = 64 l1 3.12 -> 2.90 ms,
// l2 3.35 -> 2.99 ms).  At d = 128 the second buffer leaves room for two blocks
// per SM instead of three, and the scan was slower (5.0 -> 5.5 ms).
static bool scan_double_buffered(int dtype, int d) { return dtype == CH_F32 && d <= 64; }

static size_t scan_smem(int d, bool db) {
  const TileShape t = tile_for(d);
  return size_t(d) * ((t.QT + 4) + (db ? 2 : 1) * (t.BT * t.SUB + 4)) * sizeof(float);
}

static bool scan_fits(int d) { return scan_smem(d, false) <= 220 * 1024; }

bool scan_list_fits(int64_t T, int d) { return T < (int64_t(1) << 31) && scan_fits(d); }

// Blocks of k_scan_exact one SM holds at once for dimension d: the dynamic
// tiles, the static per-row minima (16 thread rows x QT x (4 + 8) bytes) and
// the 1 KB reserved per block, out of 228 KB of shared memory per SM.
static int scan_blocks_per_sm(int d, bool db) {
  const TileShape t = tile_for(d);
  const size_t per_block = scan_smem(d, db) + size_t(16) * t.QT * 12 + 1024;
  return static_cast<int>(std::max<size_t>(1, std::min<size_t>(kScanBlocksPerSM, (228u * 1024u) / per_block)));
}

int scan_exact_chunks(int64_t T, int64_t nB, int d, int dtype, int sm_count) {
  if (d <= kSmallMaxD) {  // k_scan_small: about 4 blocks per SM, chunks of >= 256 points
    const int64_t qblocks = ceil_div(std::max<int64_t>(T, 1), kSmallQ);
    int64_t chunks = ceil_div(int64_t(sm_count) * 4, qblocks);
    chunks = std::min<int64_t>(chunks, ceil_div(nB, 256));
    return static_cast<int>(std::max<int64_t>(chunks, 1));
  }
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

template <int DT, int METRIC, int QT, int BT, int PQ, int PB, int NJ = 0, int SUB = 1>
static void scan_launch(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, ScanPart part,
                        cudaStream_t s, const ScanList& list) {
  constexpr bool kDB = DT == CH_F32 && NJ > 0 && NJ <= 2;  // the launches of scan_double_buffered(DT, d)
  const bool db = kDB;
  CHX_CHECK(tile_for(A->d).BT == BT && tile_for(A->d).SUB == SUB, CH_ENOTSUP, "scan tile mismatch");
  const size_t smem = scan_smem(A->d, db);
  if (list.list) {
    // the two-sided instantiations would double the build: l1 and FP8 samples, which the
    // chained scan hardly ever leaves over, take the forms with runtime loops
    if constexpr ((METRIC == CH_L2 && DT != CH_FP8E4M3) || NJ == 0) {
      auto kern = k_scan_exact<DT, METRIC, QT, BT, PQ, PB, NJ, SUB, kDB, true>;
      CHX_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
      launch_k(kern, part.chunks * scan_blocks_per_sm(A->d, db), 256, smem, s, A->data, A->scales, qidx, T, A->n,
               B->data, B->scales, B->n, A->d, int64_t(0), part.val, part.idx, list);
    }
    return;
  }
  // a constant value, so concurrent callers on other threads never race on it
  auto kern = k_scan_exact<DT, METRIC, QT, BT, PQ, PB, NJ, SUB, kDB, false>;
  CHX_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  const int64_t chunk_len = ceil_div(ceil_div(B->n, part.chunks), BT * SUB) * (BT * SUB);
  dim3 grid(static_cast<unsigned>(ceil_div(T, QT)), static_cast<unsigned>(part.chunks));
  launch_k(kern, grid, 256, smem, s, A->data, A->scales, qidx, T, A->n, B->data, B->scales, B->n, A->d, chunk_len,
           part.val, part.idx, list);
}

template <int DT, int METRIC>
static void scan_shape(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, ScanPart part,
                       cudaStream_t s, const ScanList& list = ScanList{nullptr, nullptr, nullptr}) {
  const TileShape t = tile_for(A->d);
  constexpr bool kListNJ = METRIC == CH_L2 && DT != CH_FP8E4M3;
  if (list.list && !kListNJ && A->d <= 32) {
    scan_launch<DT, METRIC, 32, 64, 2, 4, 0, 4>(A, qidx, T, B, part, s, list);
  } else if (A->d <= 128 && (!list.list || kListNJ)) {  // terms per partial fixed at compile time
    switch ((A->d + 31) / 32) {
      case 1: scan_launch<DT, METRIC, 32, 64, 2, 4, 1, 4>(A, qidx, T, B, part, s, list); break;
      case 2: scan_launch<DT, METRIC, 32, 64, 2, 4, 2>(A, qidx, T, B, part, s, list); break;
      case 3: scan_launch<DT, METRIC, 32, 64, 2, 4, 3>(A, qidx, T, B, part, s, list); break;
      default: scan_launch<DT, METRIC, 32, 64, 2, 4, 4>(A, qidx, T, B, part, s, list); break;
    }
  } else if (t.BT == 64)
    scan_launch<DT, METRIC, 32, 64, 2, 4>(A, qidx, T, B, part, s, list);
  else if (t.BT == 32)
    scan_launch<DT, METRIC, 32, 32, 2, 2>(A, qidx, T, B, part, s, list);
  else
    scan_launch<DT, METRIC, 16, 16, 1, 1>(A, qidx, T, B, part, s, list);
}

template <int METRIC>
static void scan_small(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, ScanPart part,
                       cudaStream_t s) {
  const int segs = scan_small_segments(B->n);
  CHX_CUDA(cudaMemsetAsync(part.best, 0xFF, size_t(segs) * T * sizeof(unsigned long long), s));
  for (int g = 0; g < segs; ++g) {
    const int64_t n0 = int64_t(g) * kSmallSegment, n = std::min(kSmallSegment, B->n - n0);
    const char* base = static_cast<const char*>(B->data) + size_t(n0) * A->d * elem_size(B->dtype);
    const float* sc = B->scales ? B->scales + n0 : nullptr;
    const int64_t chunk_len = ceil_div(n, part.chunks);
    const dim3 grid(static_cast<unsigned>(ceil_div(T, kSmallQ)), static_cast<unsigned>(part.chunks));
    auto go = [&](auto kern) {
      launch_k(kern, grid, 256, 0, s, A->dtype, A->data, A->scales, qidx, T, A->n, base, sc, n, chunk_len,
               part.best + size_t(g) * T);
    };
    switch (A->d) {
      case 1: go(k_scan_small<METRIC, 1>); break;
      case 2: go(k_scan_small<METRIC, 2>); break;
      case 3: go(k_scan_small<METRIC, 3>); break;
      default: go(k_scan_small<METRIC, 4>); break;
    }
  }
}

template <int DT>
static void scan_metric(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, int metric, ScanPart part,
                        cudaStream_t s) {
  if (A->d <= kSmallMaxD) {
    if (metric == CH_L1)
      scan_small<CH_L1>(A, qidx, T, B, part, s);
    else
      scan_small<CH_L2>(A, qidx, T, B, part, s);
    return;
  }
  if (metric == CH_L1)
    scan_shape<DT, CH_L1>(A, qidx, T, B, part, s);
  else
    scan_shape<DT, CH_L2>(A, qidx, T, B, part, s);
}

void launch_scan_exact(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, int metric, ScanPart part,
                       int sm_count, cudaStream_t s) {
  (void)sm_count;
  if (T == 0) return;
  CHX_CHECK(scan_fits(A->d), CH_ENOTSUP, "dimension too large for the exact scan");
  switch (A->dtype) {
    case CH_F32: scan_metric<CH_F32>(A, qidx, T, B, metric, part, s); break;
    case CH_BF16: scan_metric<CH_BF16>(A, qidx, T, B, metric, part, s); break;
    default: scan_metric<CH_FP8E4M3>(A, qidx, T, B, metric, part, s); break;
  }
  launch_check("scan_exact");
}

int scan_small_segments(int64_t nB) { return static_cast<int>(std::max<int64_t>(1, ceil_div(nB, kSmallSegment))); }

void launch_scan_merge(ScanPart part, int64_t T, int64_t nB, const int64_t* qidx, float* min_d, int64_t* argmin,
                       cudaStream_t s) {
  if (T == 0) return;
  if (part.best) {
    launch_k(k_scan_best_out, static_cast<int>(ceil_div(T, 256)), 256, 0, s, part.best, scan_small_segments(nB), T, qidx,
             min_d, argmin);
    launch_check("scan_best_out");
    return;
  }
  launch_k(k_scan_merge, static_cast<int>(ceil_div(T, 256)), 256, 0, s, part.val, part.idx, part.chunks, T, qidx, min_d,
                                                                  argmin);
  launch_check("scan_merge");
}

void launch_scan_list(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, int metric, const int32_t* list,
                      const uint32_t* ctl, unsigned long long* best, float* min_d, int64_t* argmin, int sm_count,
                      cudaStream_t s) {
  const ScanList sl{list, ctl, best};
  const ScanPart grid{nullptr, nullptr, sm_count, nullptr};  // the list form's grid: sm_count x resident blocks
  auto go = [&](auto dt) {
    constexpr int DT = decltype(dt)::value;
    metric == CH_L1 ? scan_shape<DT, CH_L1>(A, qidx, T, B, grid, s, sl) : scan_shape<DT, CH_L2>(A, qidx, T, B, grid, s, sl);
  };
  if (A->dtype == CH_F32) go(std::integral_constant<int, CH_F32>{});
  else if (A->dtype == CH_BF16) go(std::integral_constant<int, CH_BF16>{});
  else go(std::integral_constant<int, CH_FP8E4M3>{});
  launch_check("scan_list");
  launch_k(k_scan_list_out, static_cast<int>(std::min<int64_t>(ceil_div(T, 256), sm_count)), 256, 0, s, sl, min_d,
           argmin);
  launch_check("scan_list_out");
}

int small_scan_max_groups() { return kBatchPQ; }

template <int METRIC>
static void small_batch_d(const SmallScanPair* pairs, const SmallScanItem* items, int64_t n, int64_t chunk_len,
                          int dtype, int d, int grid, unsigned int* next, cudaStream_t s) {
  auto go = [&](auto kern) { launch_k(kern, grid, 256, 0, s, dtype, pairs, items, n, chunk_len, next); };
  switch (d) {
    case 1: go(k_scan_small_batch<METRIC, 1>); break;
    case 2: go(k_scan_small_batch<METRIC, 2>); break;
    case 3: go(k_scan_small_batch<METRIC, 3>); break;
    default: go(k_scan_small_batch<METRIC, 4>); break;
  }
}

void launch_scan_small_batch(const SmallScanPair* pairs, const SmallScanItem* items, int64_t n_items,
                             int64_t chunk_len, int dtype, int metric, int d, unsigned int* next, int sm_count,
                             cudaStream_t s) {
  if (n_items == 0) return;
  CHX_CHECK(d >= 1 && d <= kSmallMaxD, CH_EINVAL, "batched small scan: d must be in 1..4");
  CHX_CUDA(cudaMemsetAsync(next, 0, sizeof(unsigned int), s));
  // a persistent grid of two resident blocks per SM
  const int grid = static_cast<int>(std::min<int64_t>(n_items, int64_t(sm_count) * 2));
  if (metric == CH_L1)
    small_batch_d<CH_L1>(pairs, items, n_items, chunk_len, dtype, d, grid, next, s);
  else
    small_batch_d<CH_L2>(pairs, items, n_items, chunk_len, dtype, d, grid, next, s);
  launch_check("scan_small_batch");
}

}  // namespace chx
