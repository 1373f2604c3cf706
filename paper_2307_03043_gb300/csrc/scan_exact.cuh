// scan_exact.cuh -- exact sampled nearest-neighbour scan (Fig. 1, step 3) and the
// exact brute force (Section 1) on CUDA cores: the kernel, in its plain form (k_scan.cu)
// and its list form (k_scan_list.cu; two files, so that they compile side by side).
//
// Every (q, b) pair is evaluated with the canonical binary32 distance: 32
// strided partials p_r = sum_{j = r mod 32} term_j in increasing j, combined
// by the halving tree p_r += p_{r+s}, s = 16, 8, 4, 2, 1.  A thread holds a
// PQ x PB block of pairs and walks the tree depth first (leaves in bit-reversed
// order), so each pair needs ~6 live registers instead of 32; subtrees whose
// leaves are all beyond d are +0 and skipped (adding +0 to a non-negative
// partial is exact).  The result is bit-identical to the definition, for both
// the minimum and the smallest-index argmin.
#pragma once
#include "common.cuh"

namespace chx {

namespace {

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
// LIST (what the certified and chained scans leave over): the samples are the *count
// listed ones, known only on the device, so a persistent grid cuts B by the rule of
// scan_exact_chunks for that count (none listed: every block returns), the minima fold
// into best[] as (distance bits, index) words by atomicMin, and the last block to end
// writes them to their places (min_d null: k_scan_list_out does).  (Cut for four items per block instead, a fifth, nearly
// empty wave cost T = 4606 x 100k, d = 128 l2 6.7 ms where the plain form takes 5.4;
// l1 and FP8 in run-time loops, d = 64 l1 6.3 ms against 2.9.)
struct ScanList {
  const int32_t* list;
  const uint32_t* count;
  uint32_t* ended;  // blocks that have ended, 0 before
  unsigned long long* best;
  float* min_d;
  int64_t* argmin;
};

// the minimum of the i-th listed sample to its place
__device__ __forceinline__ void list_out(const ScanList& sl, int64_t i) {
  const unsigned long long v = __ldcg(&sl.best[i]);
  const int64_t l = sl.list[i];
  sl.min_d[l] = v == ~0ull ? __int_as_float(0x7F800000) : __uint_as_float(static_cast<uint32_t>(v >> 32));
  if (sl.argmin) sl.argmin[l] = v == ~0ull ? INT64_MAX : static_cast<int64_t>(v & 0xFFFFFFFFull);
}

// chunks of B for qtiles x stages on a grid that runs at once: the fewest of those with
// the least waves x stages per block (the block's threads agree on one)
__device__ __forceinline__ int64_t list_chunks(int64_t qtiles, int64_t stages, unsigned long long* s_best) {
  const int64_t grid = gridDim.x, most = max(int64_t(1), min((stages + 3) / 4, (8 * grid + qtiles - 1) / qtiles));
  if (threadIdx.x == 0) *s_best = ~0ull;
  __syncthreads();
  unsigned long long best = ~0ull;  // cost and, in the low 16 bits (most <= 8 grid < 2^16), chunks
  for (int64_t c = 1 + threadIdx.x; c <= most; c += blockDim.x)
    best = min(best, static_cast<unsigned long long>((qtiles * c + grid - 1) / grid * ((stages + c - 1) / c)) << 16 |
                         static_cast<unsigned long long>(c));
  atomicMin(s_best, best);
  __syncthreads();
  return static_cast<int64_t>(*s_best & 0xFFFFu);
}

template <int DT, int METRIC, int QT, int BT, int PQ, int PB, int NJ, int SUB, bool DB, bool LIST>
__global__ void __launch_bounds__(256, kScanBlocksPerSM)
    k_scan_exact(const void* __restrict__ A, const float* __restrict__ scA, const int64_t* __restrict__ qidx, int64_t T,
                 int64_t nA, const void* __restrict__ B, const float* __restrict__ scB, int64_t nB, int d,
                 int64_t chunk_len, float* part_val, int64_t* part_idx, ScanList sl) {
  pdl_entry();
  int64_t qtiles = 1, items = 1;
  if constexpr (LIST) {
    __shared__ unsigned long long s_plan;
    T = *sl.count;
    if (T == 0) return;
    qtiles = (T + QT - 1) / QT;
    const int64_t stages = (nB + BT * SUB - 1) / (BT * SUB);
    const int64_t want = list_chunks(qtiles, stages, &s_plan);
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
  if constexpr (LIST) {
    __shared__ bool s_last;
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = sl.min_d && atomicAdd(sl.ended, 1u) == gridDim.x - 1;
    __syncthreads();
    if (!s_last) return;
    __threadfence();
#pragma unroll 8
    for (int64_t i = tid; i < T; i += 256) list_out(sl, i);
  }
}

struct TileShape {
  int QT, BT, SUB;  // samples, rows per sub-tile, sub-tiles per stage
};

// small d stages more rows per barrier pair, so the copy of a stage is not
// short next to its latency
TileShape tile_for(int d) {
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
bool scan_double_buffered(int dtype, int d) { return dtype == CH_F32 && d <= 64; }

size_t scan_smem(int d, bool db) {
  const TileShape t = tile_for(d);
  return size_t(d) * ((t.QT + 4) + (db ? 2 : 1) * (t.BT * t.SUB + 4)) * sizeof(float);
}

bool scan_fits(int d) { return scan_smem(d, false) <= 220 * 1024; }

// Blocks of k_scan_exact one SM holds at once for dimension d: the dynamic
// tiles, the per-row minima (16 thread rows x QT x (4 + 8) bytes) and
// the 1 KB reserved per block, out of 228 KB of shared memory per SM.
int scan_blocks_per_sm(int d, bool db) {
  const TileShape t = tile_for(d);
  const size_t per_block = scan_smem(d, db) + size_t(16) * t.QT * 12 + 1024;
  return static_cast<int>(std::max<size_t>(1, std::min<size_t>(kScanBlocksPerSM, (228u * 1024u) / per_block)));
}

template <int DT, int METRIC, bool LIST, int QT, int BT, int PQ, int PB, int NJ = 0, int SUB = 1>
void scan_launch(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, ScanPart part, cudaStream_t s,
                 const ScanList& list) {
  constexpr bool kDB = DT == CH_F32 && NJ > 0 && NJ <= 2;  // the launches of scan_double_buffered(DT, d)
  CHX_CHECK(tile_for(A->d).BT == BT && tile_for(A->d).SUB == SUB, CH_ENOTSUP, "scan tile mismatch");
  const size_t smem = scan_smem(A->d, kDB);
  // a constant value, so concurrent callers on other threads never race on it
  auto kern = k_scan_exact<DT, METRIC, QT, BT, PQ, PB, NJ, SUB, kDB, LIST>;
  CHX_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  const int64_t chunk_len = LIST ? 0 : ceil_div(ceil_div(B->n, part.chunks), BT * SUB) * (BT * SUB);
  dim3 grid(static_cast<unsigned>(ceil_div(T, QT)), static_cast<unsigned>(part.chunks));
  if (LIST) grid = dim3(part.chunks * scan_blocks_per_sm(A->d, kDB));  // part.chunks: the SMs
  launch_k(kern, grid, 256, smem, s, A->data, A->scales, qidx, T, A->n, B->data, B->scales, B->n, A->d, chunk_len,
           part.val, part.idx, list);
}

template <int DT, int METRIC, bool LIST>
void scan_shape(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, ScanPart part, cudaStream_t s,
                const ScanList& list) {
  const TileShape t = tile_for(A->d);
  if (A->d <= 128) {  // terms per partial fixed at compile time
    switch ((A->d + 31) / 32) {
      case 1: scan_launch<DT, METRIC, LIST, 32, 64, 2, 4, 1, 4>(A, qidx, T, B, part, s, list); break;
      case 2: scan_launch<DT, METRIC, LIST, 32, 64, 2, 4, 2>(A, qidx, T, B, part, s, list); break;
      case 3: scan_launch<DT, METRIC, LIST, 32, 64, 2, 4, 3>(A, qidx, T, B, part, s, list); break;
      default: scan_launch<DT, METRIC, LIST, 32, 64, 2, 4, 4>(A, qidx, T, B, part, s, list); break;
    }
  } else if (t.BT == 64)
    scan_launch<DT, METRIC, LIST, 32, 64, 2, 4>(A, qidx, T, B, part, s, list);
  else if (t.BT == 32)
    scan_launch<DT, METRIC, LIST, 32, 32, 2, 2>(A, qidx, T, B, part, s, list);
  else
    scan_launch<DT, METRIC, LIST, 16, 16, 1, 1>(A, qidx, T, B, part, s, list);
}

// the instantiations of one form, by storage type and metric
template <bool LIST>
void scan_form(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, int metric, ScanPart part,
               cudaStream_t s, const ScanList& list) {
  auto go = [&](auto dt) {
    constexpr int DT = decltype(dt)::value;
    metric == CH_L1 ? scan_shape<DT, CH_L1, LIST>(A, qidx, T, B, part, s, list)
                    : scan_shape<DT, CH_L2, LIST>(A, qidx, T, B, part, s, list);
  };
  if (A->dtype == CH_F32) go(std::integral_constant<int, CH_F32>{});
  else if (A->dtype == CH_BF16) go(std::integral_constant<int, CH_BF16>{});
  else go(std::integral_constant<int, CH_FP8E4M3>{});
}

}  // namespace

}  // namespace chx
