// k_small.cu -- the exact scan of d <= 4 (Fig. 1, step 3, and the brute force): lone, and
// batched over many pairs.  Same minima and argmins as the general scan, bit for bit.
#include "common.cuh"

namespace chx {

namespace {

// Small dimensions (d <= 4, known at compile time): every partial p_r of the
// canonical distance holds the single term of coordinate r, so the halving tree
// reduces to a fixed expression, folded here at compile time.
constexpr int64_t kSmallSegment = int64_t(1) << 31;  // rows whose index fits best[]'s low word
constexpr int kSmallBT = 1024;   // rows of B per shared-memory stage
constexpr int kSmallSub = 32;    // rows per sub-tile: the unit the minima are tracked and evaluated in
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

// 64-bit words per staged row pair (even, for 16-byte reads)
template <int METRIC, int D>
constexpr int small_words() {
  const int w = METRIC == CH_L2 ? D + 1 : D;
  return w + (w & 1);
}

template <int METRIC, int D>
struct SmallShared {
  __align__(16) uint64_t rows[kSmallBT / 2 * small_words<METRIC, D>()];  // the stage of B
  float c[D];  // the block's first sample
  int wide;    // samples with three sub-tiles within the bound
};

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
//   l2: the value is L = |b'|^2 shrink - 2 q'.b' (d packed fused multiply-adds for two
//       rows, the norms staged with the rows) instead of the canonical 3 d - 1
//       operations per row, where q' = fl(q - c), b' = fl(b - c) and c is the block's
//       first sample: the bound below scales with |q'|^2, so it must not see how far
//       the cloud lies from the origin.  With u = 2^-24 and D = |q - b|:
//       each coordinate of q' and b' is off by at most u of itself, so D >= |q' - b'| -
//       u (|q'| + |b'|) and D^2 >= |q' - b'|^2 - 4.01 u (|q'|^2 + |b'|^2); the norm's
//       chain is within d u |b'|^2, the d fmas within 1.01 d u (|b'|^2 + 2 |q'||b'|) and
//       2 |q'||b'| <= |q'|^2 + |b'|^2.  With shrink = 1 - (4 d + 5) u every row then has
//       D^2 >= L + |q'|^2 (1 - (1.01 d + 4.01) u).  A row that ties with or beats a
//       canonical squared distance P (itself within 10 u, and equal square roots within
//       2^-22) therefore has
//         L <= P (1 + 2^-19) - |q'|^2 (1 - (2 d + 6) u) + 2^-100
//       (d u of it for |q'|^2's own chain).  The best sub-tile gives P; the second is
//       evaluated where it meets this.  Where the third does too (ties: lattices,
//       repeated points; or magnitudes out of the bound's range), every sub-tile may:
//       a few such samples of a block have their chunk's rows evaluated by a warp
//       each, a row per lane; from 1 / kSecondWalk of the block's samples on, a second
//       walk evaluates the sub-tiles that meet the bound.
// 512 pairs of d = 3 surfaces (2.1e10 distances), the whole batched call: 12.1 ms with
// the earlier scan of one row at a time, 6.48 ms.  256 such pairs 10, 30 and 1000 extents
// from the origin: 5.9 ms with the earlier scan; 6.8, 19.3 and 19.6 ms with raw
// coordinates in the bound; 3.2 ms each with the pivot (3.2 ms at the origin).  Lattice
// points, T = 5527 x 1M on 16^3 cells: 2.75, 6.6 and, with the second walk, 1.8 ms.
// In warp instructions a look over one sample's rows is about 0.5 a row, the second walk
// 8 x (5 PQ + 3) / 2 a row for a block: equal from about a quarter of the samples on.
constexpr int kSecondWalk = 4;

template <int METRIC, int D, int PQ>
__device__ __forceinline__ void small_item(int dtype, const void* __restrict__ A, const float* __restrict__ scA,
                                           int64_t nA, const int64_t* __restrict__ qidx, int64_t T,
                                           const void* __restrict__ B, const float* __restrict__ scB, int64_t b_begin,
                                           int64_t b_end, int64_t l0, unsigned long long* __restrict__ best,
                                           SmallShared<METRIC, D>& sh) {
  constexpr bool kL2 = METRIC == CH_L2;
  constexpr int W = small_words<METRIC, D>();
  const float kInf = __int_as_float(0x7F800000);
  const int lane = threadIdx.x & 31;
  const float u = 0x1p-24f;
  uint64_t* Bs = sh.rows;
  // sample l0 + 256 p; false where there is none to look for (past the end, no draw)
  auto load_q = [&](int p, float (&q)[D]) {
    const int64_t l = l0 + 256 * p;
    const int64_t a = l < T ? (qidx ? qidx[l] : l) : -1;
#pragma unroll
    for (int j = 0; j < D; ++j) q[j] = (a >= 0 && a < nA) ? elem_of(dtype, A, a, D, j, scA) : 0.0f;
    return a >= 0;
  };
  uint64_t q2[PQ][D];
  float b1[PQ], b2[PQ], b3[PQ];
  int i1[PQ], i2[PQ];
  float c[D];
#pragma unroll
  for (int j = 0; j < D; ++j) c[j] = 0.0f;
  if constexpr (kL2) {  // the block's first sample, by every thread (one address)
    const int64_t l = l0 - threadIdx.x;
    const int64_t a = qidx ? qidx[l] : l;
    if (a >= 0 && a < nA) {
#pragma unroll
      for (int j = 0; j < D; ++j) {
        c[j] = elem_of(dtype, A, a, D, j, scA);
        if (!(fabsf(c[j]) < kInf)) c[j] = 0.0f;
      }
    }
    if (threadIdx.x == 0) {  // read again from here on, past the barrier before the first stage
#pragma unroll
      for (int j = 0; j < D; ++j) sh.c[j] = c[j];
      sh.wide = 0;
    }
  }
#pragma unroll
  for (int p = 0; p < PQ; ++p) {
    float q[D];
    load_q(p, q);
#pragma unroll
    for (int j = 0; j < D; ++j) {
      const float t = kL2 ? -2.0f * __fsub_rn(q[j], c[j]) : q[j];
      q2[p][j] = f2_pack(t, t);
    }
  }
#pragma unroll
  for (int p = 0; p < PQ; ++p) {
    b1[p] = b2[p] = b3[p] = kInf;
    i1[p] = i2[p] = -1;
  }
  // the rows of sub-tile `sub`, one per lane (+inf past the end)
  auto row_of = [&](int sub, float (&b)[D]) {
    const int64_t r = b_begin + int64_t(sub) * kSmallSub + lane;
    const bool ok = sub >= 0 && r < b_end;
#pragma unroll
    for (int j = 0; j < D; ++j) b[j] = ok ? elem_of(dtype, B, r, D, j, scB) : kInf;
    return static_cast<uint32_t>(ok ? r : 0xFFFFFFFFll);
  };
  // the smallest distance of the warp's rows b (index r, one per lane) to a sample qs:
  // bits and, in at, its index
  auto least_of = [&](const float (&qs)[D], const float (&b)[D], uint32_t r, uint32_t& at, float& least_p) {
    const float v = small_canon<METRIC, D>(qs, b);
    const uint32_t bits = r != 0xFFFFFFFFu ? __float_as_uint(kL2 ? __fsqrt_rn(v) : v) : 0xFFFFFFFFu;
    const uint32_t least = __reduce_min_sync(0xFFFFFFFFu, bits);
    at = __reduce_min_sync(0xFFFFFFFFu, bits == least ? r : 0xFFFFFFFFu);
    if constexpr (kL2)
      least_p = __uint_as_float(__reduce_min_sync(0xFFFFFFFFu, r != 0xFFFFFFFFu ? __float_as_uint(v) : 0x7F800000u));
    return least;
  };
  auto post = [&](int p, uint32_t bits, uint32_t at) {
    const int64_t l = l0 + 256 * p;
    // +inf and NaN (bits from 0x7F800000 on) are no minimum, as for the other scans
    if (bits >= 0x7F800000u) {
      bits = 0x7F800000u;
      at = 0xFFFFFFFFu;
    }
    if (l < T) atomicMin(&best[l], (static_cast<unsigned long long>(bits) << 32) | at);
  };
#pragma unroll 1
  for (int walk = 0;; ++walk) {
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
            v[h][j] = ok ? elem_of(dtype, B, s0 + 2 * f + h, D, j, scB) : (kL2 ? sh.c[j] : kInf);
            if constexpr (kL2) {
              v[h][j] = __fsub_rn(v[h][j], sh.c[j]);
              if (ok) n[h] = __fmaf_rn(v[h][j], v[h][j], n[h]);
            }
          }
          if (kL2) n[h] = __fmul_rd(n[h], 1.0f - (4 * D + 5) * u);
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
        if (kL2 && walk) {
          // the second walk: b1 = the bound (-inf: nothing to look for), i1 = the sub-tile
          // from which on a point at distance 0 leaves nothing to find
#pragma unroll
          for (int p = 0; p < PQ; ++p) {
            unsigned hit = __ballot_sync(0xFFFFFFFFu, m[p] <= b1[p] && sub0 + sub < i1[p]);
            if (!hit) continue;
            float q[D], b[D];
            load_q(p, q);
            const uint32_t r = row_of(sub0 + sub, b);
            for (; hit; hit &= hit - 1) {
              const int s = __ffs(hit) - 1;
              float qs[D], least_p;
#pragma unroll
              for (int j = 0; j < D; ++j) qs[j] = __shfl_sync(0xFFFFFFFFu, q[j], s);
              uint32_t at;
              const uint32_t least = least_of(qs, b, r, at, least_p);
              if (lane == s) {
                post(p, least, at);
                if (least == 0u) i1[p] = sub0 + sub;
              }
            }
          }
          continue;
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
    if (walk) return;
    int wide = 0;  // this warp's samples whose third sub-tile meets the bound
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
      const bool some = load_q(p, q);
      uint32_t dmin = 0xFFFFFFFFu, imin = 0xFFFFFFFFu;  // this lane's sample: distance bits and index
      float P = kInf;
      // folds the warp's rows b (index r) into sample s
      auto fold = [&](int s, const float (&qs)[D], const float (&b)[D], uint32_t r) {
        uint32_t at;
        float least_p = 0.0f;
        const uint32_t least = least_of(qs, b, r, at, least_p);
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
        for (int j = 0; j < D; ++j) {
          const float t = __fsub_rn(q[j], sh.c[j]);
          qn = __fmaf_rn(t, t, qn);
        }
        const bool ranged = qn < 1e37f && P < 1e37f;
        const float thr = ranged ? __fadd_ru(__fsub_ru(__fmul_ru(P, 1.0f + 0x1p-19f),
                                                       __fmul_rd(qn, 1.0f - (2 * D + 6) * u)),
                                             0x1p-100f)
                                 : kInf;
        const bool far = some && t3 <= thr;
        for (unsigned rest = __ballot_sync(0xFFFFFFFFu, some && !far && t2 <= thr); rest; rest &= rest - 1) {
          const int s = __ffs(rest) - 1;
          float qs[D], b[D];
#pragma unroll
          for (int j = 0; j < D; ++j) qs[j] = __shfl_sync(0xFFFFFFFFu, q[j], s);
          const uint32_t r = row_of(__shfl_sync(0xFFFFFFFFu, e2, s), b);
          fold(s, qs, b, r);
        }
        wide += __popc(__ballot_sync(0xFFFFFFFFu, far));
        // what the wide samples' rows are looked over with (see the second walk)
        const int stop = dmin == 0u ? static_cast<int>((imin - b_begin) / kSmallSub) : INT_MAX;
#pragma unroll
        for (int k = 0; k < PQ; ++k)
          if (k == p) {
            b1[k] = far ? thr : -kInf;
            i1[k] = far ? stop : 0;
          }
      }
      post(p, dmin, imin);
    }
    if constexpr (!kL2) return;
    if (lane == 0 && wide) atomicAdd(&sh.wide, wide);
    __syncthreads();
    const int all_wide = sh.wide;
    if (all_wide == 0) return;
    if (all_wide >= 256 * PQ / kSecondWalk) continue;
#pragma unroll 1
    for (int p = 0; p < PQ; ++p) {
      int stop = 0;
#pragma unroll
      for (int k = 0; k < PQ; ++k)
        if (k == p) stop = l0 + 256 * k < T ? i1[k] : 0;
      unsigned rest = __ballot_sync(0xFFFFFFFFu, stop > 0);
      if (!rest) continue;
      float q[D];
      load_q(p, q);
      for (; rest; rest &= rest - 1) {
        const int s = __ffs(rest) - 1;
        const int64_t end = min(b_end, b_begin + int64_t(__shfl_sync(0xFFFFFFFFu, stop, s)) * kSmallSub);
        float qs[D];
#pragma unroll
        for (int j = 0; j < D; ++j) qs[j] = __shfl_sync(0xFFFFFFFFu, q[j], s);
        // a row per lane; equal square roots of unequal squares keep the smaller index
        float best_p = kInf, best_v = kInf;
        uint32_t best_r = 0xFFFFFFFFu;
#pragma unroll 4
        for (int64_t r = b_begin + lane; r < end; r += 32) {
          float b[D];
#pragma unroll
          for (int j = 0; j < D; ++j) b[j] = elem_of(dtype, B, r, D, j, scB);
          const float v = small_canon<METRIC, D>(qs, b);
          if (v < best_p) {
            best_p = v;
            const float root = __fsqrt_rn(v);
            if (root < best_v) {
              best_v = root;
              best_r = static_cast<uint32_t>(r);
            }
          }
        }
        const uint32_t least = __reduce_min_sync(0xFFFFFFFFu, __float_as_uint(best_v));
        const uint32_t at = __reduce_min_sync(0xFFFFFFFFu, __float_as_uint(best_v) == least ? best_r : 0xFFFFFFFFu);
        if (lane == s) post(p, least, at);
      }
    }
    return;
  }
}

// one pair: blockIdx.x = block of samples, blockIdx.y = chunk of B
template <int METRIC, int D, int PQ>
__global__ void __launch_bounds__(256, 3) k_scan_small(int dtype, const void* __restrict__ A,
                                                       const float* __restrict__ scA, const int64_t* __restrict__ qidx,
                                                       int64_t T, int64_t nA, const void* __restrict__ B,
                                                       const float* __restrict__ scB, int64_t nB, int64_t chunk_len,
                                                       unsigned long long* best) {
  pdl_entry();
  __shared__ SmallShared<METRIC, D> sh;
  const int64_t b_begin = int64_t(blockIdx.y) * chunk_len;
  small_item<METRIC, D, PQ>(dtype, A, scA, nA, qidx, T, B, scB, b_begin, min(nB, b_begin + chunk_len),
                                  int64_t(blockIdx.x) * (256 * PQ) + threadIdx.x, best, sh);
}

// The batched form: one persistent launch over items (pair, groups of 256 samples,
// chunk of B) of many pairs of one storage type, metric and dimension, largest
// first, each block taking the next one from a counter.
template <int METRIC, int D>
__global__ void __launch_bounds__(256, 2) k_scan_small_batch(int dtype, const SmallScanPair* __restrict__ pairs,
                                                             const SmallScanItem* __restrict__ items, int64_t n_items,
                                                             int64_t chunk_len, unsigned int* next) {
  pdl_entry();
  __shared__ SmallShared<METRIC, D> sh;
  __shared__ unsigned int s_w;
  for (;;) {
    __syncthreads();  // sh and s_w are free again
    if (threadIdx.x == 0) s_w = atomicAdd(next, 1u);
    __syncthreads();
    const int64_t w = s_w;
    if (w >= n_items) return;
    const SmallScanItem it = items[w];
    const SmallScanPair pr = pairs[it.pair];
    const int64_t l0 = int64_t(it.group) * 256 + threadIdx.x, b_end = min(pr.nB, it.b0 + chunk_len);
    const auto run = [&](auto pq) {
      small_item<METRIC, D, decltype(pq)::value>(dtype, pr.A, pr.scA, pr.nA, pr.qidx, pr.T, pr.B, pr.scB, it.b0, b_end,
                                                 l0, pr.best, sh);
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

}  // namespace

// Samples per thread and blocks of a lone scan.  More samples per thread share each read
// of a row; fewer, and fewer blocks, leave longer chunks to each sample, of which one
// 32-row sub-tile is evaluated whatever their length.  Measured at d = 3, T = 4606 (5527
// at 1M), us for 1, 2 and 4 samples at 4 blocks per SM (8 in brackets):
//            2k            20k                100k                 1M
//   l2   18  26  43    49  61  71    146 135 161 (141 145 196)  1511 1173 1104 (1368 1067 1016)
//   l1   16  20  28    43  49  55    136 135 155 (129 133 162)  1439 1312 1425 (1278 1199 1292)
// (the earlier scan of one row at a time: l2 67, 104, 356, 3302; l1 24, 65, 241, 2455).
static int small_pq(int64_t T, int64_t nB) { return double(T) * double(nB) < double(1 << 28) ? 1 : 2; }

int scan_small_chunks(int64_t T, int64_t nB, int sm_count) {
  const int64_t qblocks = ceil_div(std::max<int64_t>(T, 1), 256 * small_pq(T, nB));
  const int per_sm = double(T) * double(nB) < double(int64_t(1) << 31) ? 4 : 8;
  const int64_t chunks = std::min<int64_t>(ceil_div(int64_t(sm_count) * per_sm, qblocks), ceil_div(nB, 256));
  return static_cast<int>(std::max<int64_t>(chunks, 1));
}

int scan_small_segments(int64_t nB) { return static_cast<int>(std::max<int64_t>(1, ceil_div(nB, kSmallSegment))); }

template <int METRIC, int PQ>
static void scan_small(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, ScanPart part,
                       cudaStream_t s) {
  const int segs = scan_small_segments(B->n);
  CHX_CUDA(cudaMemsetAsync(part.best, 0xFF, size_t(segs) * T * sizeof(unsigned long long), s));
  for (int g = 0; g < segs; ++g) {
    const int64_t n0 = int64_t(g) * kSmallSegment, n = std::min(kSmallSegment, B->n - n0);
    const char* base = static_cast<const char*>(B->data) + size_t(n0) * A->d * elem_size(B->dtype);
    const float* sc = B->scales ? B->scales + n0 : nullptr;
    const int64_t chunk_len = ceil_div(n, part.chunks);
    const dim3 grid(static_cast<unsigned>(ceil_div(T, 256 * PQ)), static_cast<unsigned>(part.chunks));
    auto go = [&](auto kern) {
      launch_k(kern, grid, 256, 0, s, A->dtype, A->data, A->scales, qidx, T, A->n, base, sc, n, chunk_len,
               part.best + size_t(g) * T);
    };
    switch (A->d) {
      case 1: go(k_scan_small<METRIC, 1, PQ>); break;
      case 2: go(k_scan_small<METRIC, 2, PQ>); break;
      case 3: go(k_scan_small<METRIC, 3, PQ>); break;
      default: go(k_scan_small<METRIC, 4, PQ>); break;
    }
  }
}

void launch_scan_small(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, int metric, ScanPart part,
                       cudaStream_t s) {
  auto go = [&](auto pq) {
    constexpr int PQ = decltype(pq)::value;
    metric == CH_L1 ? scan_small<CH_L1, PQ>(A, qidx, T, B, part, s) : scan_small<CH_L2, PQ>(A, qidx, T, B, part, s);
  };
  if (small_pq(T, B->n) == 1) go(std::integral_constant<int, 1>{});
  else go(std::integral_constant<int, 2>{});
  launch_check("scan_small");
}

void launch_scan_small_out(ScanPart part, int64_t T, int64_t nB, const int64_t* qidx, float* min_d, int64_t* argmin,
                           cudaStream_t s) {
  launch_k(k_scan_best_out, static_cast<int>(ceil_div(T, 256)), 256, 0, s, part.best, scan_small_segments(nB), T, qidx,
           min_d, argmin);
  launch_check("scan_best_out");
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
  CHX_CHECK(d >= 1 && d <= kScanSmallMaxD, CH_EINVAL, "batched small scan: d must be in 1..4");
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
