// k_chain.cu -- the exact scan of d > 4 on CUDA cores (every l1 scan, and the l2 sets
// whose rows the tensor-core screen cannot read), in two steps.
//
// The canonical distance fixes a summation order (32 strided partials and a tree) that
// costs 31 extra additions a pair and, walked depth first, ties up registers, so that a
// thread could hold only 2 x 4 pairs and read shared memory 5 wavefronts per coordinate
// for them.  k_chain instead sums each pair in one chain, in whatever order the
// coordinates come: a thread holds PQ x 4 pairs with one register each, K is cut into
// slabs of 32 coordinates (any d, two slabs in flight), and only the smallest chain
// value of each four-row group is tracked, per sample and thread row.  A chain value S
// and the canonical value C of the same pair satisfy, for the exact distance D and
// u = 2^-24 (every term is non-negative, so relative errors add up plainly):
//   |S - D| <= (d + 3) u D,   |C - D| <= (d / 32 + 9) u D.
// So a row that ties with or beats a canonical C has S <= C (1 + 2 (d + d / 32 + 12) u
// + 2^-20) + 2^-100 (2^-20: square roots of nearby squares may round to one distance;
// 2^-100: underflow).  k_certify evaluates the canonical distance of every row that
// meets this -- a few per sample -- so minima and argmins are exact, bit for bit.
//
// Bound: FP32 issue, 2 pipe operations (l1: 1.5 issue slots, l2: 1) per pair and
// coordinate.  At T = 4.6k x 100k, d = 64 l1 with scalar subtractions: issue 85 %, FMA
// pipe 73 % busy, 2.12 ms; packed subtractions 2.0 ms; k_scan_exact 2.78 ms.
#include "common.cuh"

namespace chx {

namespace {

constexpr int kKS = 32;          // coordinates per slab
constexpr int kCBT = 128;        // rows of B per tile
constexpr int kCBS = kCBT + 4;   // tile strides = 4 mod 8 words: conflict-free transposed stores
constexpr int kChainSlice = 16384;  // samples per launch, which bounds the scratch
constexpr int kChainResident = 2;   // blocks per SM (register cap 128)

constexpr int PQ = 8;            // samples per thread
constexpr int QT = 8 * PQ;       // samples per block
constexpr int QS = QT + 4;
constexpr int kSmem = 2 * kKS * (QS + kCBS) * 4;

// Thread (tq, tb) = (tid % 8, tid / 8) owns samples 4 tq .. + 3 and 32 + 4 tq .. + 3 of
// the block's 64 (a warp then reads whole 128-byte rows of them) and rows 4 tb .. + 3 of
// every 128-row tile of its chunk.
template <int DT, int METRIC>
__global__ void __launch_bounds__(256, kChainResident)
    k_chain(const void* __restrict__ A, const float* __restrict__ scA, const int64_t* __restrict__ qidx, int64_t l0,
            int64_t T, int64_t nA, const void* __restrict__ B, const float* __restrict__ scB, int64_t nB, int d,
            int64_t chunk_len, float* __restrict__ part_s, int32_t* __restrict__ part_i, float* __restrict__ part_2) {
  pdl_entry();
  extern __shared__ __align__(16) float smem[];
  __shared__ int64_t s_a[QT];
  const int tid = threadIdx.x, tq = tid & 7, tb = tid >> 3;
  const int warp = tid >> 5, rl = tid & 3, jl = (tid & 31) >> 2;
  const int64_t q0 = int64_t(blockIdx.x) * QT;
  const int64_t b_begin = int64_t(blockIdx.y) * chunk_len;
  const int64_t b_end = min(nB, b_begin + chunk_len);
  const int nslab = (d + kKS - 1) / kKS;
  const int ntile = static_cast<int>((b_end - b_begin + kCBT - 1) / kCBT);
  if (tid < QT) {
    const int64_t l = q0 + tid;
    int64_t a = l < T ? (qidx ? qidx[l0 + l] : l0 + l) : -1;
    s_a[tid] = a < nA ? a : -1;
  }
  __syncthreads();
  // slab s of tile `tile` into buffer buf, transposed: lanes (rl, jl) take 4 rows x 8
  // coordinates per instruction; rows past the end become zeros, coordinates past d are
  // not read by the sums.  Binary32 goes by asynchronous 4-byte copies; the narrow types
  // are widened on the way, every load of the slab (from clamped places, so that none
  // waits on a branch) issued before the first store.
  constexpr int kQG = (QT / 4 + 7) / 8, kBG = kCBT / 32;  // row groups per warp
  auto stage = [&](int tile, int s, int buf) {
    float* Qs = smem + buf * kKS * (QS + kCBS);
    float* Bs = Qs + kKS * QS;
    const int64_t r0 = b_begin + int64_t(tile) * kCBT;
    int64_t row[kQG + kBG];
#pragma unroll
    for (int g = 0; g < kQG; ++g) {
      const int r = 4 * (warp + 8 * g) + rl;
      row[g] = r < QT ? s_a[r] : -1;
    }
#pragma unroll
    for (int g = 0; g < kBG; ++g) {
      const int64_t r = r0 + 4 * (warp + 8 * g) + rl;
      row[kQG + g] = r < b_end ? r : -1;
    }
    auto to = [&](int g, int k) {
      const int c = jl + 8 * k;
      return g < kQG ? Qs + c * QS + 4 * (warp + 8 * g) + rl : Bs + c * kCBS + 4 * (warp + 8 * (g - kQG)) + rl;
    };
    auto wanted = [&](int g, int k) {
      return s * kKS + jl + 8 * k < d && (g >= kQG || 4 * (warp + 8 * g) + rl < QT);
    };
    if constexpr (DT == CH_F32) {
#pragma unroll
      for (int g = 0; g < kQG + kBG; ++g)
#pragma unroll
        for (int k = 0; k < kKS / 8; ++k) {
          if (!wanted(g, k)) continue;
          const float* src = static_cast<const float*>(g < kQG ? A : B) + (row[g] >= 0 ? row[g] : 0) * int64_t(d) +
                             s * kKS + jl + 8 * k;
          asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                           static_cast<uint32_t>(__cvta_generic_to_shared(to(g, k)))),
                       "l"(src), "r"(row[g] >= 0 ? 4u : 0u)
                       : "memory");
        }
      asm volatile("cp.async.commit_group;" ::: "memory");
    } else {
      float v[kQG + kBG][kKS / 8];
#pragma unroll
      for (int g = 0; g < kQG + kBG; ++g)
#pragma unroll
        for (int k = 0; k < kKS / 8; ++k) {
          const int j = min(s * kKS + jl + 8 * k, d - 1);
          // a row past the end reads the chunk's first row of B, which exists
          v[g][k] = g < kQG && row[g] >= 0 ? load_elem<DT>(A, row[g], d, j, scA)
                                           : load_elem<DT>(B, row[g] >= 0 ? row[g] : b_begin, d, j, scB);
        }
#pragma unroll
      for (int g = 0; g < kQG + kBG; ++g)
#pragma unroll
        for (int k = 0; k < kKS / 8; ++k)
          if (wanted(g, k)) *to(g, k) = row[g] >= 0 ? v[g][k] : 0.0f;
    }
  };
  const float kInf = __int_as_float(0x7F800000);
  float acc[4][PQ], b1[PQ], b2[PQ];
  int i1[PQ];
#pragma unroll
  for (int p = 0; p < PQ; ++p) {
    b1[p] = b2[p] = kInf;
    i1[p] = -1;
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[b][p] = 0.0f;
  }
  int buf = 0;
  if (ntile > 0) stage(0, 0, 0);
  for (int tile = 0; tile < ntile; ++tile) {
    for (int s = 0; s < nslab; ++s, buf ^= 1) {
      const int nt = s + 1 < nslab ? tile : tile + 1, ns = s + 1 < nslab ? s + 1 : 0;
      __syncthreads();  // the other buffer's readers are done
      if (nt < ntile) {
        stage(nt, ns, buf ^ 1);
        asm volatile("cp.async.wait_group 1;" ::: "memory");
      } else {
        asm volatile("cp.async.wait_group 0;" ::: "memory");
      }
      __syncthreads();
      const float* Qs = smem + buf * kKS * (QS + kCBS);
      const float* Bs = Qs + kKS * QS + tb * 4;
      auto coord = [&](int k) {
        float q[PQ];
#pragma unroll
        for (int h = 0; h < PQ / 4; ++h) {
          const float4 t = *reinterpret_cast<const float4*>(Qs + k * QS + 32 * h + 4 * tq);
          q[4 * h] = t.x;
          q[4 * h + 1] = t.y;
          q[4 * h + 2] = t.z;
          q[4 * h + 3] = t.w;
        }
        const float4 t = *reinterpret_cast<const float4*>(Bs + k * kCBS);
        const float bv[4] = {t.x, t.y, t.z, t.w};
        // two samples per packed subtraction (b * -1 + q rounds like q - b); l1's |t| is a
        // modifier of the scalar addition, which packed ones lack
        constexpr uint64_t kNeg = 0xBF800000BF800000ull;  // (-1, -1)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          const uint64_t b2 = f2_pack(bv[b], bv[b]);
#pragma unroll
          for (int p = 0; p < PQ; p += 2) {
            uint64_t v = f2_pack(q[p], q[p + 1]);
            f2_fma(v, b2, kNeg);
            if constexpr (METRIC == CH_L1) {
              const float2 t = f2_unpack(v);
              acc[b][p] = __fadd_rn(acc[b][p], fabsf(t.x));
              acc[b][p + 1] = __fadd_rn(acc[b][p + 1], fabsf(t.y));
            } else {
              uint64_t a = f2_pack(acc[b][p], acc[b][p + 1]);
              f2_fma(a, v, v);
              const float2 t = f2_unpack(a);
              acc[b][p] = t.x;
              acc[b][p + 1] = t.y;
            }
          }
        }
      };
      const int kn = min(kKS, d - s * kKS);
      if (kn == kKS) {
#pragma unroll 8
        for (int k = 0; k < kKS; ++k) coord(k);
      } else {
#pragma unroll 2
        for (int k = 0; k < kn; ++k) coord(k);
      }
    }
    // this thread's four rows of the tile, folded into its samples' minima
    const int64_t left = b_end - b_begin - int64_t(tile) * kCBT - 4 * tb;
#pragma unroll
    for (int p = 0; p < PQ; ++p) {
      if (left < 4) {
#pragma unroll
        for (int b = 0; b < 4; ++b)
          if (b >= left) acc[b][p] = kInf;
      }
      const float v = fminf(fmin3(acc[0][p], acc[1][p], acc[2][p]), acc[3][p]);
      b2[p] = fminf(b2[p], fmaxf(b1[p], v));
      i1[p] = v < b1[p] ? tile : i1[p];
      b1[p] = fminf(b1[p], v);
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[b][p] = 0.0f;
    }
  }
#pragma unroll
  for (int p = 0; p < PQ; ++p) {
    const int64_t l = q0 + 32 * (p / 4) + 4 * tq + p % 4;
    if (l < T) {
      const size_t at = (size_t(blockIdx.y) * T + l) * 32 + tb;
      part_s[at] = b1[p];
      part_i[at] = i1[p] < 0 ? -1 : static_cast<int32_t>(b_begin + int64_t(i1[p]) * kCBT + 4 * tb);
      part_2[at] = b2[p];
    }
  }
}

struct ChainPlan {
  int chunks;
  int64_t chunk_len;
};

// chunks of B: the count that minimises waves x tiles per block (ties: fewer)
ChainPlan chain_plan(int64_t T, int64_t nB, int sm_count) {
  ChainPlan p;
  const int64_t qtiles = ceil_div(T, QT), resident = int64_t(sm_count) * kChainResident;
  const int64_t btiles = ceil_div(nB, kCBT), most = std::max<int64_t>(1, std::min<int64_t>(ceil_div(btiles, 4), 64));
  int64_t best = 1, best_cost = INT64_MAX;
  for (int64_t c = 1; c <= most; ++c) {
    const int64_t cost = ceil_div(qtiles * c, resident) * (ceil_div(btiles, c) + 1);
    if (cost < best_cost) {
      best_cost = cost;
      best = c;
    }
    if (qtiles * c >= 8 * resident) break;
  }
  p.chunk_len = ceil_div(btiles, best) * kCBT;
  p.chunks = static_cast<int>(ceil_div(nB, p.chunk_len));
  return p;
}

template <int DT, int METRIC>
void chain_launch(const ch_set* A, const int64_t* qidx, int64_t l0, int64_t n, const ch_set* B, const ChainPlan& p,
                  const CertArgs& c, cudaStream_t s) {
  auto kern = k_chain<DT, METRIC>;
  CHX_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem));
  const dim3 grid(static_cast<unsigned>(ceil_div(n, QT)), static_cast<unsigned>(p.chunks));
  launch_k(kern, grid, 256, kSmem, s, A->data, A->scales, qidx, l0, n, A->n, B->data, B->scales, B->n, A->d, p.chunk_len,
           const_cast<float*>(c.part_s), const_cast<int32_t*>(c.part_i), const_cast<float*>(c.part_2));
}

}  // namespace

// From 512 samples (64-sample blocks) and 2^29 (sample, point, coordinate) terms on;
// k_scan_exact is one launch and fills the SMs with less (l1, k_scan_exact / chained:
// T = 2000 x 4000, d = 64, 2^28.9: 63.6 / 63.7 us; T = 128 x 20k, d = 64: 45 / 64 us;
// T = 64 x 50k, d = 128: 82 / 111 us; T = 4.6k x 100k, d = 64: 2.90 / 2.0 ms; T = 3k x
// 20k, d = 300 bf16: 2.47 / 1.46 ms).  A sample with hundreds of rows at one distance
// other than 0 is listed and pays for both (T = 4.6k x 100k, every row of B the same: d =
// 8 0.73 / 1.29 ms, d = 64 2.90 / 5.15 ms); small whole coordinates do not come to that
// (in [0, 4) or [0, 16): 0.53 ms at d = 8), nor does B a hundred times over (0.54 ms).
bool exact_chain_pays(const ch_set* A, const ch_set* B, int64_t T) {
  return A->d > 4 && A->dtype == B->dtype && T >= 512 && B->n < (int64_t(1) << 31) && scan_list_fits(T, A->d) &&
         double(T) * double(B->n) * A->d >= double(1 << 29);
}

size_t exact_chain_workspace(int64_t T, int64_t nB, int sm_count) {
  size_t parts = 0;
  for (int64_t t : {std::min<int64_t>(T, kChainSlice), T % kChainSlice})
    if (t > 0) parts = std::max(parts, size_t(chain_plan(t, nB, sm_count).chunks) * t * 32);
  return 3 * ((parts * 4 + 255) & ~size_t(255)) + ((size_t(T) * 4 + 255) & ~size_t(255)) +
         ((size_t(T) * 8 + 255) & ~size_t(255)) + 1024;
}

void launch_exact_chain(const ch_set* A, const int64_t* qidx, int64_t T, const ch_set* B, int metric, void* work,
                        float* min_d, int64_t* argmin, int sm_count, cudaStream_t s) {
  if (T == 0) return;
  const int d = A->d;
  auto al = [](size_t b) { return (b + 255) & ~size_t(255); };
  char* w = static_cast<char*>(work);
  CertArgs c;
  c.ctl = reinterpret_cast<uint32_t*>(w);
  w += 256;
  c.list = reinterpret_cast<int32_t*>(w);
  w += al(size_t(T) * 4);
  c.best = reinterpret_cast<unsigned long long*>(w);
  w += al(size_t(T) * 8);
  CHX_CUDA(cudaMemsetAsync(c.ctl, 0, 12, s));
  c.d = d;
  c.nB = B->n;
  c.p_scale = 1.0 + 0x1p-20 + 2.0 * (d + d / 32 + 12) * 0x1p-24;
  c.q_scale = 0.0;  // S is the distance itself, with no share of |q|^2
  c.limit = std::min<int64_t>(2048, std::max<int64_t>(256, B->n / 8));
  c.slices = 1;
  c.slice_cols = 0;
  c.tile = kCBT;
  c.class_cols = 4;
  c.occ_cols = 1;
  for (int64_t l0 = 0; l0 < T; l0 += kChainSlice) {
    const int64_t n = std::min<int64_t>(kChainSlice, T - l0);
    const ChainPlan p = chain_plan(n, B->n, sm_count);
    const size_t parts = size_t(p.chunks) * n * 32;
    c.l0 = l0;
    c.T = n;
    c.parts = p.chunks;
    c.chunk_len = p.chunk_len;
    c.part_s = reinterpret_cast<float*>(w);
    c.part_i = reinterpret_cast<int32_t*>(w + al(parts * 4));
    c.part_2 = reinterpret_cast<float*>(w + 2 * al(parts * 4));
    auto go = [&](auto dt) {
      constexpr int DT = decltype(dt)::value;
      metric == CH_L1 ? chain_launch<DT, CH_L1>(A, qidx, l0, n, B, p, c, s)
                      : chain_launch<DT, CH_L2>(A, qidx, l0, n, B, p, c, s);
    };
    if (A->dtype == CH_F32) go(std::integral_constant<int, CH_F32>{});
    else if (A->dtype == CH_BF16) go(std::integral_constant<int, CH_BF16>{});
    else go(std::integral_constant<int, CH_FP8E4M3>{});
    launch_check("chain");
    launch_certify(A, qidx, B, metric, c, min_d, argmin, s);
  }
  launch_scan_list(A, qidx, T, B, metric, c.list, c.ctl, c.best, min_d, argmin, sm_count, s);
}

}  // namespace chx
