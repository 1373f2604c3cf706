// k_sort.cu -- CrudeNN grouping by a device radix sort (CH_GROUP_SORT, SimHash and
// the k x W variant).
//
// B's entries of every scale, (high 32 bits of the key, index) words in index order,
// go through a stable LSD radix sort by those 32 bits (4 passes of 8 bits, every
// scale a segment of its own).  A bucket is then a run of equal prefixes in
// increasing index; two keys that share a prefix lie in one run, so a reader
// compares the whole key of each entry.  A itself is not sorted: a warp per point of
// A finds its runs by binary search, a scale per lane, and reads them off in scale
// order (Fig. 2, step 3: the first b is the first entry of the first run that holds
// the point's key).  Same b(a) as the bucket tables, by definition.
//
// Sorting B alone by 32 bits moves 4 x 16 bytes per (point of B, scale); sorting A and
// B by the full key and scale moved 9 x 24 bytes per (point, scale) and needed run
// heads and positions besides.  50k x 50k, d = 128, ten scales, four structures of window
// 16, the whole call: 3.22 -> 0.98 ms.
#include "common.cuh"

namespace chx {

namespace {

constexpr int kST = 256;               // threads per sort block
constexpr int kSWarps = kST / 32;
constexpr int kSPer = 16;              // entries per thread: a warp ranks 512 consecutive ones
constexpr int kSTile = kST * kSPer;    // 4096 entries per tile
constexpr int kIdxBits = 26;           // point indices (sort_group_supported)

// entry i of scale l before the first pass (prefix from the key), or as sorted so far
__device__ __forceinline__ uint64_t sort_entry(const uint64_t* keysB, const uint64_t* in, int64_t i) {
  return in ? in[i] : (keysB[i] & 0xFFFFFFFF00000000ull) | static_cast<uint32_t>(i);
}

// per-tile digit counts, hist[l][digit][tile] (blockIdx = (tile, scale))
__global__ void __launch_bounds__(kST) k_sort_hist(const uint64_t* keysB, const uint64_t* in, int64_t n, int shift,
                                                   uint32_t* hist) {
  pdl_entry();
  __shared__ uint32_t h[256];
  h[threadIdx.x] = 0;
  __syncthreads();
  const int64_t l = blockIdx.y;
  const int64_t base = int64_t(blockIdx.x) * kSTile + threadIdx.x;
  uint64_t e[kSPer];
#pragma unroll
  for (int r = 0; r < kSPer; ++r) {
    const int64_t i = base + r * kST;
    e[r] = i < n ? (in ? in[l * n + i] : keysB[l * n + i]) : 0;
  }
#pragma unroll
  for (int r = 0; r < kSPer; ++r) {
    const bool ok = base + r * kST < n;
    const uint32_t dg = ok ? static_cast<uint32_t>(e[r] >> shift) & 0xFFu : 256u;
    // equal digits of a warp count once (coarse scales hold a handful of keys)
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, dg);
    if (ok && (threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(&h[dg], __popc(peers));
  }
  __syncthreads();
  hist[(l * 256 + threadIdx.x) * gridDim.x + blockIdx.x] = h[threadIdx.x];
}

// exclusive scan of each scale's digit-major counts (a block per scale)
__global__ void __launch_bounds__(1024) k_sort_scan(uint32_t* hist, int64_t M) {
  pdl_entry();
  __shared__ uint32_t s_warp[32];
  uint32_t* h = hist + blockIdx.x * M;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t carry = 0;
  for (int64_t c0 = 0; c0 < M; c0 += 4096) {
    const int64_t i = c0 + 4 * threadIdx.x;
    uint32_t v[4], run = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[k] = i + k < M ? h[i + k] : 0u;
      run += v[k];
    }
    uint32_t x = run;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, x, o);
      if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[warp] = x;
    __syncthreads();
    uint32_t w = s_warp[lane];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, w, o);
      if (lane >= o) w += y;
    }
    const uint32_t before = __shfl_sync(0xFFFFFFFFu, w, (warp + 31) & 31);
    uint32_t at = carry + (warp ? before : 0u) + x - run;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (i + k < M) h[i + k] = at;
      at += v[k];
    }
    carry += __shfl_sync(0xFFFFFFFFu, w, 31);
    __syncthreads();  // s_warp is rewritten
  }
}

// Stable scatter of a tile: each warp ranks its 512 consecutive entries in order
// against its own digit counts (no block barriers), one prefix over the warps per
// digit, then every entry's place is offset + warps before + rank.
__global__ void __launch_bounds__(kST) k_sort_scatter(const uint64_t* keysB, const uint64_t* in, uint64_t* out,
                                                      int64_t n, int shift, const uint32_t* hist) {
  pdl_entry();
  __shared__ uint32_t wc[kSWarps][256];
  const int64_t l = blockIdx.y;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  for (int k = tid; k < kSWarps * 256; k += kST) (&wc[0][0])[k] = 0;
  const int64_t base = int64_t(blockIdx.x) * kSTile + warp * (32 * kSPer) + lane;
  const uint64_t* src = in ? in + l * n : nullptr;
  const uint64_t* keys = keysB + l * n;
  uint64_t e[kSPer];
#pragma unroll
  for (int r = 0; r < kSPer; ++r) e[r] = base + 32 * r < n ? sort_entry(keys, src, base + 32 * r) : 0;
  const uint32_t off = hist[(l * 256 + tid) * gridDim.x + blockIdx.x];
  __syncthreads();
  uint32_t rank[kSPer];
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int r = 0; r < kSPer; ++r) {
    const bool ok = base + 32 * r < n;
    const uint32_t dg = ok ? static_cast<uint32_t>(e[r] >> shift) & 0xFFu : 256u;
    const unsigned peers = __match_any_sync(0xFFFFFFFFu, dg);
    const int lead = __ffs(peers) - 1;
    uint32_t seen = 0;
    if (ok && lane == lead) {
      seen = wc[warp][dg];
      wc[warp][dg] = seen + __popc(peers);
    }
    rank[r] = __shfl_sync(0xFFFFFFFFu, seen, lead) + __popc(peers & lt);
    __syncwarp();
  }
  __syncthreads();
  uint32_t at = off;  // digit tid: its offset, then the entries of each warp before
#pragma unroll
  for (int w = 0; w < kSWarps; ++w) {
    const uint32_t c = wc[w][tid];
    wc[w][tid] = at;
    at += c;
  }
  __syncthreads();
  uint64_t* dst = out + l * n;
#pragma unroll
  for (int r = 0; r < kSPer; ++r)
    if (base + 32 * r < n) dst[wc[warp][static_cast<uint32_t>(e[r] >> shift) & 0xFFu] + rank[r]] = e[r];
}

// A warp per point of A.  Lane l < L finds scale l's run (first entry whose prefix is
// at least the key's); then the scales in increasing order: 32 entries of the run at
// a time, those of a's own key that no finer scale gave, in index order, until W are
// taken.  A point that finds nothing takes B[0] at level L.
// Outputs: cand[a * stride + r W ..] (null: none), bidx[a] = the first taken point
// (null: none), level[a] = the finest scale any structure so far found a point at
// (set by r = 0).
__global__ void __launch_bounds__(256) k_window(const uint64_t* keysA, int64_t nA, const uint64_t* keysB,
                                                const uint64_t* ent, int64_t nB, int L, int W, int r, int stride,
                                                int32_t* cand, int64_t* bidx, uint8_t* level) {
  pdl_entry();
  __shared__ int32_t s_taken[8][kWindowMax];
  const int64_t a = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  int32_t* taken = s_taken[threadIdx.x >> 5];  // the points taken so far
  if (a >= nA) return;
  uint64_t key = 0;
  int64_t lo = 0;
  if (lane < L) {
    key = keysA[lane * nA + a];
    const uint64_t want = key & 0xFFFFFFFF00000000ull;
    const uint64_t* e = ent + lane * nB;
    int64_t hi = nB;
    while (lo < hi) {
      const int64_t m = (lo + hi) >> 1;
      if (__ldg(&e[m]) < want) lo = m + 1;
      else hi = m;
    }
  }
  int cnt = 0, first = L;
  for (int l = 0; l < L && cnt < W; ++l) {
    const uint64_t k = __shfl_sync(0xFFFFFFFFu, key, l);
    const int64_t at = __shfl_sync(0xFFFFFFFFu, lo, l);
    const uint64_t* e = ent + l * nB;
    for (int64_t j0 = at; j0 < nB && cnt < W; j0 += 32) {
      const uint64_t v = j0 + lane < nB ? __ldg(&e[j0 + lane]) : ~k;
      const bool run = (v >> 32) == (k >> 32);
      const int32_t b = static_cast<int32_t>(v & ((1u << kIdxBits) - 1u));
      bool take = run && __ldg(&keysB[l * nB + b]) == k;
      for (int q = 0; q < cnt; ++q) take = take && taken[q] != b;
      const unsigned m = __ballot_sync(0xFFFFFFFFu, take);
      const int got = min(__popc(m), W - cnt);
      if (got) first = min(first, l);
      const int place = cnt + __popc(m & ((1u << lane) - 1u));
      if (take && place < W) taken[place] = b;
      __syncwarp();
      cnt += got;
      if (!__all_sync(0xFFFFFFFFu, run)) break;  // the run ends here
    }
  }
  if (cnt == 0) {
    if (lane == 0) taken[0] = 0;
    cnt = 1;
    __syncwarp();
  }
  if (cand) {
    int32_t* out = cand + a * stride + int64_t(r) * W;
    for (int q = lane; q < W; q += 32) out[q] = q < cnt ? taken[q] : -1;
  }
  if (lane == 0) {
    if (bidx) bidx[a] = taken[0];
    if (r == 0 || first < level[a]) level[a] = static_cast<uint8_t>(first);
  }
}

struct SortWork {
  uint64_t *e0, *e1;
  uint32_t* hist;
  int tiles;
};

SortWork carve_sort(void* work, int64_t nB, int L) {
  SortWork w;
  w.tiles = static_cast<int>(ceil_div(nB, kSTile));
  char* p = static_cast<char*>(work);
  auto take = [&](size_t bytes) {
    char* q = p;
    p += (bytes + 255) & ~size_t(255);
    return q;
  };
  w.e0 = reinterpret_cast<uint64_t*>(take(size_t(nB) * L * 8));
  w.e1 = reinterpret_cast<uint64_t*>(take(size_t(nB) * L * 8));
  w.hist = reinterpret_cast<uint32_t*>(take(size_t(256) * w.tiles * L * 4));
  return w;
}

}  // namespace

size_t sort_group_workspace(int64_t nB, int L) {
  return size_t(nB) * L * 16 + size_t(256) * ceil_div(nB, kSTile) * L * 4 + 4 * 256;
}

bool sort_group_supported(int64_t nA, int64_t nB, int L) {
  return nA < (int64_t(1) << kIdxBits) && nB < (int64_t(1) << kIdxBits) && L <= 32 &&
         (nA + nB) * L < (int64_t(1) << 31);
}

// B's entries of every scale sorted by (prefix, index): [L][nB]
static const uint64_t* sort_entries(const uint64_t* keysB, int64_t nB, int L, const SortWork& w, cudaStream_t s) {
  const dim3 grid(static_cast<unsigned>(w.tiles), static_cast<unsigned>(L));
  const uint64_t* in = nullptr;  // the first pass reads the keys
  uint64_t* out = w.e0;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 32 + 8 * pass;
    launch_k(k_sort_hist, grid, kST, 0, s, keysB, in, nB, shift, w.hist);
    launch_check("sort_hist");
    launch_k(k_sort_scan, L, 1024, 0, s, w.hist, int64_t(256) * w.tiles);
    launch_check("sort_scan");
    launch_k(k_sort_scatter, grid, kST, 0, s, keysB, in, out, nB, shift, w.hist);
    launch_check("sort_scatter");
    in = out;
    out = out == w.e0 ? w.e1 : w.e0;
  }
  return in;
}

void launch_sort_group(const uint64_t* keysA, int64_t nA, const uint64_t* keysB, int64_t nB, int L, void* work,
                       int64_t* bidx, uint8_t* level, cudaStream_t s) {
  if (nA == 0) return;
  const uint64_t* ent = sort_entries(keysB, nB, L, carve_sort(work, nB, L), s);
  launch_k(k_window, static_cast<int>(ceil_div(nA, 8)), 256, 0, s, keysA, nA, keysB, ent, nB, L, 1, 0, 0,
           static_cast<int32_t*>(nullptr), bidx, level);
  launch_check("window");
}

void launch_sort_window(const uint64_t* keysA, int64_t nA, const uint64_t* keysB, int64_t nB, int L, int W, int r,
                        void* work, int32_t* cand, int stride, uint8_t* level, cudaStream_t s) {
  if (nA == 0) return;
  CHX_CHECK(W >= 1 && W <= kWindowMax, CH_EINVAL, "window must be in 1..64");
  const uint64_t* ent = sort_entries(keysB, nB, L, carve_sort(work, nB, L), s);
  launch_k(k_window, static_cast<int>(ceil_div(nA, 8)), 256, 0, s, keysA, nA, keysB, ent, nB, L, W, r, stride, cand,
           static_cast<int64_t*>(nullptr), level);
  launch_check("window");
}

}  // namespace chx
