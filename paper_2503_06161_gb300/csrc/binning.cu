// Integer stage of the pass: the tile-based binning of 3DGS that the paper
// builds on (Sec. 2.1), reorganised for one GPU:
//   1. stable LSD radix sort of the P depth keys (4 x 8-bit passes, in one
//      launch for few keys);
//   2. exclusive scan of tiles_touched in depth order (decoupled look-back)
//      and, per block of depth-ordered Gaussians, its count of entries per
//      tile (a tile-major (tile, block) table);
//   3. exclusive scan of that table: the start of every (tile, block)
//      segment of the final list, and the tile ranges;
//   4. a scatter in which a block marks, per tile, which of its Gaussians
//      touch it (bit masks); an entry's place is its segment's start plus the
//      number of earlier Gaussians in the tile's mask, so the entries are
//      taken in any order.
// The result is the order of a stable sort on (tile << 32 | depth bits) with
// ties by index, built with one write per entry instead of radix passes over
// 64-bit keys.  Every inter-block wait is a bounded spin that records
// kErrTimeout and carries on, so no launch can hang.
#include <atomic>

#include "common.cuh"
#include "kernels.h"

namespace fe {

namespace {

constexpr uint32_t kFlagAgg = 1u << 30, kFlagPre = 2u << 30, kValMask = (1u << 30) - 1;
constexpr uint64_t kFlagAgg64 = 1ull << 62, kFlagPre64 = 2ull << 62, kValMask64 = (1ull << 62) - 1;
constexpr int kSpinLimit = 1 << 22;

__device__ __forceinline__ uint32_t ld_vol(const uint32_t* p) { return *reinterpret_cast<const volatile uint32_t*>(p); }
__device__ __forceinline__ void st_vol(uint32_t* p, uint32_t v) { *reinterpret_cast<volatile uint32_t*>(p) = v; }
__device__ __forceinline__ uint64_t ld_vol64(const uint64_t* p) { return *reinterpret_cast<const volatile uint64_t*>(p); }
__device__ __forceinline__ void st_vol64(uint64_t* p, uint64_t v) { *reinterpret_cast<volatile uint64_t*>(p) = v; }

__device__ __forceinline__ uint32_t lanemask_lt() {
  uint32_t m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// Exclusive scan of one value per thread over a 256-thread block.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t x, uint32_t* s_warp, uint32_t& total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_warp[warp] = incl;
  __syncthreads();
  uint32_t wpre = 0, tot = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    const uint32_t v = s_warp[w];
    if (w < warp) wpre += v;
    tot += v;
  }
  __syncthreads();
  total = tot;
  return wpre + incl - x;
}

// ---------------------------------------------------------------------------
// Global digit histograms of the depth keys (all four passes at once).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kThreads) depth_hist_kernel(const uint32_t* keys, int n, uint32_t* hist) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ uint32_t s[4][256];
  for (int i = threadIdx.x; i < 4 * 256; i += kThreads) (&s[0][0])[i] = 0;
  __syncthreads();
  const int start = blockIdx.x * kPChunk;
  const int end = min(n, start + kPChunk);
  for (int i = start + threadIdx.x; i < end; i += kThreads) {
    const uint32_t k = keys[i];
#pragma unroll
    for (int p = 0; p < 4; ++p) atomicAdd(&s[p][(k >> (8 * p)) & 255], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 4 * 256; i += kThreads) {
    const uint32_t v = (&s[0][0])[i];
    if (v) atomicAdd(hist + i, v);
  }
}

// ---------------------------------------------------------------------------
// One stable LSD radix pass (8-bit digit at `shift`) with decoupled look-back.
// Block b (taken from an atomic ticket so predecessors are always running)
// handles elements [256 ITEMS b, 256 ITEMS (b + 1)); warp w 32 ITEMS of them.
// ---------------------------------------------------------------------------
template <int ITEMS>
struct PassSmem {
  uint32_t wcnt[8][256];
  uint32_t gbase[256];
  uint32_t bstart[256];
  uint32_t keys[kThreads * ITEMS];
  uint32_t vals[kThreads * ITEMS];
  uint32_t scan[8];
  uint32_t ticket;
};

template <bool kIdentVals, int ITEMS>
__global__ void __launch_bounds__(kThreads) onesweep_kernel(const uint32_t* keys_in, const uint32_t* vals_in,
                                                            uint32_t* keys_out, uint32_t* vals_out,
                                                            int64_t n_elems, int shift,
                                                            const uint32_t* hist, uint32_t* status,
                                                            uint32_t* ticket, uint32_t* err) {
  constexpr int CHUNK = kThreads * ITEMS;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PassSmem<ITEMS>& sm = *reinterpret_cast<PassSmem<ITEMS>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // Before the wait for the previous pass: the counters' zeros and the
  // ticket (its counter is cleared ahead of the whole chain of launches).
  for (int i = tid; i < 8 * 256; i += kThreads) (&sm.wcnt[0][0])[i] = 0;
  if (tid == 0) sm.ticket = atomicAdd(ticket, 1u);
  __syncthreads();
  grid_dep_wait();
  grid_dep_launch();
  const uint32_t b = sm.ticket;
  const uint64_t n = (uint64_t)n_elems;
  const uint64_t start = (uint64_t)b * CHUNK;
  if (start >= n) return;
  const uint32_t cnt = (uint32_t)min((uint64_t)CHUNK, n - start);

  uint32_t k[ITEMS], v[ITEMS], rk[ITEMS];
  int dg[ITEMS];
  const uint64_t wbase = start + (uint64_t)warp * (CHUNK / 8);
  // All loads in flight before the first key is ranked.
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const uint64_t idx = wbase + (uint64_t)r * 32 + lane;
    k[r] = idx < n ? keys_in[idx] : 0u;
    v[r] = idx < n ? (kIdentVals ? (uint32_t)idx : vals_in[idx]) : 0u;
  }
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    const uint64_t idx = wbase + (uint64_t)r * 32 + lane;
    const bool valid = idx < n;
    const uint32_t key = k[r];
    const int d = valid ? (int)((key >> shift) & 255u) : 256;
    const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
    const int lead = __ffs(peers) - 1;
    uint32_t base = 0;
    if (valid) base = sm.wcnt[warp][d];
    __syncwarp();
    if (valid && lane == lead) sm.wcnt[warp][d] = base + __popc(peers);
    __syncwarp();
    rk[r] = base + __popc(peers & lanemask_lt());
    dg[r] = d;
  }
  __syncthreads();
  // Digit `tid`: prefix over warps and the block count.
  uint32_t bcount = 0;
#pragma unroll
  for (int w = 0; w < 8; ++w) {
    const uint32_t c = sm.wcnt[w][tid];
    sm.wcnt[w][tid] = bcount;
    bcount += c;
  }
  // Publish the aggregate; the two block scans, which do not need the
  // prefix, run before the look-back for the exclusive prefix of this digit,
  // so predecessors have more time to resolve theirs.  Predecessors are read
  // four at a time (independent loads, overlapping latencies), then taken in
  // order until the first inclusive prefix.
  st_vol(status + (size_t)b * 256 + tid, (b == 0 ? kFlagPre : kFlagAgg) | bcount);
  uint32_t tot;
  const uint32_t gexcl = block_excl_scan(hist[tid], sm.scan, tot);
  const uint32_t bst = block_excl_scan(bcount, sm.scan, tot);
  sm.bstart[tid] = bst;
  uint32_t excl = 0;
  if (b > 0) {
    bool fin = false;
    for (int64_t j = (int64_t)b - 1; !fin && j >= 0; j -= 4) {
      uint32_t sv[4];
#pragma unroll
      for (int w = 0; w < 4; ++w) sv[w] = j - w >= 0 ? ld_vol(status + (size_t)(j - w) * 256 + tid) : 0u;
#pragma unroll
      for (int w = 0; w < 4; ++w) {
        if (!fin && j - w >= 0) {
          uint32_t s = sv[w];
          int spins = 0;
          while ((s & ~kValMask) == 0u) {
            if (++spins > kSpinLimit) {
              set_err(err, kErrTimeout);
              s = kFlagPre;
              break;
            }
            __nanosleep(32);
            s = ld_vol(status + (size_t)(j - w) * 256 + tid);
          }
          excl += s & kValMask;
          if (s & kFlagPre) fin = true;
        }
      }
    }
    st_vol(status + (size_t)b * 256 + tid, kFlagPre | ((excl + bcount) & kValMask));
  }
  sm.gbase[tid] = gexcl + excl;
  __syncthreads();
#pragma unroll
  for (int r = 0; r < ITEMS; ++r) {
    if (dg[r] < 256) {
      const uint32_t lp = sm.bstart[dg[r]] + sm.wcnt[warp][dg[r]] + rk[r];
      sm.keys[lp] = k[r];
      sm.vals[lp] = v[r];
    }
  }
  __syncthreads();
  for (uint32_t i = tid; i < cnt; i += kThreads) {
    const uint32_t key = sm.keys[i];
    const uint32_t d = (key >> shift) & 255u;
    const uint32_t gp = sm.gbase[d] + (i - sm.bstart[d]);
    keys_out[gp] = key;
    vals_out[gp] = sm.vals[i];
  }
}

// ---------------------------------------------------------------------------
// The same sort in one launch, for the few keys that one cluster of blocks
// holds in registers: per pass every block ranks its keys, the blocks exchange
// their digit counts through distributed shared memory behind a cluster
// barrier, and the keys move by way of L2, in runs ordered in shared memory.
// Bound by the latency of a pass (1.6 us in one block, 2.8 in sixteen with two
// keys a thread); the five launches above, four of them with a chain of
// look-back, are too, at 20 us for 1,000 keys and 37 for 30k, where this one
// takes 6 and 11.  With more keys a thread the sixteen SMs fall behind the
// whole chip (a frame of 100k 8 us slower, of 200k 48), so the line lies at
// three a thread (640 x 512 frames, this sort against the passes: 1,000
// Gaussians 53 and 57 us, 10k 104 and 111, 32k 177 and 179, 48k 196 and 198,
// 64k 209 and 208).
// ---------------------------------------------------------------------------
constexpr int kSortThreads = 1024, kSortWarps = kSortThreads / 32;
constexpr int kSortBlocks = 16;  // more than the eight that every device takes: see sort_blocks
constexpr int kSortMaxItems = 3;

template <int ITEMS>
struct SortSmem {
  uint32_t wcnt[kSortWarps][256];  // digit counts, then prefixes, per warp
  uint32_t cnt[256];               // the block's digit counts (read by the cluster)
  uint32_t gbase[256], bstart[256];
  uint64_t scan[8];
  uint32_t keys[kSortThreads * ITEMS], vals[kSortThreads * ITEMS];
};

struct SortArgs {
  uint32_t *key0, *key1, *val0, *val1;  // key0: input; result in val0 (the last pass writes no keys)
  int n;
};

// Word of block `rank` of the cluster at this block's shared address p.
__device__ __forceinline__ uint32_t ld_cluster(const uint32_t* p, uint32_t rank) {
  uint32_t a, v;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;" ::: "memory");
}

// Block b of the cluster holds elements [b * 1024 items, ...), warp w of it 32
// items consecutive ones; items <= ITEMS and gridDim.x * 1024 * items >= n.
template <int ITEMS>
__global__ void __launch_bounds__(kSortThreads, 1) cluster_sort_kernel(const SortArgs a, const int items) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SortSmem<ITEMS>& sm = *reinterpret_cast<SortSmem<ITEMS>*>(smem_raw);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t b = blockIdx.x, nb = gridDim.x;
  const int first = (int)b * kSortThreads * items;
  const int cnt = max(0, min(kSortThreads * items, a.n - first));
  const int wfirst = warp * 32 * items + lane;  // within the block
  grid_dep_wait();
  grid_dep_launch();
#pragma unroll 1
  for (int p = 0; p < 4; ++p) {
    const int shift = 8 * p;
    const bool odd = p & 1;
    const uint32_t* kin = odd ? a.key1 : a.key0;
    const uint32_t* vin = odd ? a.val1 : a.val0;
    uint32_t* kout = odd ? a.key0 : a.key1;
    uint32_t* vout = odd ? a.val0 : a.val1;
    uint32_t k[ITEMS], v[ITEMS], rk[ITEMS];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      const int i = wfirst + 32 * r;
      const bool valid = r < items && i < cnt;
      k[r] = valid ? __ldcg(kin + first + i) : 0u;
      v[r] = valid ? (p == 0 ? (uint32_t)(first + i) : __ldcg(vin + first + i)) : 0u;
    }
    for (int i = tid; i < kSortWarps * 256; i += kSortThreads) (&sm.wcnt[0][0])[i] = 0u;
    __syncthreads();
    uint32_t* wc = sm.wcnt[warp];
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      rk[r] = 0u;
      if (r < items) {
        const bool valid = wfirst + 32 * r < cnt;
        const int d = valid ? (int)((k[r] >> shift) & 255u) : 256;
        const uint32_t peers = __match_any_sync(0xFFFFFFFFu, d);
        const uint32_t base = valid ? wc[d] : 0u;
        __syncwarp();
        if (valid && lane == __ffs(peers) - 1) wc[d] = base + __popc(peers);
        __syncwarp();
        rk[r] = base + __popc(peers & lanemask_lt());
      }
    }
    __syncthreads();
    // Digit tid: prefix over the warps and the block's count.
    uint32_t bcount = 0;
    if (tid < 256) {
#pragma unroll
      for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t c = sm.wcnt[w][tid];
        sm.wcnt[w][tid] = bcount;
        bcount += c;
      }
      sm.cnt[tid] = bcount;
    }
    cluster_barrier();
    // Digit tid's count in the cluster and in the blocks before this one;
    // exclusive scans over the digits of the cluster's and the block's counts.
    uint32_t tot = 0, before = 0;
    uint64_t own = 0, incl = 0;
    if (tid < 256) {
#pragma unroll
      for (int c = 0; c < kSortBlocks; ++c) {
        const uint32_t x = c < (int)nb ? ld_cluster(&sm.cnt[tid], (uint32_t)c) : 0u;
        tot += x;
        if (c < (int)b) before += x;
      }
      incl = own = ((uint64_t)tot << 32) | bcount;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint64_t y = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31) sm.scan[warp] = incl;
    }
    __syncthreads();
    if (tid < 256) {
      uint64_t ex = incl - own;
      for (int w = 0; w < warp; ++w) ex += sm.scan[w];
      sm.gbase[tid] = (uint32_t)(ex >> 32) + before;
      sm.bstart[tid] = (uint32_t)ex;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < ITEMS; ++r) {
      if (r < items && wfirst + 32 * r < cnt) {
        const uint32_t d = (k[r] >> shift) & 255u;
        const uint32_t lp = sm.bstart[d] + wc[d] + rk[r];
        sm.keys[lp] = k[r];
        sm.vals[lp] = v[r];
      }
    }
    __syncthreads();
    for (int i = tid; i < cnt; i += kSortThreads) {
      const uint32_t key = sm.keys[i], d = (key >> shift) & 255u;
      const uint32_t gp = sm.gbase[d] + ((uint32_t)i - sm.bstart[d]);
      if (p < 3) kout[gp] = key;
      vout[gp] = sm.vals[i];
    }
    // The pass's output is in place, and no block of the cluster still reads
    // this one's counts.
    cluster_barrier();
  }
}

template <int ITEMS>
void sort_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int nb, cudaStream_t st) {
  cfg = cudaLaunchConfig_t{};
  cfg.gridDim = dim3((unsigned)nb);
  cfg.blockDim = dim3(kSortThreads);
  cfg.dynamicSmemBytes = sizeof(SortSmem<ITEMS>);
  cfg.stream = st;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)nb;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
}

template <int ITEMS>
cudaError_t sort_attributes() {
  auto k = cluster_sort_kernel<ITEMS>;
  const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortSmem<ITEMS>));
  return e != cudaSuccess ? e : cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
}

// Blocks a cluster of the sort can have on the current device: kSortBlocks if
// the device can hold such a cluster, else the portable eight.
int sort_blocks() {
  static std::atomic<int> known[64];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 8;
  int nb = known[dev].load(std::memory_order_relaxed);
  if (nb) return nb;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  sort_config<kSortMaxItems>(cfg, attr, kSortBlocks, nullptr);
  int n = 0;
  const bool fits = sort_attributes<kSortMaxItems>() == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&n, cluster_sort_kernel<kSortMaxItems>, &cfg) == cudaSuccess && n > 0;
  if (!fits) cudaGetLastError();
  nb = fits ? kSortBlocks : 8;
  known[dev].store(nb, std::memory_order_relaxed);
  return nb;
}

template <int ITEMS>
cudaError_t launch_cluster_sort(const SortArgs& a, int nb, int items, cudaStream_t st) {
  const cudaError_t e = sort_attributes<ITEMS>();
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg;
  cudaLaunchAttribute attr[2];
  sort_config<ITEMS>(cfg, attr, nb, st);
  return cudaLaunchKernelEx(&cfg, cluster_sort_kernel<ITEMS>, a, items);
}

// ---------------------------------------------------------------------------
// Decoupled look-back over a 64-bit running total: block b publishes its
// aggregate, then one warp sums its predecessors back to the first inclusive
// prefix, 32 at a time (a chain of blocks that start together is walked in
// few rounds of latency: one thread reading eight at a time held a scan of
// 3 M words at 32 us, 47 of 53 stall cycles at the barrier behind it).
// In two halves, so a block can do independent work between them: publish
// the aggregate (block 0: its inclusive prefix), then resolve the exclusive
// prefix from the predecessors (all 32 lanes of a warp; all get it).
__device__ __forceinline__ void lookback64_publish(uint64_t* status, uint32_t b, uint64_t aggregate) {
  st_vol64(status + b, (b == 0 ? kFlagPre64 : kFlagAgg64) | aggregate);
}

__device__ __forceinline__ uint64_t lookback64_resolve(uint64_t* status, uint32_t b, uint64_t aggregate, uint32_t* err) {
  if (b == 0) return 0;
  const int lane = threadIdx.x & 31;
  uint64_t excl = 0;
  for (int64_t j = (int64_t)b - 1;; j -= 32) {
    // Lane l: predecessor j - l (before block 0: an empty prefix).
    uint64_t s = j - lane >= 0 ? ld_vol64(status + (j - lane)) : kFlagPre64;
    int spins = 0;
    while ((s & ~kValMask64) == 0ull) {
      if (++spins > kSpinLimit) {
        set_err(err, kErrTimeout);
        s = kFlagPre64;
        break;
      }
      __nanosleep(32);
      s = ld_vol64(status + (j - lane));
    }
    const uint32_t pre = __ballot_sync(0xFFFFFFFFu, (s & kFlagPre64) != 0ull);
    // The words up to the nearest inclusive prefix count.
    uint64_t v = (pre == 0u || lane < __ffs(pre)) ? s & kValMask64 : 0ull;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
    excl += v;
    if (pre) break;
  }
  if (lane == 0) st_vol64(status + b, kFlagPre64 | (excl + aggregate));
  return excl;
}

// Tiles of a rectangle (first and last tile of each axis; none: last < first).
__device__ __forceinline__ uint32_t rect_tiles(const ushort4 rc) {
  return ((uint32_t)(rc.z + 1) - rc.x) * ((uint32_t)(rc.w + 1) - rc.y);
}

// Row-major walk over the tiles of a rectangle by T threads: thread `sub` takes
// tiles sub, sub + T, ...  One division per walk, a few additions per step (with
// a division per step the scatter of 1.2 M entries took 35 us from its early
// launch, now 27).
struct TileWalk {
  uint32_t dx, tile, width, r, inc, skip;
  __device__ __forceinline__ TileWalk(const ushort4 rc, uint32_t sub, uint32_t T, uint32_t tiles_x) {
    width = (uint32_t)(rc.z + 1) - rc.x;
    // Exact: sub, T < 2^12 lie at least 0.5 / 2^12 of themselves from the next quotient.
    const float iw = __fdividef(1.0f, (float)width);
    const uint32_t dy = (uint32_t)(((float)sub + 0.5f) * iw), q = (uint32_t)(((float)T + 0.5f) * iw);
    dx = sub - dy * width;
    tile = (rc.y + dy) * tiles_x + rc.x + dx;
    r = T - q * width;
    inc = q * tiles_x + r;
    skip = tiles_x - width;
  }
  __device__ __forceinline__ void next() {
    dx += r;
    tile += inc;
    if (dx >= width) {
      dx -= width;
      tile += skip;
    }
  }
};

// The Gaussians of a block (or round) that cover many tiles.  The few threads
// that a Gaussian has in the two kernels below would walk a screen-sized
// rectangle in hundreds of dependent steps with the whole block waiting for
// them, so beyond kNarrow steps a thread a Gaussian goes to a whole warp (they
// are dealt to the warps in turn), beyond kHuge tiles to all of the block.
// The binning stage of 100k Gaussians at 640 x 512, 0.5% of them screen-sized:
// 104 us, 287 without the lists (equal footprints with as many entries: 92);
// 200k at 1280 x 1024: 225 and 937 us (205).  A limit of 16 or 64 steps is even
// (a frame of 100k Gaussians of 55 tiles on average: 285 us at 32, 290 at 16
// and at 64); kHuge only matters for a few in a block, as many make every warp
// busy either way.
template <int N>
struct WideList {
  uint32_t n[2];    // wide ones from the front of id, huge ones from its end
  uint16_t id[N];
  __device__ __forceinline__ void clear() { n[0] = n[1] = 0u; }
  __device__ __forceinline__ void add(int i, bool huge) {
    const int at = (int)atomicAdd(&n[huge], 1u);
    id[huge ? N - 1 - at : at] = (uint16_t)i;
  }
  // Number of a warp's items, and the j-th of them.
  __device__ __forceinline__ int mine(int warp, int warps) const { return ((int)n[0] - warp + warps - 1) / warps; }
  __device__ __forceinline__ int items(int warp, int warps) const { return mine(warp, warps) + (int)n[1]; }
  __device__ __forceinline__ int item(int j, int warp, int warps, bool& huge) const {
    const int m = mine(warp, warps);
    huge = j >= m;
    return id[huge ? N - 1 - (j - m) : warp + j * warps];
  }
};
constexpr int kNarrow = 32;     // steps of a thread
constexpr int kHuge = 2048;     // tiles
constexpr int kCountTPG = 4;    // threads per Gaussian in the count kernel

// Step 2: block b (ticket) owns depth ranks [chunk b, chunk b + chunk), chunk
// <= 256 ITEMS; thread t scans ranks ITEMS t, ...  Writes offs / offs_by_gid and
// column b of the tile-major count table.
struct CountArgs {
  int P, tiles_x, ntiles, nblocks, chunk;
  int64_t cap;
  const uint32_t* order;  // depth-sorted Gaussian ids
  const uint32_t* touched;
  const ushort4* rect;
  uint32_t *offs, *offs_by_gid, *table;
  uint64_t* status;
  uint32_t* ticket;
  Header* hdr;
};

template <int ITEMS>
__global__ void __launch_bounds__(kThreads) bin_count_kernel(const CountArgs a) {
  grid_dep_wait();
  grid_dep_launch();
  extern __shared__ uint32_t s_cnt[];  // [ntiles]
  __shared__ uint32_t s_scan[8];
  __shared__ uint32_t s_ticket;
  __shared__ uint64_t s_prefix;
  __shared__ uint32_t s_c[kThreads * ITEMS];
  __shared__ ushort4 s_rect[kThreads * ITEMS];
  __shared__ WideList<kThreads * ITEMS> s_wide;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  for (int i = tid; i < a.ntiles; i += kThreads) s_cnt[i] = 0;
  if (tid == 0) {
    s_ticket = atomicAdd(a.ticket, 1u);
    s_wide.clear();
  }
  __syncthreads();
  const uint32_t b = s_ticket;
  const int64_t start = (int64_t)b * a.chunk;
  if (start >= a.P) return;
  const int nloc = (int)min((int64_t)a.chunk, (int64_t)a.P - start);
  uint32_t gid[ITEMS], cnt[ITEMS];
  uint32_t tsum = 0;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int li = tid * ITEMS + i;
    gid[i] = li < nloc ? a.order[start + li] : 0u;
    cnt[i] = li < nloc ? a.touched[gid[i]] : 0u;
    s_c[li] = cnt[i];
    s_rect[li] = cnt[i] ? a.rect[gid[i]] : make_ushort4(0, 0, 0, 0);
    if (cnt[i] > kNarrow * kCountTPG) s_wide.add(li, cnt[i] > kHuge);
    tsum += cnt[i];
  }
  uint32_t btot;
  const uint32_t texcl = block_excl_scan(tsum, s_scan, btot);
  // The block's total goes out at once; its tile counts, which do not need
  // the prefix, are taken while the predecessors resolve theirs.
  if (tid == 0) lookback64_publish(a.status, b, btot);
  // Tile counts, in any order: four threads to a Gaussian, a warp or the block
  // to a wide one.
  for (int w = tid; w < kCountTPG * nloc; w += kThreads) {
    const uint32_t c = s_c[w / kCountTPG], sub = (uint32_t)w % kCountTPG;
    if (sub >= c || c > kNarrow * kCountTPG) continue;
    TileWalk t(s_rect[w / kCountTPG], sub, kCountTPG, a.tiles_x);
    for (uint32_t k = sub; k < c; k += kCountTPG, t.next()) atomicAdd(&s_cnt[t.tile], 1u);
  }
  const int items = s_wide.items(warp, kThreads / 32);
  for (int j = 0; j < items; ++j) {
    bool huge;
    const int i = s_wide.item(j, warp, kThreads / 32, huge);
    const uint32_t c = s_c[i], sub = huge ? tid : lane, T = huge ? kThreads : 32;
    TileWalk t(s_rect[i], sub, T, a.tiles_x);
    for (uint32_t k = sub; k < c; k += T, t.next()) atomicAdd(&s_cnt[t.tile], 1u);
  }
  if (tid < 32) {
    __syncwarp();
    const uint64_t pre = lookback64_resolve(a.status, b, btot, &a.hdr->err);
    if (tid == 0) s_prefix = pre;
  }
  __syncthreads();
  uint64_t run = s_prefix + texcl;
#pragma unroll
  for (int i = 0; i < ITEMS; ++i) {
    const int li = tid * ITEMS + i;
    if (li < nloc) {
      const uint32_t o32 = (uint32_t)min(run, (uint64_t)0xFFFFFFFFu);
      a.offs[start + li] = o32;
      a.offs_by_gid[gid[i]] = o32;
    }
    run += cnt[i];
  }
  if (start + a.chunk >= a.P && tid == kThreads - 1) {
    a.offs[a.P] = (uint32_t)min(run, (uint64_t)0xFFFFFFFFu);
    a.hdr->num_dups = (uint32_t)min(run, (uint64_t)0xFFFFFFFFu);
    if (run > (uint64_t)a.cap) set_err(&a.hdr->err, kErrOverflow);
  }
  __syncthreads();
  for (int t = tid; t < a.ntiles; t += kThreads) a.table[(size_t)t * a.nblocks + b] = s_cnt[t];
}

// Step 3: in-place exclusive scan of the (tile, block) table, tile-major.
__global__ void __launch_bounds__(kThreads) table_scan_kernel(uint32_t* table, int64_t n, uint64_t* status,
                                                             uint32_t* ticket, uint32_t* err) {
  grid_dep_wait();
  grid_dep_launch();
  __shared__ uint32_t s_scan[8];
  __shared__ uint32_t s_ticket;
  __shared__ uint64_t s_prefix;
  const int tid = threadIdx.x;
  if (tid == 0) s_ticket = atomicAdd(ticket, 1u);
  __syncthreads();
  const uint32_t b = s_ticket;
  const int64_t start = (int64_t)b * kPChunk;
  if (start >= n) return;
  // Eight consecutive words per thread, two 16-byte accesses where they are
  // all there (the table starts on a 256-byte boundary).
  static_assert(kPItems == 8, "two 16-byte accesses per thread");
  const int64_t r0 = start + tid * kPItems;
  const bool full = r0 + kPItems <= n;
  uint32_t v[kPItems], tsum = 0;
  if (full) {
    const uint4 x = *reinterpret_cast<const uint4*>(table + r0), y = *reinterpret_cast<const uint4*>(table + r0 + 4);
    v[0] = x.x; v[1] = x.y; v[2] = x.z; v[3] = x.w; v[4] = y.x; v[5] = y.y; v[6] = y.z; v[7] = y.w;
  } else {
#pragma unroll
    for (int i = 0; i < kPItems; ++i) v[i] = r0 + i < n ? table[r0 + i] : 0u;
  }
#pragma unroll
  for (int i = 0; i < kPItems; ++i) tsum += v[i];
  uint32_t btot;
  const uint32_t texcl = block_excl_scan(tsum, s_scan, btot);
  if (tid == 0) lookback64_publish(status, b, btot);
  if (tid < 32) {
    const uint64_t pre = lookback64_resolve(status, b, btot, err);
    if (tid == 0) s_prefix = pre;
  }
  __syncthreads();
  uint64_t run = s_prefix + texcl;
#pragma unroll
  for (int i = 0; i < kPItems; ++i) {
    const uint32_t c = v[i];
    v[i] = (uint32_t)min(run, (uint64_t)0xFFFFFFFFu);
    run += c;
  }
  if (full) {
    *reinterpret_cast<uint4*>(table + r0) = make_uint4(v[0], v[1], v[2], v[3]);
    *reinterpret_cast<uint4*>(table + r0 + 4) = make_uint4(v[4], v[5], v[6], v[7]);
  } else {
#pragma unroll
    for (int i = 0; i < kPItems; ++i)
      if (r0 + i < n) table[r0 + i] = v[i];
  }
}

// Step 4: block b (= blockIdx.x) takes the ranks of count block b, 128
// Gaussians (a round) at a time.  Per tile it keeps a 128-bit mask of the
// round's Gaussians that touch it (atomic ors: no order among them), and the
// position in the list where the round's entries of the tile begin; an
// entry's place is that position plus the mask bits of earlier Gaussians.
// Gaussian i of the round is bit i / 4 of word i % 4: a warp's Gaussians lie
// in different words and a Gaussian's threads on consecutive tiles, so the
// ors of a warp spread over all banks, and the second visit reads a mask with
// one 16-byte load.  Several threads take a Gaussian's entries, a warp or the
// block those of a wide one (WideList); the next round's Gaussians (three
// dependent loads) are fetched while a round is worked on.
// Bound by the scattered 8-byte stores (a third to half of it: one sector
// each) and by issue (two visits of every entry and a sweep of the tiles per
// round).  1M Gaussians at 1280 x 1024, 33 M entries: 512 us from its early
// launch, 543 with suffix counts beside the masks and blocks of 512; 100k at
// 640 x 512, 1.2 M entries: 27 us; 1,000 Gaussians: 3 us, 27 with a warp walking
// its 64 Gaussians one after another.
// Block 0 also writes the tile ranges and marks the workspace as holding a
// forward's state.
struct ScatterArgs {
  int P, tiles_x, ntiles, nblocks, chunk;
  int64_t cap;
  const uint32_t *order, *touched, *offs, *table;
  const ushort4* rect;
  uint2* sorted;
  uint2* ranges;
  Header* hdr;
};
// Threads per block: with the masks of more tiles than this only one or two
// blocks fit on an SM, so they get more threads.
constexpr int kScatTiles = 2048;
constexpr int kRound = 128;  // Gaussians per round (four 32-bit mask words)
__host__ __device__ constexpr size_t scatter_smem(int ntiles) { return (size_t)ntiles * (16 + 4); }

template <int NT>
__global__ void __launch_bounds__(NT) bin_scatter_kernel(const ScatterArgs a) {
  grid_dep_wait();
  grid_dep_launch();
  extern __shared__ __align__(16) uint32_t s_dyn[];
  uint4* s_mask = reinterpret_cast<uint4*>(s_dyn);  // [ntiles]
  uint32_t* s_word = s_dyn;                         // the same, [ntiles][4]
  uint32_t* s_pos = s_dyn + 4 * a.ntiles;           // [ntiles]: next position of the tile's segment
  __shared__ uint2 s_id[2][kRound];  // id, first emission index
  __shared__ ushort4 s_rect[2][kRound];
  __shared__ WideList<kRound> s_wide[2];
  constexpr int TPG = NT / kRound;  // threads per Gaussian
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int b = blockIdx.x;
  const int64_t start = (int64_t)b * a.chunk;
  const int nloc = (int)min((int64_t)a.chunk, (int64_t)a.P - start);
  const uint64_t cap = (uint64_t)a.cap;
  // Past capacity the list is incomplete (and flagged): every range is
  // published empty so no later kernel follows an index beyond capacity.
  const bool overflow = (uint64_t)a.hdr->num_dups > cap;
  const uint64_t K = overflow ? 0 : (uint64_t)a.hdr->num_dups;
  // Rectangle of Gaussian g (width 0 where it touches no tile).
  const auto rect_of = [&](bool have, uint32_t g) {
    return have && a.touched[g] != 0u ? a.rect[g] : make_ushort4(1, 0, 0, 0);
  };
  const auto put = [&](int to, const uint2 id, const ushort4 rc) {
    s_id[to][tid] = id;
    s_rect[to][tid] = rc;
    const uint32_t c = rect_tiles(rc);
    if (c > kNarrow * TPG) s_wide[to].add(tid, c > kHuge);
  };
  if (tid < 2) s_wide[tid].clear();
  __syncthreads();
  if (tid < kRound) {
    const bool have = tid < nloc;
    const uint32_t g = have ? a.order[start + tid] : 0u;
    put(0, make_uint2(g, have ? a.offs[start + tid] : 0u), rect_of(have, g));
  }
  for (int t = tid; t < a.ntiles; t += NT) {
    s_pos[t] = a.table[(size_t)t * a.nblocks + b];
    s_mask[t] = make_uint4(0u, 0u, 0u, 0u);
    if (b == 0) {
      const uint64_t lo = min((uint64_t)a.table[(size_t)t * a.nblocks], K);
      const uint64_t hi = t + 1 < a.ntiles ? min((uint64_t)a.table[(size_t)(t + 1) * a.nblocks], K) : K;
      a.ranges[t] = make_uint2((uint32_t)lo, (uint32_t)hi);
    }
  }
  if (b == 0 && tid == 0) a.hdr->has_forward = 1u;
  // Visits of Gaussian i of the round: its bit in the masks of its tiles k,
  // k + step, ...; its entries of these tiles.
  const auto mark = [&](int i, const ushort4 rc, uint32_t c, uint32_t k, uint32_t step) {
    const uint32_t bit = 1u << (i >> 2);
    for (TileWalk t(rc, k, step, a.tiles_x); k < c; k += step, t.next()) atomicOr(&s_word[4 * t.tile + (i & 3)], bit);
  };
  const auto emit = [&](int i, const uint2 id, const ushort4 rc, uint32_t c, uint32_t k, uint32_t step) {
    // Bits of the Gaussians before i in the four words.
    const int word = i & 3, bit = i >> 2;
    const uint32_t below = (1u << bit) - 1u, upto = (2u << bit) - 1u;
    const uint32_t m0 = word > 0 ? upto : below, m1 = word > 1 ? upto : below, m2 = word > 2 ? upto : below;
    for (TileWalk t(rc, k, step, a.tiles_x); k < c; k += step, t.next()) {
      const uint4 m = s_mask[t.tile];
      const uint32_t pos = s_pos[t.tile] + __popc(m.x & m0) + __popc(m.y & m1) + __popc(m.z & m2) + __popc(m.w & below);
      if ((uint64_t)pos < cap) a.sorted[pos] = make_uint2(id.y + k, id.x);
    }
  };
  const int i = tid / TPG, sub = tid % TPG;
  __syncthreads();
  int buf = 0;
  for (int r0 = 0; r0 < nloc; r0 += kRound, buf ^= 1) {
    // The next round's Gaussian of this thread: ids now, rectangles below.
    const int rn = r0 + kRound + tid;
    const bool have = tid < kRound && rn < nloc;
    uint2 nid = make_uint2(0u, 0u);
    if (have) nid = make_uint2(a.order[start + rn], a.offs[start + rn]);
    // A thread's own Gaussian, unless it is a wide one; then the wide ones.
    const ushort4 rc = s_rect[buf][i];
    const uint32_t c = rect_tiles(rc) <= kNarrow * TPG ? rect_tiles(rc) : 0u;
    const int items = s_wide[buf].items(warp, NT / 32);
    mark(i, rc, c, sub, TPG);
    for (int j = 0; j < items; ++j) {
      bool huge;
      const int w = s_wide[buf].item(j, warp, NT / 32, huge);
      const ushort4 wrc = s_rect[buf][w];
      mark(w, wrc, rect_tiles(wrc), huge ? tid : lane, huge ? NT : 32);
    }
    __syncthreads();
    const ushort4 nrc = rect_of(have, nid.x);
    if (sub < c) emit(i, s_id[buf][i], rc, c, sub, TPG);
    for (int j = 0; j < items; ++j) {
      bool huge;
      const int w = s_wide[buf].item(j, warp, NT / 32, huge);
      const ushort4 wrc = s_rect[buf][w];
      emit(w, s_id[buf][w], wrc, rect_tiles(wrc), huge ? tid : lane, huge ? NT : 32);
    }
    if (r0 + kRound >= nloc) break;
    if (tid < kRound) put(buf ^ 1, nid, nrc);
    __syncthreads();
    if (tid == 0) s_wide[buf].clear();  // of the round after the next
    for (int t = tid; t < a.ntiles; t += NT) {
      const uint4 m = s_mask[t];
      s_pos[t] += __popc(m.x) + __popc(m.y) + __popc(m.z) + __popc(m.w);
      s_mask[t] = make_uint4(0u, 0u, 0u, 0u);
    }
    __syncthreads();
  }
}

__global__ void bin_prep_kernel(int P, const float* __restrict__ uv, const int* __restrict__ radius,
                                const float* __restrict__ depth, int W, int H, int tw, int th, ushort4* rect,
                                uint32_t* touched, uint32_t* dkey, uint32_t* num_visible) {
  const int g = blockIdx.x * blockDim.x + threadIdx.x;
  bool vis = false;
  if (g < P) {
    ushort4 rc = make_ushort4(1, 1, 0, 0);
    uint32_t t = 0, key = 0xFFFFFFFFu;
    const int r = radius[g];
    const float u = uv[2 * g], v = uv[2 * g + 1];
    int x0, y0, x1, y1;
    if (r > 0 && isfinite(u) && isfinite(v) && pixel_rect(u, v, r, W, H, x0, y0, x1, y1)) {
      const int tx0 = x0 / tw, tx1 = x1 / tw, ty0 = y0 / th, ty1 = y1 / th;
      rc = make_ushort4(tx0, ty0, tx1, ty1);
      t = (uint32_t)((tx1 - tx0 + 1) * (ty1 - ty0 + 1));
      key = __float_as_uint(depth[g]);
      vis = true;
    }
    rect[g] = rc;
    touched[g] = t;
    dkey[g] = key;
  }
  const unsigned vote = __ballot_sync(0xFFFFFFFFu, vis);
  if ((threadIdx.x & 31) == 0 && vote) atomicAdd(num_visible, (uint32_t)__popc(vote));
}

int grid_for(int64_t n, int per_block) {
  const int64_t b = (n + per_block - 1) / per_block;
  const int64_t c = b < 152 * 16 ? b : 152 * 16;
  return (int)(c > 1 ? c : 1);
}

}  // namespace

cudaError_t launch_bin_prep(int P, const float* uv, const int* radius, const float* depth, int W, int H, int tw,
                            int th, ushort4* rect, uint32_t* touched, uint32_t* dkey, uint32_t* num_visible,
                            cudaStream_t st) {
  if (P <= 0) return cudaSuccess;
  bin_prep_kernel<<<ceil_div(P, kThreads), kThreads, 0, st>>>(P, uv, radius, depth, W, H, tw, th, rect, touched,
                                                              dkey, num_visible);
  return cudaGetLastError();
}

cudaError_t launch_binning(BinArgs& b, cudaStream_t st) {
  Header* hdr = static_cast<Header*>(b.hdr);
  const size_t ppass_smem = sizeof(PassSmem<kPItems>);
  const int P = b.P;
  if (P <= 0) return cudaSuccess;  // K = 0: the cleared header and ranges already say so
  cudaError_t e;
  const int pblocks = b.pblocks;
  uint32_t* status_depth = b.status;
  const int bblocks = b.bblocks;
  uint64_t* status_count = reinterpret_cast<uint64_t*>(b.status + (size_t)pblocks * 256 * 4);
  uint64_t* status_table = status_count + bblocks;
  // 1. depth sort (values: Gaussian ids; an even number of passes, so the
  // result is in dval[0] either way)
  const int max_nb = P <= kSortBlocks * kSortThreads * kSortMaxItems ? sort_blocks() : 0;
  if (P <= max_nb * kSortThreads * kSortMaxItems) {
    SortArgs so;
    so.key0 = b.dkey[0];
    so.key1 = b.dkey[1];
    so.val0 = b.dval[0];
    so.val1 = b.dval[1];
    so.n = P;
    int nb = 1;  // blocks: one key a thread first, then more keys a thread
    while (nb < max_nb && nb * kSortThreads < P) nb *= 2;
    const int items = ceil_div(P, nb * kSortThreads);
    e = items <= 1 ? launch_cluster_sort<1>(so, nb, items, st) : launch_cluster_sort<kSortMaxItems>(so, nb, items, st);
    if (e != cudaSuccess) return e;
  } else {
    if ((e = launch_pdl(depth_hist_kernel, pblocks, kThreads, 0, st, (const uint32_t*)b.dkey[0], P, b.hist)) != cudaSuccess)
      return e;
    for (int p = 0; p < 4; ++p) {
      const int i = p & 1, o = i ^ 1;
      e = launch_pdl(p == 0 ? onesweep_kernel<true, kPItems> : onesweep_kernel<false, kPItems>, pblocks, kThreads,
                     ppass_smem, st, (const uint32_t*)b.dkey[i], p == 0 ? (const uint32_t*)nullptr : (const uint32_t*)b.dval[i],
                     b.dkey[o], b.dval[o], (int64_t)P, 8 * p, (const uint32_t*)(b.hist + 256 * p),
                     status_depth + (size_t)p * pblocks * 256, hdr->ticket + kTicketDepth0 + p, &hdr->err);
      if (e != cudaSuccess) return e;
    }
  }
  // 2. tiles_touched scan + per-block tile counts
  CountArgs ca;
  ca.P = P;
  ca.tiles_x = b.tiles_x;
  ca.ntiles = b.ntiles;
  ca.nblocks = bblocks;
  ca.chunk = b.bchunk;
  ca.cap = b.cap;
  ca.order = b.dval[0];
  ca.touched = b.touched;
  ca.rect = b.rect;
  ca.offs = b.offs;
  ca.offs_by_gid = b.offs_by_gid;
  ca.table = b.table;
  ca.status = status_count;
  ca.ticket = hdr->ticket + kTicketScan;
  ca.hdr = hdr;
  const size_t count_smem = (size_t)b.ntiles * 4;
  auto count = b.bchunk <= 2 * kThreads ? bin_count_kernel<2> : bin_count_kernel<kBinChunk / kThreads>;
  cudaFuncSetAttribute(count, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)count_smem);
  if ((e = launch_pdl(count, bblocks, kThreads, count_smem, st, ca)) != cudaSuccess) return e;
  // 3. scan of the (tile, block) table
  const int64_t tn = (int64_t)b.ntiles * bblocks;
  e = launch_pdl(table_scan_kernel, ceil_div(tn, kPChunk), kThreads, 0, st, b.table, tn, status_table,
                 hdr->ticket + kTicketTable, &hdr->err);
  if (e != cudaSuccess) return e;
  // 4. scatter into the final list
  ScatterArgs sa;
  sa.P = P;
  sa.tiles_x = b.tiles_x;
  sa.ntiles = b.ntiles;
  sa.nblocks = bblocks;
  sa.chunk = b.bchunk;
  sa.cap = b.cap;
  sa.order = b.dval[0];
  sa.touched = b.touched;
  sa.offs = b.offs;
  sa.table = b.table;
  sa.rect = b.rect;
  sa.sorted = b.sorted;
  sa.ranges = b.ranges;
  sa.hdr = hdr;
  const size_t smem = scatter_smem(b.ntiles);
  const int nt = b.ntiles <= kScatTiles ? 512 : 1024;
  auto scat = nt == 512 ? bin_scatter_kernel<512> : bin_scatter_kernel<1024>;
  cudaFuncSetAttribute(scat, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  return launch_pdl(scat, bblocks, nt, smem, st, sa);
}

// ---------------------------------------------------------------------------
// Debug dump of the forward state (parity tests).
// ---------------------------------------------------------------------------
__global__ void dump_kernel(const DumpArgs d) {
  const Header* hdr = static_cast<const Header*>(d.hdr);
  const uint64_t K = min((uint64_t)hdr->num_dups, (uint64_t)d.cap);
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  const uint64_t i0 = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (uint64_t i = i0; i < K; i += stride) {
    const uint32_t g = d.sorted[i].y;
    if (d.keys) {
      // Tile of list position i: the last tile whose range starts at or
      // before i (empty tiles share the start of the next tile).
      int lo = 0, hi = d.ntiles;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (d.ranges[mid].x <= i) lo = mid; else hi = mid;
      }
      const float dep = d.rec[3 * (size_t)g + 1].z;
      d.keys[i] = ((uint64_t)(uint32_t)lo << 32) | __float_as_uint(dep);
    }
    if (d.gauss) d.gauss[i] = g;
  }
  for (uint64_t i = i0; i < (uint64_t)d.ntiles; i += stride)
    if (d.ranges_out) { d.ranges_out[2 * i] = d.ranges[i].x; d.ranges_out[2 * i + 1] = d.ranges[i].y; }
  for (uint64_t i = i0; i < (uint64_t)d.HW; i += stride) {
    if (d.ncontrib_out) d.ncontrib_out[i] = d.ncontrib[i];
    if (d.tfinal_out) d.tfinal_out[i] = d.tfinal[i];
  }
  for (uint64_t g = i0; g < (uint64_t)d.P; g += stride) {
    const float4 r0 = d.rec[3 * g], r1 = d.rec[3 * g + 1], r2 = d.rec[3 * g + 2];
    if (d.uv) { d.uv[2 * g] = r0.x; d.uv[2 * g + 1] = r0.y; }
    if (d.conic) {
      // Stored scaled conic back to (a, b, c).
      d.conic[3 * g] = r0.z / (-0.5f * kLog2e);
      d.conic[3 * g + 1] = r0.w / (-kLog2e);
      d.conic[3 * g + 2] = r1.x / (-0.5f * kLog2e);
    }
    if (d.opacity) d.opacity[g] = r1.y;
    if (d.depth) d.depth[g] = r1.z;
    if (d.rgb) { d.rgb[3 * g] = r1.w; d.rgb[3 * g + 1] = r2.x; d.rgb[3 * g + 2] = r2.y; }
    if (d.radius) d.radius[g] = (int32_t)r2.z;
    if (d.touched_out) d.touched_out[g] = d.touched[g];
  }
}

cudaError_t launch_dump(const DumpArgs& d, cudaStream_t st) {
  int64_t n = d.cap;
  if (d.P > n) n = d.P;
  if (d.HW > n) n = d.HW;
  if (d.ntiles > n) n = d.ntiles;
  dump_kernel<<<grid_for(n, 256), 256, 0, st>>>(d);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// FP32 FMA throughput probe: 8 independent FMA chains per thread.
// ---------------------------------------------------------------------------
__device__ float g_probe_sink[1];

__global__ void __launch_bounds__(256) fma_probe_kernel(int iters, float seed, float* out) {
  float a0 = seed + threadIdx.x, a1 = a0 + 1, a2 = a0 + 2, a3 = a0 + 3, a4 = a0 + 4, a5 = a0 + 5, a6 = a0 + 6,
        a7 = a0 + 7;
  const float m = 0.999999f, c = 1e-7f;
#pragma unroll 1
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      a0 = fmaf(a0, m, c); a1 = fmaf(a1, m, c); a2 = fmaf(a2, m, c); a3 = fmaf(a3, m, c);
      a4 = fmaf(a4, m, c); a5 = fmaf(a5, m, c); a6 = fmaf(a6, m, c); a7 = fmaf(a7, m, c);
    }
  }
  const float s = a0 + a1 + a2 + a3 + a4 + a5 + a6 + a7;
  if (s == 12345.678f) out[0] = s;  // keeps the chains alive
}

cudaError_t probe_fp32(int iters, double* flops, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int blocks = sms * 8;
  // The sink's address first: nothing to release if the lookup fails.
  float* sink = nullptr;
  cudaError_t e = cudaGetSymbolAddress(reinterpret_cast<void**>(&sink), g_probe_sink);
  if (e != cudaSuccess) return e;
  if (!sink) return cudaErrorInvalidSymbol;
  cudaEvent_t e0, e1;
  if ((e = cudaEventCreate(&e0)) != cudaSuccess) return e;
  if ((e = cudaEventCreate(&e1)) != cudaSuccess) {
    cudaEventDestroy(e0);
    return e;
  }
  fma_probe_kernel<<<blocks, 256, 0, st>>>(iters / 8 + 1, 1.0f, sink);  // warm-up
  cudaEventRecord(e0, st);
  fma_probe_kernel<<<blocks, 256, 0, st>>>(iters, 1.0f, sink);
  cudaEventRecord(e1, st);
  e = cudaEventSynchronize(e1);
  float ms = 0.f;
  if (e == cudaSuccess) e = cudaEventElapsedTime(&ms, e0, e1);
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (e != cudaSuccess) return e;
  *flops = (double)blocks * 256.0 * iters * 16.0 * 8.0 * 2.0 / (ms * 1e-3);
  return cudaGetLastError();
}

}  // namespace fe
