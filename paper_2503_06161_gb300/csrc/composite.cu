// Per-tile front-to-back compositing of colour, semantic feature and depth
// (Sec. 3.3, Eq. 7-8) and its reverse pass.
//
// Forward: one 256-thread block per tile, one pixel per thread.  Batches of
// the tile's sorted list are staged in shared memory; each pixel walks them
// in order, accumulating w = alpha*T into rgb, depth and the D feature
// channels, and stops before a Gaussian that would take T below 1e-4.  The
// block leaves as soon as every pixel is done (__syncthreads_count).
//
// Reverse: the same block walks the list backwards from the largest
// n_contrib of the tile, replaying T_i = T_{i+1} / (1 - alpha_i) from
// T_final (no per-pixel lists are stored).  Per batch, the terms of each
// warp's (pixel, Gaussian) pairs are summed over its pixels by tensor-core
// products and then over the tile's warps in a fixed order, one partial row
// per (tile, Gaussian) entry: no floating-point atomics, bitwise
// deterministic.
#include "common.cuh"
#include "kernels.h"
#include "mma.cuh"

namespace fe {

namespace {

// Gaussians per staged batch of the forward (two batches are in flight) and
// blocks per SM, by the channels and the tiles of the launch.  Most tiles end
// within the first 200 entries of their list, so batches of 64 land sooner and
// load less past the end, but stop the block twice as often: with several
// waves of tiles D = 32 takes 64 (frames of 200k Gaussians at 640 x 512: 279 us,
// 282 with 128, 289 with 32; 100k at 1280 x 1024: 661, 671, 687), with all tiles
// resident at once 128 (1,500 at 96 x 72: 57 us, 61 with 64; 30k at 160 x 128:
// 169 and 176).  D = 16 takes two blocks per SM, whose registers suffice, while
// the tiles fit about one such wave, else three (frames at two and three
// blocks: 30k at 320 x 240, 300 tiles, 98 and 111 us; at 333 x 251, 336 tiles,
// 102 and 114; at 352 x 288, 396 tiles, 111 and 111; at 384 x 288 117 and 109;
// at 640 x 512 171 and 160; 100k at 352 x 288 141 and 125).  At three blocks
// D = 32 spills 28 bytes (64-entry batches) or 56 (128); two blocks, without
// spills, are 1% slower (200k at 640 x 512: 350 us for 347).
constexpr int kSMs = 152;
template <int D>
constexpr int fwd_batch() { return D <= 16 ? 128 : (D <= 64 ? 64 : 32); }
template <int D>
int fwd_batch_for(int tiles) { return D == 32 && tiles <= 3 * kSMs ? 128 : fwd_batch<D>(); }
template <int D>
constexpr int fwd_blocks() { return D <= 32 ? 3 : (D <= 64 ? 2 : 1); }
constexpr int kTwoBlockTiles = 2 * kSMs + kSMs / 4;

// Bytes of one staged batch: B render records (48 bytes each), then B
// feature rows in their stored format (fp32 or bf16).
__host__ __device__ constexpr uint32_t stage_bytes(int B, int D, int bf16) {
  return (uint32_t)B * (uint32_t)(kRec * 4 + D * (bf16 ? 2 : 4));
}

// Bulk copies of one batch into a staging buffer, completing on `bar`:
// thread 0 arms the barrier with the batch's byte count, thread t < nb copies
// the record and the feature row of its Gaussian g.  Sources start at
// 48 g and g * row bytes of 16-byte aligned arrays, destinations at
// multiples of 16 bytes, and every size is a multiple of 16 bytes.
template <int D>
__device__ __forceinline__ void stage_issue(const CompositeArgs& a, unsigned char* buf, int B, int nb, uint32_t g,
                                            uint64_t* bar) {
  const int tid = threadIdx.x;
  const uint32_t rowb = (uint32_t)D * (a.feat_bf16 ? 2u : 4u);
  if (tid == 0) mbar_arrive_expect_tx(bar, (uint32_t)nb * ((uint32_t)kRec * 4u + rowb));
  if (tid < nb) {
    fence_proxy_async();  // earlier generic reads of this buffer come first
    tma_load_1d(buf + (size_t)tid * kRec * 4, a.rec + 3 * (size_t)g, (uint32_t)kRec * 4u, bar);
    tma_load_1d(buf + (size_t)B * kRec * 4 + (size_t)tid * rowb,
                static_cast<const unsigned char*>(a.feat) + (size_t)g * a.feat_row_bytes, rowb, bar);
  }
}

// bf16 feature rows of a landed batch -> fp32 rows (whole block).
template <int D>
__device__ __forceinline__ void widen_bf16(const unsigned char* raw, float* dst, int nb) {
  const uint4* src = reinterpret_cast<const uint4*>(raw);
  float4* d4 = reinterpret_cast<float4*>(dst);
  for (int i = threadIdx.x; i < nb * (D / 8); i += kThreads) {
    const uint4 q = src[i];
    d4[2 * i] = make_float4(__uint_as_float(q.x << 16), __uint_as_float(q.x & 0xFFFF0000u),
                            __uint_as_float(q.y << 16), __uint_as_float(q.y & 0xFFFF0000u));
    d4[2 * i + 1] = make_float4(__uint_as_float(q.z << 16), __uint_as_float(q.z & 0xFFFF0000u),
                                __uint_as_float(q.w << 16), __uint_as_float(q.w & 0xFFFF0000u));
  }
}

// Shared memory of the forward with B-Gaussian batches: two staging
// buffers, then (bf16 features) one fp32 copy of the current batch's rows.
__host__ __device__ constexpr size_t fwd_smem_bytes(int B, int D, int bf16) {
  return 2 * (size_t)stage_bytes(B, D, bf16) + (bf16 ? (size_t)B * D * 4 : 0);
}

// Staging state a block carries from tile to tile: how many times each of
// its two staging buffers has been armed.  Arming is block-uniform, so
// every thread derives the same wait parity from it: batch j of a tile sits
// in buffer j & 1 and completes that buffer's (arms[b] + j / 2)-th phase.
struct StageState {
  uint32_t arms[2];
  bool dead;  // a drain gave up: shared memory may still receive a copy
};

__device__ __forceinline__ uint32_t stage_parity(const StageState& st, uint32_t j) {
  return (st.arms[j & 1] + (j >> 1)) & 1u;
}

// A tile is done with its staging buffers: the last two batches it issued
// (any earlier one completed before its buffer was re-armed) must land
// before shared memory is reused, whether the tile finished, left early or
// gave up on a wait.  The drain has its own, long bound; if even that runs
// out the block stops taking tiles.
__device__ __forceinline__ void stage_drain(StageState& st, uint64_t* s_bar, uint32_t issued, uint32_t* err) {
  bool ok = true;
  for (uint32_t j = issued > 2 ? issued - 2 : 0; j < issued; ++j)
    ok &= mbar_wait(&s_bar[j & 1], stage_parity(st, j), kDrainPolls);
  if (__syncthreads_or(!ok)) {
    if (threadIdx.x == 0) set_err(err, kErrTimeout);
    st.dead = true;
  }
  st.arms[0] += (issued + 1) / 2;
  st.arms[1] += issued / 2;
}

// True when no pixel centre of the rectangle [x0, x1] x [y0, y1] can blend
// record `rec` (so a warp covering it may skip the entry without changing
// anything): either the 3-sigma square misses the rectangle -- the per-pixel
// test, at the rectangle's nearest centres, with the same subtractions -- or
// the record's blend box (word 11) does.
__device__ __forceinline__ bool block_misses(const float* rec, float x0, float x1, float y0, float y1) {
  const float2 uv = *reinterpret_cast<const float2*>(rec);
  const float2 rb = *reinterpret_cast<const float2*>(rec + 10);  // radius, packed box
  const float u = uv.x, v = uv.y, r = rb.x;
  if (__fsub_rn(x0, u) > r || __fsub_rn(u, x1) > r || __fsub_rn(y0, v) > r || __fsub_rn(v, y1) > r) return true;
  const uint32_t hb = __float_as_uint(rb.y);
  const __half2 h = *reinterpret_cast<const __half2*>(&hb);
  const float hx = __low2float(h), hy = __high2float(h);
  return hx < 0.0f || x0 - u > hx || u - x1 > hx || y0 - v > hy || v - y1 > hy;
}

// Forward compositing of one tile by the whole block (see the file comment).
template <int D, int B, bool kCount>
__device__ __forceinline__ void fwd_tile(const CompositeArgs& a, const int tile, unsigned char* smem, uint64_t* s_bar,
                                         int* s_abort, StageState& stg) {
  const int tid = threadIdx.x;
  const bool bf16 = a.feat_bf16 != 0;
  const uint32_t sbytes = stage_bytes(B, D, a.feat_bf16);
  float* s_wide = reinterpret_cast<float*>(smem + 2 * (size_t)sbytes);
  const int tx = tile % a.tiles_x, ty = tile / a.tiles_x;
  int lx, ly;
  tile_pixel(tid, a.tw, lx, ly);
  const int px = tx * a.tw + lx, py = ty * a.th + ly;
  const bool inside = px < a.W && py < a.H;
  const float pxc = (float)px + 0.5f, pyc = (float)py + 0.5f;
  const uint2 rg = a.ranges[tile];
  const uint32_t n = rg.y - rg.x;
  const uint32_t nbatch = (n + B - 1) / B;
  // Gaussian of this thread's slot in batch k (prefetched a batch ahead).
  auto slot_gid = [&](uint32_t k) -> uint32_t {
    const uint32_t p = k * B + (uint32_t)tid;
    return (k < nbatch && tid < B && p < n) ? a.sorted[rg.x + p].y : 0u;
  };
  auto batch_len = [&](uint32_t k) -> int { return (int)min((uint32_t)B, n - k * B); };
  uint32_t issued = 0;
  if (nbatch > 0) {
    stage_issue<D>(a, smem, B, batch_len(0), slot_gid(0), &s_bar[0]);
    issued = 1;
  }
  uint32_t g_next = slot_gid(1);
  float T = 1.0f, C0 = 0.f, C1 = 0.f, C2 = 0.f, Z = 0.f;
  float2 F[D / 2];  // feature channels in pairs (packed FP32 FMA)
#pragma unroll
  for (int d = 0; d < D / 2; ++d) F[d] = make_float2(0.0f, 0.0f);
  uint32_t last = 0;
  uint32_t visits = 0, contribs = 0;  // only used by the counting variant
  bool done = !inside;
  // Entries of the current batch this pixel blended, per 32-entry group
  // (up to four groups: B <= 128).
  constexpr int NG = B / 32;
  static_assert(NG >= 1 && NG <= 4, "blend masks cover at most four groups");
  uint32_t cm0 = 0u, cm1 = 0u, cm2 = 0u, cm3 = 0u;
  const bool track = !kCount && a.cmask != nullptr && a.aux;
  const size_t cslot0 = (size_t)(rg.x >> 5) + (size_t)tile;
  const int lane = tid & 31, warp = tid >> 5;
  // Pixel centres of this warp's 8 x 4 block.
  const float bx0 = (float)(tx * a.tw + ((warp % (a.tw >> 3)) << 3)) + 0.5f;
  const float by0 = (float)(ty * a.th + ((warp / (a.tw >> 3)) << 2)) + 0.5f;
  for (uint32_t k = 0; k < nbatch; ++k) {
    // Every thread is past batch k-1 here, so its buffer may be refilled.
    // A wait on batch k-1 that gave up (s_abort[(k-1) & 1], written before
    // this barrier; a failure in this iteration writes the other slot, so
    // no thread can see it change) ends the tile for the whole block before
    // anything is re-armed.
    if (__syncthreads_count(done) == kThreads || (k > 0 && ((volatile int*)s_abort)[(k - 1) & 1])) break;
    if (k + 1 < nbatch) {
      stage_issue<D>(a, smem + ((k + 1) & 1) * (size_t)sbytes, B, batch_len(k + 1), g_next, &s_bar[(k + 1) & 1]);
      issued = k + 2;
      g_next = slot_gid(k + 2);
    }
    const unsigned char* buf = smem + (k & 1) * (size_t)sbytes;
    const bool landed = mbar_wait(&s_bar[k & 1], stage_parity(stg, k), a.polls);
    if (!landed) {
      ((volatile int*)s_abort)[k & 1] = 1;
      set_err(a.err, kErrTimeout);
      done = true;
    }
    const int nb = batch_len(k);
    const float* s_rec = reinterpret_cast<const float*>(buf);
    const float* s_feat = reinterpret_cast<const float*>(buf + (size_t)B * kRec * 4);
    if (bf16) {
      // Every thread widens its share of the rows (also threads whose pixel
      // is outside the image or done), unless its wait gave up.
      if (landed) widen_bf16<D>(buf + (size_t)B * kRec * 4, s_wide, nb);
      __syncthreads();
      s_feat = s_wide;
    }
    uint32_t cur = 0u;  // blended entries of the current 32-entry group
    // Entries of each 32-entry group that some pixel of this warp's block
    // may blend (the others leave every pixel of the block unchanged).
    uint32_t em0 = 0u, em1 = 0u, em2 = 0u, em3 = 0u;
    if (!kCount && __any_sync(0xFFFFFFFFu, !done)) {
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        const int j = 32 * g + lane;
        const bool ev = j < nb && !block_misses(s_rec + j * kRec, bx0, bx0 + 7.0f, by0, by0 + 3.0f);
        const uint32_t m = __ballot_sync(0xFFFFFFFFu, ev);
        if (g == 0) em0 = m;
        if (g == 1) em1 = m;
        if (g == 2) em2 = m;
        if (g == 3) em3 = m;
      }
    }
    // Blend entry j (pe: its evaluation); true once the pixel is done.
    auto blend = [&](int j, const PairEval& pe) -> bool {
      const float* rec = s_rec + j * kRec;
      const float Tn = __fmul_rn(T, __fsub_rn(1.0f, pe.alpha));
      if (Tn < kTMin) {
        done = true;
        return true;
      }
      if (kCount) ++contribs;
      const float w = pe.alpha * T;
      C0 = fmaf(w, rec[7], C0);
      C1 = fmaf(w, rec[8], C1);
      C2 = fmaf(w, rec[9], C2);
      Z = fmaf(w, rec[6], Z);
      const float4* f4 = reinterpret_cast<const float4*>(s_feat + j * D);
      const float2 w2 = make_float2(w, w);
#pragma unroll
      for (int d4 = 0; d4 < D / 4; ++d4) {
        const float4 f = f4[d4];
        F[2 * d4] = __ffma2_rn(w2, make_float2(f.x, f.y), F[2 * d4]);
        F[2 * d4 + 1] = __ffma2_rn(w2, make_float2(f.z, f.w), F[2 * d4 + 1]);
      }
      T = Tn;
      last = k * B + (uint32_t)j + 1u;
      cur |= 1u << (j & 31);
      return false;
    };
    if (!done) {
      if (kCount) {
        // Counting form: every listed pair up to termination.
        for (int j = 0; j < nb; ++j) {
          PairEval pe;
          ++visits;
          if (eval_pair(s_rec + j * kRec, pxc, pyc, pe) && blend(j, pe)) break;
        }
      } else {
        // Groups of 32 entries; the entries the warp's block may blend are
        // taken in order, two at a time: both evaluated ahead of their
        // (ordered) blending -- the two evaluations are independent, only
        // the blend carries T.  One code path for full and half pairs and one
        // exit (a second path for a single last entry and breaks out of each
        // cost 5 to 14%: 30k Gaussians at 333 x 251, D = 16, 66 -> 57 us;
        // 90k, D = 128, 483 -> 453; 1M at 1280 x 1024, D = 64, 744 -> 717).
        // Bound by the latency of this loop (evaluation, then the blends in
        // order); four at a time are no faster, and evaluating a pair ahead
        // of the previous one's blends is slower (61 us for the 57).
        for (int g = 0; g < NG && !done; ++g) {
          uint32_t t = g == 0 ? em0 : g == 1 ? em1 : g == 2 ? em2 : em3;
          cur = 0u;
          while (t) {
            // Evaluations without early exits, so that they interleave
            // (identical arithmetic and decisions to eval_pair); a missing
            // second entry evaluates the group's first and is not blended.
            int j[2];
            bool h[2];
            PairEval pe[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const bool have = t != 0u;
              j[u] = 32 * g + (have ? __ffs(t) - 1 : 0);
              t &= t - 1u;
              h[u] = eval_pair_flat(s_rec + j[u] * kRec, pxc, pyc, pe[u]) && have;
            }
#pragma unroll
            for (int u = 0; u < 2; ++u)
              if (h[u] && blend(j[u], pe[u])) goto ended;
          }
        ended:
          cm0 |= g == 0 ? cur : 0u;
          if (NG > 1) cm1 |= g == 1 ? cur : 0u;
          if (NG > 2) cm2 |= g == 2 ? cur : 0u;
          if (NG > 3) cm3 |= g == 3 ? cur : 0u;
        }
      }
    }
    if (track) {
      // The warp's blended entries of each group of this batch.
#pragma unroll
      for (int g = 0; g < NG; ++g) {
        const uint32_t m = __reduce_or_sync(0xFFFFFFFFu, g == 0 ? cm0 : g == 1 ? cm1 : g == 2 ? cm2 : cm3);
        if (lane == 0 && k * B + 32u * g < n) a.cmask[(cslot0 + (k * B) / 32 + g) * 8 + warp] = m;
      }
      cm0 = cm1 = cm2 = cm3 = 0u;
    }
  }
  stage_drain(stg, s_bar, issued, a.err);
  if (kCount) {
    // Block sums of the pair counts, one 64-bit atomic per warp.
    unsigned long long v = visits, c = contribs;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
      c += __shfl_xor_sync(0xFFFFFFFFu, c, o);
    }
    if ((tid & 31) == 0) {
      atomicAdd(reinterpret_cast<unsigned long long*>(a.counts), v);
      atomicAdd(reinterpret_cast<unsigned long long*>(a.counts) + 1, c);
    }
    return;
  }
  if (inside) {
    const size_t HW = (size_t)a.W * a.H, p = (size_t)py * a.W + px;
    if (a.aux) {
      a.out_rgb[p] = C0 + T * a.bg[0];
      a.out_rgb[HW + p] = C1 + T * a.bg[1];
      a.out_rgb[2 * HW + p] = C2 + T * a.bg[2];
      a.out_depth[p] = Z;
      a.out_alpha[p] = 1.0f - T;
      a.t_final[p] = T;
      a.n_contrib[p] = last;
    }
    float4* fo = reinterpret_cast<float4*>(a.out_feat + p * a.out_ld);
#pragma unroll
    for (int d4 = 0; d4 < D / 4; ++d4) fo[d4] = make_float4(F[2 * d4].x, F[2 * d4].y, F[2 * d4 + 1].x, F[2 * d4 + 1].y);
    if (a.out_feat_bf16) {
      uint4* fb = reinterpret_cast<uint4*>(a.out_feat_bf16 + p * a.out_ld);
#pragma unroll
      for (int q = 0; q < D / 8; ++q) {
        uint32_t w4[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const __nv_bfloat162 h = __floats2bfloat162_rn(F[4 * q + e].x, F[4 * q + e].y);
          w4[e] = *reinterpret_cast<const uint32_t*>(&h);
        }
        fb[q] = make_uint4(w4[0], w4[1], w4[2], w4[3]);
      }
    }
  }
}

// Barriers and the abort flag of a compositing block, initialised once.
__device__ __forceinline__ void stage_init(uint64_t* s_bar) {
  if (threadIdx.x == 0) {
    mbar_init(&s_bar[0], 1);
    mbar_init(&s_bar[1], 1);
    mbar_init_fence();
  }
}

// One block per tile.
template <int D, int B, bool kCount, int NB>
__global__ void __launch_bounds__(kThreads, NB) composite_fwd_kernel(const CompositeArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ int s_abort[2];
  stage_init(s_bar);
  if (threadIdx.x == 0) s_abort[0] = s_abort[1] = 0;
  __syncthreads();
  grid_dep_wait();
  grid_dep_launch();
  StageState stg{{0u, 0u}, false};
  fwd_tile<D, B, kCount>(a, blockIdx.x, smem, s_bar, s_abort, stg);
}

// (view, tile) work item `item` of a batch: the view whose item range holds it.
__device__ __forceinline__ int batch_view(const BatchCompositeArgs& ba, int item) {
  int v = 0;
  while (v + 1 < ba.V && item >= ba.item_start[v + 1]) ++v;
  return v;
}

// Persistent form over a batch of views: each block takes (view, tile)
// items from a device counter until the batch is exhausted (no block waits
// for another: items are independent).
template <int D, int B, int NB>
__global__ void __launch_bounds__(kThreads, NB)
    composite_fwd_batch_kernel(const __grid_constant__ BatchCompositeArgs ba) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ int s_abort[2], s_item;
  stage_init(s_bar);
  grid_dep_wait();
  grid_dep_launch();
  StageState stg{{0u, 0u}, false};
  for (;;) {
    // Every thread is past the previous tile (its drain ended in a barrier).
    if (threadIdx.x == 0) {
      s_item = (int)atomicAdd(ba.queue, 1u);
      s_abort[0] = s_abort[1] = 0;
    }
    __syncthreads();
    const int item = s_item;
    if (item >= ba.nitems || stg.dead) break;
    const int v = batch_view(ba, item);
    fwd_tile<D, B, false>(ba.view[v], item - ba.item_start[v], smem, s_bar, s_abort, stg);
  }
}

// ---------------------------------------------------------------------------
// Reverse pass.  Per batch of 32 list entries (walked backwards), each warp
// takes the entries some pixel of its 8 x 4 block blended (the forward's
// masks), up to 16 at a time (a chunk), and forms three matrix products over
// them on the tensor cores (mma.sync, warp-local: no block barrier and no
// operand shared between warps but the staged entries):
//   S[entry][pixel]  = feature . feature gradient      (K = D channels)
//   P[entry][channel] = sum over pixels of w G           (K = 32 pixels)
//   M[entry][6]       = sum over pixels of e (1 x y xx xy yy)
// with w the blend weight, G the pixel's upstream gradient and e =
// dL/dalpha alpha.  Between S and the other two, each lane replays its
// pixel's recurrence over the chunk's entries (T_i = T_{i+1} / (1 - alpha_i)).
// The geometric sums of an entry (du .. dopacity) follow from its six
// moments M, taken about the centre of the warp's block, where the
// pixel coordinates and their products are exact in BF16.
//
// Every FP32 operand is carried as three BF16 terms x = hi + mid + lo (24
// significant bits) and a product as the six term products down to 2^-16 of
// |x||y|, smallest first, accumulated in FP32; a BF16-stored feature and the
// moments' coordinates are exact in one term (three products).
//
// The pass is bound by instruction issue and the latency of the few warps
// that its shared memory leaves room for.  With FP32 FMAs for the products
// and shuffles for the geometric sums an entry cost a warp 256 instructions
// at D = 32 (75 the product with G, 46 the geometric terms, 30 the feature
// dot), now about 180; at D = 128 the gradient rows had to be re-read from
// shared memory for every entry.  Measured, before and now: 200k Gaussians at
// 640 x 512, D = 32: 365 -> 330 us; 90k, D = 128: 1520 -> 1345 us; 1M at
// 1280 x 1024, D = 64 BF16: 2135 -> 1811 us; eight views of 100k, D = 32
// BF16, in one launch: 1960 -> 1528 us.  At D = 32 the second block per SM costs
// 56 bytes of spills; one block takes 976 us for the 842 of a whole forward and
// reverse (200k).  (tcgen05 products over the whole
// tile were costed: they take every entry of a batch for every pixel where a
// warp needs half of them, and their operands in three terms leave one block
// per SM at D = 32 too.)
template <int D>
struct BwdCfg {
  static_assert(D == 16 || D == 32 || D == 64, "channels of one reverse pass");
  static constexpr int B = 32;          // entries per batch
  static constexpr int CH = 16;         // entries per chunk (MMA rows)
  static constexpr int KS = D / 16;     // K steps of S
  static constexpr int NT = D / 8;      // channel tiles of P (one more for colour and depth)
  static constexpr int SS = 36;         // row stride of the [entry][pixel] slices (floats)
  static constexpr int PR = D + 12;     // a warp's partial row: features | du dv dA dB dCc dopacity r g b depth 0 0
  // A warp's area (floats): its partial rows of the batch from the start,
  // and the two slices of the chunk in flight (S, overwritten by w; e) at
  // the end, which end up under the chunk's own rows.  A later chunk of the
  // batch takes at most as many entries as the place behind the rows so far
  // has slices for: 16 at D = 16 and 64; at D = 32, where two blocks per SM
  // leave less, 26 entries are two chunks and 32 are four (of the synthetic
  // scenes' warps and batches under 5% have more than 26).
  static constexpr int AREA = D == 16 ? CH * PR + 2 * CH * SS : D == 32 ? 1472 : B * PR;
  static_assert(AREA >= B * PR && AREA >= 2 * CH * SS && AREA % 4 == 0, "partial rows and slices of a warp");
  // Upstream gradients of a warp's pixels, per term [channel][32 pixels]
  // BF16 (64-byte rows, 16-byte chunk t of row c at t ^ ((c >> 2) & 3): the
  // fragment loads below touch every bank once).
  static constexpr int GTERM = (D + 4) * 64;
  static constexpr int GWARP = 3 * GTERM;
  static constexpr size_t off_G = 0;
  static constexpr size_t off_area = off_G + (size_t)8 * GWARP;
  static constexpr size_t off_stage = (off_area + (size_t)8 * AREA * 4 + 127) / 128 * 128;
  __host__ __device__ static constexpr size_t off_e(int bf16) { return off_stage + 2 * (size_t)stage_bytes(B, D, bf16); }
  // List entries of the two staged batches, the warps' entry masks, the
  // warps' entry lists.
  __host__ __device__ static constexpr size_t smem_bytes(int bf16) { return off_e(bf16) + (size_t)(2 * B + 8 + 8 * B) * 4; }
};

static_assert(BwdCfg<64>::smem_bytes(0) <= 232448, "reverse compositing shared memory per block");
static_assert(2 * (BwdCfg<32>::smem_bytes(0) + 128 + 1024) <= 233472, "two reverse blocks per SM at D <= 32");

// 1 / x by the hardware approximation (about 1 ulp).
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Terms (of the first operand, of the second) of the six products, smallest first.
__device__ constexpr int kTermA[6] = {2, 1, 0, 1, 0, 0};
__device__ constexpr int kTermB[6] = {0, 1, 2, 0, 1, 0};

// Byte offset of 16-byte chunk t (pixels 8 t .. 8 t + 7) of row c of a term.
__device__ __forceinline__ uint32_t g_chunk(int c, int t) { return (uint32_t)(c * 64 + ((t ^ ((c >> 2) & 3)) << 4)); }

// Reverse compositing of one tile by the whole block.
template <int D>
__device__ __forceinline__ void bwd_tile(const CompositeArgs& a, const int tile, unsigned char* smem, uint64_t* s_bar,
                                         int* s_abort, StageState& stg) {
  using K = BwdCfg<D>;
  constexpr int B = K::B, CH = K::CH, SS = K::SS, PR = K::PR, KS = K::KS, NT = K::NT;
  const bool bf16 = a.feat_bf16 != 0;
  const uint32_t sbytes = stage_bytes(B, D, a.feat_bf16);
  float* s_area = reinterpret_cast<float*>(smem + K::off_area);  // [8][AREA]
  unsigned char* s_stage = smem + K::off_stage;                   // [2][sbytes]
  uint32_t* s_e = reinterpret_cast<uint32_t*>(smem + K::off_e(a.feat_bf16));  // [2][B]
  uint32_t* s_jact = s_e + 2 * B;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  uint32_t* s_list = s_jact + 8 + warp * B;  // this warp's entries of the batch, latest first
  unsigned char* s_G = smem + K::off_G + warp * K::GWARP;
  float* area = s_area + warp * K::AREA;
  const int tx = tile % a.tiles_x, ty = tile / a.tiles_x;
  int lx, ly;
  tile_pixel(tid, a.tw, lx, ly);
  const int px = tx * a.tw + lx, py = ty * a.th + ly;
  const bool inside = px < a.W && py < a.H;
  const float pxc = (float)px + 0.5f, pyc = (float)py + 0.5f;
  const size_t HW = (size_t)a.W * a.H, pix = inside ? (size_t)py * a.W + px : 0;
  const uint2 rg = a.ranges[tile];
  const float Tf = inside ? a.t_final[pix] : 1.0f;
  const uint32_t nc = inside ? a.n_contrib[pix] : 0u;
  // Upstream gradients of this pixel: every load is issued before the first
  // is used, and the first batches are on their way before the split below.
  float g0 = 0.f, g1 = 0.f, g2 = 0.f, gz = 0.f, ga = 0.f;
  if (inside) {
    if (a.g_rgb) { g0 = a.g_rgb[pix]; g1 = a.g_rgb[HW + pix]; g2 = a.g_rgb[2 * HW + pix]; }
    if (a.g_depth) gz = a.g_depth[pix];
    if (a.g_alpha) ga = a.g_alpha[pix];
  }
  float4 gf[D / 4];
  {
    const bool has = inside && a.g_feat != nullptr;
    const float4* src = reinterpret_cast<const float4*>(a.g_feat + (has ? pix * a.out_ld : 0));
#pragma unroll
    for (int d4 = 0; d4 < D / 4; ++d4) gf[d4] = has ? __ldg(src + d4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  const uint32_t wmax = __reduce_max_sync(0xFFFFFFFFu, nc);
  if (lane == 0) s_jact[warp] = wmax;
  __syncthreads();
  // Batches aligned to multiples of B from the tile start, walked backwards
  // from the largest n_contrib (the first one processed, the last in list
  // order, may be short).
  uint32_t n = 0;
#pragma unroll
  for (int w8 = 0; w8 < 8; ++w8) n = max(n, s_jact[w8]);
  const uint32_t nbatch = (n + B - 1) / B;
  auto batch_lo = [&](uint32_t k) -> uint32_t { return (nbatch - 1 - k) * (uint32_t)B; };
  auto batch_len = [&](uint32_t k) -> int { return (int)min((uint32_t)B, n - batch_lo(k)); };
  const size_t cslot0 = (size_t)(rg.x >> 5) + (size_t)tile;
  // List entry and Gaussian of this thread's slot in batch k.
  auto slot = [&](uint32_t k, uint32_t& e, uint32_t& g) {
    e = 0u;
    g = 0u;
    if (k < nbatch && tid < batch_len(k)) {
      const uint32_t p = rg.x + batch_lo(k) + (uint32_t)tid;
      const uint2 eg = a.sorted[p];
      e = eg.x;
      g = eg.y;
    }
  };
  // The forward's blend mask of this warp for batch k: the entries some
  // pixel of its block blended (read a batch ahead, so its global latency
  // overlaps the previous batch).
  auto mask_word = [&](uint32_t k) -> uint32_t {
    return (k < nbatch && batch_lo(k) < wmax) ? a.cmask[(cslot0 + batch_lo(k) / 32) * 8 + warp] : 0u;
  };
  uint32_t mask_next = mask_word(0);
  uint32_t e_next, g_next;
  slot(0, e_next, g_next);
  uint32_t issued = 0;
  if (nbatch > 0) {
    stage_issue<D>(a, s_stage, B, batch_len(0), g_next, &s_bar[0]);
    if (tid < B) s_e[tid] = e_next;
    issued = 1;
  }
  slot(1, e_next, g_next);
  // The gradients as the warp's operand rows (features, then r g b depth).
  auto put_pair = [&](int c, float x, float y) {  // rows c and c + 1, this lane's pixel
    uint32_t t3[3];
    split3(x, y, t3[0], t3[1], t3[2]);
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      unsigned char* p = s_G + t * K::GTERM + 2 * (lane & 7);
      *reinterpret_cast<uint16_t*>(p + g_chunk(c, lane >> 3)) = (uint16_t)(t3[t] & 0xFFFFu);
      *reinterpret_cast<uint16_t*>(p + g_chunk(c + 1, lane >> 3)) = (uint16_t)(t3[t] >> 16);
    }
  };
#pragma unroll
  for (int d4 = 0; d4 < D / 4; ++d4) {
    put_pair(4 * d4, gf[d4].x, gf[d4].y);
    put_pair(4 * d4 + 2, gf[d4].z, gf[d4].w);
  }
  put_pair(D, g0, g1);
  put_pair(D + 2, g2, gz);
  __syncwarp();
  float T = Tf;
  float Q = (g0 * a.bg[0] + g1 * a.bg[1] + g2 * a.bg[2]) * Tf;
  const float gaTf = ga * Tf;
  // Fragment coordinates of this lane: rows fr and fr + 8, columns 2 ft and
  // 2 ft + 1 of an accumulator.
  const int fr = lane >> 2, ft = lane & 3;
  // S: the second operand G[channel][pixel], read transposed.  K index
  // 2 t + e (+ 8 h) of a step is channel 4 t + 2 h + e, so that a lane's four
  // first-operand values of a row are one 16-byte load.
  const uint32_t g_addr = smem_addr(s_G);
  const int lm_c = 4 * ((lane & 7) >> 1) + 2 * ((lane >> 3) & 1) + (lane & 1), lm_t = lane >> 4;
  // Moments: the second operand, moment fr of pixels 8 ft + i (row ft of the
  // block, column i), about the block's centre.  K index 2 t + e (+ 8 h) of
  // step s is pixel 8 t + 4 s + 2 h + e, for P and M alike.
  uint32_t mom[4];
  {
    const float y = (float)ft - 1.5f;
    auto moment = [&](int i) -> float {
      const float x = (float)i - 3.5f;
      return fr == 0 ? 1.0f : fr == 1 ? x : fr == 2 ? y : fr == 3 ? x * x : fr == 4 ? x * y : fr == 5 ? y * y : 0.0f;
    };
#pragma unroll
    for (int i = 0; i < 4; ++i) mom[i] = pack_bf16(moment(2 * i), moment(2 * i + 1));
  }
  // Centre of this warp's block.
  const float cxw = (float)(tx * a.tw + ((warp % (a.tw >> 3)) << 3)) + 4.0f;
  const float cyw = (float)(ty * a.th + ((warp / (a.tw >> 3)) << 2)) + 2.0f;
  for (uint32_t k = 0; k < nbatch; ++k) {
    // Every thread is past batch k-1 (and its combine) here.  A wait on
    // batch k-1 that gave up ends the tile for the whole block (the flag
    // slots alternate by batch, as in the forward).
    __syncthreads();
    if (k > 0 && ((volatile int*)s_abort)[(k - 1) & 1]) break;
    if (k + 1 < nbatch) {
      stage_issue<D>(a, s_stage + ((k + 1) & 1) * (size_t)sbytes, B, batch_len(k + 1), g_next, &s_bar[(k + 1) & 1]);
      if (tid < B) s_e[((k + 1) & 1) * B + tid] = e_next;
      issued = k + 2;
      slot(k + 2, e_next, g_next);
    }
    bool live = true;
    if (!mbar_wait(&s_bar[k & 1], stage_parity(stg, k), a.polls)) {
      ((volatile int*)s_abort)[k & 1] = 1;
      set_err(a.err, kErrTimeout);
      live = false;
    }
    const unsigned char* buf = s_stage + (k & 1) * (size_t)sbytes;
    const float* s_rec = reinterpret_cast<const float*>(buf);
    const unsigned char* s_feat = buf + (size_t)B * kRec * 4;  // rows as stored (fp32 or bf16)
    const int nb = batch_len(k);
    const uint32_t rel0 = batch_lo(k);
    const uint32_t jact = mask_next & (nb >= 32 ? 0xFFFFFFFFu : ((1u << nb) - 1u));
    mask_next = mask_word(k + 1);
    const int cnt = __popc(jact);
    if (cnt > 0) {
      // Entry list, latest first: slot = number of later entries.
      if ((jact >> lane) & 1u) s_list[__popc((jact >> lane) >> 1)] = (uint32_t)lane;
      __syncwarp();
    }
    uint32_t todo = jact;
    for (int c0 = 0, m; c0 < cnt; c0 += m) {
      m = min(min(CH, cnt - c0), (K::AREA - c0 * PR) / (2 * SS));  // entries of this chunk
      float* sl_w = area + (K::AREA - 2 * SS * m);  // [m][SS]: S, then w
      float* sl_e = sl_w + SS * m;                  // [m][SS]: e
      // ---- S[entry][pixel] ----
      {
        // First operand: the feature rows of entries fr and fr + 8 (slots past
        // the chunk repeat its last entry; their results are not used).
        const int ra = (int)s_list[c0 + min(fr, m - 1)], rb = (int)s_list[c0 + min(fr + 8, m - 1)];
        uint32_t xa[3][KS][4];
        if (bf16) {
#pragma unroll
          for (int ks = 0; ks < KS; ++ks) {
            const uint2 va = *reinterpret_cast<const uint2*>(s_feat + ra * (2 * D) + 32 * ks + 8 * ft);
            const uint2 vb = *reinterpret_cast<const uint2*>(s_feat + rb * (2 * D) + 32 * ks + 8 * ft);
            xa[0][ks][0] = va.x; xa[0][ks][2] = va.y; xa[0][ks][1] = vb.x; xa[0][ks][3] = vb.y;
          }
        } else {
#pragma unroll
          for (int ks = 0; ks < KS; ++ks) {
            const float4 va = *reinterpret_cast<const float4*>(s_feat + ra * (4 * D) + 64 * ks + 16 * ft);
            const float4 vb = *reinterpret_cast<const float4*>(s_feat + rb * (4 * D) + 64 * ks + 16 * ft);
            split3(va.x, va.y, xa[0][ks][0], xa[1][ks][0], xa[2][ks][0]);
            split3(va.z, va.w, xa[0][ks][2], xa[1][ks][2], xa[2][ks][2]);
            split3(vb.x, vb.y, xa[0][ks][1], xa[1][ks][1], xa[2][ks][1]);
            split3(vb.z, vb.w, xa[0][ks][3], xa[1][ks][3], xa[2][ks][3]);
          }
        }
        // The four pixel tiles' chains run side by side.
        float sa[4][4];
        auto step = [&](int tx, int tg, int ks, bool first) {
          uint32_t v[2][4];
          ldmatrix_x4_trans(g_addr + tg * K::GTERM + g_chunk(16 * ks + lm_c, lm_t), v[0]);
          ldmatrix_x4_trans(g_addr + tg * K::GTERM + g_chunk(16 * ks + lm_c, 2 + lm_t), v[1]);
#pragma unroll
          for (int pt = 0; pt < 4; ++pt) {
            const uint32_t b0 = v[pt >> 1][2 * (pt & 1)], b1 = v[pt >> 1][2 * (pt & 1) + 1];
            if (first) mma_bf16_16816_first(sa[pt], xa[tx][ks], b0, b1);
            else mma_bf16_16816(sa[pt], xa[tx][ks], b0, b1);
          }
        };
        if (bf16) {
#pragma unroll
          for (int t = 2; t >= 0; --t)
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) step(0, t, ks, t == 2 && ks == 0);
        } else {
#pragma unroll
          for (int p = 0; p < 6; ++p)
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) step(kTermA[p], kTermB[p], ks, p == 0 && ks == 0);
        }
#pragma unroll
        for (int pt = 0; pt < 4; ++pt) {
          float* o = sl_w + fr * SS + 8 * pt + 2 * ft;
          if (fr < m) *reinterpret_cast<float2*>(o) = make_float2(sa[pt][0], sa[pt][1]);
          if (fr + 8 < m) *reinterpret_cast<float2*>(o + 8 * SS) = make_float2(sa[pt][2], sa[pt][3]);
        }
      }
      __syncwarp();
      // ---- replay of the chunk's entries, two at a time ----
      // Entries of this batch the pixel reached (none if the wait gave up).
      const uint32_t nc_rel = live && nc > rel0 ? nc - rel0 : 0u;
      float clamp_sum = 0.0f;  // lane q: opacity sum of slot q's clamped pixels
      auto evaluate = [&](int j, PairEval& pe) -> bool {
        const bool h = eval_pair_flat(s_rec + j * kRec, pxc, pyc, pe);
        return h & ((uint32_t)j < nc_rel);
      };
      // Entry j (slot q of the chunk) given its evaluation (hit: the pixel
      // includes it), without branches so that the two entries of a pair
      // interleave: a lane that did not blend takes alpha = 0, which leaves
      // T and Q exactly as they were (1 / (1 - 0) = 1, w = 0).
      auto entry = [&](int j, int q, bool hit, const PairEval& pe) {
        const float2 zr = *reinterpret_cast<const float2*>(s_rec + j * kRec + 6);  // depth, r
        const float2 gbl = *reinterpret_cast<const float2*>(s_rec + j * kRec + 8);  // g, b
        float s = sl_w[q * SS + lane];
        s = fmaf(zr.x, gz, fmaf(zr.y, g0, s)) + fmaf(gbl.x, g1, gbl.y * g2);
        const float al = hit ? pe.alpha : 0.0f;
        const float inv = rcp_approx(1.0f - al);  // 1 - alpha >= 0.01
        T = T * inv;  // transmittance before this Gaussian
        const float w = al * T;
        const float dalpha = T * s - (Q - gaTf) * inv;
        Q = fmaf(w, s, Q);
        sl_w[q * SS + lane] = w;
        sl_e[q * SS + lane] = hit && !pe.clamped ? dalpha * pe.alpha : 0.0f;
        const bool over = hit && pe.clamped;
        if (__any_sync(0xFFFFFFFFu, over)) {
          // Pixels whose alpha was clamped add to the opacity sum alone.
          float v = over ? dalpha * pe.G : 0.0f;
#pragma unroll
          for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
          if (lane == q) clamp_sum = v;
        }
      };
      int q = 0;
      for (; q + 1 < m; q += 2) {
        const int ja = 31 - __clz(todo);
        todo &= ~(1u << ja);
        const int jb = 31 - __clz(todo);
        todo &= ~(1u << jb);
        PairEval pa, pb;
        const bool ha = evaluate(ja, pa);
        const bool hb = evaluate(jb, pb);
        entry(ja, q, ha, pa);
        entry(jb, q + 1, hb, pb);
      }
      if (q < m) {
        const int ja = 31 - __clz(todo);
        todo &= ~(1u << ja);
        PairEval pa;
        const bool ha = evaluate(ja, pa);
        entry(ja, q, ha, pa);
      }
      __syncwarp();
      // ---- P[entry][channel] and M[entry][moment] ----
      // First operands: rows fr and fr + 8 of the slices (slots past the
      // chunk repeat its last entry or are zero; their results are not used).
      auto load_rows = [&](const float* sl, uint32_t (&v)[3][2][4]) {
#pragma unroll
        for (int s = 0; s < 2; ++s) {
          const float4 va = *reinterpret_cast<const float4*>(sl + min(fr, m - 1) * SS + 8 * ft + 4 * s);
          split3(va.x, va.y, v[0][s][0], v[1][s][0], v[2][s][0]);
          split3(va.z, va.w, v[0][s][2], v[1][s][2], v[2][s][2]);
          if (m > 8) {
            const float4 vb = *reinterpret_cast<const float4*>(sl + min(fr + 8, m - 1) * SS + 8 * ft + 4 * s);
            split3(vb.x, vb.y, v[0][s][1], v[1][s][1], v[2][s][1]);
            split3(vb.z, vb.w, v[0][s][3], v[1][s][3], v[2][s][3]);
          } else {
#pragma unroll
            for (int t = 0; t < 3; ++t) v[t][s][1] = v[t][s][3] = 0u;
          }
        }
      };
      float mo[4] = {0.f, 0.f, 0.f, 0.f};
      {
        uint32_t ea[3][2][4];
        load_rows(sl_e, ea);
#pragma unroll
        for (int t = 2; t >= 0; --t)
#pragma unroll
          for (int s = 0; s < 2; ++s) mma_bf16_16816(mo, ea[t][s], mom[2 * s], mom[2 * s + 1]);
      }
      uint32_t wa[3][2][4];
      load_rows(sl_w, wa);
      __syncwarp();  // every lane has its rows: partial rows may take their place
      // Channel tiles, then colour and depth as four more channels (columns
      // 4-7 of their tile zero).
      float acc[NT + 1][4];
      // The tiles' chains run side by side.
#pragma unroll
      for (int p = 0; p < 6; ++p) {
        uint4 g[NT + 1];
#pragma unroll
        for (int nt = 0; nt <= NT; ++nt)
          g[nt] = nt < NT || fr < 4 ? *reinterpret_cast<const uint4*>(s_G + kTermB[p] * K::GTERM + g_chunk(8 * nt + fr, ft))
                                    : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int nt = 0; nt <= NT; ++nt) {
          if (p == 0) mma_bf16_16816_first(acc[nt], wa[kTermA[p]][0], g[nt].x, g[nt].y);
          else mma_bf16_16816(acc[nt], wa[kTermA[p]][0], g[nt].x, g[nt].y);
        }
#pragma unroll
        for (int nt = 0; nt <= NT; ++nt) mma_bf16_16816(acc[nt], wa[kTermA[p]][1], g[nt].z, g[nt].w);
      }
      // Geometric sums of rows fr and fr + 8 from their moments (spread over
      // the quad: lane ft holds moments 2 ft and 2 ft + 1): two columns to a
      // lane.
      float2 geo[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float lo = mo[2 * h], hi = mo[2 * h + 1];
        const float m0 = __shfl_sync(0xFFFFFFFFu, lo, 0, 4), mx = __shfl_sync(0xFFFFFFFFu, hi, 0, 4);
        const float my = __shfl_sync(0xFFFFFFFFu, lo, 1, 4), mxx = __shfl_sync(0xFFFFFFFFu, hi, 1, 4);
        const float mxy = __shfl_sync(0xFFFFFFFFu, lo, 2, 4), myy = __shfl_sync(0xFFFFFFFFu, hi, 2, 4);
        const int r = fr + 8 * h;
        const float cl = __shfl_sync(0xFFFFFFFFu, clamp_sum, r);
        const float* rec = s_rec + s_list[c0 + min(r, m - 1)] * kRec;
        const float4 r0 = *reinterpret_cast<const float4*>(rec);      // u, v, A, B
        const float2 r4 = *reinterpret_cast<const float2*>(rec + 4);  // Cc, opacity
        const float ox = cxw - r0.x, oy = cyw - r0.y;
        // Sums of e dx^i dy^j, dx = x + ox, dy = y + oy.
        const float ex = fmaf(ox, m0, mx), ey = fmaf(oy, m0, my);
        const float exx = fmaf(ox, mx + ex, mxx);
        const float exy = fmaf(ox, my, fmaf(oy, ex, mxy));
        const float eyy = fmaf(oy, my + ey, myy);
        // power2 = log2(alpha / opacity): dL/dpower2 = e ln 2.
        if (ft == 0) geo[h] = make_float2(-kLn2 * fmaf(2.0f * r0.z, ex, r0.w * ey), -kLn2 * fmaf(2.0f * r4.x, ey, r0.w * ex));
        else if (ft == 1) geo[h] = make_float2(kLn2 * exx, kLn2 * exy);
        else geo[h] = make_float2(kLn2 * eyy, __fdividef(m0, r4.y) + cl);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (fr + 8 * h < m) {
          float* row = area + (c0 + fr + 8 * h) * PR + 2 * ft;
#pragma unroll
          for (int nt = 0; nt < NT; ++nt)
            *reinterpret_cast<float2*>(row + 8 * nt) = make_float2(acc[nt][2 * h], acc[nt][2 * h + 1]);
          if (ft < 3) {
            // du dv | dA dB | dCc dopacity, then r g | b depth | 0 0.
            *reinterpret_cast<float2*>(row + D) = geo[h];
            *reinterpret_cast<float2*>(row + D + 6) = make_float2(acc[NT][2 * h], acc[NT][2 * h + 1]);
          }
        }
      }
      __syncwarp();  // the area may be written again
    }
    if (lane == 0) s_jact[warp] = jact;
    __syncthreads();
    // Fixed-order sum of the warp partials: one row per (tile, entry) that
    // some pixel of the tile blended (the other rows stay unwritten and
    // unflagged, i.e. zero).
    const uint32_t* se = s_e + (k & 1) * B;
    uint32_t jm[8], bm = 0;
#pragma unroll
    for (int w8 = 0; w8 < 8; ++w8) {
      jm[w8] = s_jact[w8];
      bm |= jm[w8];
    }
    // A group of lanes takes one active entry at a time, each lane four
    // consecutive columns of its partial row [features | du dv dA dB dCc
    // dopacity | r g b | depth | 0 0]: the warps' rows of that entry (in warp
    // w at the number of its later entries) summed in warp order, one 16-byte
    // store.  A channel-split pass that is not the first adds its geometric
    // terms (du .. dopacity) to the row the first pass wrote and leaves
    // colour and depth (the last four columns) alone.
    constexpr int NQ = PR / 4, GL = NQ <= 8 ? 8 : NQ <= 16 ? 16 : 32;
    const int q4 = tid % GL;
    const bool col = q4 < NQ && (a.aux || q4 < NQ - 1);
    for (int j = tid / GL; j < B; j += kThreads / GL) {
      if (!((bm >> j) & 1u) || !col) continue;
      const float* src = s_area + 4 * q4;
      float4 acc = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int w8 = 0; w8 < 8; ++w8) {
        const uint32_t later = jm[w8] >> j;
        float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        if (later & 1u) v = *reinterpret_cast<const float4*>(src + w8 * K::AREA + __popc(later >> 1) * PR);
        acc.x += v.x;
        acc.y += v.y;
        acc.z += v.z;
        acc.w += v.w;
      }
      if ((int64_t)se[j] < a.cap) {
        float* row = a.partials + (size_t)se[j] * a.prow;
        float4* dst = reinterpret_cast<float4*>(q4 < D / 4 ? row + a.pcol0 + 4 * q4 : row + a.pscal + 4 * (q4 - D / 4));
        if (!a.aux && q4 >= D / 4) {
          const float4 prev = *dst;
          acc.x += prev.x;
          acc.y += prev.y;
          if (q4 == D / 4) {
            acc.z += prev.z;
            acc.w += prev.w;
          } else {
            acc.z = prev.z;  // colour: the first pass's
            acc.w = prev.w;
          }
        }
        *dst = acc;
      }
    }
    if (tid < nb && ((bm >> tid) & 1u) && (int64_t)se[tid] < a.cap)
      atomicOr(a.pflags + (se[tid] >> 5), 1u << (se[tid] & 31u));
  }
  stage_drain(stg, s_bar, issued, a.err);
}

// One block per tile.
template <int D>
__global__ void __launch_bounds__(kThreads, D <= 32 ? 2 : 1) composite_bwd_kernel(const CompositeArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ int s_abort[2];
  stage_init(s_bar);
  if (threadIdx.x == 0) s_abort[0] = s_abort[1] = 0;
  __syncthreads();
  grid_dep_wait();
  grid_dep_launch();
  StageState stg{{0u, 0u}, false};
  bwd_tile<D>(a, blockIdx.x, smem, s_bar, s_abort, stg);
}

// Persistent form over a batch of views, as the forward's.
template <int D>
__global__ void __launch_bounds__(kThreads, D <= 32 ? 2 : 1)
    composite_bwd_batch_kernel(const __grid_constant__ BatchCompositeArgs ba) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t s_bar[2];
  __shared__ int s_abort[2], s_item;
  stage_init(s_bar);
  grid_dep_wait();
  grid_dep_launch();
  StageState stg{{0u, 0u}, false};
  for (;;) {
    if (threadIdx.x == 0) {
      s_item = (int)atomicAdd(ba.queue, 1u);
      s_abort[0] = s_abort[1] = 0;
    }
    __syncthreads();
    const int item = s_item;
    if (item >= ba.nitems || stg.dead) break;
    const int v = batch_view(ba, item);
    bwd_tile<D>(ba.view[v], item - ba.item_start[v], smem, s_bar, s_abort, stg);
  }
}

template <int D, int B, bool kCount, int NB = fwd_blocks<D>()>
cudaError_t launch_fwd_t(const CompositeArgs& a, cudaStream_t st) {
  const size_t smem = fwd_smem_bytes(B, D, a.feat_bf16);
  auto k = composite_fwd_kernel<D, B, kCount, NB>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  return launch_pdl(k, a.ntiles, kThreads, smem, st, a);
}

// Batch sizes: 32, 64, 128 Gaussians (128 only up to D = 64); the counting
// form runs with the default batch only.
template <int D>
cudaError_t launch_fwd_d(const CompositeArgs& a, int B, cudaStream_t st) {
  if (a.counts && B == 0) B = fwd_batch<D>();
  if (B == 0) B = fwd_batch_for<D>(a.ntiles);
  if (a.counts) return B == fwd_batch<D>() ? launch_fwd_t<D, fwd_batch<D>(), true>(a, st) : cudaErrorInvalidValue;
  switch (B) {
    case 32: return launch_fwd_t<D, 32, false>(a, st);
    case 64: return launch_fwd_t<D, 64, false>(a, st);
    case 128:
      if constexpr (D == 16) {
        if (a.ntiles <= kTwoBlockTiles) return launch_fwd_t<D, 128, false, 2>(a, st);
      }
      if constexpr (D <= 64) return launch_fwd_t<D, 128, false>(a, st);
      break;
  }
  return cudaErrorInvalidValue;
}

template <int D>
cudaError_t launch_bwd_t(const CompositeArgs& a, cudaStream_t st) {
  const size_t smem = BwdCfg<D>::smem_bytes(a.feat_bf16);
  auto k = composite_bwd_kernel<D>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  return launch_pdl(k, a.ntiles, kThreads, smem, st, a);
}

// Grid of a persistent launch: as many blocks as fit on the GPU at once
// (occupancy x SMs), never more than there are work items.
template <typename Kern>
cudaError_t persistent_grid(Kern k, size_t smem, int nitems, int& grid) {
  int dev = 0, sms = 0, per_sm = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, kThreads, smem);
  if (e != cudaSuccess) return e;
  grid = per_sm * sms;
  if (grid > nitems) grid = nitems;
  if (grid < 1) grid = 1;
  return cudaSuccess;
}

template <int D, int B, int NB = fwd_blocks<D>()>
cudaError_t launch_fwd_batch_t(const BatchCompositeArgs& b, int bf16, cudaStream_t st) {
  const size_t smem = fwd_smem_bytes(B, D, bf16);
  auto k = composite_fwd_batch_kernel<D, B, NB>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int grid = 1;
  if (e == cudaSuccess) e = persistent_grid(k, smem, b.nitems, grid);
  if (e != cudaSuccess) return e;
  return launch_pdl(k, grid, kThreads, smem, st, b);
}

template <int D>
cudaError_t launch_fwd_batch_d(const BatchCompositeArgs& b, int bf16, int B, cudaStream_t st) {
  if (B == 0) B = fwd_batch_for<D>(b.nitems);
  switch (B) {
    case 32: return launch_fwd_batch_t<D, 32>(b, bf16, st);
    case 64: return launch_fwd_batch_t<D, 64>(b, bf16, st);
    case 128:
      if constexpr (D == 16) {
        if (b.nitems <= kTwoBlockTiles) return launch_fwd_batch_t<D, 128, 2>(b, bf16, st);
      }
      if constexpr (D <= 64) return launch_fwd_batch_t<D, 128>(b, bf16, st);
      break;
  }
  return cudaErrorInvalidValue;
}

template <int D>
cudaError_t launch_bwd_batch_t(const BatchCompositeArgs& b, int bf16, cudaStream_t st) {
  const size_t smem = BwdCfg<D>::smem_bytes(bf16);
  auto k = composite_bwd_batch_kernel<D>;
  cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  int grid = 1;
  if (e == cudaSuccess) e = persistent_grid(k, smem, b.nitems, grid);
  if (e != cudaSuccess) return e;
  return launch_pdl(k, grid, kThreads, smem, st, b);
}

// Wide features run as several passes over `width` channels each (part h of
// them): the same list, the same per-pixel decisions, each pass staging and
// accumulating its part of every feature row.  Part 0 owns colour, depth,
// alpha, T_final, n_contrib, the blend masks and (reverse) the colour / depth
// / alpha / background terms; the reverse's geometric terms are linear in the
// dot products g . x, so a later part adds the share of its channels to the
// rows the earlier ones wrote (same stream, in order: a fixed order).  The
// forward takes 128 channels a pass, the reverse 64 (its operands of 128
// channels do not fit in shared memory; two 64-channel passes repeat the
// evaluation and the replay but not the products, which dominate).
CompositeArgs channel_part(const CompositeArgs& a, int width, int h) {
  CompositeArgs c = a;
  const size_t elem = a.feat_bf16 ? 2 : 4;
  c.D = width;
  c.feat = static_cast<const unsigned char*>(a.feat) + (size_t)h * width * elem;
  if (a.out_feat) c.out_feat = a.out_feat + h * width;
  if (a.out_feat_bf16) c.out_feat_bf16 = a.out_feat_bf16 + h * width;
  if (a.g_feat) c.g_feat = a.g_feat + h * width;
  c.pcol0 = a.pcol0 + h * width;
  if (h > 0) {
    c.aux = 0;
    c.g_rgb = c.g_depth = c.g_alpha = nullptr;
  }
  return c;
}
constexpr int kFwdPart = 128, kBwdPart = 64;

}  // namespace

bool fwd_batch_supported(int B) { return B == 0 || B == 32 || B == 64 || B == 128; }

cudaError_t launch_composite_fwd(const CompositeArgs& a, int fwd_batch, cudaStream_t st) {
  if (a.ntiles <= 0) return cudaSuccess;
  switch (a.D) {
    case 16: return launch_fwd_d<16>(a, fwd_batch, st);
    case 32: return launch_fwd_d<32>(a, fwd_batch, st);
    case 64: return launch_fwd_d<64>(a, fwd_batch, st);
    case 128: return launch_fwd_d<128>(a, fwd_batch, st);
    case 256: {
      const cudaError_t e = launch_fwd_d<128>(channel_part(a, kFwdPart, 0), fwd_batch, st);
      if (e != cudaSuccess || a.counts) return e;
      return launch_fwd_d<128>(channel_part(a, kFwdPart, 1), fwd_batch, st);
    }
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_composite_bwd(const CompositeArgs& a, cudaStream_t st) {
  if (a.ntiles <= 0) return cudaSuccess;
  switch (a.D) {
    case 16: return launch_bwd_t<16>(a, st);
    case 32: return launch_bwd_t<32>(a, st);
    case 64: return launch_bwd_t<64>(a, st);
    case 128:
    case 256: {
      cudaError_t e = cudaSuccess;
      for (int h = 0; h < a.D / kBwdPart && e == cudaSuccess; ++h) e = launch_bwd_t<64>(channel_part(a, kBwdPart, h), st);
      return e;
    }
  }
  return cudaErrorInvalidValue;
}

// The batch's per-view arguments for channel part h, its own work counter.
static BatchCompositeArgs batch_part(const BatchCompositeArgs& b, int width, int h) {
  BatchCompositeArgs c = b;
  for (int v = 0; v < b.V; ++v) c.view[v] = channel_part(b.view[v], width, h);
  c.queue = b.queue + h;
  return c;
}

cudaError_t launch_composite_fwd_batch(const BatchCompositeArgs& b, int D, int feat_bf16, int fwd_batch,
                                       cudaStream_t st) {
  if (b.nitems <= 0) return cudaSuccess;
  switch (D) {
    case 16: return launch_fwd_batch_d<16>(b, feat_bf16, fwd_batch, st);
    case 32: return launch_fwd_batch_d<32>(b, feat_bf16, fwd_batch, st);
    case 64: return launch_fwd_batch_d<64>(b, feat_bf16, fwd_batch, st);
    case 128: return launch_fwd_batch_d<128>(b, feat_bf16, fwd_batch, st);
    case 256: {
      const cudaError_t e = launch_fwd_batch_d<128>(batch_part(b, kFwdPart, 0), feat_bf16, fwd_batch, st);
      return e != cudaSuccess ? e : launch_fwd_batch_d<128>(batch_part(b, kFwdPart, 1), feat_bf16, fwd_batch, st);
    }
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_composite_bwd_batch(const BatchCompositeArgs& b, int D, int feat_bf16, cudaStream_t st) {
  if (b.nitems <= 0) return cudaSuccess;
  switch (D) {
    case 16: return launch_bwd_batch_t<16>(b, feat_bf16, st);
    case 32: return launch_bwd_batch_t<32>(b, feat_bf16, st);
    case 64: return launch_bwd_batch_t<64>(b, feat_bf16, st);
    case 128:
    case 256: {
      cudaError_t e = cudaSuccess;
      for (int h = 0; h < D / kBwdPart && e == cudaSuccess; ++h)
        e = launch_bwd_batch_t<64>(batch_part(b, kBwdPart, h), feat_bf16, st);
      return e;
    }
  }
  return cudaErrorInvalidValue;
}

}  // namespace fe
