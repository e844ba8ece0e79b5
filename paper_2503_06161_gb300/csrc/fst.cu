// Full FST deformation module (Sec. 3.2, Eq. 4-6; Appendix A): the
// multi-resolution HexPlane encoding of (mu, t), the decoder MLP F_out
// (width 64, depth 8), the four branches (mu, R, S, o) with their feature
// extractors and heads, and the semantic updater F_feat giving dz; forward
// and reverse, including the gradients of the planes and of every weight.
//
// Kernels, in launch order:
//   fst_pack_kernel     16-byte-aligned transposed and row-major copies of
//                       the weights in the workspace;
//   fst_sample_kernel   HexPlane features f, eight lanes to a Gaussian (four
//                       channels each), so a corner fetch is one coalesced
//                       128-byte line of the channels-last planes, written
//                       Gaussian-major;
//   fst_fwd_tc_kernel   the MLP of a forward without reverse state, on the
//                       tensor cores (three BF16 terms per operand);
//   fst_fwd_kernel      the MLP in training: a block holds 128 Gaussians and
//                       every layer is a block product -- activations in
//                       shared memory (a row per Gaussian), lanes over rows,
//                       packed FP32 FMAs, weight tiles staged by cp.async --
//                       writing the deformed Gaussians and relu(z) of every
//                       hidden layer for the reverse;
//   fst_bwd_kernel      (persistent blocks, tensor cores) per layer the input
//                       gradient delta W, masked by the stored relu(z), and
//                       the weight gradient sum_g delta_g x_g^T added into
//                       the block's own partial; writes d f;
//   fst_hex_bwd_kernel  the HexPlane reverse: plane gradients by vector
//                       float atomics (the only order-dependent sum of this
//                       file), the time planes' as lines over the spatial
//                       axis (spread by fst_lines_out_kernel), and the
//                       canonical mean's gradient;
//   fst_reduce_kernel   the weight gradients: the blocks' partials summed in
//                       block order (reproducible bit for bit);
//   fst_tv_kernel       the TV term and its plane gradient.
#include <cstdint>

#include "common.cuh"
#include "mma.cuh"

namespace fe {

namespace {

constexpr int kFW = 64, kFHalf = 32, kFDepth = 8, kFC = 32, kFMaxL = 4;
constexpr int kFLayers = kFDepth + 12 + 2;
constexpr int kFM = 128;           // Gaussians per block (chunk) of the product kernels
constexpr int kFwdThreads = 256;   // threads of the forward product kernel
constexpr int kFRow = 68;  // shared-memory row stride (floats) of the block products
constexpr int kLZ1 = kFDepth + 12, kLZ2 = kFDepth + 13;

__host__ __device__ constexpr int branch_e1(int g) { return kFDepth + 3 * g; }
// Offset sizes of the branches mu, R, S, o (Eq. 4).
__host__ __device__ constexpr int branch_out(int g) { return g == 1 ? 4 : (g == 3 ? 1 : 3); }
// Coordinate pairs of the planes xy, xz, yz, xt, yt, zt.
__host__ __device__ constexpr int pair_a(int k) { return k == 2 || k == 4 ? 1 : (k == 5 ? 2 : 0); }
__host__ __device__ constexpr int pair_b(int k) { return k == 0 ? 1 : (k == 1 || k == 2 ? 2 : 3); }

struct FstGeom {
  int levels, rs, rt, D, P;
  int nslots, sz, se1, shg, sv;  // a Gaussian's activations ([P][nslots] float32)
  int nout[kFLayers], nin[kFLayers];
  int64_t pw[kFLayers], pb[kFLayers];  // offsets in the caller's packed array
  int64_t aw[kFLayers], ab[kFLayers];  // offsets in the aligned copies
  int64_t mlp_packed, mlp_aligned;
  int64_t poff[kFMaxL * 6];
  int pra[kFMaxL * 6], prb[kFMaxL * 6];
  float lo[3], scale[3];  // coordinate = (mu - lo) * scale - 1, scale = 2 / (hi - lo)
};

bool make_geom(const fe_fst* f, int P, FstGeom& g) {
  if (!f || f->levels < 1 || f->levels > kFMaxL || f->rs < 2 || f->rt < 2 || P < 0) return false;
  if (!(f->D == 16 || f->D == 32 || f->D == 64 || f->D == 128)) return false;
  if (((int64_t)f->rs << (f->levels - 1)) > (1 << 20) || f->rt > (1 << 20)) return false;
  g = FstGeom{};
  g.levels = f->levels;
  g.rs = f->rs;
  g.rt = f->rt;
  g.D = f->D;
  g.P = P;
  int l = 0;
  auto add = [&](int o, int i) { g.nout[l] = o; g.nin[l] = i; ++l; };
  add(kFW, f->levels * kFC);
  for (int j = 1; j < kFDepth; ++j) add(kFW, kFW);
  for (int b = 0; b < 4; ++b) {
    add(kFHalf, kFW);
    add(kFHalf, kFHalf);
    add(branch_out(b), kFHalf);
  }
  add(kFW, 4 * kFHalf);
  add(f->D, kFW);
  int64_t p = 0, a = 0;
  for (int k = 0; k < kFLayers; ++k) {
    const int64_t nw = (int64_t)g.nout[k] * g.nin[k];
    g.pw[k] = p;
    g.pb[k] = p + nw;
    p += nw + g.nout[k];
    g.aw[k] = a;
    a += (nw + 3) / 4 * 4;
    g.ab[k] = a;
    a += (g.nout[k] + 3) / 4 * 4;
  }
  g.mlp_packed = p;
  g.mlp_aligned = a;
  int64_t off = 0;
  for (int lv = 0; lv < f->levels; ++lv) {
    const int res[4] = {f->rs << lv, f->rs << lv, f->rs << lv, f->rt};
    for (int k = 0; k < 6; ++k) {
      g.poff[lv * 6 + k] = off;
      g.pra[lv * 6 + k] = res[pair_a(k)];
      g.prb[lv * 6 + k] = res[pair_b(k)];
      off += (int64_t)res[pair_a(k)] * res[pair_b(k)] * kFC;
    }
  }
  for (int k = 0; k < f->levels * 6; ++k)
    if ((int64_t)g.pra[k] * g.prb[k] * kFC > (int64_t)0x7FFFFFFF) return false;  // 32-bit plane indexing
  g.sz = 0;
  g.se1 = g.sz + kFDepth * kFW;
  g.shg = g.se1 + 4 * kFHalf;
  g.sv = g.shg + 4 * kFHalf;
  g.nslots = g.sv + kFW;
  for (int a3 = 0; a3 < 3; ++a3) {
    const float ext = f->bbox_max[a3] - f->bbox_min[a3];
    if (!(ext > 0.0f)) return false;
    g.lo[a3] = f->bbox_min[a3];
    g.scale[a3] = 2.0f / ext;
  }
  return true;
}

__host__ __device__ int64_t plane_floats(const FstGeom& g) {
  const int last = g.levels * 6 - 1;
  return g.poff[last] + (int64_t)g.pra[last] * g.prb[last] * kFC;
}

// Workspace: header | transposed weights (aligned) | row-major weights
// (aligned) | f [P][levels*32] | with the reverse: relu activations
// [P][nslots], F_feat delta [P][64], d f [P][levels*32], per-block partials
// of the weight gradients [nblk][mlp_aligned], the reverse's packed weights.
constexpr size_t kWsHeader = 256;
int bwd_blocks(int P) {
  const int chunks = (P + kFM - 1) / kFM;
  return chunks < 2 * 152 ? chunks : 2 * 152;
}
size_t al256(size_t x) { return (x + 255) / 256 * 256; }
// The reverse's packed weights (fst_pack_bwd_kernel): byte offset of each
// layer, 768 bytes per (32-column group, 16 outputs, 8 columns); the heads
// (at most four outputs) are not packed.
struct BwdPack {
  int off[kFLayers + 1], bytes;
};
__host__ __device__ constexpr bool is_head(int l) { return l >= kFDepth && l < kLZ1 && (l - kFDepth) % 3 == 2; }
BwdPack bwd_pack(const FstGeom& g) {
  BwdPack p{};
  for (int l = 0; l < kFLayers; ++l) {
    p.off[l] = p.bytes;
    if (!is_head(l)) p.bytes += g.nin[l] / 32 * (g.nout[l] / 16) * 4 * 768;
  }
  p.off[kFLayers] = p.bytes;
  return p;
}
// The time planes' gradient lines: three axes per level, kFC floats a
// position, in kLineCopies copies that blocks take in turn (a line's few
// positions get terms from every Gaussian: shorter sums round less).
constexpr int kLineCopies = 16;
size_t line_bytes(const FstGeom& g) { return (size_t)kLineCopies * 3 * g.rs * ((1u << g.levels) - 1u) * kFC * 4; }
// acc: with the reverse pass, the exact plane-gradient accumulators, two
// uint64 arrays (hi, lo) of one entry per plane float (see fixed_add).
struct WsLayout {
  size_t wt, wn, f, act, dv, df, part, wp, lines, acc, total;
};
WsLayout ws_layout(const FstGeom& g, int with_backward) {
  WsLayout w{};
  w.wt = kWsHeader;
  w.wn = w.wt + al256((size_t)g.mlp_aligned * 4);
  w.f = w.wn + al256((size_t)g.mlp_aligned * 4);
  w.act = w.f + al256((size_t)g.levels * kFC * g.P * 4);
  w.dv = w.act + (with_backward ? al256((size_t)g.nslots * g.P * 4) : 0);
  w.df = w.dv + (with_backward ? al256((size_t)kFW * g.P * 4) : 0);
  w.part = w.df + (with_backward ? al256((size_t)g.levels * kFC * g.P * 4) : 0);
  w.wp = w.part + (with_backward ? al256((size_t)bwd_blocks(g.P) * g.mlp_aligned * 4) : 0);
  w.lines = w.wp + (with_backward ? al256((size_t)bwd_pack(g).bytes) : 0);
  w.acc = w.lines + (with_backward ? al256(line_bytes(g)) : 0);
  w.total = w.acc + (with_backward == 2 ? al256((size_t)plane_floats(g) * 16) : 0);
  return w;
}

// ---------------------------------------------------------------------------
// Weight copies: transposed [in][out] and row-major [out][in], each layer at
// a 16-byte-aligned offset (biases copied beside both).
// ---------------------------------------------------------------------------
__global__ void fst_pack_kernel(const FstGeom g, const float* __restrict__ mlp, float* __restrict__ wt,
                                float* __restrict__ wn) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < g.mlp_packed;
       e += (int64_t)gridDim.x * blockDim.x) {
    int k = 0;
    while (k + 1 < kFLayers && e >= g.pw[k + 1]) ++k;
    const float v = mlp[e];
    if (e < g.pb[k]) {
      const int64_t r = e - g.pw[k];
      const int o = (int)(r / g.nin[k]), i = (int)(r % g.nin[k]);
      wt[g.aw[k] + (int64_t)i * g.nout[k] + o] = v;
      wn[g.aw[k] + r] = v;
    } else {
      wt[g.ab[k] + (e - g.pb[k])] = v;
      wn[g.ab[k] + (e - g.pb[k])] = v;
    }
  }
}

// ---------------------------------------------------------------------------
// Block products.  A block holds 128 Gaussians; activations live in shared
// memory row-major per Gaussian ([128][kFRow] floats).
//
// Eight warps: warp w owns TN consecutive columns from w TN, lane l the rows
// l + 32 r (r < 4).  Per step of four inputs a lane reads four 16-byte row
// slices (four wavefronts each) and, uniformly over the warp, TN weights per
// input (16-byte broadcasts, one wavefront each), and issues 4 TN / 2 packed
// FMAs per input.  The shared-memory pipe decides the shape: at TN = 8 it is
// 24 wavefronts per 64 FMAs.
// ---------------------------------------------------------------------------
template <int TN>
__device__ __forceinline__ void tile_zero(float2 (&acc)[4][TN / 2]) {
#pragma unroll
  for (int r = 0; r < 4; ++r)
#pragma unroll
    for (int c = 0; c < TN / 2; ++c) acc[r][c] = make_float2(0.0f, 0.0f);
}

// N consecutive floats of shared memory as pairs, in the widest loads.
template <int N>
__device__ __forceinline__ void lds_pairs(const float* p, float2 (&v)[N / 2]) {
  if constexpr (N % 4 == 0) {
#pragma unroll
    for (int i = 0; i < N / 4; ++i) {
      const float4 q = reinterpret_cast<const float4*>(p)[i];
      v[2 * i] = make_float2(q.x, q.y);
      v[2 * i + 1] = make_float2(q.z, q.w);
    }
  } else {
#pragma unroll
    for (int i = 0; i < N / 2; ++i) v[i] = reinterpret_cast<const float2*>(p)[i];
  }
}

// acc[r][c] += sum_k X[(row0 + 32 r) * kFRow + k] * B[k * ldb + n0 + (2c, 2c+1)],
// k < K (multiple of 8) in increasing order; B in shared memory, its rows
// aligned to the widest load at n0.
template <int TN>
__device__ __forceinline__ void tile_mma(const float* X, int K, const float* B, int ldb, int row0, int n0,
                                         float2 (&acc)[4][TN / 2]) {
#pragma unroll 2
  for (int k = 0; k < K; k += 4) {
    float4 xv[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) xv[r] = *reinterpret_cast<const float4*>(X + (row0 + 32 * r) * kFRow + k);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      float2 b[TN / 2];
      lds_pairs<TN>(B + (size_t)(k + kk) * ldb + n0, b);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const float xk = kk == 0 ? xv[r].x : (kk == 1 ? xv[r].y : (kk == 2 ? xv[r].z : xv[r].w));
        const float2 x2 = make_float2(xk, xk);
#pragma unroll
        for (int c = 0; c < TN / 2; ++c) acc[r][c] = __ffma2_rn(x2, b[c], acc[r][c]);
      }
    }
  }
}

// Layer epilogue of the forward: z = acc + bias; relu(z) -> Y (shared, column
// offset yc).
template <int TN>
__device__ __forceinline__ void tile_out(const float2 (&acc)[4][TN / 2], const float* __restrict__ bias, int row0,
                                         int n0, float* Y, int yc) {
  float2 bb[TN / 2];
#pragma unroll
  for (int c = 0; c < TN / 2; ++c) bb[c] = __ldg(reinterpret_cast<const float2*>(bias + n0) + c);
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    float z[TN];
#pragma unroll
    for (int c = 0; c < TN / 2; ++c) {
      z[2 * c] = fmaxf(acc[r][c].x + bb[c].x, 0.0f);
      z[2 * c + 1] = fmaxf(acc[r][c].y + bb[c].y, 0.0f);
    }
#pragma unroll
    for (int c = 0; c < TN; c += 4)
      *reinterpret_cast<float4*>(Y + (row0 + 32 * r) * kFRow + yc + n0 + c) = make_float4(z[c], z[c + 1], z[c + 2], z[c + 3]);
  }
}

// Columns [yc, yc + N) of the block's rows of Y -> the Gaussians' activation
// rows from `slot` (whole 16-byte units, consecutive lanes along a row).  The
// reverse pass needs only relu(z): it is the next layer's input, and z > 0 iff
// relu(z) > 0.
template <int N>
__device__ __forceinline__ void keep_rows(const float* Y, int yc, float* act, int nslots, int slot, int p0, int P) {
#pragma unroll 4
  for (int i = threadIdx.x; i < kFM * (N / 4); i += kFwdThreads) {
    const int r = i / (N / 4), q = i % (N / 4);
    if (p0 + r < P)
      *reinterpret_cast<float4*>(act + (size_t)(p0 + r) * nslots + slot + 4 * q) =
          *reinterpret_cast<const float4*>(Y + r * kFRow + yc + 4 * q);
  }
}

__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }

// Weight tiles staged into shared memory with cp.async, two buffers: the
// tile of the next product is in flight while the current one runs.  (The
// waits are the hardware's group waits: no spinning.)
struct WTile {
  int64_t off;           // float offset of the tile's first element
  int rows, cols, ld;    // copied as [rows][cols] from rows of `ld` floats
};
constexpr int kMaxWTiles = 40;
constexpr int kWBuf = 4096;   // floats per staging buffer

__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(smem_addr(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async16_zfill(void* dst, const void* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_addr(dst)), "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
__device__ __forceinline__ void cp_async_wait1() { asm volatile("cp.async.wait_group 1;\n" ::: "memory"); }

// Issue the copy of tile t (if any) into buffer t & 1; always commits a
// group so that "all but the newest group" names tile t - 1.  The caller
// guarantees no thread still reads buffer t & 1.
__device__ __forceinline__ void stage_tile(const WTile* tiles, int ntiles, int t, const float* __restrict__ base,
                                           float* wbuf) {
  if (t < ntiles) {
    const WTile w = tiles[t];
    float* dst = wbuf + (t & 1) * kWBuf;
    const int c4 = w.cols / 4, n = w.rows * c4;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
      const int r = i / c4, c = i - r * c4;
      cp_async16(dst + r * w.cols + 4 * c, base + w.off + (size_t)r * w.ld + 4 * c);
    }
  }
  cp_async_commit();
}

// Tile t: start tile t + 1, wait for tile t, make it visible to the block.
__device__ __forceinline__ const float* next_tile(const WTile* tiles, int ntiles, int& t, const float* base,
                                                  float* wbuf) {
  stage_tile(tiles, ntiles, t + 1, base, wbuf);
  cp_async_wait1();
  __syncthreads();
  const float* w = wbuf + (t & 1) * kWBuf;
  ++t;
  return w;
}

struct FwdArgs {
  FstGeom g;
  const float* wt;
  WTile tiles[kMaxWTiles];
  int ntiles;
  const float *means, *quats, *log_scales, *logits;
  const void* feat;
  int feat_bf16;
  float *means_t, *quats_t, *log_scales_t, *logits_t;
  void* feat_t;
  float* act;
  const float* f;  // [P][levels * 32] HexPlane features from fst_sample_kernel
};

__device__ __forceinline__ float load_feat(const void* f, int bf16, size_t i) {
  if (bf16) {
    const uint16_t b = reinterpret_cast<const uint16_t*>(f)[i];
    return __uint_as_float((uint32_t)b << 16);
  }
  return reinterpret_cast<const float*>(f)[i];
}
__device__ __forceinline__ void store_feat(void* f, int bf16, size_t i, float v) {
  if (bf16) {
    const __nv_bfloat16 h = __float2bfloat16_rn(v);
    reinterpret_cast<uint16_t*>(f)[i] = *reinterpret_cast<const uint16_t*>(&h);
  } else {
    reinterpret_cast<float*>(f)[i] = v;
  }
}

// Position of a coordinate in [-1, 1] on R nodes, clamped to the border: cell,
// fraction, and whether it was clamped.
struct Node {
  int i;
  float f;
  bool clamped;
};
__device__ __forceinline__ Node node_of(float c, int R) {
  float x = (c + 1.0f) * 0.5f * (float)(R - 1);
  Node n;
  n.clamped = false;
  if (!(x >= 0.0f)) { x = 0.0f; n.clamped = true; }  // also catches NaN
  if (x > (float)(R - 1)) { x = (float)(R - 1); n.clamped = true; }
  n.i = (int)floorf(x);
  if (n.i > R - 2) n.i = R - 2;
  n.f = x - (float)n.i;
  return n;
}

// The gathers (and their reverse) give a Gaussian eight consecutive lanes,
// four channels to a lane: a warp's 16-byte load instruction covers four
// Gaussians' texels, each a whole 128-byte line, and every lane works out
// its own positions, so nothing is exchanged.
constexpr int kGLanes = kFC / 4;

// Nodes of the four axes at level lv.
__device__ __forceinline__ void level_nodes(const FstGeom& g, const float c[4], int lv, Node n[4]) {
#pragma unroll
  for (int a = 0; a < 4; ++a) n[a] = node_of(c[a], a < 3 ? (g.rs << lv) : g.rt);
}

// Offset (in 16-byte units) of the corner (i, j) of plane k of level lv,
// channel quad q, and the plane's row stride.
__device__ __forceinline__ size_t corner_off(const FstGeom& g, int lv, int k, const Node n[4], int q, uint32_t& row) {
  const int rb = g.prb[lv * 6 + k];
  row = (uint32_t)rb * kGLanes;
  return (size_t)(g.poff[lv * 6 + k] / 4) + ((size_t)n[pair_a(k)].i * rb + n[pair_b(k)].i) * kGLanes + q;
}

__device__ __forceinline__ void gauss_coords(const FstGeom& g, const float* __restrict__ means, int p, float t,
                                             float c[4]) {
#pragma unroll
  for (int a = 0; a < 3; ++a) c[a] = (__ldg(means + (size_t)p * 3 + a) - g.lo[a]) * g.scale[a] - 1.0f;
  c[3] = 2.0f * t - 1.0f;
}

// HexPlane features f of every Gaussian, written Gaussian-major
// [P][levels * 32] for the MLP kernel: block row y takes level y, so the
// blocks in flight read one level's planes.  Bound by the texel gathers
// (2.46 GB through L1 and L2 at 200k Gaussians, 4 levels): 128 us, 218 us with
// a warp per four Gaussians, lanes over channels and 4-byte loads.
constexpr int kSampThreads = 256;
struct SampArgs {
  FstGeom g;
  const float *planes, *means;
  float t;
  float* f;
};

__global__ void __launch_bounds__(kSampThreads) fst_sample_kernel(const SampArgs a) {
  const FstGeom& g = a.g;
  const int64_t tid = (int64_t)blockIdx.x * kSampThreads + threadIdx.x;
  const int p = (int)(tid / kGLanes), q = (int)(tid % kGLanes), lv = blockIdx.y;
  if (p >= g.P) return;
  float c[4];
  gauss_coords(g, a.means, p, a.t, c);
  Node n[4];
  level_nodes(g, c, lv, n);
  const float4* planes = reinterpret_cast<const float4*>(a.planes);
  float f[4] = {1.0f, 1.0f, 1.0f, 1.0f};
#pragma unroll
  for (int k = 0; k < 6; ++k) {
    uint32_t row;
    const float4* base = planes + corner_off(g, lv, k, n, q, row);
    const float4 v00 = __ldg(base), v01 = __ldg(base + kGLanes), v10 = __ldg(base + row), v11 = __ldg(base + row + kGLanes);
    const float fa = n[pair_a(k)].f, fb = n[pair_b(k)].f;
    const float ga = 1.0f - fa, gb = 1.0f - fb;
    // Explicit roundings: f feeds the ReLUs of the MLP, whose decisions must
    // not depend on how the compiler contracts this expression.
    auto sample = [&](float p00, float p01, float p10, float p11) -> float {
      const float s0 = __fmaf_rn(gb, p00, __fmul_rn(fb, p01)), s1 = __fmaf_rn(gb, p10, __fmul_rn(fb, p11));
      return __fmaf_rn(ga, s0, __fmul_rn(fa, s1));
    };
    f[0] *= sample(v00.x, v01.x, v10.x, v11.x);
    f[1] *= sample(v00.y, v01.y, v10.y, v11.y);
    f[2] *= sample(v00.z, v01.z, v10.z, v11.z);
    f[3] *= sample(v00.w, v01.w, v10.w, v11.w);
  }
  reinterpret_cast<float4*>(a.f)[((size_t)p * g.levels + lv) * kGLanes + q] = make_float4(f[0], f[1], f[2], f[3]);
}

constexpr size_t kFwdSmem = ((size_t)2 * kFM * kFRow + 2 * kWBuf) * 4;

template <int D>
__global__ void __launch_bounds__(kFwdThreads, 2) fst_fwd_kernel(const FwdArgs a) {
  // 256 threads over 128 Gaussians: rows and columns of the products as above;
  // threads below 128 also own Gaussian p0 + tid for the per-Gaussian parts (f
  // rows, heads, outputs).
  extern __shared__ __align__(16) float s_buf[];
  float* A = s_buf;                        // [128][kFRow]
  float* B = s_buf + kFM * kFRow;          // [128][kFRow]
  float* wbuf = s_buf + 2 * kFM * kFRow;   // [2][kWBuf] staged weight tiles
  int wt_i = 0;
  stage_tile(a.tiles, a.ntiles, 0, a.wt, wbuf);
  const FstGeom& g = a.g;
  const int tid = threadIdx.x;
  const int row0 = tid & 31, nt = tid >> 5;
  const int p0 = blockIdx.x * kFM;
  const int p = p0 + tid;
  const bool owner = tid < kFM;
  const bool valid = owner && p < g.P;
  const int P = g.P;
  float* act = a.act;
  float mu[3] = {0.0f, 0.0f, 0.0f};
  if (valid) {
#pragma unroll
    for (int k = 0; k < 3; ++k) mu[k] = a.means[(size_t)p * 3 + k];
  }
  // F_out layer 0 over f (written Gaussian-major by the sampling kernel),
  // two levels (64 columns) at a time, copied into A asynchronously.
  const int nf = g.levels * kFC;
  float2 acc[4][4];
  tile_zero<8>(acc);
  for (int l0 = 0; l0 < g.levels; l0 += 2) {
    const int nl = g.levels - l0 < 2 ? g.levels - l0 : 2;
    if (owner) {
      const float* src = a.f + (size_t)(valid ? p : 0) * nf + l0 * kFC;
      for (int q = 0; q < nl * kFC; q += 4) cp_async16_zfill(A + tid * kFRow + q, src + q, valid);
      cp_async_wait_all();
    }
    __syncthreads();
    {
      const float* w = next_tile(a.tiles, a.ntiles, wt_i, a.wt, wbuf);
      tile_mma<8>(A, nl * kFC, w, kFW, row0, nt * 8, acc);
    }
    __syncthreads();
  }
  tile_out<8>(acc, a.wt + g.ab[0], row0, nt * 8, B, 0);
  __syncthreads();
  keep_rows<kFW>(B, 0, act, g.nslots, g.sz, p0, P);
  // z_j = W_j relu(z_{j-1}) + b_j; layer j reads (j odd ? B : A).
  for (int j = 1; j < kFDepth; ++j) {
    float* src = (j & 1) ? B : A;
    float* dst = (j & 1) ? A : B;
    tile_zero<8>(acc);
    tile_mma<8>(src, kFW, next_tile(a.tiles, a.ntiles, wt_i, a.wt, wbuf), kFW, row0, nt * 8, acc);
    tile_out<8>(acc, a.wt + g.ab[j], row0, nt * 8, dst, 0);
    __syncthreads();
    keep_rows<kFW>(dst, 0, act, g.nslots, g.sz + j * kFW, p0, P);
  }
  // relu(h) is in A.  Branches: e1 -> B[0, 32), h_g -> B[32, 64); the
  // semantic updater's first layer accumulates over the branches.
  float2 v[4][4];
  tile_zero<8>(v);
  float out[11];
#pragma unroll
  for (int b = 0; b < 4; ++b) {
    const int l1 = branch_e1(b);
    {
      float2 e[4][2];
      tile_zero<4>(e);
      tile_mma<4>(A, kFW, next_tile(a.tiles, a.ntiles, wt_i, a.wt, wbuf), kFHalf, row0, nt * 4, e);
      tile_out<4>(e, a.wt + g.ab[l1], row0, nt * 4, B, 0);
    }
    __syncthreads();
    {
      float2 e[4][2];
      tile_zero<4>(e);
      tile_mma<4>(B, kFHalf, next_tile(a.tiles, a.ntiles, wt_i, a.wt, wbuf), kFHalf, row0, nt * 4, e);
      tile_out<4>(e, a.wt + g.ab[l1 + 1], row0, nt * 4, B, kFHalf);
    }
    __syncthreads();
    keep_rows<kFHalf>(B, 0, act, g.nslots, g.se1 + b * kFHalf, p0, P);
    keep_rows<kFHalf>(B, kFHalf, act, g.nslots, g.shg + b * kFHalf, p0, P);
    // Head (the owner thread's own Gaussian): offset = H relu(h_g) + b.
    constexpr int dgs[4] = {3, 4, 3, 1}, oos[4] = {0, 3, 7, 10};
    if (owner) {
      const float* hgr = B + tid * kFRow + kFHalf;
      const float* wt_h = a.wt + g.aw[l1 + 2];  // [32][dg]
      const float* bh = a.wt + g.ab[l1 + 2];
#pragma unroll
      for (int o = 0; o < 4; ++o)
        if (o < dgs[b]) out[oos[b] + o] = __ldg(bh + o);
#pragma unroll 4
      for (int i4 = 0; i4 < kFHalf; i4 += 4) {
        const float4 h4 = *reinterpret_cast<const float4*>(hgr + i4);
        const float hv[4] = {h4.x, h4.y, h4.z, h4.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int o = 0; o < 4; ++o)
            if (o < dgs[b]) out[oos[b] + o] = fmaf(__ldg(wt_h + (i4 + i) * dgs[b] + o), hv[i], out[oos[b] + o]);
      }
    }
    tile_mma<8>(B + kFHalf, kFHalf, next_tile(a.tiles, a.ntiles, wt_i, a.wt, wbuf), kFW, row0, nt * 8, v);
    __syncthreads();
  }
  tile_out<8>(v, a.wt + g.ab[kLZ1], row0, nt * 8, A, 0);
  __syncthreads();
  keep_rows<kFW>(A, 0, act, g.nslots, g.sv, p0, P);
  // dz = Z2 relu(v) + b, 64 columns at a time.
  constexpr int ZN = D < 64 ? D : 64, ZT = ZN / 8;
#pragma unroll
  for (int c0 = 0; c0 < D; c0 += ZN) {
    float2 z[4][ZT / 2];
    tile_zero<ZT>(z);
    tile_mma<ZT>(A, kFW, next_tile(a.tiles, a.ntiles, wt_i, a.wt, wbuf), ZN, row0, nt * ZT, z);
    float2 bb[ZT / 2];
#pragma unroll
    for (int c = 0; c < ZT / 2; ++c) bb[c] = __ldg(reinterpret_cast<const float2*>(a.wt + g.ab[kLZ2] + c0 + nt * ZT) + c);
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int pm = p0 + row0 + 32 * r;
      if (pm < P) {
#pragma unroll
        for (int c = 0; c < ZT / 2; ++c) {
          const size_t i0 = (size_t)pm * D + c0 + nt * ZT + 2 * c;
          store_feat(a.feat_t, a.feat_bf16, i0, load_feat(a.feat, a.feat_bf16, i0) + z[r][c].x + bb[c].x);
          store_feat(a.feat_t, a.feat_bf16, i0 + 1, load_feat(a.feat, a.feat_bf16, i0 + 1) + z[r][c].y + bb[c].y);
        }
      }
    }
    __syncthreads();
  }
  if (!valid) return;
  // Deformed Gaussian (Eq. 6): offsets added to the canonical parameters.
#pragma unroll
  for (int k = 0; k < 3; ++k) a.means_t[(size_t)p * 3 + k] = mu[k] + out[k];
#pragma unroll
  for (int k = 0; k < 4; ++k) a.quats_t[(size_t)p * 4 + k] = a.quats[(size_t)p * 4 + k] + out[3 + k];
#pragma unroll
  for (int k = 0; k < 3; ++k) a.log_scales_t[(size_t)p * 3 + k] = a.log_scales[(size_t)p * 3 + k] + out[7 + k];
  a.logits_t[p] = a.logits[p] + out[10];
}

// ---------------------------------------------------------------------------
// Forward without reverse state: the MLP on the tensor cores.
//
// Every operand is three BF16 terms (24 significant bits), every product the
// six term products down to 2^-16 of |x||w|: the five small ones and hi.hi in
// accumulators of their own, added at the end, so that the small ones are
// not rounded away against the large sum.  A warp takes 16 Gaussians
// through all 22 layers: a layer's accumulators (rows = Gaussians) have the
// register layout of the next layer's first operand, so activations stay in
// registers (h, which four branches read, waits in shared memory), and only
// the weights are shared by the block: packed by fst_pack_tc_kernel in the
// order the products read them, staged 32 output columns at a time through
// three shared-memory buffers (one barrier per stage).
//
// The products alone need 236 us (200k Gaussians, 4 levels: 35 M products of
// 16 x 8 x 16 at the measured 607 TFLOP/s of mma.sync); the kernel takes 405,
// with the tensor pipe 58% busy: two blocks per SM cannot hide all of the
// fragment loads and splits.  With FP32 FMAs (fst_fwd_kernel), which training keeps --
// the reverse's ReLU masks are decisions that a different rounding would take
// differently -- they are bound by FMA issue: 592 us, with the same error against
// 64 bits (1e-7 of the outputs).
// ---------------------------------------------------------------------------
constexpr int kTcWarps = 8, kTcThreads = 32 * kTcWarps, kTcRows = 16 * kTcWarps;
constexpr int kTcBuf = 4 * 4 * 768;   // bytes of the largest stage: K = 64, 32 columns
constexpr int kTcMaxItems = 48;
constexpr size_t kTcSmem = 3 * (size_t)kTcBuf + (size_t)kTcWarps * 12 * 512;

// One stage of weights: output columns [n0, n0 + 8 nt) and inputs [k0, k0 + 16 ks)
// of layer `layer`, 768 bytes per (16 inputs, 8 columns): per lane the two
// registers of the hi and mid terms (16 bytes), then of the lo term (8).
struct TcItem {
  int layer, k0, ks, n0, nt;
  int off;  // bytes
};
struct TcPlan {
  TcItem item[kTcMaxItems];
  int n, bytes;
};

TcPlan make_tc_plan(const FstGeom& g) {
  TcPlan p{};
  auto add = [&](int layer, int k0, int k, int n0, int n) {
    p.item[p.n++] = TcItem{layer, k0, k / 16, n0, (n + 7) / 8, p.bytes};
    p.bytes += k / 16 * ((n + 7) / 8) * 768;
  };
  // In the order of use: the first layer per half of its columns and per 64
  // inputs, a hidden layer per half of its columns, a branch's three layers
  // and its share of F_feat's first layer, F_feat's second layer.
  for (int h = 0; h < 2; ++h)
    for (int k0 = 0; k0 < g.levels * kFC; k0 += 64) add(0, k0, g.levels * kFC - k0 < 64 ? 32 : 64, 32 * h, 32);
  for (int j = 1; j < kFDepth; ++j)
    for (int h = 0; h < 2; ++h) add(j, 0, kFW, 32 * h, 32);
  for (int b = 0; b < 4; ++b) {
    add(branch_e1(b), 0, kFW, 0, 32);
    add(branch_e1(b) + 1, 0, kFHalf, 0, 32);
    add(branch_e1(b) + 2, 0, kFHalf, 0, branch_out(b));
    for (int h = 0; h < 2; ++h) add(kLZ1, b * kFHalf, kFHalf, 32 * h, 32);
  }
  for (int n0 = 0; n0 < g.D; n0 += 32) add(kLZ2, 0, kFW, n0, g.D < 32 ? g.D : 32);
  return p;
}

// A thread per (16 inputs, 8 columns, lane) of the plan.
__global__ void fst_pack_tc_kernel(const FstGeom g, const TcPlan plan, const float* __restrict__ mlp,
                                   unsigned char* __restrict__ out) {
  const int u = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (u * 768 >= plan.bytes) return;
  int i = 0;
  while (i + 1 < plan.n && u * 768 >= plan.item[i + 1].off) ++i;
  const TcItem it = plan.item[i];
  const int v = u - it.off / 768, ks = v / it.nt, nt = v % it.nt;
  const int n = it.n0 + 8 * nt + (lane >> 2), k = it.k0 + 16 * ks + 2 * (lane & 3);
  float x[4] = {0.f, 0.f, 0.f, 0.f};
  if (n < g.nout[it.layer]) {
    const float* w = mlp + g.pw[it.layer] + (int64_t)n * g.nin[it.layer] + k;
    x[0] = w[0]; x[1] = w[1]; x[2] = w[8]; x[3] = w[9];
  }
  uint32_t h[2], m[2], l[2];
  split3(x[0], x[1], h[0], m[0], l[0]);
  split3(x[2], x[3], h[1], m[1], l[1]);
  unsigned char* o = out + (size_t)u * 768;
  reinterpret_cast<uint4*>(o)[lane] = make_uint4(h[0], h[1], m[0], m[1]);
  reinterpret_cast<uint2*>(o + 512)[lane] = make_uint2(l[0], l[1]);
}

struct TcArgs {
  FstGeom g;
  const float* mlp;           // biases (the caller's packed array)
  const unsigned char* wpack;
  int bytes[kTcMaxItems];     // of each stage; they follow one another in wpack
  int nitems;
  const float *means, *quats, *log_scales, *logits;
  const void* feat;
  int feat_bf16;
  float *means_t, *quats_t, *log_scales_t, *logits_t;
  void* feat_t;
  const float* f;
};

// First operand of KS steps (16 inputs each), three terms.
template <int KS>
using TcFrag = uint32_t[3][KS][4];

// acc_h += hi.hi, acc_s += the five smaller term products of one 16-input
// step with NT column tiles of staged weights at w.
template <int NT>
__device__ __forceinline__ void tc_step(const uint32_t (&ah)[4], const uint32_t (&am)[4], const uint32_t (&al)[4],
                                        const unsigned char* w, int lane, float (&acc_h)[NT][4], float (&acc_s)[NT][4]) {
  uint4 hm[NT];
  uint2 lo[NT];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    hm[nt] = reinterpret_cast<const uint4*>(w + nt * 768)[lane];
    lo[nt] = reinterpret_cast<const uint2*>(w + nt * 768 + 512)[lane];
  }
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc_s[nt], al, hm[nt].x, hm[nt].y);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc_s[nt], am, hm[nt].z, hm[nt].w);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc_s[nt], ah, lo[nt].x, lo[nt].y);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc_s[nt], am, hm[nt].x, hm[nt].y);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc_s[nt], ah, hm[nt].z, hm[nt].w);
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(acc_h[nt], ah, hm[nt].x, hm[nt].y);
}

template <int NT>
__device__ __forceinline__ void tc_zero(float (&a)[NT][4], float (&b)[NT][4]) {
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int i = 0; i < 4; ++i) a[nt][i] = b[nt][i] = 0.0f;
}

// max(x, 0) that keeps a NaN.
__device__ __forceinline__ float relu_nan(float x) {
  float y;
  asm("max.NaN.f32 %0, %1, 0f00000000;" : "=f"(y) : "f"(x));
  return y;
}

// Columns 8 nt + 2 t, + 1 of four tiles (rows fr, fr + 8) as steps k0 and
// k0 + 1 of the next layer's first operand: relu(z + bias), three terms.
template <int KS>
__device__ __forceinline__ void tc_relu(const float (&z)[4][4], const float* __restrict__ bias, int ft, TcFrag<KS>& out,
                                        int k0) {
#pragma unroll
  for (int nt = 0; nt < 4; ++nt) {
    const float b0 = __ldg(bias + 8 * nt + 2 * ft), b1 = __ldg(bias + 8 * nt + 2 * ft + 1);
    const int k = k0 + (nt >> 1), i = 2 * (nt & 1);
    split3(relu_nan(z[nt][0] + b0), relu_nan(z[nt][1] + b1), out[0][k][i], out[1][k][i], out[2][k][i]);
    split3(relu_nan(z[nt][2] + b0), relu_nan(z[nt][3] + b1), out[0][k][i + 1], out[1][k][i + 1], out[2][k][i + 1]);
  }
}

// The outputs `todo` (bit b: branch b; bit 4 + s: feature columns of stage s, zt
// columns each) of Gaussian p with FP32 products, by one warp, in the order of
// fst_fwd_kernel's sums.  For the Gaussians whose values leave the range of
// the three BF16 terms: an infinity, or anything that rounds to one in BF16,
// splits into terms that give NaN, which relu_nan carries to every output
// behind it; FP32 products keep infinities and clamp NaNs at the ReLUs.
// (What a diverged plane or weight does must not depend on whether reverse state
// is kept; the outputs that it does not reach cost 4 us of 540 at 200k.)
static_assert((2 * kFW + 2 * kFHalf) * 4 <= 12 * 512, "works in the warp's part of shared memory");
__device__ __noinline__ void fst_row_fp32(const TcArgs& a, float* buf, int p, uint32_t todo, int D, int zt) {
  const FstGeom& g = a.g;
  const int lane = threadIdx.x & 31;
  float *x = buf, *y = buf + kFW, *e = buf + 2 * kFW, *u = e + kFHalf;
  // acc + sum_k w[o][k] in[k], k ascending.
  auto dot = [&](int layer, int o, int k0, const float* in, int K, float acc) {
    const float* w = a.mlp + g.pw[layer] + (int64_t)o * g.nin[layer] + k0;
    for (int k = 0; k < K; ++k) acc = fmaf(in[k], __ldg(w + k), acc);
    return acc;
  };
  auto relu_layer = [&](int layer, const float* in, float* out) {
    for (int o = lane; o < g.nout[layer]; o += 32)
      out[o] = fmaxf(dot(layer, o, 0, in, g.nin[layer], 0.0f) + a.mlp[g.pb[layer] + o], 0.0f);
    __syncwarp();
  };
  __syncwarp();
  relu_layer(0, a.f + (size_t)p * g.levels * kFC, x);
  for (int j = 1; j < kFDepth; ++j) {
    relu_layer(j, x, y);
    float* t = x;
    x = y;
    y = t;
  }
  const float* srcs[4] = {a.means, a.quats, a.log_scales, a.logits};
  float* dsts[4] = {a.means_t, a.quats_t, a.log_scales_t, a.logits_t};
  float v[2] = {0.0f, 0.0f};
  for (int b = 0; b < 4; ++b) {
    const int l1 = branch_e1(b), dg = branch_out(b);
    relu_layer(l1, x, e);
    relu_layer(l1 + 1, e, u);
    if (((todo >> b) & 1u) && lane < dg) {
      const size_t at = (size_t)p * dg + lane;
      dsts[b][at] = srcs[b][at] + dot(l1 + 2, lane, 0, u, kFHalf, a.mlp[g.pb[l1 + 2] + lane]);
    }
    for (int h = 0; h < 2; ++h) v[h] = dot(kLZ1, lane + 32 * h, b * kFHalf, u, kFHalf, v[h]);
    __syncwarp();
  }
  for (int h = 0; h < 2; ++h) y[lane + 32 * h] = fmaxf(v[h] + a.mlp[g.pb[kLZ1] + lane + 32 * h], 0.0f);
  __syncwarp();
  for (int o = lane; o < D; o += 32) {
    if (!((todo >> (4 + o / zt)) & 1u)) continue;
    const size_t at = (size_t)p * D + o;
    const float z = dot(kLZ2, o, 0, y, kFW, 0.0f);
    store_feat(a.feat_t, a.feat_bf16, at, load_feat(a.feat, a.feat_bf16, at) + z + a.mlp[g.pb[kLZ2] + o]);
  }
  __syncwarp();
}

template <int D>
__global__ void __launch_bounds__(kTcThreads, 2) fst_fwd_tc_kernel(const __grid_constant__ TcArgs a) {
  extern __shared__ __align__(16) unsigned char s_tc[];
  const FstGeom& g = a.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, fr = lane >> 2, ft = lane & 3;
  uint4* s_h = reinterpret_cast<uint4*>(s_tc + 3 * kTcBuf) + warp * 12 * 32;  // [ks][term][lane]
  const int P = g.P;
  const int p[2] = {(int)blockIdx.x * kTcRows + warp * 16 + fr, (int)blockIdx.x * kTcRows + warp * 16 + fr + 8};
  const bool valid[2] = {p[0] < P, p[1] < P};
  // Weight stages: stage t is in buffer t % 3; two are in flight.
  int t_issue = 0, t_use = 0;
  const unsigned char* src = a.wpack;
  auto issue = [&]() {
    if (t_issue < a.nitems) {
      const int n = a.bytes[t_issue];
      unsigned char* dst = s_tc + (t_issue % 3) * kTcBuf;
      for (int i = tid; i < n / 16; i += kTcThreads) cp_async16(dst + 16 * i, src + 16 * i);
      src += n;
      ++t_issue;
    }
    cp_async_commit();
  };
  issue();
  issue();
  auto next = [&]() -> const unsigned char* {
    cp_async_wait1();
    __syncthreads();  // the stage has landed for all; the one before it is read
    issue();
    return s_tc + (t_use++ % 3) * kTcBuf;
  };
  float zh[4][4], zs[4][4];
  auto sum = [&]() {
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) zh[nt][i] += zs[nt][i];
  };
  // ---- F_out ----
  TcFrag<4> x;
  const int nf = g.levels * kFC;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    tc_zero(zh, zs);
    for (int k0 = 0; k0 < nf; k0 += 64) {
      const unsigned char* w = next();
      const int ks_n = nf - k0 < 64 ? 2 : 4;
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        if (ks < ks_n) {
          uint32_t f3[3][4];
#pragma unroll
          for (int r = 0; r < 2; ++r) {
            const float* row = a.f + (size_t)(valid[r] ? p[r] : 0) * nf + k0 + 16 * ks + 2 * ft;
            const float2 u0 = __ldg(reinterpret_cast<const float2*>(row)), u1 = __ldg(reinterpret_cast<const float2*>(row + 8));
            split3(u0.x, u0.y, f3[0][r], f3[1][r], f3[2][r]);
            split3(u1.x, u1.y, f3[0][2 + r], f3[1][2 + r], f3[2][2 + r]);
          }
          tc_step<4>(f3[0], f3[1], f3[2], w + ks * 4 * 768, lane, zh, zs);
        }
      }
    }
    sum();
    tc_relu<4>(zh, a.mlp + g.pb[0] + 32 * h, ft, x, 2 * h);
  }
  for (int j = 1; j < kFDepth; ++j) {
    TcFrag<4> y;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned char* w = next();
      tc_zero(zh, zs);
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) tc_step<4>(x[0][ks], x[1][ks], x[2][ks], w + ks * 4 * 768, lane, zh, zs);
      sum();
      tc_relu<4>(zh, a.mlp + g.pb[j] + 32 * h, ft, y, 2 * h);
    }
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
      for (int ks = 0; ks < 4; ++ks)
#pragma unroll
        for (int i = 0; i < 4; ++i) x[t][ks][i] = y[t][ks][i];
  }
  // relu(h) for the branches.
#pragma unroll
  for (int ks = 0; ks < 4; ++ks)
#pragma unroll
    for (int t = 0; t < 3; ++t) s_h[(3 * ks + t) * 32 + lane] = make_uint4(x[t][ks][0], x[t][ks][1], x[t][ks][2], x[t][ks][3]);
  // ---- branches; F_feat's first layer sums over them ----
  float v[8][4];
#pragma unroll
  for (int nt = 0; nt < 8; ++nt)
#pragma unroll
    for (int i = 0; i < 4; ++i) v[nt][i] = 0.0f;
  const float* srcs[4] = {a.means, a.quats, a.log_scales, a.logits};
  float* dsts[4] = {a.means_t, a.quats_t, a.log_scales_t, a.logits_t};
  // Outputs of rows fr and fr + 8 that are left to fst_row_fp32 (its bits).
  uint32_t todo[2] = {0u, 0u};
  auto finite = [&](const float (&x)[2], int r, uint32_t bit) -> bool {
    const uint32_t bad = __ballot_sync(0xFFFFFFFFu, valid[r] && !(isfinite(x[0]) && isfinite(x[1])));
    if ((bad >> (4 * fr)) & 15u) {
      todo[r] |= bit;
      return false;
    }
    return true;
  };
#pragma unroll 1
  for (int b = 0; b < 4; ++b) {
    const int l1 = branch_e1(b);
    TcFrag<2> e, u;
    {
      const unsigned char* w = next();
      tc_zero(zh, zs);
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        uint32_t hx[3][4];
#pragma unroll
        for (int t = 0; t < 3; ++t) {
          const uint4 q = s_h[(3 * ks + t) * 32 + lane];
          hx[t][0] = q.x; hx[t][1] = q.y; hx[t][2] = q.z; hx[t][3] = q.w;
        }
        tc_step<4>(hx[0], hx[1], hx[2], w + ks * 4 * 768, lane, zh, zs);
      }
      sum();
      tc_relu<2>(zh, a.mlp + g.pb[l1], ft, e, 0);
    }
    {
      const unsigned char* w = next();
      tc_zero(zh, zs);
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) tc_step<4>(e[0][ks], e[1][ks], e[2][ks], w + ks * 4 * 768, lane, zh, zs);
      sum();
      tc_relu<2>(zh, a.mlp + g.pb[l1 + 1], ft, u, 0);
    }
    {
      // Head: offsets added to the canonical parameters (Eq. 6).
      const unsigned char* w = next();
      float oh[1][4], os[1][4];
      tc_zero(oh, os);
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) tc_step<1>(u[0][ks], u[1][ks], u[2][ks], w + ks * 768, lane, oh, os);
      const int dg = branch_out(b);
      const float* bias = a.mlp + g.pb[l1 + 2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        float off[2];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int o = 2 * ft + i;
          off[i] = o < dg ? (oh[0][2 * r + i] + os[0][2 * r + i]) + __ldg(bias + o) : 0.0f;
        }
        if (finite(off, r, 1u << b)) {
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int o = 2 * ft + i;
            const size_t at = (size_t)p[r] * dg + o;
            if (o < dg && valid[r]) dsts[b][at] = srcs[b][at] + off[i];
          }
        }
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned char* w = next();
      tc_zero(zh, zs);
#pragma unroll
      for (int ks = 0; ks < 2; ++ks) tc_step<4>(u[0][ks], u[1][ks], u[2][ks], w + ks * 4 * 768, lane, zh, zs);
#pragma unroll
      for (int nt = 0; nt < 4; ++nt)
#pragma unroll
        for (int i = 0; i < 4; ++i) v[4 * h + nt][i] += zh[nt][i] + zs[nt][i];
    }
  }
  // ---- dz = Z2 relu(v) + b ----
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float z[4][4];
#pragma unroll
    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) z[nt][i] = v[4 * h + nt][i];
    tc_relu<4>(z, a.mlp + g.pb[kLZ1] + 32 * h, ft, x, 2 * h);
  }
  constexpr int ZT = D < 32 ? D / 8 : 4;  // column tiles per stage
#pragma unroll 1
  for (int n0 = 0; n0 < D; n0 += 8 * ZT) {
    const unsigned char* w = next();
    float dh[ZT][4], ds[ZT][4];
    tc_zero(dh, ds);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) tc_step<ZT>(x[0][ks], x[1][ks], x[2][ks], w + ks * ZT * 768, lane, dh, ds);
    const float* bias = a.mlp + g.pb[kLZ2] + n0;
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      // (A sum of the row's values is finite only if each of them is.)
      float any[2] = {0.0f, 0.0f};
#pragma unroll
      for (int nt = 0; nt < ZT; ++nt)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          dh[nt][2 * r + i] += ds[nt][2 * r + i];
          any[i] += dh[nt][2 * r + i];
        }
      if (!finite(any, r, 16u << (n0 / (8 * ZT)))) continue;
#pragma unroll
      for (int nt = 0; nt < ZT; ++nt)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int c = 8 * nt + 2 * ft + i;
          if (valid[r]) {
            const size_t at = (size_t)p[r] * D + n0 + c;
            store_feat(a.feat_t, a.feat_bf16, at, load_feat(a.feat, a.feat_bf16, at) + dh[nt][2 * r + i] + __ldg(bias + c));
          }
        }
    }
  }
  if (__any_sync(0xFFFFFFFFu, (todo[0] | todo[1]) != 0u)) {
#pragma unroll 1
    for (int r = 0; r < 16; ++r) {
      const uint32_t w = __shfl_sync(0xFFFFFFFFu, r < 8 ? todo[0] : todo[1], 4 * (r & 7));
      if (w) fst_row_fp32(a, reinterpret_cast<float*>(s_h), (int)blockIdx.x * kTcRows + warp * 16 + r, w, D, 8 * ZT);
    }
  }
}

// ---------------------------------------------------------------------------
// Reverse.
// ---------------------------------------------------------------------------
// Exact, order-independent plane-gradient sums.  Each float contribution x
// is the integer X = x 2^72 (exact for |x| >= 2^-49; smaller ones rounded to
// the nearest multiple of 2^-72), held as hi 2^32 + lo with 0 <= lo < 2^32,
// and added with 64-bit integer atomics into hi[i] (two's complement) and
// lo[i]: integer sums do not depend on the order of the additions, so the
// result is the same bits however the Gaussians are scheduled.  |sum| must
// stay below 2^23 (contributions at or above it are clamped and flagged).
__device__ __forceinline__ void fixed_add(unsigned long long* hi, unsigned long long* lo, size_t i, float x,
                                          uint32_t* err) {
  const uint32_t u = __float_as_uint(x);
  const int e = (int)((u >> 23) & 0xFFu);
  if (e == 0) return;  // zero or below 2^-126: under the resolution
  uint64_t m = (u & 0x7FFFFFu) | 0x800000u;  // |x| = m 2^(e - 150)
  int sh = e - 150 + 72;                      // |X| = m 2^sh
  if (sh > 71) {                              // |x| >= 2^23
    set_err(err, kErrOverflow);
    m = 0xFFFFFFu;
    sh = 71;
  }
  uint64_t h, l;
  if (sh >= 32) {
    h = m << (sh - 32);
    l = 0;
  } else if (sh >= 0) {
    const uint64_t X = m << sh;
    h = X >> 32;
    l = X & 0xFFFFFFFFull;
  } else if (sh > -25) {
    h = 0;
    l = (m + (1ull << (-sh - 1))) >> (-sh);  // nearest, ties up
  } else {
    return;
  }
  if (u >> 31) {  // -(h 2^32 + l)
    if (l) {
      h = ~h;            // -h - 1
      l = 0x100000000ull - l;
    } else {
      h = ~h + 1ull;     // -h
    }
  }
  if (h) atomicAdd(hi + i, (unsigned long long)h);
  if (l) atomicAdd(lo + i, (unsigned long long)l);
}

// Packed weights of the reverse's delta W products: the second operand
// B[k = output][n = input] in fragment order, three BF16 terms (as
// fst_pack_tc_kernel's, with the roles of outputs and inputs exchanged), from
// the row-major copies the forward left.
__global__ void fst_pack_bwd_kernel(const FstGeom g, const BwdPack pk, const float* __restrict__ wn,
                                    unsigned char* __restrict__ out) {
  const int u = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (u * 768 >= pk.bytes) return;
  int l = 0;
  while (u * 768 >= pk.off[l + 1]) ++l;
  const int v = u - pk.off[l] / 768, KS = g.nout[l] / 16, nt = v & 3, ks = (v >> 2) % KS, grp = (v >> 2) / KS;
  const int n = 32 * grp + 8 * nt + (lane >> 2), k = 16 * ks + 2 * (lane & 3), ld = g.nin[l];
  const float* w = wn + g.aw[l] + (int64_t)k * ld + n;
  uint32_t h[2], m[2], lo[2];
  split3(w[0], w[ld], h[0], m[0], lo[0]);
  split3(w[8 * ld], w[9 * ld], h[1], m[1], lo[1]);
  unsigned char* o = out + (size_t)u * 768;
  reinterpret_cast<uint4*>(o)[lane] = make_uint4(h[0], h[1], m[0], m[1]);
  reinterpret_cast<uint2*>(o + 512)[lane] = make_uint2(lo[0], lo[1]);
}

struct BwdArgs {
  FstGeom g;
  BwdPack pk;
  const unsigned char* wp;    // packed weights
  const float *wn, *act, *f;  // row-major weights (the heads), activations, HexPlane features
  const float *d_means_t, *d_quats_t, *d_log_scales_t, *d_logits_t, *d_feat_t;
  float* dv;    // [P][64]: delta of F_feat's first layer
  float* df;    // [P][levels * 32]: d f, read by the HexPlane reverse kernel
  float* part;  // [gridDim.x][mlp_aligned]
};

// A tile of 128 Gaussians x 64 columns in shared memory, three BF16 terms:
// rows of 128 bytes, 16-byte chunk c of row r at c ^ (r & 7), so that the
// fragment loads and stores below touch every bank once.
constexpr int kTTerm = kFM * 128;
__device__ __forceinline__ uint32_t t_off(int r, int chunk) { return (uint32_t)(r * 128 + ((chunk ^ (r & 7)) << 4)); }

// Lane's pair of values (columns c, c + 1; c even) of row r into a tile.
__device__ __forceinline__ void put_pair(unsigned char* tile, int r, int c, float x, float y) {
  uint32_t t3[3];
  split3(x, y, t3[0], t3[1], t3[2]);
  const uint32_t o = t_off(r, c >> 3) + 2 * (c & 7);
#pragma unroll
  for (int t = 0; t < 3; ++t) *reinterpret_cast<uint32_t*>(tile + t * kTTerm + o) = t3[t];
}

// What a lane holds of its warp's 16 rows: columns 8 nt + 2 ft, + 1 of rows fr
// (elements 0, 1) and fr + 8 (2, 3), the accumulator layout.
template <int NT>
__device__ __forceinline__ void load_rows(const float* a, const float* b, int ft, float (&v)[NT][4]) {
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    const float2 x = a ? __ldg(reinterpret_cast<const float2*>(a + 8 * nt + 2 * ft)) : make_float2(0.0f, 0.0f);
    const float2 y = b ? __ldg(reinterpret_cast<const float2*>(b + 8 * nt + 2 * ft)) : make_float2(0.0f, 0.0f);
    v[nt][0] = x.x; v[nt][1] = x.y; v[nt][2] = y.x; v[nt][3] = y.y;
  }
}
template <int NT>
__device__ __forceinline__ void put_rows(unsigned char* tile, int row, int c0, int ft, const float (&v)[NT][4]) {
#pragma unroll
  for (int nt = 0; nt < NT; ++nt) {
    put_pair(tile, row, c0 + 8 * nt + 2 * ft, v[nt][0], v[nt][1]);
    put_pair(tile, row + 8, c0 + 8 * nt + 2 * ft, v[nt][2], v[nt][3]);
  }
}
// v where the activation x (>= 0) is positive, else 0.
template <int NT>
__device__ __forceinline__ void mask_rows(float (&v)[NT][4], const float (&x)[NT][4]) {
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int i = 0; i < 4; ++i) v[nt][i] = x[nt][i] > 0.0f ? v[nt][i] : 0.0f;
}

// acc (32 columns) = delta W for the warp's rows: delta in columns
// [16 kc, 16 (kc + KS)) of the tile, packed weights at w ([KS][4] units).
template <int KS>
__device__ __forceinline__ void delta_w(uint32_t tile, int warp, int kc, const unsigned char* __restrict__ w, int lane,
                                        float (&acc)[4][4]) {
  float zs[4][4];
  tc_zero(acc, zs);
  const int r = warp * 16 + (lane & 7) + 8 * ((lane >> 3) & 1), ch = lane >> 4;
#pragma unroll
  for (int ks = 0; ks < KS; ++ks) {
    uint32_t a[3][4];
#pragma unroll
    for (int t = 0; t < 3; ++t) ldmatrix_x4(tile + t * kTTerm + t_off(r, 2 * (kc + ks) + ch), a[t]);
    tc_step<4>(a[0], a[1], a[2], w + ks * 4 * 768, lane, acc, zs);
  }
#pragma unroll
  for (int nt = 0; nt < 4; ++nt)
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[nt][i] += zs[nt][i];
}

// Weight gradient block of one warp: outputs [16 om, + 16) (columns oc0 + ...
// of the delta tile) x inputs [8 in0, + 8 NT) (columns of the input tile),
// summed over the tile's 128 Gaussians and added to pw (row stride ldw); with
// pb also the bias gradient.  rows: outputs that exist.
template <int NT>
__device__ __forceinline__ void weight_grad(uint32_t sd, int oc, uint32_t sx, int ic, int rows, float* pw, int ldw, float* pb,
                                            bool first, int lane) {
  const int fr = lane >> 2, ft = lane & 3, mi = lane >> 3, r = lane & 7;
  float2 prev[NT][2];
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      prev[nt][h] = !first && fr + 8 * h < rows ? *reinterpret_cast<const float2*>(pw + (size_t)(fr + 8 * h) * ldw + 8 * nt + 2 * ft)
                                                : make_float2(0.0f, 0.0f);
  float zh[NT][4], zs[NT][4], bh[1][4], bs[1][4];
  tc_zero(zh, zs);
  tc_zero(bh, bs);
  const uint32_t one = fr == 0 ? 0x3F803F80u : 0u;  // column 0 of the bias tile
#pragma unroll 1
  for (int g0 = 0; g0 < kFM; g0 += 16) {
    uint32_t a[3][4];
#pragma unroll
    for (int t = 0; t < 3; ++t) ldmatrix_x4_trans(sd + t * kTTerm + t_off(g0 + r + 8 * (mi >> 1), oc + (mi & 1)), a[t]);
    if (pb) {
      mma_bf16_16816(bs[0], a[2], one, one);
      mma_bf16_16816(bs[0], a[1], one, one);
      mma_bf16_16816(bh[0], a[0], one, one);
    }
    constexpr int NP = (NT + 1) / 2;
    uint32_t b[3][NP][4];
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
      for (int q = 0; q < NP; ++q)
        ldmatrix_x4_trans(sx + t * kTTerm + t_off(g0 + r + 8 * (mi & 1), NT == 1 ? ic : ic + 2 * q + (mi >> 1)), b[t][q]);
#define FST_WG(za, ta, tb)                                                                                     \
  _Pragma("unroll") for (int nt = 0; nt < NT; ++nt)                                                            \
      mma_bf16_16816(za[nt], a[ta], b[tb][nt >> 1][2 * (nt & 1)], b[tb][nt >> 1][2 * (nt & 1) + 1]);
    FST_WG(zs, 2, 0)
    FST_WG(zs, 1, 1)
    FST_WG(zs, 0, 2)
    FST_WG(zs, 1, 0)
    FST_WG(zs, 0, 1)
    FST_WG(zh, 0, 0)
#undef FST_WG
  }
#pragma unroll
  for (int nt = 0; nt < NT; ++nt)
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (fr + 8 * h < rows) {
        const float2 v = prev[nt][h];
        *reinterpret_cast<float2*>(pw + (size_t)(fr + 8 * h) * ldw + 8 * nt + 2 * ft) =
            make_float2(v.x + (zh[nt][2 * h] + zs[nt][2 * h]), v.y + (zh[nt][2 * h + 1] + zs[nt][2 * h + 1]));
      }
  if (pb && ft == 0) {
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (fr + 8 * h < rows) pb[fr + 8 * h] = (first ? 0.0f : pb[fr + 8 * h]) + (bh[0][2 * h] + bs[0][2 * h]);
  }
}

constexpr int kBwdThreads = 256;
constexpr int kBwdW = 4 * 4 * 768;  // staged weights: 64 outputs x 32 columns
constexpr size_t kBwdSmem = 6 * (size_t)kTTerm + kBwdW + 1024;

// Reverse of the MLP for 128 Gaussians at a time (persistent blocks).  Layers
// are walked backwards; a round holds a layer's delta and input tiles in
// shared memory (three BF16 terms), from which the block's eight warps take
// the weight gradient (each a 16-output block, all 128 Gaussians) and each
// warp the input delta of its own 16 Gaussians, masked by the stored
// relu(z).  The same term products and accumulators as the forward without
// reverse state.
//
// The products alone need 472 us (200k Gaussians, 4 levels: 70 M products of
// 16 x 8 x 16 at 607 TFLOP/s); the kernel takes 1094, the tensor pipe half
// busy: the rounds' barriers and fragment loads are the rest.  The FP32 form
// (8 x 8 register tiles of packed FMAs, 249 registers, 8 warps per SM) took
// 1555 us.  Two blocks per SM leave 128 registers and 236 (D = 16) to 508
// (D = 128) bytes of spills; one block without them is slower (module forward +
// reverse + TV 2625 us for 2435).
template <int D>
__global__ void __launch_bounds__(kBwdThreads, 2) fst_bwd_kernel(const __grid_constant__ BwdArgs a) {
  extern __shared__ unsigned char s_raw[];
  unsigned char* sD = s_raw + ((1024u - (smem_addr(s_raw) & 1023u)) & 1023u);
  unsigned char* sX = sD + 3 * kTTerm;
  unsigned char* sW = sX + 3 * kTTerm;
  const uint32_t uD = smem_addr(sD), uX = smem_addr(sX);
  const FstGeom& g = a.g;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, fr = lane >> 2, ft = lane & 3;
  const int P = g.P, nf = g.levels * kFC, row = warp * 16 + fr;
  const int nchunk = (P + kFM - 1) / kFM;
  float* part = a.part + (size_t)blockIdx.x * g.mlp_aligned;
  // Weight-gradient blocks: output tile om and input columns of this warp.
  auto wgrad = [&](int l, int oc, int O, int ic, int I, int i0, bool bias, bool first) {
    // Outputs O (64, 32 or 16 of the tile's columns from oc), inputs I (64 or
    // 32 of the tile's columns from ic) that are inputs i0 .. of layer l.
    const int om = warp % (O / 16), grp = warp / (O / 16);
    float* pw = part + g.aw[l] + (size_t)(16 * om) * g.nin[l] + i0;
    float* pb = bias && grp == 0 ? part + g.ab[l] + 16 * om : nullptr;
    if (O == 64 && I == 64)
      weight_grad<4>(uD, oc + 2 * om, uX, ic + 4 * grp, 16, pw + 32 * grp, g.nin[l], pb, first, lane);
    else if ((O == 64 && I == 32) || (O == 32 && I == 64))
      weight_grad<2>(uD, oc + 2 * om, uX, ic + 2 * grp, 16, pw + 16 * grp, g.nin[l], pb, first, lane);
    else
      weight_grad<1>(uD, oc + 2 * om, uX, ic + grp, 16, pw + 8 * grp, g.nin[l], pb, first, lane);
  };
  // Weights of the next delta W product into sW (every thread is past the
  // product before it); landed() completes the copy for the whole block, with
  // the tiles written meanwhile.
  auto stage = [&](int l, int off, int bytes) {
    const unsigned char* src = a.wp + a.pk.off[l] + off;
    for (int i = tid; i < bytes / 16; i += kBwdThreads) cp_async16(sW + 16 * i, src + 16 * i);
  };
  auto landed = [&]() {
    cp_async_wait_all();
    __syncthreads();
  };
  for (int chunk = blockIdx.x; chunk < nchunk; chunk += gridDim.x) {
    const bool first = chunk == (int)blockIdx.x;
    const int p[2] = {chunk * kFM + row, chunk * kFM + row + 8};
    const bool valid[2] = {p[0] < P, p[1] < P};
    const float* act[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) act[h] = valid[h] ? a.act + (size_t)p[h] * g.nslots : nullptr;
    // A round's activation rows are fetched to L2 a round ahead: a lane takes
    // one 128-byte line of its warp's 16 rows of 64 floats.
    const int pf = chunk * kFM + warp * 16 + (lane >> 1);
    auto fetch = [&](int slot) {
      if (pf < P) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.act + (size_t)pf * g.nslots + slot + 32 * (lane & 1)));
    };
    auto act_rows = [&](int slot, auto& v) { load_rows(act[0] ? act[0] + slot : nullptr, act[1] ? act[1] + slot : nullptr, ft, v); };
    float d[8][4];  // delta of 64 columns (or the sum that becomes it)
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) d[nt][i] = 0.0f;
    float x[8][4];
    // ---- F_feat second layer: delta = d dz, input relu(v).
    constexpr int NC = D < 64 ? D : 64;
    act_rows(g.sv, x);
#pragma unroll 1
    for (int c0 = 0; c0 < D; c0 += NC) {
      __syncthreads();  // the tiles are free (previous chunk or part)
      // Packed [group][outputs / 16][4]: the outputs of this part.
      stage(kLZ2, (c0 / 16) * 4 * 768, NC / 16 * 4 * 768);
      {
        float z[NC / 8][4];
        load_rows(valid[0] ? a.d_feat_t + (size_t)p[0] * D + c0 : nullptr, valid[1] ? a.d_feat_t + (size_t)p[1] * D + c0 : nullptr, ft, z);
        put_rows(sD, row, 0, ft, z);
      }
      if (c0 == 0) put_rows(sX, row, 0, ft, x);
      fetch(g.shg);
      landed();
      auto product = [&](int h) {
        float z[4][4];
        delta_w<NC / 16>(uD, warp, 0, sW, lane, z);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
          for (int i = 0; i < 4; ++i) d[4 * h + nt][i] += z[nt][i];
      };
      product(0);
      __syncthreads();
      stage(kLZ2, (D / 16 + c0 / 16) * 4 * 768, NC / 16 * 4 * 768);
      {
        float* pw = part + g.aw[kLZ2] + (size_t)c0 * kFW;
        float* pb = part + g.ab[kLZ2] + c0;
        constexpr int OT = NC / 16;
        const int om = warp % OT, grp = warp / OT;
        constexpr int NTW = OT;  // 64 columns over 8 / OT groups: OT tiles each
        weight_grad<NTW>(uD, 2 * om, uX, NTW * grp, 16, pw + (size_t)(16 * om) * kFW + 8 * NTW * grp, kFW, grp == 0 ? pb + 16 * om : nullptr, first, lane);
      }
      landed();
      product(1);
    }
    mask_rows(d, x);
    // ---- F_feat first layer: input u = [h_mu, h_R, h_S, h_o] (relu).  Its
    // delta goes to the tile and to the workspace (for the branches).
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (valid[h])
#pragma unroll
        for (int nt = 0; nt < 8; ++nt)
          *reinterpret_cast<float2*>(a.dv + (size_t)p[h] * kFW + 8 * nt + 2 * ft) = make_float2(d[nt][2 * h], d[nt][2 * h + 1]);
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      act_rows(g.shg + half * kFW, x);
      fetch(half == 0 ? g.shg + kFW : g.se1);
      __syncthreads();
      if (half == 0) put_rows(sD, row, 0, ft, d);
      put_rows(sX, row, 0, ft, x);
      __syncthreads();
      wgrad(kLZ1, 0, 64, 0, 64, half * kFW, half == 0, first);
    }
    // ---- branches; d relu(h) accumulates over them.
#pragma unroll
    for (int nt = 0; nt < 8; ++nt)
#pragma unroll
      for (int i = 0; i < 4; ++i) d[nt][i] = 0.0f;
#pragma unroll 1
    for (int b = 0; b < 4; ++b) {
      const int dg = branch_out(b), l1 = branch_e1(b);
      const float* dsrc = b == 0 ? a.d_means_t : b == 1 ? a.d_quats_t : b == 2 ? a.d_log_scales_t : a.d_logits_t;
      float off[2][4];  // head deltas of the two rows
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int o = 0; o < 4; ++o) off[h][o] = valid[h] && o < dg ? __ldg(dsrc + (size_t)p[h] * dg + o) : 0.0f;
      // delta of h_g: Z1[:, branch]^T delta_v + H^T d offset, masked.
      __syncthreads();
      stage(kLZ1, b * 4 * 4 * 768, 4 * 4 * 768);
      landed();
      float du[4][4];
      {
        float zs[4][4];
        tc_zero(du, zs);
#pragma unroll
        for (int ks = 0; ks < 4; ++ks) {
          uint32_t f3[3][4];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const float* r = a.dv + (size_t)(valid[h] ? p[h] : 0) * kFW + 16 * ks + 2 * ft;
            const float2 u0 = valid[h] ? *reinterpret_cast<const float2*>(r) : make_float2(0.f, 0.f);
            const float2 u1 = valid[h] ? *reinterpret_cast<const float2*>(r + 8) : make_float2(0.f, 0.f);
            split3(u0.x, u0.y, f3[0][h], f3[1][h], f3[2][h]);
            split3(u1.x, u1.y, f3[0][2 + h], f3[1][2 + h], f3[2][2 + h]);
          }
          tc_step<4>(f3[0], f3[1], f3[2], sW + ks * 4 * 768, lane, du, zs);
        }
        const float* wh = a.wn + g.aw[l1 + 2];  // [dg][32]
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
          for (int i = 0; i < 4; ++i) du[nt][i] += zs[nt][i];
#pragma unroll
        for (int o = 0; o < 4; ++o)
          if (o < dg)
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) {
              const float2 w2 = __ldg(reinterpret_cast<const float2*>(wh + o * kFHalf + 8 * nt + 2 * ft));
              du[nt][0] = fmaf(off[0][o], w2.x, du[nt][0]);
              du[nt][1] = fmaf(off[0][o], w2.y, du[nt][1]);
              du[nt][2] = fmaf(off[1][o], w2.x, du[nt][2]);
              du[nt][3] = fmaf(off[1][o], w2.y, du[nt][3]);
            }
      }
      float u[4][4], e1[4][4];
      act_rows(g.shg + b * kFHalf, u);
      act_rows(g.se1 + b * kFHalf, e1);
      mask_rows(du, u);
      __syncthreads();
      stage(l1 + 1, 0, 2 * 4 * 768);
      // Round 1: delta of h_g and the head deltas (columns 32..47 of the
      // tile, zeros past dg); inputs e1 and h_g.
      put_rows(sD, row, 0, ft, du);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        put_pair(sD, row + 8 * h, 32 + 2 * ft, ft == 0 ? off[h][0] : ft == 1 ? off[h][2] : 0.0f,
                 ft == 0 ? off[h][1] : ft == 1 ? off[h][3] : 0.0f);
        put_pair(sD, row + 8 * h, 40 + 2 * ft, 0.0f, 0.0f);
      }
      put_rows(sX, row, 0, ft, e1);
      put_rows(sX, row, 32, ft, u);
      fetch(g.sz + (kFDepth - 1) * kFW);
      landed();
      wgrad(l1 + 1, 0, 32, 0, 32, 0, true, first);
      if (warp < 4)
        weight_grad<1>(uD, 4, uX, 4 + warp, dg, part + g.aw[l1 + 2] + 8 * warp, kFHalf, warp == 0 ? part + g.ab[l1 + 2] : nullptr, first, lane);
      float de[4][4];
      delta_w<2>(uD, warp, 0, sW, lane, de);
      mask_rows(de, e1);
      act_rows(g.sz + (kFDepth - 1) * kFW, x);
      __syncthreads();
      stage(l1, 0, 2 * 2 * 4 * 768);
      // Round 2: delta of e1, input relu(h).
      put_rows(sD, row, 0, ft, de);
      put_rows(sX, row, 0, ft, x);
      fetch(b < 3 ? (b == 1 ? g.se1 + kFW : g.se1) : g.sz + (kFDepth - 2) * kFW);
      landed();
      wgrad(l1, 0, 32, 0, 64, 0, true, first);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float z[4][4];
        delta_w<2>(uD, warp, 0, sW + h * 2 * 4 * 768, lane, z);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
          for (int i = 0; i < 4; ++i) d[4 * h + nt][i] += z[nt][i];
      }
    }
    // ---- F_out, last layer first (x holds relu(h)).
    mask_rows(d, x);
#pragma unroll 1
    for (int j = kFDepth - 1; j >= 1; --j) {
      act_rows(g.sz + (j - 1) * kFW, x);
      __syncthreads();
      stage(j, 0, kBwdW);
      put_rows(sD, row, 0, ft, d);
      put_rows(sX, row, 0, ft, x);
      if (j >= 2) fetch(g.sz + (j - 2) * kFW);
      landed();
      auto product = [&](int h) {
        float z[4][4];
        delta_w<4>(uD, warp, 0, sW, lane, z);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
#pragma unroll
          for (int i = 0; i < 4; ++i) d[4 * h + nt][i] = x[4 * h + nt][i] > 0.0f ? z[nt][i] : 0.0f;
      };
      product(0);
      __syncthreads();
      stage(j, kBwdW, kBwdW);
      wgrad(j, 0, 64, 0, 64, 0, true, first);
      landed();
      product(1);
    }
    // First layer: input f, 64 columns (two levels) at a time; d f.
#pragma unroll 1
    for (int c0 = 0; c0 < nf; c0 += kFW) {
      const bool wide = nf - c0 >= kFW;
#pragma unroll
      for (int nt = 0; nt < 8; ++nt) {
        const bool in = wide || nt < 4;
        const float2 u0 = in && valid[0] ? __ldg(reinterpret_cast<const float2*>(a.f + (size_t)p[0] * nf + c0 + 8 * nt + 2 * ft)) : make_float2(0.f, 0.f);
        const float2 u1 = in && valid[1] ? __ldg(reinterpret_cast<const float2*>(a.f + (size_t)p[1] * nf + c0 + 8 * nt + 2 * ft)) : make_float2(0.f, 0.f);
        x[nt][0] = u0.x; x[nt][1] = u0.y; x[nt][2] = u1.x; x[nt][3] = u1.y;
      }
      __syncthreads();
      stage(0, c0 / 32 * kBwdW, kBwdW);
      if (c0 == 0) put_rows(sD, row, 0, ft, d);
      put_rows(sX, row, 0, ft, x);
      landed();
      for (int h = 0; h < (wide ? 2 : 1); ++h) {
        if (h == 1) landed();
        float z[4][4];
        delta_w<4>(uD, warp, 0, sW, lane, z);
#pragma unroll
        for (int r2 = 0; r2 < 2; ++r2)
          if (valid[r2])
#pragma unroll
            for (int nt = 0; nt < 4; ++nt)
              *reinterpret_cast<float2*>(a.df + (size_t)p[r2] * nf + c0 + 32 * h + 8 * nt + 2 * ft) = make_float2(z[nt][2 * r2], z[nt][2 * r2 + 1]);
        if (h == 0) {
          __syncthreads();
          if (wide) stage(0, (c0 / 32 + 1) * kBwdW, kBwdW);
          wgrad(0, 0, 64, 0, wide ? 64 : 32, c0, c0 == 0, first);
        }
      }
    }
  }
}

// HexPlane reverse: per Gaussian and level, d f (Gaussian-major rows) through
// the channel-wise product and the bilinear weights -- plane gradients by
// 16-byte vector atomics (a corner is one 128-byte line), the canonical mean's
// gradient (the product's derivatives, carried from plane to plane) summed
// over the lanes by a fixed shuffle tree (reproducible).  Every Gaussian has
// the same time, so a time plane's gradient is a line over the spatial axis
// times the two time weights: the lines are added here (two corners instead
// of four) and spread over the planes by fst_lines_out_kernel.  The exact sums
// keep the four corners.  Bound by the gathers (250 us of it without the
// atomics) and the 18 atomic lines per level: 200k Gaussians, 4 levels: 349 us,
// 432 with four corners for every plane, 633 with lanes over channels, 4-byte
// atomics and five shuffles per sum.  At three blocks per SM (80 registers)
// it spills: 410 us; a block row per level, which the forward takes, meets
// the coarse levels' atomics all at once: 396 to 411; with one copy of the
// lines: 357.
constexpr int kHexThreads = 256;
struct HexArgs {
  FstGeom g;
  const float *planes, *means, *df, *d_means_t;
  float t;
  float* d_means;
  float* d_planes;                      // float-atomic plane sums (acc_hi == NULL)
  float4* lines;                        // and those of the time planes' lines
  unsigned long long *acc_hi, *acc_lo;  // or exact plane-gradient sums (fixed_add)
  uint32_t* err;
};

// Line of axis a of level lv (in 16-byte units; a position is kGLanes of them).
__host__ __device__ __forceinline__ size_t line_off(const FstGeom& g, int lv, int a) {
  return ((size_t)3 * g.rs * ((1u << lv) - 1u) + (size_t)a * (g.rs << lv)) * kGLanes;
}

// The time planes' gradients from the lines (n 16-byte units a copy): the two
// time rows around t.
__global__ void __launch_bounds__(256) fst_lines_out_kernel(const FstGeom g, const float4* __restrict__ lines, float t,
                                                            float* __restrict__ d_planes, int64_t n) {
  const int64_t e = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (e >= n) return;
  int lv = 0;
  while (lv + 1 < g.levels && e >= (int64_t)line_off(g, lv + 1, 0)) ++lv;
  const int64_t r = e - (int64_t)line_off(g, lv, 0);
  const int64_t per = (int64_t)(g.rs << lv) * kGLanes;
  const int a = (int)(r / per), i = (int)(r % per) / kGLanes, q = (int)(r % kGLanes);
  const Node nt = node_of(2.0f * t - 1.0f, g.rt);
  float4 v = lines[e];
#pragma unroll
  for (int c = 1; c < kLineCopies; ++c) {
    const float4 x = __ldg(lines + e + c * n);
    v = make_float4(v.x + x.x, v.y + x.y, v.z + x.z, v.w + x.w);
  }
  // Plane 3 + a is (axis a, time).
  float* o = d_planes + g.poff[lv * 6 + 3 + a] + ((int64_t)i * g.rt + nt.i) * kFC + 4 * q;
  const float w0 = 1.0f - nt.f, w1 = nt.f;
  o[0] = w0 * v.x; o[1] = w0 * v.y; o[2] = w0 * v.z; o[3] = w0 * v.w;
  o[kFC] = w1 * v.x; o[kFC + 1] = w1 * v.y; o[kFC + 2] = w1 * v.z; o[kFC + 3] = w1 * v.w;
}

// d_planes[i] = the exact sum hi 2^32 + lo, times 2^-72, rounded to float.
__global__ void __launch_bounds__(256) fst_planes_out_kernel(const unsigned long long* __restrict__ hi,
                                                             const unsigned long long* __restrict__ lo, int64_t n,
                                                             float* __restrict__ d_planes) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double v = (double)(long long)hi[i] * 0x1p-40 + (double)lo[i] * 0x1p-72;
    d_planes[i] = (float)v;
  }
}

__device__ __forceinline__ void red_add4(float4* p, float x, float y, float z, float w) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(p), "f"(x), "f"(y), "f"(z), "f"(w) : "memory");
}

// How plane gradients are added: 16-byte atomics, 4-byte atomics (planes or a
// gradient array that are not 16-byte aligned), or exactly (fixed_add).  With the
// element-wise atomics lane q has channels q, q + 8, ..., so that each
// instruction covers whole 32- or 64-byte pieces of a corner; with four
// neighbouring channels to a lane they take four times the sectors (50k
// Gaussians, 4 levels, forward + reverse + TV: exact sums 2777 us, now 1857;
// 4-byte atomics 850, now 813).
enum class PlaneAdd { kVector, kScalar, kExact };

template <PlaneAdd kAdd>
__global__ void __launch_bounds__(kHexThreads, 2) fst_hex_bwd_kernel(const HexArgs a) {
  const FstGeom& g = a.g;
  const int64_t tid = (int64_t)blockIdx.x * kHexThreads + threadIdx.x;
  const int p = (int)(tid / kGLanes), q = (int)(tid % kGLanes);
  const bool valid = p < g.P;
  float dmu[3] = {0.0f, 0.0f, 0.0f};
  if (valid) {
    float c[4];
    gauss_coords(g, a.means, p, a.t, c);
    // This lane's channels of a position (32 floats).
    constexpr bool kQuads = kAdd == PlaneAdd::kVector;
    auto load = [&](const float* x) -> float4 {
      if (kQuads) return __ldg(reinterpret_cast<const float4*>(x) + q);
      return make_float4(__ldg(x + q), __ldg(x + q + kGLanes), __ldg(x + q + 2 * kGLanes), __ldg(x + q + 3 * kGLanes));
    };
    for (int lv = 0; lv < g.levels; ++lv) {
      const float4 df4 = load(a.df + ((size_t)p * g.levels + lv) * kFC);
      const float df[4] = {df4.x, df4.y, df4.z, df4.w};
      Node n[4];
      level_nodes(g, c, lv, n);
      // Samples of the six planes; their product's derivatives along x, y, z
      // (product rule, plane by plane).
      uint32_t loc[6];  // the first corner within its plane (floats)
      float smp[6][4], pr[4], dp[3][4];
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const int ia = pair_a(k), ib = pair_b(k);
        const uint32_t row = (uint32_t)g.prb[lv * 6 + k] * kFC;
        loc[k] = (uint32_t)n[ia].i * row + (uint32_t)n[ib].i * kFC;
        const float* base = a.planes + g.poff[lv * 6 + k] + loc[k];
        const float4 v00 = load(base), v01 = load(base + kFC), v10 = load(base + row), v11 = load(base + row + kFC);
        const float p00[4] = {v00.x, v00.y, v00.z, v00.w}, p01[4] = {v01.x, v01.y, v01.z, v01.w};
        const float p10[4] = {v10.x, v10.y, v10.z, v10.w}, p11[4] = {v11.x, v11.y, v11.z, v11.w};
        const float fa = n[ia].f, fb = n[ib].f;
#pragma unroll
        for (int ch = 0; ch < 4; ++ch) {
          const float sv = (1.0f - fa) * ((1.0f - fb) * p00[ch] + fb * p01[ch]) + fa * ((1.0f - fb) * p10[ch] + fb * p11[ch]);
          const float da = (1.0f - fb) * (p10[ch] - p00[ch]) + fb * (p11[ch] - p01[ch]);
          const float db = (1.0f - fa) * (p01[ch] - p00[ch]) + fa * (p11[ch] - p10[ch]);
          smp[k][ch] = sv;
#pragma unroll
          for (int i = 0; i < 3; ++i) {
            const bool on_a = i == ia, on_b = i == ib;  // (axis 3 is time)
            if (k == 0) {
              dp[i][ch] = on_a ? da : on_b ? db : 0.0f;
            } else {
              const float t = dp[i][ch] * sv;
              dp[i][ch] = on_a ? fmaf(pr[ch], da, t) : on_b ? fmaf(pr[ch], db, t) : t;
            }
          }
          pr[ch] = k == 0 ? sv : pr[ch] * sv;
        }
      }
      float dg[3];  // d L / d(grid position) per axis, over this lane's channels
#pragma unroll
      for (int i = 0; i < 3; ++i) dg[i] = df[0] * dp[i][0] + df[1] * dp[i][1] + df[2] * dp[i][2] + df[3] * dp[i][3];
      float ds[6][4];
#pragma unroll
      for (int ch = 0; ch < 4; ++ch) {
        // The product of the other five samples by prefix / suffix products.
        float pre[6], suf = df[ch];
        pre[0] = 1.0f;
#pragma unroll
        for (int k = 1; k < 6; ++k) pre[k] = pre[k - 1] * smp[k - 1][ch];
#pragma unroll
        for (int k = 5; k >= 0; --k) {
          ds[k][ch] = pre[k] * suf;
          suf *= smp[k][ch];
        }
      }
#pragma unroll
      for (int ax = 0; ax < 3; ++ax)
        if (!n[ax].clamped) dmu[ax] = fmaf(dg[ax], 0.5f * (float)((g.rs << lv) - 1), dmu[ax]);
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const float fa = n[pair_a(k)].f, fb = n[pair_b(k)].f;
        if (kAdd != PlaneAdd::kExact && pair_b(k) == 3) {
          float4* line = a.lines + (size_t)(blockIdx.x % kLineCopies) * line_off(g, g.levels, 0) +
                         line_off(g, lv, pair_a(k)) + (size_t)n[pair_a(k)].i * kGLanes;
          const float w0 = 1.0f - fa;
          if (kQuads) {
            red_add4(line + q, w0 * ds[k][0], w0 * ds[k][1], w0 * ds[k][2], w0 * ds[k][3]);
            red_add4(line + kGLanes + q, fa * ds[k][0], fa * ds[k][1], fa * ds[k][2], fa * ds[k][3]);
          } else {
            float* x = reinterpret_cast<float*>(line) + q;
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) {
              atomicAdd(x + kGLanes * ch, w0 * ds[k][ch]);
              atomicAdd(x + kFC + kGLanes * ch, fa * ds[k][ch]);
            }
          }
          continue;
        }
        const float w[4] = {(1.0f - fa) * (1.0f - fb), (1.0f - fa) * fb, fa * (1.0f - fb), fa * fb};
        const uint32_t row = (uint32_t)g.prb[lv * 6 + k] * kFC;
        const size_t at0 = (size_t)g.poff[lv * 6 + k] + loc[k];
        const size_t at[4] = {at0, at0 + kFC, at0 + row, at0 + row + kFC};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float x[4] = {w[e] * ds[k][0], w[e] * ds[k][1], w[e] * ds[k][2], w[e] * ds[k][3]};
          if (kAdd == PlaneAdd::kExact) {
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) fixed_add(a.acc_hi, a.acc_lo, at[e] + q + kGLanes * ch, x[ch], a.err);
          } else if (kAdd == PlaneAdd::kScalar) {
#pragma unroll
            for (int ch = 0; ch < 4; ++ch) atomicAdd(a.d_planes + at[e] + q + kGLanes * ch, x[ch]);
          } else {
            red_add4(reinterpret_cast<float4*>(a.d_planes + at[e]) + q, x[0], x[1], x[2], x[3]);
          }
        }
      }
    }
  }
#pragma unroll
  for (int o = kGLanes / 2; o > 0; o >>= 1)
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) dmu[ax] += __shfl_xor_sync(0xFFFFFFFFu, dmu[ax], o);
  if (valid && q < 3) {
    const float d = q == 0 ? dmu[0] : q == 1 ? dmu[1] : dmu[2];
    a.d_means[(size_t)p * 3 + q] = a.d_means_t[(size_t)p * 3 + q] + d * g.scale[q];
  }
}

// d_mlp (caller's packed layout) = sum over blocks, in block order, of the
// partials (aligned layout).
__global__ void fst_reduce_kernel(const FstGeom g, const float* __restrict__ part, int nblk, float* __restrict__ out) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < g.mlp_packed;
       e += (int64_t)gridDim.x * blockDim.x) {
    int k = 0;
    while (k + 1 < kFLayers && e >= g.pw[k + 1]) ++k;
    const int64_t src = e < g.pb[k] ? g.aw[k] + (e - g.pw[k]) : g.ab[k] + (e - g.pb[k]);
    // Sixteen loads in flight, added in block order.
    float s = 0.0f;
    int b = 0;
    for (; b + 16 <= nblk; b += 16) {
      float v[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) v[u] = __ldg(part + (size_t)(b + u) * g.mlp_aligned + src);
#pragma unroll
      for (int u = 0; u < 16; ++u) s += v[u];
    }
    for (; b < nblk; ++b) s += part[(size_t)b * g.mlp_aligned + src];
    out[e] = s;
  }
}

// ---------------------------------------------------------------------------
// Total variation of the planes (L_TV of Eq. 11).
// ---------------------------------------------------------------------------
constexpr int kTvMaxBlocks = 1024;  // loss partials (the caller's scratch)

struct TvArgs {
  FstGeom g;
  const float* planes;
  float* d_planes;
  float weight;
  float* partial;                   // [gridDim.x]
  int bstart[kFMaxL * 6 + 1];       // first block of each plane (blocks in proportion to plane size)
};

template <bool kQuads>
__device__ __forceinline__ float4 load4(const float* p) {
  return kQuads ? *reinterpret_cast<const float4*>(p) : make_float4(p[0], p[1], p[2], p[3]);
}

// Each plane gets a share of the blocks in proportion to its size; each
// thread takes four channels of a node (the planes are channels-last, so a
// float4 per neighbour; kQuads: both arrays are 16-byte aligned, else four
// 4-byte accesses of the same sums).  One loss partial per block, summed in a
// fixed order afterwards.
template <bool kQuads>
__global__ void __launch_bounds__(256) fst_tv_kernel(const TvArgs a) {
  __shared__ float s_w[8];
  const FstGeom& g = a.g;
  int k = 0;
  while (k + 1 < g.levels * 6 && (int)blockIdx.x >= a.bstart[k + 1]) ++k;
  const int b0 = a.bstart[k], nb = a.bstart[k + 1] - b0;
  const int ra = g.pra[k], rb = g.prb[k];
  const float* planes = a.planes + g.poff[k];
  float* d_planes = a.d_planes + g.poff[k];
  const auto pl = [&](int e) { return load4<kQuads>(planes + 4 * (int64_t)e); };
  const int q4 = kFC / 4;
  const int total = ra * rb * q4;
  const float ia = 1.0f / (float)((int64_t)(ra - 1) * rb * kFC), ib = 1.0f / (float)((int64_t)ra * (rb - 1) * kFC);
  float acc = 0.0f;
  for (int e = ((int)blockIdx.x - b0) * blockDim.x + threadIdx.x; e < total; e += nb * blockDim.x) {
    const int node = e / q4;
    const int i = node / rb, j = node - i * rb;
    const float4 v = pl(e);
    float4 gr = make_float4(0.f, 0.f, 0.f, 0.f);
    auto term = [&](const float4 n, float w, bool forward) {
      // forward: n is the next node (difference n - v, counted in the loss)
      const float4 d = forward ? make_float4(n.x - v.x, n.y - v.y, n.z - v.z, n.w - v.w)
                               : make_float4(v.x - n.x, v.y - n.y, v.z - n.z, v.w - n.w);
      if (forward) acc += (d.x * d.x + d.y * d.y + d.z * d.z + d.w * d.w) * w;
      const float s = forward ? -2.0f * w : 2.0f * w;
      gr.x += s * d.x; gr.y += s * d.y; gr.z += s * d.z; gr.w += s * d.w;
    };
    if (i + 1 < ra) term(pl(e + rb * q4), ia, true);
    if (i > 0) term(pl(e - rb * q4), ia, false);
    if (j + 1 < rb) term(pl(e + q4), ib, true);
    if (j > 0) term(pl(e - q4), ib, false);
    float* dp = d_planes + 4 * (int64_t)e;
    float4 o = load4<kQuads>(dp);
    o.x += a.weight * gr.x; o.y += a.weight * gr.y; o.z += a.weight * gr.z; o.w += a.weight * gr.w;
    if (kQuads) {
      *reinterpret_cast<float4*>(dp) = o;
    } else {
      dp[0] = o.x; dp[1] = o.y; dp[2] = o.z; dp[3] = o.w;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xFFFFFFFFu, acc, o);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int w = 0; w < 8; ++w) t += s_w[w];
    a.partial[blockIdx.x] = t;
  }
}

__global__ void fst_tv_finish(const float* __restrict__ partial, int n, float weight, float* __restrict__ loss) {
  // Staged by the whole block, then added in order by one thread.
  __shared__ float s_part[kTvMaxBlocks];
  for (int b = threadIdx.x; b < n; b += blockDim.x) s_part[b] = partial[b];
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.0f;
    for (int b = 0; b < n; ++b) s += s_part[b];
    *loss = weight * s;
  }
}

bool al16p(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

}  // namespace

}  // namespace fe

using namespace fe;

extern "C" int64_t fe_fst_plane_floats(int levels, int rs, int rt) {
  fe_fst f{};
  f.levels = levels;
  f.rs = rs;
  f.rt = rt;
  f.D = 32;
  for (int a = 0; a < 3; ++a) f.bbox_max[a] = 1.0f;
  FstGeom g;
  return make_geom(&f, 0, g) ? plane_floats(g) : 0;
}

extern "C" int64_t fe_fst_mlp_floats(int levels, int D) {
  fe_fst f{};
  f.levels = levels;
  f.rs = 2;
  f.rt = 2;
  f.D = D;
  for (int a = 0; a < 3; ++a) f.bbox_max[a] = 1.0f;
  FstGeom g;
  return make_geom(&f, 0, g) ? g.mlp_packed : 0;
}

extern "C" fe_status fe_fst_workspace_size(int P, int levels, int rs, int rt, int D, int with_backward,
                                           size_t* bytes) {
  if (!bytes) return FE_ERR_INVALID_ARG;
  fe_fst f{};
  f.levels = levels;
  f.rs = rs;
  f.rt = rt;
  f.D = D;
  for (int a = 0; a < 3; ++a) f.bbox_max[a] = 1.0f;
  FstGeom g;
  if (!make_geom(&f, P, g)) return (D == 16 || D == 32 || D == 64 || D == 128) ? FE_ERR_INVALID_ARG : FE_ERR_UNSUPPORTED;
  if (with_backward < 0 || with_backward > 2) return FE_ERR_INVALID_ARG;
  *bytes = ws_layout(g, with_backward).total;
  return FE_OK;
}

namespace {

template <int D>
cudaError_t launch_fst_fwd(const FwdArgs& a, cudaStream_t st) {
  const int blocks = (a.g.P + kFM - 1) / kFM;
  const size_t smem = kFwdSmem;
  auto k = fst_fwd_kernel<D>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k<<<blocks, kFwdThreads, smem, st>>>(a);
  return cudaGetLastError();
}

template <int D>
cudaError_t launch_fst_fwd_tc(const TcArgs& a, cudaStream_t st) {
  auto k = fst_fwd_tc_kernel<D>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kTcSmem);
  k<<<(a.g.P + kTcRows - 1) / kTcRows, kTcThreads, kTcSmem, st>>>(a);
  return cudaGetLastError();
}

template <int D>
cudaError_t launch_fst_bwd(const BwdArgs& a, int nblk, cudaStream_t st) {
  const size_t smem = kBwdSmem;
  auto k = fst_bwd_kernel<D>;
  cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k<<<nblk, kBwdThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

extern "C" fe_status fe_fst_forward(const fe_fst* fst, int P, const float* means, const float* quats,
                                    const float* log_scales, const float* opacity_logits, const void* feat,
                                    int feat_bf16, float t, float* means_t, float* quats_t, float* log_scales_t,
                                    float* opacity_logits_t, void* feat_t, void* workspace, size_t workspace_bytes,
                                    int with_backward, void* stream) {
  FstGeom g;
  if (!fst || !make_geom(fst, P, g)) {
    if (fst && !(fst->D == 16 || fst->D == 32 || fst->D == 64 || fst->D == 128)) return FE_ERR_UNSUPPORTED;
    return FE_ERR_INVALID_ARG;
  }
  if (!workspace || !al16p(workspace)) return FE_ERR_INVALID_ARG;
  const WsLayout w = ws_layout(g, with_backward ? 1 : 0);
  if (workspace_bytes < w.total) return FE_ERR_WORKSPACE;
  if (P == 0) return FE_OK;
  if (!fst->planes || !fst->mlp || !means || !quats || !log_scales || !opacity_logits || !feat || !means_t ||
      !quats_t || !log_scales_t || !opacity_logits_t || !feat_t || !al16p(fst->planes) || !al16p(fst->mlp))
    return FE_ERR_INVALID_ARG;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  float* wt = reinterpret_cast<float*>(ws + w.wt);
  float* wn = reinterpret_cast<float*>(ws + w.wn);
  {
    SampArgs sa{};
    sa.g = g;
    sa.planes = fst->planes;
    sa.means = means;
    sa.t = t;
    sa.f = reinterpret_cast<float*>(ws + w.f);
    const dim3 grid((unsigned)(((int64_t)P * kGLanes + kSampThreads - 1) / kSampThreads), (unsigned)g.levels);
    fst_sample_kernel<<<grid, kSampThreads, 0, st>>>(sa);
  }
  if (!with_backward) {
    // Packed weights in the place of the FP32 copies (6 bytes a weight
    // against 8: checked, for the heads are padded to eight columns).
    const TcPlan plan = make_tc_plan(g);
    if ((size_t)plan.bytes > w.f - w.wt) return FE_ERR_WORKSPACE;
    fst_pack_tc_kernel<<<(plan.bytes / 768 * 32 + 255) / 256, 256, 0, st>>>(g, plan, fst->mlp, ws + w.wt);
    TcArgs a{};
    a.g = g;
    a.mlp = fst->mlp;
    a.wpack = ws + w.wt;
    a.nitems = plan.n;
    for (int i = 0; i < plan.n; ++i) a.bytes[i] = plan.item[i].ks * plan.item[i].nt * 768;
    a.means = means; a.quats = quats; a.log_scales = log_scales; a.logits = opacity_logits;
    a.feat = feat; a.feat_bf16 = feat_bf16 ? 1 : 0;
    a.means_t = means_t; a.quats_t = quats_t; a.log_scales_t = log_scales_t; a.logits_t = opacity_logits_t;
    a.feat_t = feat_t;
    a.f = reinterpret_cast<const float*>(ws + w.f);
    cudaError_t e = cudaErrorInvalidValue;
    switch (g.D) {
      case 16: e = launch_fst_fwd_tc<16>(a, st); break;
      case 32: e = launch_fst_fwd_tc<32>(a, st); break;
      case 64: e = launch_fst_fwd_tc<64>(a, st); break;
      case 128: e = launch_fst_fwd_tc<128>(a, st); break;
    }
    return e == cudaSuccess ? FE_OK : FE_ERR_CUDA;
  }
  if (cudaMemsetAsync(wt, 0, w.f - w.wt, st) != cudaSuccess) return FE_ERR_CUDA;
  fst_pack_kernel<<<(int)((g.mlp_packed + 255) / 256), 256, 0, st>>>(g, fst->mlp, wt, wn);
  FwdArgs a{};
  a.g = g;
  a.wt = wt;
  a.means = means;
  a.quats = quats;
  a.log_scales = log_scales;
  a.logits = opacity_logits;
  a.feat = feat;
  a.feat_bf16 = feat_bf16 ? 1 : 0;
  a.means_t = means_t;
  a.quats_t = quats_t;
  a.log_scales_t = log_scales_t;
  a.logits_t = opacity_logits_t;
  a.feat_t = feat_t;
  a.act = reinterpret_cast<float*>(ws + w.act);
  a.f = reinterpret_cast<const float*>(ws + w.f);
  // Weight tiles of the transposed copy in the order the kernel uses them.
  {
    int n = 0;
    auto add = [&](int64_t off, int rows, int cols, int ld) { a.tiles[n++] = WTile{off, rows, cols, ld}; };
    for (int l0 = 0; l0 < g.levels; l0 += 2) {
      const int nl = g.levels - l0 < 2 ? g.levels - l0 : 2;
      add(g.aw[0] + (int64_t)l0 * kFC * kFW, nl * kFC, kFW, kFW);
    }
    for (int j = 1; j < kFDepth; ++j) add(g.aw[j], kFW, kFW, kFW);
    for (int b = 0; b < 4; ++b) {
      add(g.aw[branch_e1(b)], kFW, kFHalf, kFHalf);
      add(g.aw[branch_e1(b) + 1], kFHalf, kFHalf, kFHalf);
      add(g.aw[kLZ1] + (int64_t)b * kFHalf * kFW, kFHalf, kFW, kFW);
    }
    const int zn = g.D < 64 ? g.D : 64;
    for (int c0 = 0; c0 < g.D; c0 += zn) add(g.aw[kLZ2] + c0, kFW, zn, g.D);
    a.ntiles = n;
  }
  cudaError_t e = cudaErrorInvalidValue;
  switch (g.D) {
    case 16: e = launch_fst_fwd<16>(a, st); break;
    case 32: e = launch_fst_fwd<32>(a, st); break;
    case 64: e = launch_fst_fwd<64>(a, st); break;
    case 128: e = launch_fst_fwd<128>(a, st); break;
  }
  return e == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

extern "C" fe_status fe_fst_backward(const fe_fst* fst, int P, const float* means, float t, const float* d_means_t,
                                     const float* d_quats_t, const float* d_log_scales_t,
                                     const float* d_opacity_logits_t, const float* d_feat_t, float* d_means,
                                     float* d_planes, float* d_mlp, void* workspace, size_t workspace_bytes,
                                     void* stream) {
  FstGeom g;
  if (!fst || !make_geom(fst, P, g)) {
    if (fst && !(fst->D == 16 || fst->D == 32 || fst->D == 64 || fst->D == 128)) return FE_ERR_UNSUPPORTED;
    return FE_ERR_INVALID_ARG;
  }
  if (!workspace || !al16p(workspace) || !d_planes || !d_mlp) return FE_ERR_INVALID_ARG;
  const bool exact = fst->exact_planes != 0;
  const WsLayout w = ws_layout(g, exact ? 2 : 1);
  if (workspace_bytes < w.total) return FE_ERR_WORKSPACE;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int64_t npl = plane_floats(g);
  if (P == 0) {
    if (cudaMemsetAsync(d_planes, 0, (size_t)npl * 4, st) != cudaSuccess) return FE_ERR_CUDA;
    return cudaMemsetAsync(d_mlp, 0, (size_t)g.mlp_packed * 4, st) == cudaSuccess ? FE_OK : FE_ERR_CUDA;
  }
  if (!fst->planes || !means || !d_means_t || !d_quats_t || !d_log_scales_t || !d_opacity_logits_t || !d_feat_t ||
      !d_means || !al16p(d_feat_t))
    return FE_ERR_INVALID_ARG;
  unsigned char* ws = static_cast<unsigned char*>(workspace);
  unsigned long long* acc_hi = exact ? reinterpret_cast<unsigned long long*>(ws + w.acc) : nullptr;
  unsigned long long* acc_lo = exact ? acc_hi + npl : nullptr;
  if (cudaMemsetAsync(ws, 0, kWsHeader, st) != cudaSuccess) return FE_ERR_CUDA;
  if (exact) {
    if (cudaMemsetAsync(acc_hi, 0, (size_t)npl * 16, st) != cudaSuccess) return FE_ERR_CUDA;
  } else if (cudaMemsetAsync(d_planes, 0, (size_t)npl * 4, st) != cudaSuccess) {
    return FE_ERR_CUDA;
  }
  BwdArgs a{};
  a.g = g;
  a.pk = bwd_pack(g);
  a.wp = ws + w.wp;
  a.wn = reinterpret_cast<const float*>(ws + w.wn);
  a.act = reinterpret_cast<const float*>(ws + w.act);
  a.f = reinterpret_cast<const float*>(ws + w.f);
  a.d_means_t = d_means_t;
  a.d_quats_t = d_quats_t;
  a.d_log_scales_t = d_log_scales_t;
  a.d_logits_t = d_opacity_logits_t;
  a.d_feat_t = d_feat_t;
  a.dv = reinterpret_cast<float*>(ws + w.dv);
  a.df = reinterpret_cast<float*>(ws + w.df);
  a.part = reinterpret_cast<float*>(ws + w.part);
  fst_pack_bwd_kernel<<<(a.pk.bytes / 768 * 32 + 255) / 256, 256, 0, st>>>(g, a.pk, a.wn, ws + w.wp);
  const int nblk = bwd_blocks(P);
  cudaError_t e = cudaErrorInvalidValue;
  switch (g.D) {
    case 16: e = launch_fst_bwd<16>(a, nblk, st); break;
    case 32: e = launch_fst_bwd<32>(a, nblk, st); break;
    case 64: e = launch_fst_bwd<64>(a, nblk, st); break;
    case 128: e = launch_fst_bwd<128>(a, nblk, st); break;
  }
  if (e != cudaSuccess) return FE_ERR_CUDA;
  {
    HexArgs h{};
    h.g = g;
    h.planes = fst->planes;
    h.means = means;
    h.df = a.df;
    h.d_means_t = d_means_t;
    h.t = t;
    h.d_means = d_means;
    h.d_planes = d_planes;
    h.lines = reinterpret_cast<float4*>(ws + w.lines);
    h.acc_hi = acc_hi;
    h.acc_lo = acc_lo;
    h.err = reinterpret_cast<uint32_t*>(ws);
    const int hb = (int)(((int64_t)P * kGLanes + kHexThreads - 1) / kHexThreads);
    if (exact) {
      fst_hex_bwd_kernel<PlaneAdd::kExact><<<hb, kHexThreads, 0, st>>>(h);
      const int64_t nb = (npl + 255) / 256;
      fst_planes_out_kernel<<<(int)(nb < 152 * 16 ? nb : 152 * 16), 256, 0, st>>>(acc_hi, acc_lo, npl, d_planes);
    } else {
      const size_t lb = line_bytes(g);
      if (cudaMemsetAsync(h.lines, 0, lb, st) != cudaSuccess) return FE_ERR_CUDA;
      if (al16p(d_planes) && al16p(fst->planes)) fst_hex_bwd_kernel<PlaneAdd::kVector><<<hb, kHexThreads, 0, st>>>(h);
      else fst_hex_bwd_kernel<PlaneAdd::kScalar><<<hb, kHexThreads, 0, st>>>(h);
      const int64_t nl = (int64_t)(lb / 16 / kLineCopies);
      fst_lines_out_kernel<<<(int)((nl + 255) / 256), 256, 0, st>>>(g, h.lines, t, d_planes, nl);
    }
  }
  fst_reduce_kernel<<<(int)((g.mlp_packed + 255) / 256), 256, 0, st>>>(g, a.part, nblk, d_mlp);
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}

extern "C" fe_status fe_fst_tv(const fe_fst* fst, float weight, float* loss, float* d_planes, float* scratch,
                               void* stream) {
  FstGeom g;
  if (!fst || !make_geom(fst, 0, g)) return FE_ERR_INVALID_ARG;
  if (!fst->planes || !loss || !d_planes || !scratch) return FE_ERR_INVALID_ARG;
  {
    // The gradient array must not overlap the planes (the kernel reads the
    // planes while it updates the gradient).
    const uintptr_t p0 = reinterpret_cast<uintptr_t>(fst->planes), d0 = reinterpret_cast<uintptr_t>(d_planes);
    const uintptr_t n = (uintptr_t)plane_floats(g) * sizeof(float);
    if (p0 < d0 + n && d0 < p0 + n) return FE_ERR_INVALID_ARG;
  }
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  TvArgs a{};
  a.g = g;
  a.planes = fst->planes;
  a.d_planes = d_planes;
  a.weight = weight;
  a.partial = scratch;
  // Blocks per plane in proportion to its size (at least one), at most
  // kTvMaxBlocks in all.
  const int np = g.levels * 6;
  const double total = (double)plane_floats(g);
  const int budget = kTvMaxBlocks - np;
  a.bstart[0] = 0;
  for (int k = 0; k < np; ++k) {
    const double n = (double)g.pra[k] * g.prb[k] * kFC;
    a.bstart[k + 1] = a.bstart[k] + 1 + (int)(budget * n / total);
  }
  const int nblk = a.bstart[np];
  if (al16p(fst->planes) && al16p(d_planes)) fst_tv_kernel<true><<<nblk, 256, 0, st>>>(a);
  else fst_tv_kernel<false><<<nblk, 256, 0, st>>>(a);
  fst_tv_finish<<<1, 256, 0, st>>>(scratch, nblk, weight, loss);
  return cudaGetLastError() == cudaSuccess ? FE_OK : FE_ERR_CUDA;
}
