// Packed draft-graph attention (Sec. 4.3; mask of Fig. 3) on the fp32 CUDA
// cores.  This is the kernel for fp32 inputs (tensor cores would need TF32,
// whose 10-bit mantissa cannot hold a 1e-4 tolerance), and for bf16 where it is
// asked for by name or more than 128 query heads share a kv head.
//
// Work decomposition.  For one sequence and one key/value head the query rows are
// all (node, position, query head of the group) triples; they share the context
// keys.  A CTA owns M consecutive rows and walks over tiles of 64 keys: context
// tiles, then the tiles covering the block keys of the nodes its rows belong to.
// The mask is never materialised: in a block-key tile a row sees the contiguous
// column range of its own node.  The key tiles of one row tile are split over the
// CTAs of a cluster, which merge their partials through each other's shared
// memory; M and the cluster size are chosen so that short problems still spread
// over the machine (see choose()).
//
// Inside a CTA 128 threads form an 8 x 16 grid: thread (rg, kg) computes the
// scores of rows rg, rg + 8, ... against keys kg, kg + 16, ..., and then the
// output columns 4 kg .. 4 kg + 3 (and + 64) of the same rows, so that the
// probabilities pass through shared memory inside one half-warp only.  All
// operands come as 16-byte loads from shared memory (chunks XOR-swizzled by row:
// no bank conflicts, no padding) and feed packed fp32x2 multiply-adds; K of the
// next tile is fetched under P V, V under Q K^T, by asynchronous copies.
//
// Bound: the fp32 multiply-add pipe when there is enough work (20 TFLOP/s at 288
// positions x 12 heads over 1000 keys, d = 128; a quarter of the pipe's rate, the
// rest goes to padding, to doubling P for the packed instructions and to the last
// wave); for the shortest calls one tile's latency chain and the launch.  The
// kernel before this one (a CTA per node and head, a warp per row) took 24.1 us for
// 4 nodes x 8 positions x 4 heads over 128 keys and 433 us for 2 x 2 x 4 positions
// x 24 heads on 8 over 3249 keys, d = 64; this one 5.9 and 34.2 us.  (Some twenty divisions of the set-up and
// the rows' places by multiplication: 0.45 us of the former's step, 9.5 -> 9.05.)
#include <math.h>

#include "common.cuh"
#include "sm100_ptx.cuh"

namespace spiffy {
namespace {

constexpr int kThreads = 128;
constexpr int kKeys = 64;  // keys per tile
constexpr int kMaxCluster = 8;

struct SimtParams {
  int NL, L, P, Hq, Hkv, group;
  int rows;      // NL * group rows per (sequence, kv head)
  int ctx_tiles; // context key tiles
  int row_tiles; // tiles of M rows
  int slices;    // CTAs the key tiles of a row tile are split over
  float scale;
  FastDiv by_slices, by_row_tiles, by_Hkv, by_group, by_L;
};

// Float offset of 16-byte chunk c of row r in a swizzled [rows][W] tile.
template <int W>
__device__ __forceinline__ int chunk_at(int r, int c) {
  return r * W + ((c ^ (r & 7)) << 2);
}

// Four elements (one chunk) of a row into shared memory as fp32; zeros when !valid.
__device__ __forceinline__ void stage4(float* dst, const float* src, bool valid) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(valid ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void stage4(float* dst, const __nv_bfloat16* src, bool valid) {
  uint2 w = valid ? *reinterpret_cast<const uint2*>(src) : make_uint2(0u, 0u);
  *reinterpret_cast<float4*>(dst) = make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u),
                                                __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ void stage_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// grid = slices (the cluster size) * row tiles * Hkv * B, slices innermost.
template <typename T, int D, int M>
__global__ void __launch_bounds__(kThreads)
graph_attention_simt_kernel(const SimtParams p, const T* __restrict__ q, const T* __restrict__ kp,
                            const T* __restrict__ vp, const T* __restrict__ kb, const T* __restrict__ vb,
                            T* __restrict__ out) {
  constexpr int R = M / 8;    // rows per thread
  constexpr int C = D / 64;   // output chunks of 4 columns per thread
  constexpr int kChunks = D / 4;
  extern __shared__ __align__(16) float simt_smem[];
  float* sq = simt_smem;        // [M][D]
  float* sk = sq + M * D;       // [64][D]
  float* sv = sk + kKeys * D;   // [64][D]
  float* sp = sv + kKeys * D;   // [M][64]
  float2* sml = reinterpret_cast<float2*>(sp);  // [M] (maximum, sum) of this slice, once P is done with

  const int tid = threadIdx.x, rg = tid >> 4, kg = tid & 15;
  const int slices = p.slices, at = p.by_slices.div((int)blockIdx.x), slice = (int)blockIdx.x - at * slices;
  const int bg = p.by_row_tiles.div(at), tile = at - bg * p.row_tiles;
  const int b = p.by_Hkv.div(bg), g = bg - b * p.Hkv;
  const int row0 = tile * M;
  const int n_rows = min(M, p.rows - row0);
  const int n_lo = p.by_L.div(p.by_group.div(row0)), n_hi = p.by_L.div(p.by_group.div(row0 + n_rows - 1));
  const int kb_start = n_lo * p.L, kb_count = (n_hi - n_lo + 1) * p.L;
  const int T_all = p.ctx_tiles + (kb_count + kKeys - 1) / kKeys;
  const int t0 = p.by_slices.div(slice * T_all), t1 = p.by_slices.div((slice + 1) * T_all);

  cudaGridDependencySynchronize();  // inputs written by earlier kernels are visible
  pdl_launch_dependents();
  for (int i = tid; i < M * kChunks; i += kThreads) {
    const int r = i / kChunks, c = i % kChunks;
    const int rr = min(row0 + r, p.rows - 1);
    const int nl = p.by_group.div(rr), hh = rr - nl * p.group;
    stage4(sq + chunk_at<D>(r, c), q + (((int64_t)b * p.NL + nl) * p.Hq + g * p.group + hh) * D + 4 * c, r < n_rows);
  }
  // K or V of key tile t into `dst`; keys beyond the segment's end are zeros
  auto stage_tile = [&](float* dst, const T* ctx, const T* blk, int t) {
    const bool in_ctx = t < p.ctx_tiles;
    const int first = in_ctx ? t * kKeys : kb_start + (t - p.ctx_tiles) * kKeys;
    const int last = in_ctx ? p.P : kb_start + kb_count;
    const T* src = (in_ctx ? ctx + (int64_t)b * p.P * p.Hkv * D : blk + (int64_t)b * p.NL * p.Hkv * D) + (int64_t)g * D;
    for (int i = tid; i < kKeys * kChunks; i += kThreads) {
      const int r = i / kChunks, c = i % kChunks;
      const int key = first + r;
      stage4(dst + chunk_at<D>(r, c), src + (int64_t)min(key, last - 1) * p.Hkv * D + 4 * c, key < last);
    }
  };
  if (t0 < t1) stage_tile(sk, kp, kb, t0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  if (t0 < t1) stage_tile(sv, vp, vb, t0);
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 1;" ::: "memory");  // Q and the first K are here
  __syncthreads();

  float m[R], l[R];
  uint64_t o[R][C][2];
  int node_lo[R];  // first block key of the row's own node, relative to kb_start
#pragma unroll
  for (int i = 0; i < R; ++i) {
    m[i] = -INFINITY;
    l[i] = 0.f;
    node_lo[i] = p.by_L.div(p.by_group.div(min(row0 + rg + 8 * i, p.rows - 1))) * p.L - kb_start;
#pragma unroll
    for (int c = 0; c < C; ++c) o[i][c][0] = o[i][c][1] = pack2(0.f, 0.f);
  }

  for (int t = t0; t < t1; ++t) {
    // scores: sums over even and odd dimensions in the two halves of a pair
    uint64_t acc[R][4];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = pack2(0.f, 0.f);
#pragma unroll 2
    for (int c = 0; c < kChunks; ++c) {
      ulonglong2 qv[R], kv[4];
#pragma unroll
      for (int i = 0; i < R; ++i) qv[i] = *reinterpret_cast<const ulonglong2*>(sq + chunk_at<D>(rg + 8 * i, c));
#pragma unroll
      for (int j = 0; j < 4; ++j) kv[j] = *reinterpret_cast<const ulonglong2*>(sk + chunk_at<D>(kg + 16 * j, c));
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fma2(qv[i].x, kv[j].x, acc[i][j]);
          acc[i][j] = fma2(qv[i].y, kv[j].y, acc[i][j]);
        }
    }
    const bool in_ctx = t < p.ctx_tiles;
    const int rel = in_ctx ? 0 : (t - p.ctx_tiles) * kKeys;
#pragma unroll
    for (int i = 0; i < R; ++i) {
      // the columns of this tile the row sees
      const int lo = in_ctx ? 0 : node_lo[i] - rel;
      const int hi = in_ctx ? p.P - t * kKeys : lo + p.L;
      float s[4], mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        float a0, a1;
        unpack2(acc[i][j], a0, a1);
        const int col = kg + 16 * j;
        s[j] = (col >= lo && col < hi) ? (a0 + a1) * p.scale : -INFINITY;
        mx = fmaxf(mx, s[j]);
      }
#pragma unroll
      for (int off = 8; off > 0; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
      const float m_new = fmaxf(m[i], mx);
      const float m_use = m_new == -INFINITY ? 0.f : m_new;
      if (m_new > m[i]) {
        const float corr = expf(m[i] - m_use);  // 0 for a row that had seen nothing yet
        l[i] *= corr;
        m[i] = m_new;
        const uint64_t c2 = pack2(corr, corr);
#pragma unroll
        for (int c = 0; c < C; ++c) {
          o[i][c][0] = fma2(o[i][c][0], c2, pack2(0.f, 0.f));
          o[i][c][1] = fma2(o[i][c][1], c2, pack2(0.f, 0.f));
        }
      }
      const int r = rg + 8 * i;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float e = expf(s[j] - m_use);
        l[i] += e;
        const int col = kg + 16 * j;
        sp[chunk_at<kKeys>(r, col >> 2) + (col & 3)] = e;
      }
    }
    stage_wait();     // V of this tile
    __syncthreads();  // ... of every thread; K has been read
    if (t + 1 < t1) stage_tile(sk, kp, kb, t + 1);
#pragma unroll 4  // 1 to 2 % over two (64 x 32 positions x 32 heads on 8 over 4000 keys 3175 us, 3132 so)
    for (int c4 = 0; c4 < kKeys / 4; ++c4) {
      float4 pv[R];
#pragma unroll
      for (int i = 0; i < R; ++i) pv[i] = *reinterpret_cast<const float4*>(sp + chunk_at<kKeys>(rg + 8 * i, c4));
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        ulonglong2 vv[C];
#pragma unroll
        for (int c = 0; c < C; ++c)
          vv[c] = *reinterpret_cast<const ulonglong2*>(sv + chunk_at<D>(4 * c4 + e, kg + 16 * c));
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const float pe = e == 0 ? pv[i].x : e == 1 ? pv[i].y : e == 2 ? pv[i].z : pv[i].w;
          const uint64_t p2 = pack2(pe, pe);
#pragma unroll
          for (int c = 0; c < C; ++c) {
            o[i][c][0] = fma2(p2, vv[c].x, o[i][c][0]);
            o[i][c][1] = fma2(p2, vv[c].y, o[i][c][1]);
          }
        }
      }
    }
    stage_wait();     // K of the next tile
    __syncthreads();  // V and P have been read
    if (t + 1 < t1) stage_tile(sv, vp, vb, t + 1);
  }
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int off = 8; off > 0; off >>= 1) l[i] += __shfl_xor_sync(0xffffffffu, l[i], off);

  auto store4 = [&](int r, int col, float a0, float a1, float a2, float a3) {
    const int rr = row0 + r, nl = p.by_group.div(rr), hh = rr - nl * p.group;
    T* at = out + (((int64_t)b * p.NL + nl) * p.Hq + g * p.group + hh) * D + col;
    if constexpr (sizeof(T) == 4) {
      *reinterpret_cast<float4*>(at) = make_float4(a0, a1, a2, a3);
    } else {
      const __nv_bfloat162 lo = __floats2bfloat162_rn(a0, a1), hi = __floats2bfloat162_rn(a2, a3);
      *reinterpret_cast<uint2*>(at) = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
    }
  };
  if (slices == 1) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const float inv = 1.0f / l[i];
      if (rg + 8 * i < n_rows)
#pragma unroll
        for (int c = 0; c < C; ++c) {
          float a0, a1, a2, a3;
          unpack2(o[i][c][0], a0, a1);
          unpack2(o[i][c][1], a2, a3);
          store4(rg + 8 * i, 4 * (kg + 16 * c), a0 * inv, a1 * inv, a2 * inv, a3 * inv);
        }
    }
    return;
  }
  // This slice's partial into its own shared memory (over Q), then every CTA of the
  // cluster merges its share of the rows, slices in ascending order.
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = rg + 8 * i;
#pragma unroll
    for (int c = 0; c < C; ++c)
      *reinterpret_cast<ulonglong2*>(sq + chunk_at<D>(r, kg + 16 * c)) = make_ulonglong2(o[i][c][0], o[i][c][1]);
    if (kg == 0) sml[r] = make_float2(m[i], l[i]);
  }
  sm100::cluster_arrive();
  sm100::cluster_wait();
  const uint32_t q_addr = sm100::smem_u32(sq), ml_addr = sm100::smem_u32(sml);
  for (int i = slice * kThreads + tid; i < n_rows * kChunks; i += slices * kThreads) {
    const int r = i / kChunks, c = i % kChunks;
    float2 ml[kMaxCluster];
    float4 part[kMaxCluster];
    float mx = -INFINITY;
#pragma unroll
    for (int s = 0; s < kMaxCluster; ++s) {
      if (s >= slices) continue;
      asm volatile("ld.shared::cluster.v2.f32 {%0,%1}, [%2];"
                   : "=f"(ml[s].x), "=f"(ml[s].y)
                   : "r"(sm100::map_to_cta(ml_addr, (uint32_t)s) + (uint32_t)r * 8u));
      asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];"
                   : "=f"(part[s].x), "=f"(part[s].y), "=f"(part[s].z), "=f"(part[s].w)
                   : "r"(sm100::map_to_cta(q_addr, (uint32_t)s) + (uint32_t)chunk_at<D>(r, c) * 4u));
      mx = fmaxf(mx, ml[s].x);
    }
    float sum = 0.f, a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
    for (int s = 0; s < kMaxCluster; ++s) {
      if (s >= slices || ml[s].x == -INFINITY) continue;  // this slice held no key the row sees
      const float w = expf(ml[s].x - mx);
      sum = fmaf(w, ml[s].y, sum);
      a0 = fmaf(w, part[s].x, a0);
      a1 = fmaf(w, part[s].y, a1);
      a2 = fmaf(w, part[s].z, a2);
      a3 = fmaf(w, part[s].w, a3);
    }
    const float inv = 1.0f / sum;
    store4(r, 4 * c, a0 * inv, a1 * inv, a2 * inv, a3 * inv);
  }
  sm100::cluster_arrive();  // nobody leaves while its shared memory may still be read
  sm100::cluster_wait();
}

struct Choice {
  int m, slices;
};
// Rows per CTA and slices of the key tiles: the pair that a small model of the
// kernel's time finds cheapest.  A CTA alone on its SM takes `alone` us per key
// tile (a latency chain), several CTAs together `shared` us per tile and CTA (the
// SM's throughput), as measured at head dimension 128; 64 takes 0.85 and 0.6 of
// that; the exchange between slices costs 2.5 us.  Fewer rows per CTA read the
// keys more often and feed the multiply-adds worse, but short problems would
// leave most SMs idle otherwise.  Clusters of 2, 4 and 8 pack the machine; other
// sizes are taken only where they give every key tile a CTA of its own.
Choice choose(const spiffy_attn_desc& d) {
  constexpr int kRows[3] = {64, 32, 16};
  constexpr float alone[3] = {9.6f, 6.4f, 3.4f}, shared[3] = {8.8f, 4.7f, 4.3f};
  const int sms = sm_count() > 0 ? sm_count() : 1;
  const int64_t rows = (int64_t)d.n_nodes * d.block_len * (d.n_q_heads / d.n_kv_heads);
  const int64_t bg = (int64_t)d.batch * d.n_kv_heads;
  const int tiles = (d.prefix_len + kKeys - 1) / kKeys + 1;  // at least
  Choice best = {64, 1};
  float best_cost = INFINITY;
  for (int i = 0; i < 3; ++i) {
    const int64_t ctas = bg * ((rows + kRows[i] - 1) / kRows[i]);
    for (int s = 1; s <= kMaxCluster && s <= tiles; ++s) {
      const int64_t per_sm = (ctas * s + sms - 1) / sms;
      const int per_slice = (tiles + s - 1) / s;
      if ((s & (s - 1)) != 0 && (s != tiles || per_sm > 1)) continue;
      const bool narrow = d.head_dim == 64;
      const float tile = per_sm > 1 ? (float)per_sm * shared[i] * (narrow ? 0.6f : 1.0f)
                                    : alone[i] * (narrow ? 0.85f : 1.0f);
      const float cost = (s > 1 ? 2.5f : 0.f) + tile * (float)per_slice;
      if (cost < best_cost) {
        best_cost = cost;
        best = {kRows[i], s};
      }
    }
  }
  return best;
}

template <typename T, int D, int M>
spiffy_status launch(const spiffy_attn_desc& d, int slices, const void* q, const void* kp, const void* vp,
                     const void* kb, const void* vb, void* out, cudaStream_t stream) {
  constexpr int kSmem = (M * D + 2 * kKeys * D + M * kKeys) * 4;
  auto kern = graph_attention_simt_kernel<T, D, M>;
  static std::atomic<bool> smem_allowed[64];
  if (!allow_smem(kern, kSmem, smem_allowed)) return SPIFFY_ECUDA;
  SimtParams p;
  p.NL = d.n_nodes * d.block_len;
  p.L = d.block_len;
  p.P = d.prefix_len;
  p.Hq = d.n_q_heads;
  p.Hkv = d.n_kv_heads;
  p.group = d.n_q_heads / d.n_kv_heads;
  p.rows = p.NL * p.group;
  p.ctx_tiles = (d.prefix_len + kKeys - 1) / kKeys;
  p.row_tiles = (p.rows + M - 1) / M;
  p.slices = slices;
  p.scale = d.scale != 0.f ? d.scale : 1.0f / sqrtf((float)d.head_dim);
  p.by_slices = FastDiv::by(slices);
  p.by_row_tiles = FastDiv::by(p.row_tiles);
  p.by_Hkv = FastDiv::by(p.Hkv);
  p.by_group = FastDiv::by(p.group);
  p.by_L = FastDiv::by(p.L);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((int64_t)slices * p.row_tiles * d.n_kv_heads * d.batch));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = kSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)slices;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = slices > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kern, p, static_cast<const T*>(q), static_cast<const T*>(kp),
                                           static_cast<const T*>(vp), static_cast<const T*>(kb),
                                           static_cast<const T*>(vb), static_cast<T*>(out));
  count_launch();
  return e == cudaSuccess ? SPIFFY_OK : SPIFFY_ECUDA;
}

template <typename T, int D>
spiffy_status launch_m(const spiffy_attn_desc& d, const void* q, const void* kp, const void* vp, const void* kb,
                       const void* vb, void* out, cudaStream_t stream) {
  const Choice c = choose(d);
  if (c.m == 64) return launch<T, D, 64>(d, c.slices, q, kp, vp, kb, vb, out, stream);
  if (c.m == 32) return launch<T, D, 32>(d, c.slices, q, kp, vp, kb, vb, out, stream);
  return launch<T, D, 16>(d, c.slices, q, kp, vp, kb, vb, out, stream);
}

}  // namespace

spiffy_status launch_attention_simt(const spiffy_attn_desc& d, const void* q, const void* kp, const void* vp,
                                    const void* kb, const void* vb, void* out, cudaStream_t stream) {
  if (d.dtype == SPIFFY_F32) {
    if (d.head_dim == 64) return launch_m<float, 64>(d, q, kp, vp, kb, vb, out, stream);
    return launch_m<float, 128>(d, q, kp, vp, kb, vb, out, stream);
  }
  if (d.head_dim == 64) return launch_m<__nv_bfloat16, 64>(d, q, kp, vp, kb, vb, out, stream);
  return launch_m<__nv_bfloat16, 128>(d, q, kp, vp, kb, vb, out, stream);
}

}  // namespace spiffy
