// octree.cu -- maintenance of the point-probability octree (Sec. 3.1:
// "Probability Updates" Eq. 2 / Eq. 3, "Subdivision", "Pruning"; App. A.4
// leaf layout) and the per-point blending weights it consumes (App. A.6).
//
// Blending weights: after a forward, every pixel's blended prefix (recorded
// by the forward in blending order) is walked once more with the product scan
// of whole warps: T_k alpha_k is bitwise the forward's for widths that whole
// warps blend, and agrees to FP32 rounding for narrower ones; each splat's
// value lands at its point's entry for the footprint corner it came from
// and a per-point pass combines a point's four splats with their bilinear
// weights.
//
// Updates: per-leaf max and min of the weights of the points drawn from the
// leaf (as FP32 bit patterns: non-negative floats order like their bits)
// with a warp-level reduction over runs of equal leaves first (the sampler
// emits points grouped by leaf), then one FP64 update per leaf.
//
// Subdivision and pruning: an exclusive scan of the per-leaf output counts
// (8 or 1; 1 or 0) gives every surviving leaf its place, so children
// replace their parent in place and the order of the list is kept.
#include "raster_impl.cuh"

namespace inpc {
namespace {

// ------------------------------------------------------ blending weights ---
// The values T_k alpha_k lie point-major, entry 4 p + c for point p's corner c
// (the memory of the backward's pairs).
__device__ __forceinline__ float* splat_values(const RasterWs& ws) { return reinterpret_cast<float*>(ws.fscal); }

// The pixels with at most 8 blended fragments (`few`: the lanes that hold their
// bucket start, size, count and place), four at a time on 8 lanes each, the next
// four's order read while these are walked.  The product scan of 8 lanes is the
// one of 32 on its first 8, so the values are the same bits.
__device__ __forceinline__ void few_splat_weights(const RP& P, const RasterWs& ws, float* __restrict__ val,
                                                  unsigned few, uint32_t s0, int m, int nb, int qx, int qy) {
  const Group<8> L;
  const int g = L.base_lane >> 3;
  int j = 0, jnb = 0;
  uint32_t js0 = 0;
  uint2 o = make_uint2(0, 0);
  const auto next = [&]() {  // this group's next pixel and its order entries
    unsigned f = few;
#pragma unroll
    for (int i = 0; i < 3; ++i)
      if (i < g) f &= f - 1;
    const bool any = f != 0;
    j = any ? __ffs(f) - 1 : 0;
    jnb = __shfl_sync(0xffffffffu, nb, j);
    js0 = __shfl_sync(0xffffffffu, s0, j);
    const int jm = __shfl_sync(0xffffffffu, m, j);
    if (!any) jnb = 0;
    if (L.lg < jnb) o = order_at(P, ws, js0, jm, L.lg);
#pragma unroll
    for (int i = 0; i < 4; ++i) few &= few - 1;  // 0 stays 0
  };
  bool more = few != 0;
  if (more) next();
  while (more) {
    const int cnb = jnb, cx = __shfl_sync(0xffffffffu, qx, j), cy = __shfl_sync(0xffffffffu, qy, j);
    const uint32_t cs0 = js0;
    const uint2 co = o;
    more = few != 0;
    if (more) next();
    const bool valid = L.lg < cnb;
    float a = 0.f;
    uint32_t dst = 0;
    if (valid) {
      a = ws.alpha[cs0 + co.x];
      dst = frag_index(ws, co.y, cx, cy);
    }
    const ChunkT<8> ct = chunk_transmittance<8>(L, P, a, valid, cnb, 1.0f);
    if (L.lg < ct.take) val[dst] = __fmul_rn(ct.Tk, a);
  }
}

// Pixels that lie a grid of warps apart (neighbouring ones, whose points they
// share, are walked at the same time), 32 to a warp: one lane each reads their
// buckets, so empty pixels cost no chain of loads; pixels of up to 8 blended
// fragments go four at a time, the others a warp each, a pixel's order entries
// read while the one before is walked.  A warp for every pixel leaves most of
// its lanes idle and most of its time in one pixel's chain of loads: 300,000
// points at 1280 x 832 141 -> 56 us (a grid-stride loop over all pixels 103),
// 600,000 at 1920 x 1080 256 -> 90, 4M there (8 fragments a pixel) 395 -> 224;
// 1M leaf-grouped points at 640 x 416 the same, near the L2's rate of partly
// written sectors (4.2M stores, 125G/s).  The times are of the whole call.
constexpr int kSplatCtas = 8;  // per SM (5, 6 and 7: 4M points 252, 233 us; leaf-grouped ones 73, 68 and 67, with 8 66)
__global__ void __launch_bounds__(256, kSplatCtas) k_pixel_splat_weights(RP P, const int32_t* __restrict__ n_contrib,
                                                                        RasterWs ws) {
  const Group<32> G;
  float* const val = splat_values(ws);
  const long long n_warps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w0 < P.n_pix; w0 += 32 * n_warps) {
    // the warp's next 32 pixels, one per lane
    const long long mine = w0 + G.lg * n_warps;
    uint32_t s0 = 0;
    int m = 0, nb = 0;
    if (mine < P.n_pix) {
      s0 = ws.pix_start[mine];
      m = (int)(ws.pix_start[mine + 1] - s0);
      nb = blended_count(n_contrib, mine, m);
    }
    const int qy = (int)((uint32_t)mine / (uint32_t)P.cam.W), qx = (int)((uint32_t)mine - (uint32_t)qy * P.cam.W);
    few_splat_weights(P, ws, val, __ballot_sync(0xffffffffu, nb > 0 && nb <= 8), s0, m, nb, qx, qy);
    unsigned todo = __ballot_sync(0xffffffffu, nb > 8);
    uint2 o_next = make_uint2(0, 0);
    const auto first_order = [&]() {  // of the next pixel
      if (!todo) return;
      const int j = __ffs(todo) - 1;
      const uint32_t js0 = G.bcast(s0, j);
      const int jm = G.bcast(m, j), jnb = G.bcast(nb, j);
      if (G.lg < jnb) o_next = order_at(P, ws, js0, jm, G.lg);
    };
    first_order();
    while (todo) {
      const int j = __ffs(todo) - 1;
      todo &= todo - 1;
      const int jqx = G.bcast(qx, j), jqy = G.bcast(qy, j);
      const uint32_t js0 = G.bcast(s0, j);
      const int jm = G.bcast(m, j), jnb = G.bcast(nb, j);
      uint2 o = o_next;
      first_order();
      float T = 1.0f;
      for (int b = 0;;) {
        const bool valid = b + G.lg < jnb;
        float a = 0.f;
        uint32_t dst = 0;
        if (valid) {
          a = ws.alpha[js0 + o.x];
          dst = frag_index(ws, o.y, jqx, jqy);
        }
        const ChunkT<32> ct = chunk_transmittance<32>(G, P, a, valid, min(32, jnb - b), T);
        if (G.lg < ct.take) val[dst] = __fmul_rn(ct.Tk, a);
        T = G.bcast(ct.Tn, ct.take - 1);
        b += 32;
        if (ct.stop || b >= jnb) break;
        if (b + G.lg < jnb) o = order_at(P, ws, js0, jm, b + G.lg);
      }
    }
  }
}

__global__ void __launch_bounds__(256) k_point_blend_weights(RP P, const float* __restrict__ pos, RasterWs ws,
                                                            float* __restrict__ b_out) {
  for (long long id = blockIdx.x * (long long)blockDim.x + threadIdx.x; id < P.n;
       id += (long long)gridDim.x * blockDim.x) {
    float b = 0.f;
    Splat s;
    if (splat_point(P, pos, id, s)) {
      // zero where nothing blended
      const float4 f = __ldg(reinterpret_cast<const float4*>(splat_values(ws)) + id);
      const float sc[4] = {f.x, f.y, f.z, f.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) b = __fmaf_rn(corner_weight(s.f, k & 1, k >> 1), sc[k], b);
    }
    b_out[id] = b;
  }
}

// --------------------------------------------------------------- updates ---
struct UpdateWs {
  uint32_t* status;
  uint32_t* bmax;  // [L] FP32 bits
  uint32_t* bmin;  // [L] the maximum of the complemented bits (so that both start from zero), 0 when no
                   // point was drawn from the leaf
  size_t bytes;
};

UpdateWs carve_update(void* base, int64_t L) {
  Carver c(base);
  UpdateWs w;
  w.status = static_cast<uint32_t*>(base);
  w.bmax = c.take<uint32_t>(std::max<int64_t>(L, 1));
  w.bmin = c.take<uint32_t>(std::max<int64_t>(L, 1));
  w.bytes = c.bytes();
  return w;
}

__global__ void __launch_bounds__(256) k_leaf_minmax(const int32_t* __restrict__ leaf_idx,
                                                    const float* __restrict__ b, long long n, long long L,
                                                    UpdateWs ws) {
  const int lane = threadIdx.x & 31;
  const long long stride = (long long)gridDim.x * blockDim.x;
  // the trip count is uniform per warp, so every lane takes part in the shuffles
  for (long long base = (long long)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < n; base += stride) {
    const long long id = base + lane;
    int leaf = -1;
    uint32_t bits = 0;
    if (id < n) {
      leaf = leaf_idx[id];
      const float v = b[id];
      bits = __float_as_uint(v);
      if (!(v >= 0.0f) || (bits & 0x80000000u)) {  // negative, -0 or NaN: counted as 0
        if (!(v == 0.0f)) raise_status(ws.status, INPC_DEV_BAD_BLEND_WEIGHT);
        bits = 0;
      }
      if (leaf < 0 || (long long)leaf >= L) {
        raise_status(ws.status, INPC_DEV_BAD_LEAF);
        leaf = -1;
      }
    }
    uint32_t mx = bits, mn = bits;
    // runs of equal leaves: lane i ends with the max / min over its run from i on
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ol = __shfl_down_sync(0xffffffffu, leaf, o);
      const uint32_t omx = __shfl_down_sync(0xffffffffu, mx, o);
      const uint32_t omn = __shfl_down_sync(0xffffffffu, mn, o);
      if (lane + o < 32 && ol == leaf) {
        mx = max(mx, omx);
        mn = min(mn, omn);
      }
    }
    const int prev = __shfl_up_sync(0xffffffffu, leaf, 1);
    if (leaf >= 0 && (lane == 0 || prev != leaf)) {
      atomicMax(ws.bmax + leaf, mx);
      atomicMax(ws.bmin + leaf, ~mn);
    }
  }
}

__global__ void k_leaf_update(double* __restrict__ p, double* __restrict__ q, long long L, double lambda_u,
                              UpdateWs ws) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < L; i += (long long)gridDim.x * blockDim.x) {
    const double dp = __dmul_rn(lambda_u, p[i]), dq = __dmul_rn(lambda_u, q[i]);
    if (ws.bmin[i] == 0u) {  // no point drawn from the leaf: decay only
      p[i] = dp;
      q[i] = dq;
    } else {
      const double mx = (double)__uint_as_float(ws.bmax[i]), mn = (double)__uint_as_float(~ws.bmin[i]);
      const double spread = __dsub_rn(mx, mn);
      p[i] = mx > dp ? mx : dp;
      q[i] = spread > dq ? spread : dq;
    }
  }
}

// ---------------------------------------------------- subdivide / prune ---
struct RefineWs {
  uint32_t* offset;  // [L] exclusive scan of the output counts
  uint32_t* tops;    // scan block totals; grand total at the end
  size_t bytes;
};

RefineWs carve_refine(void* base, int64_t L) {
  Carver c(base);
  RefineWs w;
  w.offset = c.take<uint32_t>(std::max<int64_t>(L, 1));
  w.tops = c.take<uint32_t>(scan::n_tops(std::max<int64_t>(L, 1)));
  w.bytes = c.bytes();
  return w;
}

struct SplitCount {
  const double* q;
  double tau;
  __device__ uint32_t operator()(int64_t i) const { return q[i] > tau ? 8u : 1u; }
};

struct KeepCount {
  const double* p;
  double tau;
  __device__ uint32_t operator()(int64_t i) const { return p[i] < tau ? 0u : 1u; }
};

struct LeafOut {
  float* centers;
  int32_t* levels;
  double* p;
  double* q;
};

__device__ __forceinline__ void copy_leaf(const inpc_octree& t, const double* __restrict__ q, int64_t i, LeafOut out,
                                          int64_t o) {
  out.centers[3 * o + 0] = t.centers[3 * i + 0];
  out.centers[3 * o + 1] = t.centers[3 * i + 1];
  out.centers[3 * o + 2] = t.centers[3 * i + 2];
  out.levels[o] = t.levels[i];
  out.p[o] = t.weights[i];
  out.q[o] = q[i];
}

// split = 0: copy every leaf to its place (the leaf cap was reached).
__global__ void k_subdivide(inpc_octree t, const double* __restrict__ q, double tau, int split,
                            const uint32_t* __restrict__ offset, LeafOut out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < t.n_leaves;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (!split) {
      copy_leaf(t, q, i, out, i);
      continue;
    }
    const int64_t o = offset[i];
    if (!(q[i] > tau)) {
      copy_leaf(t, q, i, out, o);
      continue;
    }
    const int l = t.levels[i];
    const double child = __dmul_rn((double)t.root_size, ldexp(1.0, -(l + 1)));  // child edge
    for (int k = 0; k < 8; ++k) {
      const int d[3] = {k & 1, (k >> 1) & 1, (k >> 2) & 1};
#pragma unroll
      for (int a = 0; a < 3; ++a)
        out.centers[3 * (o + k) + a] =
            (float)__dadd_rn((double)t.centers[3 * i + a], __dmul_rn((double)d[a] - 0.5, child));
      out.levels[o + k] = l + 1;
      out.p[o + k] = t.weights[i];
      out.q[o + k] = 0.0;
    }
  }
}

__global__ void k_prune(inpc_octree t, const double* __restrict__ q, double tau, const uint32_t* __restrict__ offset,
                        LeafOut out) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < t.n_leaves;
       i += (int64_t)gridDim.x * blockDim.x)
    if (!(t.weights[i] < tau)) copy_leaf(t, q, i, out, offset[i]);
}

inpc_status check_tree(const inpc_octree* t, const double* q) {
  if (!t || !t->centers || !t->levels || !t->weights || !q) return fail(INPC_ERR_INVALID_ARG, "null octree array");
  if (t->n_leaves < 1 || t->n_leaves > (int64_t(1) << 24))
    return fail(INPC_ERR_INVALID_ARG, "n_leaves must be in [1, 2^24]");
  if (!(t->root_size > 0.0f)) return fail(INPC_ERR_INVALID_ARG, "root_size must be positive");
  return INPC_OK;
}

inpc_status check_out(const LeafOut& o) {
  if (!o.centers || !o.levels || !o.p || !o.q) return fail(INPC_ERR_INVALID_ARG, "null output array");
  return INPC_OK;
}

unsigned grid_1d(int64_t n, int per_sm = 8) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>(ceil_div(n, 256), (int64_t)device_sm_count() * per_sm));
}

// Scan of the per-leaf output counts; returns the total on the host (the
// stream is synchronised).
template <class Load>
inpc_status count_outputs(Load ld, int64_t L, const RefineWs& ws, cudaStream_t s, int64_t* total) {
  INPC_TRY((scan::run<uint32_t, Load, false>(ld, L, ws.offset, ws.tops, s)));
  uint32_t t = 0;
  INPC_CUDA(cudaMemcpyAsync(&t, ws.tops + ceil_div(L, scan::kBlock), sizeof(t), cudaMemcpyDeviceToHost, s),
            "read output count");
  INPC_CUDA(cudaStreamSynchronize(s), "output count sync");
  *total = t;
  return INPC_OK;
}

}  // namespace
}  // namespace inpc

using namespace inpc;

extern "C" inpc_status inpc_rasterize_point_weights(const inpc_camera* cam, const inpc_raster_opts* opts,
                                                    const float* pos, int64_t n, const int32_t* n_contrib,
                                                    float* b_out, void* workspace, size_t workspace_bytes,
                                                    inpc_stream_t stream) {
  inpc::fault_arg(pos);
  RP P;
  INPC_TRY(make_rp(cam, opts, n, P));
  const RasterWs need = carve(nullptr, P.n_pix, n);
  if (!workspace || workspace_bytes < need.bytes || !aligned(workspace, 256))
    return fail(INPC_ERR_INVALID_ARG, "workspace null, unaligned or smaller than %zu bytes", need.bytes);
  if (n == 0) return INPC_OK;
  if (!pos || !n_contrib || !b_out) return fail(INPC_ERR_INVALID_ARG, "null pointer");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  RasterWs ws = carve(workspace, P.n_pix, n);
  INPC_CUDA(cudaMemsetAsync(ws.fscal, 0, sizeof(float) * 4 * n, s), "clear splat weights");
  INPC_TIMED("k_pixel_splat_weights", s,
             k_pixel_splat_weights<<<(unsigned)std::min<long long>(ceil_div(P.n_pix, 8),
                                                                    (long long)device_sm_count() * kSplatCtas),
                                     256, 0, s>>>(P, n_contrib, ws));
  INPC_TRY(check_launch("k_pixel_splat_weights"));
  INPC_TIMED("k_point_blend_weights", s,
             k_point_blend_weights<<<grid_1d(n, 16), 256, 0, s>>>(P, pos, ws, b_out));
  return check_launch("k_point_blend_weights");
}

extern "C" inpc_status inpc_octree_update_workspace_size(int64_t n_leaves, size_t* bytes) {
  if (inpc::fault_workspace_overflow())
    return inpc::fail(INPC_ERR_CAPACITY, "inpc_octree_update_workspace_size: size overflow (injected fault)");
  if (!bytes) return fail(INPC_ERR_INVALID_ARG, "bytes is null");
  if (n_leaves < 1 || n_leaves > (int64_t(1) << 24)) return fail(INPC_ERR_INVALID_ARG, "n_leaves must be in [1, 2^24]");
  *bytes = carve_update(nullptr, n_leaves).bytes;
  return INPC_OK;
}

extern "C" inpc_status inpc_octree_update(const int32_t* leaf_idx, const float* b, int64_t n, double* p, double* q,
                                          int64_t n_leaves, double lambda_u, void* workspace,
                                          size_t workspace_bytes, inpc_stream_t stream) {
  inpc::fault_arg(leaf_idx);
  if (n_leaves < 1 || n_leaves > (int64_t(1) << 24)) return fail(INPC_ERR_INVALID_ARG, "n_leaves must be in [1, 2^24]");
  if (n < 0 || n > INT32_MAX) return fail(INPC_ERR_CAPACITY, "n must be in [0, 2^31 - 1]");
  if (!p || !q || (n > 0 && (!leaf_idx || !b))) return fail(INPC_ERR_INVALID_ARG, "null pointer");
  if (!(lambda_u >= 0.0 && lambda_u <= 1.0)) return fail(INPC_ERR_INVALID_ARG, "lambda_u must be in [0, 1]");
  const UpdateWs need = carve_update(nullptr, n_leaves);
  if (!workspace || workspace_bytes < need.bytes || !aligned(workspace, 256))
    return fail(INPC_ERR_INVALID_ARG, "workspace null, unaligned or smaller than %zu bytes", need.bytes);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  UpdateWs ws = carve_update(workspace, n_leaves);
  INPC_CUDA(cudaMemsetAsync(workspace, 0, need.bytes, s), "clear header, maxima and minima");
  if (n > 0) {
    INPC_TIMED("k_leaf_minmax", s, k_leaf_minmax<<<grid_1d(n, 16), 256, 0, s>>>(leaf_idx, b, n, n_leaves, ws));
    INPC_TRY(check_launch("k_leaf_minmax"));
  }
  INPC_TIMED("k_leaf_update", s, k_leaf_update<<<grid_1d(n_leaves), 256, 0, s>>>(p, q, n_leaves, lambda_u, ws));
  return check_launch("k_leaf_update");
}

extern "C" inpc_status inpc_octree_refine_workspace_size(int64_t n_leaves, size_t* bytes) {
  if (inpc::fault_workspace_overflow())
    return inpc::fail(INPC_ERR_CAPACITY, "inpc_octree_refine_workspace_size: size overflow (injected fault)");
  if (!bytes) return fail(INPC_ERR_INVALID_ARG, "bytes is null");
  if (n_leaves < 1 || n_leaves > (int64_t(1) << 24)) return fail(INPC_ERR_INVALID_ARG, "n_leaves must be in [1, 2^24]");
  *bytes = carve_refine(nullptr, n_leaves).bytes;
  return INPC_OK;
}

extern "C" inpc_status inpc_octree_subdivide(const inpc_octree* tree, const double* q, double tau_s,
                                             int64_t max_leaves, float* centers_out, int32_t* levels_out,
                                             double* p_out, double* q_out, int64_t out_capacity, int64_t* n_out,
                                             void* workspace, size_t workspace_bytes, inpc_stream_t stream) {
  inpc::fault_arg(tree);
  INPC_TRY(check_tree(tree, q));
  const LeafOut out{centers_out, levels_out, p_out, q_out};
  INPC_TRY(check_out(out));
  if (!n_out) return fail(INPC_ERR_INVALID_ARG, "n_out is null");
  const int64_t L = tree->n_leaves;
  const RefineWs need = carve_refine(nullptr, L);
  if (!workspace || workspace_bytes < need.bytes || !aligned(workspace, 256))
    return fail(INPC_ERR_INVALID_ARG, "workspace null, unaligned or smaller than %zu bytes", need.bytes);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const RefineWs ws = carve_refine(workspace, L);
  int64_t total = 0;
  INPC_TRY(count_outputs(SplitCount{q, tau_s}, L, ws, s, &total));
  const int split = total < max_leaves ? 1 : 0;
  const int64_t n_new = split ? total : L;
  if (n_new > out_capacity)
    return fail(INPC_ERR_CAPACITY, "subdivision yields %lld leaves, output capacity is %lld", (long long)n_new,
                (long long)out_capacity);
  INPC_TIMED("k_subdivide", s, k_subdivide<<<grid_1d(L), 256, 0, s>>>(*tree, q, tau_s, split, ws.offset, out));
  INPC_TRY(check_launch("k_subdivide"));
  *n_out = n_new;
  return INPC_OK;
}

extern "C" inpc_status inpc_octree_prune(const inpc_octree* tree, const double* q, double tau_p, float* centers_out,
                                         int32_t* levels_out, double* p_out, double* q_out, int64_t out_capacity,
                                         int64_t* n_out, void* workspace, size_t workspace_bytes,
                                         inpc_stream_t stream) {
  inpc::fault_arg(tree);
  INPC_TRY(check_tree(tree, q));
  const LeafOut out{centers_out, levels_out, p_out, q_out};
  INPC_TRY(check_out(out));
  if (!n_out) return fail(INPC_ERR_INVALID_ARG, "n_out is null");
  const int64_t L = tree->n_leaves;
  const RefineWs need = carve_refine(nullptr, L);
  if (!workspace || workspace_bytes < need.bytes || !aligned(workspace, 256))
    return fail(INPC_ERR_INVALID_ARG, "workspace null, unaligned or smaller than %zu bytes", need.bytes);
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const RefineWs ws = carve_refine(workspace, L);
  int64_t total = 0;
  INPC_TRY(count_outputs(KeepCount{tree->weights, tau_p}, L, ws, s, &total));
  if (total > out_capacity)
    return fail(INPC_ERR_CAPACITY, "pruning keeps %lld leaves, output capacity is %lld", (long long)total,
                (long long)out_capacity);
  INPC_TIMED("k_prune", s, k_prune<<<grid_1d(L), 256, 0, s>>>(*tree, q, tau_p, ws.offset, out));
  INPC_TRY(check_launch("k_prune"));
  *n_out = total;
  return INPC_OK;
}
