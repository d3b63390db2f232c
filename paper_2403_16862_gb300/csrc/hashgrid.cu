// hashgrid.cu -- multi-resolution hash-grid query (Sec. 3.3, App. A.5) and
// its adjoint (the table gradient).
//
// The query runs two threads per point, each gathering the four corners on
// one side of the cell along x; a warp takes 16 consecutive points through
// all levels.  Corner rows are gathered as 16-byte vectors (FP32) or 8-byte
// vectors (BF16).  The output is written with streaming stores so that it
// does not evict the table from L2.
//
// The backward reduces 16-byte rows into an FP32 gradient table
// (red.global.add.v4.f32), after merging the coarse levels' contributions of
// consecutive points (adjoint_impl.cuh).
#include <algorithm>

#include "adjoint_impl.cuh"

namespace inpc {
namespace {

// A warp takes 16 consecutive points, two lanes per point, through the
// levels of one level group (grid y, plan_level_groups), two levels at a
// time: lane bx gathers the four corners at x + bx
// of the point's cell.  The x neighbours' rows differ only in their lowest
// bits (hashed: x is multiplied by 1 before the XOR; dense: consecutive
// rows), so they share one 128-byte line unless the carry of x + 1 reaches
// bit 3 (FP32) or bit 4 (BF16): loading both from one instruction costs one
// L1 wavefront instead of two, and the L1 wavefront rate bounds this
// kernel.  Consecutive points come from the same octree leaf, so at the
// coarse levels the 16 points of an instruction mostly fall in a few cells
// and share their lines as well (about 2.6 distinct lines per point and
// level on average over the benchmark's 16 levels, against 2.9 with 8
// points of two levels per instruction).  A group's rows stay in L2 under
// evict_last while positions and outputs stream past them.  After each pair of levels the two lanes swap halves so that each stores
// one level's whole 16-byte row: the warp writes each point's two levels
// as one full 32-byte sector.
template <class TT, class OT>
__global__ void __launch_bounds__(256) k_hash_fwd(GridParams P, LevelGroups LG, const TT* __restrict__ table,
                                                  const float* __restrict__ pos, long long n, OT* __restrict__ h) {
  const int lb = LG.begin[blockIdx.y], le = LG.begin[blockIdx.y + 1];
  const uint64_t keep = l2_evict_last();
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t bx = lane & 1u;
  // n <= 2^29 (checked by the caller): 32-bit indices do not overflow
  const uint32_t n_groups = (uint32_t)((n + 15) >> 4);
  const uint32_t n_warps = (gridDim.x * blockDim.x) >> 5;
  // warp-uniform trip counts: the pair exchanges are warp shuffles
  for (uint32_t g = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; g < n_groups; g += n_warps) {
    const uint32_t pr = g * 16u + (lane >> 1);
    const bool valid = pr < (uint32_t)n;
    const uint32_t p = valid ? pr : (uint32_t)n - 1u;  // spare lanes redo the last point
    const float x = __ldg(pos + 3 * p + 0), y = __ldg(pos + 3 * p + 1), z = __ldg(pos + 3 * p + 2);
    OT* hp = h + (long long)p * P.n_levels * 4;
    for (int l = lb; l < le; l += 2) {
      const float2 a = query_half<TT>(P, table, x, y, z, l, bx, keep);
      if (l + 1 < le) {
        const float2 b = query_half<TT>(P, table, x, y, z, l + 1, bx, keep);
        // lane 0 holds features 0-1 of both levels, lane 1 features 2-3:
        // lane 0 gives level l + 1's half away and takes level l's, lane 1
        // the other way round
        const float2 give = bx ? a : b;
        const float r0 = __shfl_xor_sync(0xffffffffu, give.x, 1), r1 = __shfl_xor_sync(0xffffffffu, give.y, 1);
        const float4 row = bx ? make_float4(r0, r1, b.x, b.y) : make_float4(a.x, a.y, r0, r1);
        if (valid) store_out<OT>(hp, l + (int)bx, row);
      } else if (valid) {
        store_half<OT>(hp, l, bx, a);
      }
    }
  }
}


// The adjoint of the query, laid out as the fused rasterizer backward's: warps
// in pairs over the same points, the even warp on the coarse half of the
// levels (AdjointLane::coarse merges the contributions of consecutive points
// that share a vertex before they are reduced into L2), the odd warp on the
// fine half (reduced directly), two adjacent lanes per level.  The L2
// reduction rate bounds it, so the merge is what pays: on leaf-grouped
// points fewer than half of the 8 n_levels contributions of a point are left
// to reduce (1,000,003 points, 16 levels, 2^19 rows: forward and backward
// 1,145 -> 661 us, of which the adjoint 0.85 -> 0.40 ms; one thread per
// point and level with eight reductions each before).  A CTA takes `chunk`
// consecutive points, its point slots interleaved over them; each lane loads
// its next point's position and gradient row before it works on the current
// one.  The coarse warps take levels 0 .. n_coarse - 1 (at most kH), the fine
// warps levels kH .. l_end - 1 (none with l_end = 0).
template <int GA>
__global__ void __launch_bounds__(256, 4) k_hash_bwd(GridParams P, const float* __restrict__ pos,
                                                     const float4* __restrict__ dh, long long n,
                                                     float* __restrict__ grad, long long chunk, int n_coarse,
                                                     int l_end) {
  constexpr int kH = GA / 2;           // levels per half
  constexpr int kPW = 16 / kH;         // points per warp
  constexpr int kGroups = 4 * kPW;     // points in flight per CTA (4 warp pairs)
  constexpr int kStride = kGroups * kH * 2;
  __shared__ float4 acc_s[4][kStride];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool coarse = (warp & 1) == 0;
  const uint32_t bx = lane & 1u;
  const int lvl = (lane >> 1) % kH;
  const int l = (coarse ? 0 : kH) + lvl;
  const int slot = (warp >> 1) * kPW + lane / (2 * kH);
  if (l >= (coarse ? n_coarse : l_end)) return;  // nothing below is collective
  const uint64_t keep = l2_evict_last(), stream = l2_evict_first();
  AdjointLane<kStride> adj(P, l, true, grad, bx, &acc_s[0][(slot * kH + lvl) * 2 + bx]);
  const long long last = min((long long)(blockIdx.x + 1) * chunk, n);
  long long id = (long long)blockIdx.x * chunk + slot;
  if (id >= last) return;
  uint4 d = ld_hint_u4(dh + id * P.n_levels + l, stream);
  float x = __ldg(pos + 3 * id), y = __ldg(pos + 3 * id + 1), z = __ldg(pos + 3 * id + 2);
  while (id < last) {
    const long long nx = id + kGroups;
    uint4 dn = make_uint4(0u, 0u, 0u, 0u);
    float xn = 0.f, yn = 0.f, zn = 0.f;
    if (nx < last) {
      dn = ld_hint_u4(dh + nx * P.n_levels + l, stream);
      xn = __ldg(pos + 3 * nx);
      yn = __ldg(pos + 3 * nx + 1);
      zn = __ldg(pos + 3 * nx + 2);
    }
    const float dc[4] = {__uint_as_float(d.x), __uint_as_float(d.y), __uint_as_float(d.z), __uint_as_float(d.w)};
    if (dc[0] != 0.f || dc[1] != 0.f || dc[2] != 0.f || dc[3] != 0.f) adj.add(coarse, x, y, z, dc, keep);
    d = dn;
    x = xn;
    y = yn;
    z = zn;
    id = nx;
  }
  if (coarse) adj.flush(keep);
}

// How the adjoint takes the levels: the first n_coarse on the coarse warps; the
// others on the fine warps or, with split, level group by level group in a
// launch of their own.  What is reduced into at a time has to stay in L2 (129
// MB): the coarse levels within 96 MB, the fine ones within kQueryL2Budget, all
// of them within 112 MB, counting the rows that the points can touch (8 a level
// each; a 16-byte row takes a 32-byte sector while its neighbour is not).
// Random positions, before and after this rule (levels, log2 of the rows):
// 1,000,000 points 9/21 690 and 370 us, 12/20 677 and 431, 24/19 1482 and 776,
// 16/19 and 16/21 the same; 1,000 points 16/20 11.0 and 6.1, 32/19 13.2 and 6.3.
struct AdjointPlan {
  int n_coarse;
  bool split;
};

AdjointPlan plan_adjoint(const GridParams& P, int kH, long long n) {
  constexpr long long kCoarseBytes = 96ll << 20, kAllBytes = 112ll << 20;
  const auto bytes = [&](int l, int per_row) {
    return std::min<long long>(16 * level_rows(P, l), 8 * per_row * n);
  };
  AdjointPlan a = {0, false};
  for (long long coarse = 0; a.n_coarse < kH; ++a.n_coarse) {
    coarse += bytes(a.n_coarse, 32);
    if (a.n_coarse > 0 && coarse > kCoarseBytes) break;
  }
  long long fine = 0, all = 0;
  for (int l = 0; l < P.n_levels; ++l) {
    if (l >= a.n_coarse) fine += bytes(l, 32);
    all += bytes(l, 16);
  }
  a.split = a.n_coarse < kH || fine > kQueryL2Budget || all > kAllBytes;
  return a;
}

template <int GA>
inpc_status launch_hash_bwd(const GridParams& P, const float* pos, const float4* dh, long long n, float* grad,
                            cudaStream_t s) {
  constexpr int kH = GA / 2, kGroups = 4 * (16 / kH);
  const AdjointPlan plan = plan_adjoint(P, kH, n);
  // whole waves of resident CTAs (4 per SM), about 48 points per slot: long
  // enough runs to merge, and no nearly empty last wave
  const long long resident = (long long)device_sm_count() * 4;
  const long long waves = std::max<long long>(1, (n + 24 * kGroups * resident) / (48 * kGroups * resident));
  const long long chunk = kGroups * std::max<long long>(1, ceil_div(n, kGroups * resident * waves));
  INPC_TIMED("k_hash_bwd", s,
             k_hash_bwd<GA><<<(unsigned)ceil_div(n, chunk), 256, 0, s>>>(P, pos, dh, n, grad, chunk, plan.n_coarse,
                                                                     plan.split ? 0 : P.n_levels));
  INPC_TRY(check_launch("k_hash_bwd"));
  if (!plan.split) return INPC_OK;
  return launch_grad_levels(P, plan.n_coarse, pos, dh + plan.n_coarse, P.n_levels, 1, n, grad, s);
}

}  // namespace
}  // namespace inpc

using namespace inpc;

extern "C" inpc_status inpc_hashgrid_n_entries(const inpc_hashgrid_desc* g, int64_t* n_entries) {
  if (!n_entries) return fail(INPC_ERR_INVALID_ARG, "n_entries is null");
  GridParams P;
  INPC_TRY(make_params(g, P, n_entries));
  return INPC_OK;
}

extern "C" inpc_status inpc_query_hashgrid(const inpc_hashgrid_desc* g, const void* table, const float* pos,
                                           int64_t n, void* h_out, inpc_stream_t stream) {
  inpc::fault_arg(table);
  GridParams P;
  int64_t total = 0;
  INPC_TRY(make_params(g, P, &total));
  if (n < 0 || n > (int64_t(1) << 29)) return fail(INPC_ERR_CAPACITY, "n must be in [0, 2^29]");
  if (n == 0) return INPC_OK;
  if (!table || !pos || !h_out) return fail(INPC_ERR_INVALID_ARG, "inpc_query_hashgrid: null pointer");
  const size_t ta = g->table_dtype == INPC_F32 ? 16 : 8, oa = g->out_dtype == INPC_F32 ? 16 : 8;
  if (!aligned(table, ta) || !aligned(h_out, oa) || !aligned(pos, 4))
    return fail(INPC_ERR_INVALID_ARG, "inpc_query_hashgrid: misaligned table/output/pos");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  // two lanes per point; grid y: the level groups
  const LevelGroups LG = plan_level_groups(P, g->table_dtype == INPC_F32 ? 16 : 8);
  const long long cap = (long long)device_sm_count() * 16;
  const dim3 grid((unsigned)std::max<long long>(1, std::min<long long>((long long)ceil_div(2 * n, 256), cap)),
                  (unsigned)LG.n);
  TimedLaunch timed("k_hash_fwd", s);
  if (g->table_dtype == INPC_F32 && g->out_dtype == INPC_F32)
    k_hash_fwd<float, float><<<grid, 256, 0, s>>>(P, LG, (const float*)table, pos, n, (float*)h_out);
  else if (g->table_dtype == INPC_F32)
    k_hash_fwd<float, __nv_bfloat16><<<grid, 256, 0, s>>>(P, LG, (const float*)table, pos, n, (__nv_bfloat16*)h_out);
  else if (g->out_dtype == INPC_F32)
    k_hash_fwd<__nv_bfloat16, float><<<grid, 256, 0, s>>>(P, LG, (const __nv_bfloat16*)table, pos, n, (float*)h_out);
  else
    k_hash_fwd<__nv_bfloat16, __nv_bfloat16>
        <<<grid, 256, 0, s>>>(P, LG, (const __nv_bfloat16*)table, pos, n, (__nv_bfloat16*)h_out);
  return check_launch("k_hash_fwd");
}

extern "C" inpc_status inpc_query_hashgrid_bwd(const inpc_hashgrid_desc* g, const float* pos, const float* dh,
                                               int64_t n, float* grad_table, inpc_stream_t stream) {
  inpc::fault_arg(pos);
  GridParams P;
  int64_t total = 0;
  INPC_TRY(make_params(g, P, &total));
  if (n < 0 || n > INT32_MAX) return fail(INPC_ERR_CAPACITY, "n out of range");
  if (n == 0) return INPC_OK;
  if (!pos || !dh || !grad_table) return fail(INPC_ERR_INVALID_ARG, "inpc_query_hashgrid_bwd: null pointer");
  if (!aligned(grad_table, 16) || !aligned(dh, 16) || !aligned(pos, 4))
    return fail(INPC_ERR_INVALID_ARG, "inpc_query_hashgrid_bwd: misaligned buffer");
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  const float4* d = reinterpret_cast<const float4*>(dh);
  // up to 4 levels would leave most lanes of the warp pairs idle: two lanes
  // per point and level instead
  if (P.n_levels <= 4) return launch_grad_levels(P, 0, pos, d, P.n_levels, 1, n, grad_table, s);
  if (P.n_levels <= 8) return launch_hash_bwd<8>(P, pos, d, n, grad_table, s);
  if (P.n_levels <= 16) return launch_hash_bwd<16>(P, pos, d, n, grad_table, s);
  return launch_hash_bwd<32>(P, pos, d, n, grad_table, s);
}
