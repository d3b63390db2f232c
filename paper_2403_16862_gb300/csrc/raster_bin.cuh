// raster_bin.cuh -- binning of the rasterizer's fragments into per-pixel
// buckets: a counting pass, a prefix sum over the pixels (scan.cuh) and a
// scattering pass.
//
// Points come grouped by octree leaf with the leaves in Morton order, so a
// few hundred consecutive points fall on a few hundred pixels and a pixel
// receives several of their fragments.  A CTA therefore counts the fragments
// of a chunk of consecutive points in a window of counters in shared memory
// (pixel (x, y) -> counter (x mod 64, y mod 64), tagged with the 64 x 64
// block it stands for) and goes to the pixel's global counter once per pixel
// and chunk.  Two pixels of one chunk that fall on the same counter (an
// unordered cloud, a jump in the Morton order) are no error: the later one
// goes to its global counter directly.
//
// With one global atomic per fragment the counting pass ran at the L2's
// atomic rate (253M atomics in 1.29 ms = 196G/s for 67M points), and the
// scattering pass waited on returning atomics and left most sectors of the
// buckets partly written.  The scattering pass now also sorts a chunk's
// fragments by pixel in shared memory, so that a bucket receives runs of
// consecutive keys.
#pragma once

namespace inpc {
namespace {

constexpr int kWinBits = 6;
constexpr int kWinSide = 1 << kWinBits;
constexpr int kWinSlots = kWinSide * kWinSide;
// Window word: 18-bit tag (block column, block row), 14-bit count.  The free
// word is no counter's: a chunk has at most kBinPoints * 4 fragments.
constexpr int kWinCountBits = 14;
constexpr uint32_t kWinCountMask = (1u << kWinCountBits) - 1;
constexpr uint32_t kWinFree = 0xFFFFFFFFu;
constexpr uint32_t kNoRank = 0xFFFFu;

// The window: words, and the list of the counters in use.
struct BinWindow {
  uint32_t* word;   // [kWinSlots]
  uint16_t* list;   // [min(kWinSlots, fragments of a chunk)]
  int* n_list;
};

// Counter of pixel (x, y); the rows are skewed so that a few pixels of
// several rows spread over the shared-memory banks.
__device__ __forceinline__ int win_slot(int x, int y) {
  return ((y & (kWinSide - 1)) << kWinBits) | ((x + 11 * y) & (kWinSide - 1));
}

__device__ __forceinline__ uint32_t win_tag(int x, int y) {
  return ((uint32_t)x >> kWinBits) | (((uint32_t)y >> kWinBits) << 9);  // images are at most 32768 wide and high
}

// Pixel index of the counter at `slot` with word w.
__device__ __forceinline__ uint32_t win_pixel(int slot, uint32_t w, int W) {
  const uint32_t tag = w >> kWinCountBits;
  const int y = (int)((tag >> 9) << kWinBits) | (slot >> kWinBits);
  const int x = (int)((tag & 511u) << kWinBits) | ((slot - 11 * y) & (kWinSide - 1));
  return (uint32_t)(y * W + x);
}

// Counts a fragment of pixel (x, y): its rank among the chunk's fragments of
// that pixel, or kNoRank when another pixel holds the counter.
__device__ __forceinline__ uint32_t win_take(const BinWindow& B, int x, int y) {
  const int slot = win_slot(x, y);
  const uint32_t fresh = win_tag(x, y) << kWinCountBits;
  uint32_t w = *(volatile uint32_t*)(B.word + slot);
  if (w == kWinFree) {
    w = atomicCAS(B.word + slot, kWinFree, fresh);
    if (w == kWinFree) {
      B.list[atomicAdd(B.n_list, 1)] = (uint16_t)slot;
      w = fresh;
    }
  }
  if ((w ^ fresh) >> kWinCountBits) return kNoRank;
  return atomicAdd(B.word + slot, 1u) & kWinCountMask;
}

// A CTA of kT threads bins chunks of kT * kPP consecutive points.
template <int kT, int kPP>
struct BinSmem {
  static constexpr int kPoints = kT * kPP;
  static constexpr int kFrags = 4 * kPoints;
  static constexpr int kList = kFrags < kWinSlots ? kFrags : kWinSlots;
  static_assert(kFrags <= (int)kWinCountMask, "a chunk's count fits its field");
  uint32_t word[kWinSlots];
  uint16_t list[kList];
  int n_list[2];   // alternate over the chunks
  int n_sorted[2];
};

template <int kT, int kPP>
__global__ void __launch_bounds__(kT) k_pix_count(RP P, const float* __restrict__ pos,
                                                  uint32_t* __restrict__ pix_count) {
  using Smem = BinSmem<kT, kPP>;
  __shared__ Smem S;
  for (int i = threadIdx.x; i < kWinSlots; i += kT) S.word[i] = kWinFree;
  if (threadIdx.x < 2) S.n_list[threadIdx.x] = 0;
  __syncthreads();
  const int n = (int)P.n;  // <= 2^28
  int turn = 0;
  for (int c0 = blockIdx.x * Smem::kPoints; c0 < n; c0 += gridDim.x * Smem::kPoints, turn ^= 1) {
    const BinWindow B{S.word, S.list, &S.n_list[turn]};
    float xyz[kPP][3];
#pragma unroll
    for (int u = 0; u < kPP; ++u) {
      const long long id = c0 + u * kT + (int)threadIdx.x;
#pragma unroll
      for (int a = 0; a < 3; ++a) xyz[u][a] = id < n ? __ldg(pos + 3 * id + a) : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kPP; ++u) {
      Splat s;
      if (c0 + u * kT + (int)threadIdx.x >= n || !splat_xyz(P, xyz[u][0], xyz[u][1], xyz[u][2], s)) continue;
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int q = corner_pixel(P, s.f, k);
        if (q >= 0 && win_take(B, s.f.i0 + (k & 1), s.f.j0 + (k >> 1)) == kNoRank) atomicAdd(pix_count + q, 1u);
      }
    }
    __syncthreads();
    const int m = S.n_list[turn];
    if (threadIdx.x == 0) S.n_list[turn ^ 1] = 0;
    for (int e = threadIdx.x; e < m; e += kT) {
      const int slot = S.list[e];
      const uint32_t w = S.word[slot];
      S.word[slot] = kWinFree;
      atomicAdd(pix_count + win_pixel(slot, w, P.cam.W), w & kWinCountMask);
    }
    __syncthreads();
  }
}

// Dynamic shared memory of the scattering pass: the window, then per counter
// the global slot of the chunk's first fragment, then the chunk's fragments
// sorted by pixel (key, alpha, global slot).
template <int kT, int kPP>
struct ScatterSmem {
  using Bin = BinSmem<kT, kPP>;
  unsigned long long key[Bin::kFrags];
  float alpha[Bin::kFrags];
  uint32_t dst[Bin::kFrags];
  uint32_t base[kWinSlots];
  Bin bin;
};

template <int kT, int kPP, class FT>
__global__ void __launch_bounds__(kT, 1024 / kT) k_pix_scatter(RP P, const float* __restrict__ pos,
                                                               const float* __restrict__ opacity,
                                                               const FT* __restrict__ feat, RasterWs ws) {
  using Smem = ScatterSmem<kT, kPP>;
  constexpr int kPoints = Smem::Bin::kPoints;
  extern __shared__ __align__(16) unsigned char dyn[];
  Smem& S = *reinterpret_cast<Smem*>(dyn);
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < kWinSlots; i += kT) S.bin.word[i] = kWinFree;
  if (threadIdx.x < 2) {
    S.bin.n_list[threadIdx.x] = 0;
    S.bin.n_sorted[threadIdx.x] = 0;
  }
  __syncthreads();
  const int n = (int)P.n;  // <= 2^28
  int turn = 0;
  // the next chunk's positions and alpha inputs are loaded while this one is
  // worked on
  float next[kPP][4];
  const auto load = [&](long long first) {
#pragma unroll
    for (int u = 0; u < kPP; ++u) {
      const long long id = first + u * kT + (int)threadIdx.x;
#pragma unroll
      for (int a = 0; a < 3; ++a) next[u][a] = id < n ? __ldg(pos + 3 * id + a) : 0.f;
      next[u][3] = id < n ? alpha_input(P, opacity, feat, id) : 0.f;
    }
  };
  load((long long)blockIdx.x * kPoints);
  for (int c0 = blockIdx.x * kPoints; c0 < n; c0 += gridDim.x * kPoints, turn ^= 1) {
    const BinWindow B{S.bin.word, S.bin.list, &S.bin.n_list[turn]};
    float xyz[kPP][3], av[kPP];
#pragma unroll
    for (int u = 0; u < kPP; ++u) {
#pragma unroll
      for (int a = 0; a < 3; ++a) xyz[u][a] = next[u][a];
      av[u] = next[u][3];
    }
    // the chunk's fragments: their rank within their pixel
    Splat s[kPP];
    uint32_t rank[kPP][2];
    unsigned ok = 0;
#pragma unroll
    for (int u = 0; u < kPP; ++u) {
      rank[u][0] = rank[u][1] = 0u;
      const int id = c0 + u * kT + (int)threadIdx.x;
      const bool in = id < n && splat_xyz(P, xyz[u][0], xyz[u][1], xyz[u][2], s[u]);
      if (in) {
        ok |= 1u << u;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int q = corner_pixel(P, s[u].f, k);
          if (q >= 0) rank[u][k >> 1] |= win_take(B, s[u].f.i0 + (k & 1), s[u].f.j0 + (k >> 1)) << (16 * (k & 1));
        }
      }
    }
    __syncthreads();
    // one global atomic per pixel in use: the bucket slots of its fragments
    // (the counts run down from the bucket size, so the buckets fill back to
    // front) and their place in the sorted chunk
    const int m = *B.n_list;
    load(c0 + (long long)gridDim.x * kPoints);
    for (int e0 = (int)threadIdx.x - lane; e0 < m; e0 += kT) {
      const int e = e0 + lane;
      int slot = 0;
      uint32_t c = 0, first = 0;
      if (e < m) {
        slot = S.bin.list[e];
        const uint32_t w = S.bin.word[slot];
        const uint32_t q = win_pixel(slot, w, P.cam.W);
        c = w & kWinCountMask;
        first = __ldg(ws.pix_start + q) + atomicSub(ws.pix_count + q, c) - c;
      }
      uint32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      int at = 0;
      if (lane == 31) at = atomicAdd(&S.bin.n_sorted[turn], (int)incl);
      at = __shfl_sync(0xffffffffu, at, 31);
      if (e < m) {
        S.bin.word[slot] = (uint32_t)at + incl - c;
        S.base[slot] = first;
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < kPP; ++u) {
      const int id = c0 + u * kT + (int)threadIdx.x;
      const bool in = (ok >> u) & 1u;
      float e_h0 = 0.f;
      if (in) {
        // head mode: alpha_h = 1 - exp(-exp(h0)) as in point_alpha_h, with
        // exp(h0) kept for the backward's opacity path
        e_h0 = P.head ? expf(av[u]) : 0.f;
        const float ah = P.head ? -expm1f(-e_h0) : av[u];
        const unsigned long long key =
            ((unsigned long long)(__float_as_uint(s[u].d) - P.dbase) << P.idb) | (unsigned long long)id;
        uint32_t to[4];  // the corners without a counter: their own atomics, all in flight together
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int q = corner_pixel(P, s[u].f, k);
          to[k] = 0;
          if (q >= 0 && ((rank[u][k >> 1] >> (16 * (k & 1))) & 0xffffu) == kNoRank)
            to[k] = __ldg(ws.pix_start + q) + atomicSub(ws.pix_count + q, 1u) - 1u;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (corner_pixel(P, s[u].f, k) < 0) continue;
          const float a = fminf(__fmul_rn(ah, corner_weight(s[u].f, k & 1, k >> 1)), P.alpha_max);
          const uint32_t r = (rank[u][k >> 1] >> (16 * (k & 1))) & 0xffffu;
          if (r != kNoRank) {
            const int slot = win_slot(s[u].f.i0 + (k & 1), s[u].f.j0 + (k >> 1));
            const uint32_t at = S.bin.word[slot] + r;
            S.key[at] = key;
            S.alpha[at] = a;
            S.dst[at] = S.base[slot] + r;
          } else {
            ws.keys[to[k]] = key;
            ws.alpha[to[k]] = a;
          }
        }
      }
      if (id < n) {
        ws.porg[id] = in ? ((uint32_t)(s[u].f.i0 + 1) & 0xffffu) | ((uint32_t)(s[u].f.j0 + 1) << 16) : 0u;
        if (P.head) ws.pexp[id] = e_h0;
      }
    }
    __syncthreads();
    const int total = S.bin.n_sorted[turn];
    for (int j = threadIdx.x; j < total; j += kT) {
      const uint32_t to = S.dst[j];
      ws.keys[to] = S.key[j];
      ws.alpha[to] = S.alpha[j];
    }
    for (int e = threadIdx.x; e < m; e += kT) S.bin.word[S.bin.list[e]] = kWinFree;
    if (threadIdx.x == 0) {
      S.bin.n_list[turn ^ 1] = 0;
      S.bin.n_sorted[turn ^ 1] = 0;
    }
    __syncthreads();
  }
}

// The scattering pass without the window, for clouds with few fragments per
// pixel: one returning atomic per run of equal pixels over consecutive lanes.
// A run of equal pixels over
// consecutive lanes is found with one shuffle and one ballot (its start is a
// lane whose pixel differs from the previous lane's), and its first lane
// updates the counter for the whole run.
struct LaneRun {
  int start;  // first lane of this lane's run
  int len;    // lanes in the run (valid in the first lane)
};

__device__ __forceinline__ LaneRun lane_run(int q, int lane) {
  const int prev = __shfl_up_sync(0xffffffffu, q, 1);
  const unsigned starts = __ballot_sync(0xffffffffu, lane == 0 || prev != q);
  const unsigned upto = lane == 31 ? 0xffffffffu : ((2u << lane) - 1u);
  const unsigned later = starts & ~upto;
  LaneRun r;
  r.start = 31 - __clz(starts & upto);
  r.len = (later ? __ffs(later) - 1 : 32) - lane;
  return r;
}

template <class FT>
__global__ void __launch_bounds__(256) k_pix_scatter_direct(RP P, const float* __restrict__ pos,
                                                     const float* __restrict__ opacity,
                                                     const FT* __restrict__ feat,
                                                     const uint32_t* __restrict__ pix_start,
                                                     uint32_t* __restrict__ pix_count,
                                                     unsigned long long* __restrict__ keys,
                                                     float* __restrict__ alpha, uint32_t* __restrict__ porg,
                                                     float* __restrict__ pexp) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int n = (int)P.n;  // <= 2^28
  const int stride = gridDim.x * blockDim.x;
  // each iteration loads the next point's position and alpha input while it
  // bins this one, so those round trips overlap this point's atomics
  float x = 0.f, y = 0.f, z = 0.f, av = 0.f;
  if (blockIdx.x * blockDim.x + threadIdx.x < n) {
    const long long id = blockIdx.x * blockDim.x + threadIdx.x;
    x = __ldg(pos + 3 * id); y = __ldg(pos + 3 * id + 1); z = __ldg(pos + 3 * id + 2);
    av = alpha_input(P, opacity, feat, id);
  }
  for (int base = blockIdx.x * blockDim.x; base < n; base += stride) {
    const int id = base + threadIdx.x;
    const long long nid = (long long)id + stride;
    float nx = 0.f, ny = 0.f, nz = 0.f, na = 0.f;
    if (nid < n) {
      nx = __ldg(pos + 3 * nid); ny = __ldg(pos + 3 * nid + 1); nz = __ldg(pos + 3 * nid + 2);
      na = alpha_input(P, opacity, feat, nid);
    }
    int q[4] = {-1, -1, -1, -1};
    Splat s;
    float ah = 0.f;
    bool splat_ok = false;
    float e_h0 = 0.f;
    if (id < n && splat_xyz(P, x, y, z, s)) {
      for (int k = 0; k < 4; ++k) q[k] = corner_pixel(P, s.f, k);
      // head mode: alpha_h = 1 - exp(-exp(h0)) as in point_alpha_h, with
      // exp(h0) kept for the backward's opacity path
      e_h0 = P.head ? expf(av) : 0.f;
      ah = P.head ? -expm1f(-e_h0) : av;
      splat_ok = true;
    }
    x = nx; y = ny; z = nz; av = na;
    const unsigned long long key = ((unsigned long long)(__float_as_uint(s.d) - P.dbase) << P.idb) | (unsigned long long)id;
    // the four corners' bucket offsets and atomics are all issued before
    // any result is used, so their round trips overlap
    LaneRun run[4];
    uint32_t start[4], top[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      run[k] = lane_run(q[k], lane);
      start[k] = q[k] >= 0 ? __ldg(pix_start + q[k]) : 0u;
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      // counts run down from the bucket size, so the buckets fill back to front
      top[k] = 0;
      if (q[k] >= 0 && run[k].start == lane) top[k] = atomicSub(pix_count + q[k], (uint32_t)run[k].len);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const uint32_t t = __shfl_sync(full, top[k], run[k].start);
      if (q[k] >= 0) {
        const uint32_t slot = start[k] + t - 1 - (uint32_t)(lane - run[k].start);
        keys[slot] = key;
        alpha[slot] = fminf(__fmul_rn(ah, corner_weight(s.f, k & 1, k >> 1)), P.alpha_max);
      }
    }
    if (id < n) porg[id] = splat_ok ? ((uint32_t)(s.f.i0 + 1) & 0xffffu) | ((uint32_t)(s.f.j0 + 1) << 16) : 0u;
    if (id < n && P.head) pexp[id] = e_h0;
  }
}

}  // namespace
}  // namespace inpc
