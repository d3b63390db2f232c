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
// atomic rate (253M atomics in 1.29 ms = 196G/s for 67M points; 0.58 ms with
// the window, now bound by issue at 69 % of the slots), and the scattering
// pass waited on returning atomics and left most sectors of the buckets partly
// written.  The scattering pass also sorts a chunk's fragments by pixel in
// shared memory, so that a bucket receives runs of consecutive keys: without
// the sort the stores alone, a sector each, take 5.0 ms for 67M points.
//
// Scattering 67M points (1280 x 832, BF16 rows): 5.44 ms direct, 3.86 ms with
// a list of the counters in use, 3.13 ms with a footprint's four counters in
// flight together and the window read as a whole in place of the list; 16M
// 1.44, 1.12 and 0.89 ms; 4M (FP32) 367, 346 and 272 us.  What bounds it now
// is the memory's handling of partly written sectors (16M points: 1.07 GB
// written, 2.56 GB read of which 0.74 GB are inputs, at 4.05 TB/s).  Larger
// chunks, more resident warps and streaming hints on the inputs measured the
// same or slower.
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

// Counts the (up to four) fragments of a footprint: the rank of each among the
// chunk's fragments of its pixel, or kNoRank when another pixel holds the
// counter (or the corner is off the image), two ranks to a word.  A footprint's
// corners have four different counters, so the reads, the claims and the
// additions of the four go out together.
__device__ __forceinline__ void win_take(const RP& P, uint32_t* word, const Footprint& f, uint32_t (&rank)[2]) {
  int slot[4];
  uint32_t fresh[4], w[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const int x = f.i0 + (k & 1), y = f.j0 + (k >> 1);
    slot[k] = win_slot(x, y);
    fresh[k] = win_tag(x, y) << kWinCountBits;
    w[k] = *(volatile uint32_t*)(word + slot[k]);
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (corner_pixel(P, f, k) < 0) {
      w[k] = ~fresh[k];  // no counter of this tag
    } else if (w[k] == kWinFree) {
      w[k] = atomicCAS(word + slot[k], kWinFree, fresh[k]);
      if (w[k] == kWinFree) w[k] = fresh[k];
    }
  }
  uint32_t r[4];
#pragma unroll
  for (int k = 0; k < 4; ++k)
    r[k] = (w[k] ^ fresh[k]) >> kWinCountBits ? kNoRank : atomicAdd(word + slot[k], 1u) & kWinCountMask;
  rank[0] = r[0] | (r[1] << 16);
  rank[1] = r[2] | (r[3] << 16);
}

__device__ __forceinline__ uint32_t rank_of(const uint32_t (&rank)[2], int k) {
  return (rank[k >> 1] >> (16 * (k & 1))) & 0xffffu;
}

// A CTA of kT threads bins chunks of kT * kPP consecutive points.
template <int kT, int kPP>
struct BinShape {
  static constexpr int kPoints = kT * kPP;
  static_assert(4 * kPoints <= (int)kWinCountMask, "a chunk's count fits its field");
  static constexpr int kScan = kWinSlots / (4 * kT);  // 16-byte groups of counters per thread
  static_assert(kScan * 4 * kT == kWinSlots, "the threads share the window evenly");
};

// What the counting pass leaves for the choice of the scattering pass: the
// fragments in the windows of a few CTAs' first chunks, and the counters they
// took.  An unordered cloud has hardly more fragments than counters; there
// the window is only work (16M points in no order at 1280 x 832: 2.74 ms with
// it, 2.36 ms without; grouped by leaf 0.89 and 1.44 ms).
struct WinSample {
  uint32_t used, frags;
};
constexpr int kSampleEvery = 16;  // CTAs per sampled one

__device__ __forceinline__ bool window_wanted(const WinSample* s) { return 4u * s->frags >= 5u * s->used; }

// sample: null where the scattering pass has no use for it.
template <int kT, int kPP>
__global__ void __launch_bounds__(kT) k_pix_count(RP P, const float* __restrict__ pos,
                                                  uint32_t* __restrict__ pix_count, WinSample* sample) {
  using Shape = BinShape<kT, kPP>;
  __shared__ __align__(16) uint32_t word[kWinSlots];
  for (int i = threadIdx.x; i < kWinSlots; i += kT) word[i] = kWinFree;
  __syncthreads();
  const int n = (int)P.n;  // <= 2^28
  for (int c0 = blockIdx.x * Shape::kPoints; c0 < n; c0 += gridDim.x * Shape::kPoints) {
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
      uint32_t rank[2];
      win_take(P, word, s.f, rank);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int q = corner_pixel(P, s.f, k);
        if (q >= 0 && rank_of(rank, k) == kNoRank) atomicAdd(pix_count + q, 1u);
      }
    }
    __syncthreads();
    if (sample && blockIdx.x % kSampleEvery == 0 && c0 == (int)blockIdx.x * Shape::kPoints) {
      unsigned used = 0, frags = 0;
      for (int i = threadIdx.x; i < kWinSlots; i += kT) {
        if (word[i] == kWinFree) continue;
        ++used;
        frags += word[i] & kWinCountMask;
      }
      used = __reduce_add_sync(0xffffffffu, used);
      frags = __reduce_add_sync(0xffffffffu, frags);
      if ((threadIdx.x & 31) == 0) {
        atomicAdd(&sample->used, used);
        atomicAdd(&sample->frags, frags);
      }
      __syncthreads();
    }
    // the counters go to the pixels and are free again
#pragma unroll
    for (int i = 0; i < Shape::kScan; ++i) {
      const int slot = 4 * (i * kT + (int)threadIdx.x);
      const uint4 w4 = *reinterpret_cast<const uint4*>(word + slot);
      if ((w4.x & w4.y & w4.z & w4.w) == kWinFree) continue;
      const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (w[j] != kWinFree) atomicAdd(pix_count + win_pixel(slot + j, w[j], P.cam.W), w[j] & kWinCountMask);
      *reinterpret_cast<uint4*>(word + slot) = make_uint4(kWinFree, kWinFree, kWinFree, kWinFree);
    }
    __syncthreads();
  }
}

// Dynamic shared memory of the scattering pass: the chunk's fragments sorted
// by pixel (key, alpha, bucket slot), the window, and per counter the bucket
// slot of the chunk's first fragment.
template <int kT, int kPP>
struct ScatterSmem {
  static constexpr int kFrags = 4 * kT * kPP;
  unsigned long long key[kFrags];
  float alpha[kFrags];
  uint32_t dst[kFrags];
  uint32_t word[kWinSlots];
  uint32_t base[kWinSlots];
  int n_sorted[2];  // alternate over the chunks
};

template <int kT, int kPP, class FT>
__global__ void __launch_bounds__(kT, 1024 / kT) k_pix_scatter(RP P, const float* __restrict__ pos,
                                                           const float* __restrict__ opacity,
                                                           const FT* __restrict__ feat, RasterWs ws) {
  using Shape = BinShape<kT, kPP>;
  constexpr int kPoints = Shape::kPoints;
  if (!window_wanted(ws.sample)) return;
  extern __shared__ __align__(16) unsigned char dyn[];
  ScatterSmem<kT, kPP>& S = *reinterpret_cast<ScatterSmem<kT, kPP>*>(dyn);
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < kWinSlots; i += kT) S.word[i] = kWinFree;
  if (threadIdx.x < 2) S.n_sorted[threadIdx.x] = 0;
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
    // the chunk's fragments: their rank within their pixel
    Splat s[kPP];
    float av[kPP];
    uint32_t rank[kPP][2];
    unsigned ok = 0;
#pragma unroll
    for (int u = 0; u < kPP; ++u) {
      av[u] = next[u][3];
      if (c0 + u * kT + (int)threadIdx.x < n && splat_xyz(P, next[u][0], next[u][1], next[u][2], s[u])) {
        ok |= 1u << u;
        win_take(P, S.word, s[u].f, rank[u]);
      }
    }
    __syncthreads();
    load(c0 + (long long)gridDim.x * kPoints);
    // one global atomic per pixel in use gives the bucket slots of its
    // fragments (the counts run down from the bucket size, so the buckets
    // fill back to front) and its place in the sorted chunk replaces the
    // counter.  The window is read as a whole: a thread's few counters are
    // all in flight together.
#pragma unroll
    for (int i = 0; i < Shape::kScan; ++i) {
      const int slot = 4 * (i * kT + (int)threadIdx.x);
      const uint4 w4 = *reinterpret_cast<const uint4*>(S.word + slot);
      const uint32_t w[4] = {w4.x, w4.y, w4.z, w4.w};
      const bool used = (w4.x & w4.y & w4.z & w4.w) != kWinFree;
      if (!__any_sync(0xffffffffu, used)) continue;
      uint32_t first[4] = {0, 0, 0, 0}, c[4], incl = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        c[j] = w[j] != kWinFree ? w[j] & kWinCountMask : 0u;
        if (c[j]) {
          const uint32_t q = win_pixel(slot + j, w[j], P.cam.W);
          first[j] = __ldg(ws.pix_start + q) + atomicSub(ws.pix_count + q, c[j]) - c[j];
        }
        incl += c[j];
      }
      const uint32_t mine = incl;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += t;
      }
      int at = 0;
      if (lane == 31) at = atomicAdd(&S.n_sorted[turn], (int)incl);
      at = __shfl_sync(0xffffffffu, at, 31) + (int)(incl - mine);
      uint4 place;
      place.x = at;
      place.y = place.x + c[0];
      place.z = place.y + c[1];
      place.w = place.z + c[2];
      if (used) {
        *reinterpret_cast<uint4*>(S.word + slot) = place;
        *reinterpret_cast<uint4*>(S.base + slot) = make_uint4(first[0], first[1], first[2], first[3]);
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
          if (q >= 0 && rank_of(rank[u], k) == kNoRank)
            to[k] = __ldg(ws.pix_start + q) + atomicSub(ws.pix_count + q, 1u) - 1u;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (corner_pixel(P, s[u].f, k) < 0) continue;
          const float a = fminf(__fmul_rn(ah, corner_weight(s[u].f, k & 1, k >> 1)), P.alpha_max);
          const uint32_t r = rank_of(rank[u], k);
          if (r != kNoRank) {
            const int slot = win_slot(s[u].f.i0 + (k & 1), s[u].f.j0 + (k >> 1));
            const uint32_t at = S.word[slot] + r;
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
    const int total = S.n_sorted[turn];
    if (threadIdx.x == 0) S.n_sorted[turn ^ 1] = 0;
#pragma unroll
    for (int i = 0; i < Shape::kScan; ++i)
      *reinterpret_cast<uint4*>(S.word + 4 * (i * kT + (int)threadIdx.x)) =
          make_uint4(kWinFree, kWinFree, kWinFree, kWinFree);
    for (int j = threadIdx.x; j < total; j += kT) {
      const uint32_t to = S.dst[j];
      ws.keys[to] = S.key[j];
      ws.alpha[to] = S.alpha[j];
    }
    __syncthreads();
  }
}

// The scattering pass without the window, for small or unordered clouds (with
// a sample, only where that does not ask for the window): one returning atomic
// per run of equal pixels over consecutive lanes.  A run is found with one
// shuffle and one ballot (its start is a lane whose pixel differs from the
// previous lane's), and its first lane updates the counter for the whole run.
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
                                                     float* __restrict__ pexp,
                                                     const WinSample* __restrict__ sample) {
  if (sample && window_wanted(sample)) return;
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
