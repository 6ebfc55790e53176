// Cell-linked list of the multi-resolution grid (the neighbour search of Algorithm 1).
//
// At a neighbour-list rebuild, particles are ordered by cell key with a
// counting sort over the dense key range: warp-aggregated atomic counts per
// cell and per tile of cells (k_rekey, sph_step_impl.cuh), an exclusive scan of
// the counts (which is also the cell-start table the list build reads), an
// atomic scatter that counts each cell back down to zero, and a gather that
// orders each cell by particle id (so the order is a function of the keys
// alone: by key, then id) while it moves the particle state into the other
// buffer and makes the views (k_gather_view, sph_step_impl.cuh). Every kernel
// here returns at once on steps without a rebuild (ctl->rebuild == 0), so one
// captured graph serves every step; an idle kernel of a graph still takes
// 1.1 us, so there are as few of them as grid-wide dependencies allow.
#include "sph_internal.h"

namespace sph {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanItems = kScanTile / kScanThreads;
// up to this many tiles every block of k_scan_down adds up the tiles before its
// own (8 sums per thread at most); beyond, one block scans them first
constexpr int kScanOwn = 2048;

__global__ void k_request_rebuild(StepCtl* __restrict__ ctl) { ctl->need_rebuild = 1; }
__global__ void k_write_ctl(StepCtl* __restrict__ ctl, StepCtl v) { *ctl = v; }

__global__ void __launch_bounds__(256) k_scatter(int n, const StepCtl* __restrict__ ctl,
                                                 const uint32_t* __restrict__ key,
                                                 const uint32_t* __restrict__ cstart,
                                                 uint32_t* __restrict__ cnt,
                                                 uint32_t* __restrict__ slots, uint32_t* __restrict__ part, int nb) {
  after_predecessor();
  if (!ctl->rebuild) return;
  // the tile counts are used up: zero for the next rebuild
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x) part[b] = 0u;
  for (int b0 = blockIdx.x * blockDim.x; b0 < n; b0 += gridDim.x * blockDim.x) {
    const int i = b0 + threadIdx.x;
    const bool active = i < n;
    const unsigned mask = __ballot_sync(0xffffffffu, active);
    if (!active) continue;
    const uint32_t k = key[i];
    const unsigned peers = __match_any_sync(mask, k);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    uint32_t top = 0;
    if (lane == leader) top = atomicSub(&cnt[k], (uint32_t)__popc(peers));
    top = __shfl_sync(peers, top, leader);
    const int rank = __popc(peers & ((1u << lane) - 1u));
    slots[cstart[k] + top - 1 - rank] = (uint32_t)i;
  }
}

// exclusive scan of the tile counts, in place (one block of 1024 threads)
__global__ void __launch_bounds__(1024) k_scan_top(const StepCtl* __restrict__ ctl, uint32_t* __restrict__ part,
                                                   int nb) {
  after_predecessor();
  if (!ctl->rebuild) return;
  __shared__ uint32_t wsum[32];
  int per = (nb + blockDim.x - 1) / blockDim.x;
  int b0 = threadIdx.x * per;
  uint32_t local = 0;
  for (int k = 0; k < per; ++k)
    if (b0 + k < nb) local += part[b0 + k];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t incl = local;
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) wsum[w] = incl;
  __syncthreads();
  if (w == 0) {
    uint32_t v = lane < (int)(blockDim.x >> 5) ? wsum[lane] : 0;
    uint32_t vi = v;
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t u = __shfl_up_sync(0xffffffffu, vi, o);
      if (lane >= o) vi += u;
    }
    wsum[lane] = vi - v;
  }
  __syncthreads();
  uint32_t run = wsum[w] + incl - local;
  for (int k = 0; k < per; ++k)
    if (b0 + k < nb) {
      uint32_t v = part[b0 + k];
      part[b0 + k] = run;
      run += v;
    }
}

// exclusive scan of each tile plus its block offset; out has n + 1 entries
__global__ void __launch_bounds__(kScanThreads) k_scan_down(const StepCtl* __restrict__ ctl,
                                                            const uint32_t* __restrict__ in, uint32_t n,
                                                            const uint32_t* __restrict__ part, int scanned,
                                                            uint32_t* __restrict__ out) {
  after_predecessor();
  if (!ctl->rebuild) return;
  __shared__ uint32_t wtot[kScanThreads / 32], wpre[kScanThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  // the counts before this tile: scanned already, or added up here
  uint32_t pre = 0;
  if (!scanned) {
    for (int b = threadIdx.x; b < (int)blockIdx.x; b += kScanThreads) pre += part[b];
    pre = __reduce_add_sync(0xffffffffu, pre);
    if (lane == 0) wpre[w] = pre;
  }
  // each warp owns kScanItems * 32 consecutive entries of the tile
  size_t wbase = (size_t)blockIdx.x * kScanTile + (size_t)w * kScanItems * 32;
  uint32_t v[kScanItems];
  uint32_t run = 0;
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    size_t idx = wbase + (size_t)k * 32 + lane;
    uint32_t x = idx < n ? in[idx] : 0u;
    uint32_t incl = x;
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    v[k] = run + incl - x;
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
  if (lane == 0) wtot[w] = run;
  __syncthreads();
  uint32_t start = 0;
  if (scanned) start = part[blockIdx.x];
  else
    for (int q = 0; q < kScanThreads / 32; ++q) start += wpre[q];
  uint32_t off = start;
  for (int q = 0; q < w; ++q) off += wtot[q];
#pragma unroll
  for (int k = 0; k < kScanItems; ++k) {
    size_t idx = wbase + (size_t)k * 32 + lane;
    if (idx < n) out[idx] = off + v[k];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == kScanThreads - 1) {
    uint32_t tot = start;
    for (int q = 0; q < kScanThreads / 32; ++q) tot += wtot[q];
    out[n] = tot;
  }
}

// feature-surface flags by particle id into the current meta words (colours kept)
__global__ void __launch_bounds__(256) k_set_surface(int n, const StepCtl* __restrict__ ctl,
                                                     const uint32_t* __restrict__ p0, const uint32_t* __restrict__ p1,
                                                     uint32_t* __restrict__ m0, uint32_t* __restrict__ m1,
                                                     const uint8_t* __restrict__ flags) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int buf = ctl->buf;
  uint32_t* __restrict__ m = buf ? m1 : m0;
  const uint32_t id = (buf ? p1 : p0)[i];
  const uint32_t v = m[i] & ~kSurfaceBit;
  m[i] = (flags && flags[id]) ? (v | kSurfaceBit) : v;
}

__global__ void __launch_bounds__(256) k_get_colors(int n, const StepCtl* __restrict__ ctl,
                                                    const uint32_t* __restrict__ m0, const uint32_t* __restrict__ m1,
                                                    const uint32_t* __restrict__ p0, const uint32_t* __restrict__ p1,
                                                    uint8_t* __restrict__ out) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int buf = ctl->buf;
  if (i < n) out[(buf ? p1 : p0)[i]] = (uint8_t)((buf ? m1 : m0)[i] & 0xFFu);
}

}  // namespace

cudaError_t launch_write_ctl(const DevState& S, const StepCtl& v, cudaStream_t st) {
  k_write_ctl<<<1, 1, 0, st>>>(S.ctl, v);
  return cudaGetLastError();
}

cudaError_t launch_request_rebuild(const DevState& S, cudaStream_t st) {
  k_request_rebuild<<<1, 1, 0, st>>>(S.ctl);
  return cudaGetLastError();
}

cudaError_t launch_set_surface(const DevState& S, const uint8_t* flags, cudaStream_t st) {
  if (S.n > 0)
    k_set_surface<<<(S.n + 255) / 256, 256, 0, st>>>(S.n, S.ctl, S.pid[0], S.pid[1], S.meta[0], S.meta[1], flags);
  return cudaGetLastError();
}

cudaError_t launch_get_colors(const DevState& S, uint8_t* out, cudaStream_t st) {
  if (S.n > 0)
    k_get_colors<<<(S.n + 255) / 256, 256, 0, st>>>(S.n, S.ctl, S.meta[0], S.meta[1], S.pid[0], S.pid[1], out);
  return cudaGetLastError();
}

cudaError_t build_cells(const DevState& S, cudaStream_t st) {
  const int n = S.n;
  if (n <= 0) return cudaSuccess;
  const int tb = 256;
  const int gb = rebuild_grid(n, tb, 8);
  const uint32_t m = S.total_cells;
  const int nb = (int)scan_tiles(m), scanned = nb > kScanOwn;
  if (scanned) launch_after(k_scan_top, 1, 1024, 0, st, S.ctl, S.scan_part, nb);
  launch_after(k_scan_down, nb, kScanThreads, 0, st, S.ctl, S.cnt, m, S.scan_part, scanned, S.cstart);
  launch_after(k_scatter, gb, tb, 0, st, n, S.ctl, S.key, S.cstart, S.cnt, S.tmp, S.scan_part, nb);
  return cudaGetLastError();
}

}  // namespace sph
