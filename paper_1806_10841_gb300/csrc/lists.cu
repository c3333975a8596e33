// The list build (lists_impl.cuh) as a kernel of its own, the device-wide scan of the sample
// collection, and the largest list length.
#include <algorithm>

#include "lists_impl.cuh"

namespace adress {

constexpr int kScanThreads = 512;
constexpr int kScanEPT = 4;
constexpr int kScanTile = kScanThreads * kScanEPT;

// ---- decision and build --------------------------------------------------------------------

// What the last block to arrive does once every block has read the control block: make the
// mapping current, clear the maxima and the network's pair count for the next step.
__device__ __forceinline__ void finish_mapping(const Bufs& b, const Decision& d, DecideArgs da) {
  Ctrl* c = b.ctrl;
  const int l = threadIdx.x & 31;
  c->ext_slot[0][0][l] = 0u;
  c->ext_slot[0][1][l] = 0u;
  if (l != 0) return;
  if (d.too_wide) set_error(c, ADRESS_ERR_EXTENT, (int)(d.ext * 1000));
  c->ext_now = d.ext;
  if (d.rebuild) c->rebuilds += 1;
  if (d.rebuild && da.build) c->force_rebuild = 0;
  if (da.advance) c->step += 1;
  c->parity ^= 1;
  if (b.npair) *b.npair = 0u;
  c->lists_err = __ldcg(&c->err);
}

// Decision only (a mapping outside a run: no lists are built for it).  A programmatic dependent of
// the mapping kernel, whose last blocks its launch overlaps: a density sample of 4000 molecules
// 23.2 us a call without, 21.3 with.
__global__ void __launch_bounds__(32) k_decide(const __grid_constant__ Sys s, Bufs b, DecideArgs da) {
  asm volatile("griddepcontrol.wait;" ::: "memory");  // the mapping is complete and visible
  const Decision d = decide_rebuild(s, b.ctrl, 0, da.force);
  if (!d.dead) finish_mapping(b, d, da);
}

// Decision and, when needed, the whole list build: one block of 768 threads per SM.  Few blocks
// keep the steps without a build cheap (two dependent L2 reads and one atomic per block; as a
// decision kernel and a conditional graph node around nine build kernels the same cost about
// 12 us a step at 800k atoms), and 80 registers keep the build's cell loop free of spills (800k
// atoms, us a build: 512 threads x 4 blocks 115, x 3 111, x 2 99, 1024 x 1 94, 768 x 1 90).
constexpr int kListThreads = 768, kListBlocksPerSm = 1;
__global__ void __launch_bounds__(kListThreads, kListBlocksPerSm) k_lists(const __grid_constant__ Sys s, const __grid_constant__ Bufs b,
                                                                        DecideArgs da) {
  Ctrl* c = b.ctrl;
  const int cur = c->parity ^ 1;
  const Decision d = decide_rebuild(s, c, 0, da.force);
  if (d.dead) return;  // (the barrier left a timeout in lists_err)
  if (d.rebuild) {
    GridBarrier bar(b, &c->bar[0]);
    if (!rebuild_lists<kListThreads / 32>(s, b, cur, bar)) return;
    // the last phase ends without a barrier: a block arrives below only with the errors of all its
    // warps set, for the host takes lists_err for the outcome of the build
    __syncthreads();
  }
  // the last block to get here (no block waits) closes the mapping
  if (threadIdx.x < 32 && last_to_arrive(c)) finish_mapping(b, d, da);
}

cudaError_t launch_lists(const Sys& s, const Bufs& b, DecideArgs da, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[1];
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (!da.build) {
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.gridDim = dim3(1);
    cfg.blockDim = dim3(32);
    return cudaLaunchKernelEx(&cfg, k_decide, s, b, da);
  }
  // two and a half cells a warp, or a block per 64 molecules where the cells are few or dense (us a
  // build, the whole call, 256 / 64 / 32 a block: 1000 tetrahedra at density 0.1 55 / 45 / 46, at 0.3
  // 94 / 69 / 70; 6000 water-like molecules 338 / 321 / 319, with steps that build no lists 20.9 / 21.0 /
  // 21.0 us each)
  const long long want = std::max(ceil_div((long long)s.ncell * 32 * 2, kListThreads * 5), ceil_div(s.M, 64));
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.gridDim = dim3((unsigned)std::min<long long>(want, (long long)s.n_sm * kListBlocksPerSm));
  cfg.blockDim = dim3(kListThreads);
  return cudaLaunchKernelEx(&cfg, k_lists, s, b, da);
}

// ---- candidate pairs of lists already built --------------------------------------------------

template <bool F64>
__global__ void __launch_bounds__(128) k_net_candidates(const __grid_constant__ Sys s, Bufs b) {
  net_candidates_of<F64>(s, b, b.ctrl->parity, (blockIdx.x * blockDim.x + threadIdx.x) >> 2, threadIdx.x & 3);
}

cudaError_t launch_net_candidates(const Sys& s, const Bufs& b, cudaStream_t st) {
  const int blocks = ceil_div((long long)s.M * 4, 128);
  if (s.fp64) k_net_candidates<true><<<blocks, 128, 0, st>>>(s, b);
  else k_net_candidates<false><<<blocks, 128, 0, st>>>(s, b);
  return cudaGetLastError();
}

// ---- exclusive scan in two launches: tile sums, then every block adds up the sums of the
// tiles before its own (at most kScanMaxTiles of them) and scans its tile ----

constexpr int kScanMaxTiles = 4096;
static_assert((long long)kScanMaxTiles * kScanTile == kMaxScan, "largest scan");

// Block-wide sum of v (every thread gets it).
__device__ __forceinline__ int block_sum(int v) {
  __shared__ int part[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  v = __reduce_add_sync(0xffffffffu, v);
  __syncthreads();  // part[] may still be read by a previous call
  if (lane == 0) part[w] = v;
  __syncthreads();
  int s = lane < (int)(blockDim.x >> 5) ? part[lane] : 0;
  return __reduce_add_sync(0xffffffffu, s);
}

// Block-wide exclusive scan of v; *total gets the block's sum.
__device__ __forceinline__ int block_exclusive_scan(int v, int* total) {
  __shared__ int warp_sums[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_sums[w] = incl;
  __syncthreads();
  if (w == 0) {
    int ws = lane < (int)(blockDim.x >> 5) ? warp_sums[lane] : 0;
    int wi = ws;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      int t = __shfl_up_sync(0xffffffffu, wi, o);
      if (lane >= o) wi += t;
    }
    warp_sums[lane] = wi - ws;  // exclusive
    if (lane == 31) warp_sums[31] = wi;  // block total in the last slot (read below)
  }
  __syncthreads();
  const int excl = incl - v + (w ? warp_sums[w] : 0);
  if (total) *total = warp_sums[31];
  return excl;
}

// The warp-0 pass stores exclusive sums in slots 0..nw-1 and the total in slot 31; with 512
// threads nw = 16 <= 31, so they never clash.
static_assert(kScanThreads / 32 < 32, "scan block too large");

__global__ void __launch_bounds__(kScanThreads) k_scan_sums(const int* in, int* tile_sums, int n) {
  const int base = blockIdx.x * kScanTile + threadIdx.x * kScanEPT;
  int sum = 0;
#pragma unroll
  for (int e = 0; e < kScanEPT; ++e) sum += (base + e < n) ? in[base + e] : 0;
  sum = block_sum(sum);
  if (threadIdx.x == 0) tile_sums[blockIdx.x] = sum;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_apply(const int* in, int* out, const int* tile_sums, int n,
                                                             int* grand) {
  int before = 0;
  for (int k = threadIdx.x; k < (int)blockIdx.x; k += blockDim.x) before += tile_sums[k];
  before = block_sum(before);
  const int base = blockIdx.x * kScanTile + threadIdx.x * kScanEPT;
  int v[kScanEPT], sum = 0;
#pragma unroll
  for (int e = 0; e < kScanEPT; ++e) {
    v[e] = (base + e < n) ? in[base + e] : 0;
    sum += v[e];
  }
  int total;
  int run = before + block_exclusive_scan(sum, &total);
#pragma unroll
  for (int e = 0; e < kScanEPT; ++e) {
    if (base + e < n) out[base + e] = run;
    run += v[e];
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) *grand = before + total;
}

static cudaError_t exclusive_scan(const int* in, int* out, int n, int* tmp, int* total, cudaStream_t st) {
  const int ntiles = std::max(1, ceil_div(n, kScanTile));
  if (ntiles > kScanMaxTiles) return cudaErrorInvalidValue;
  k_scan_sums<<<ntiles, kScanThreads, 0, st>>>(in, tmp, n);
  k_scan_apply<<<ntiles, kScanThreads, 0, st>>>(in, out, tmp, n, total);
  return cudaGetLastError();
}

// Largest neighbour count of the last build (host-side capacity check only).
__global__ void k_max_nn(const __grid_constant__ Sys s, const Bufs b) {
  int m = 0;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < s.M; t += gridDim.x * blockDim.x) m = max(m, b.nn[t]);
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(&b.ctrl->max_nn, m);
}

cudaError_t launch_max_nn(const Sys& s, const Bufs& b, cudaStream_t st) {
  cudaMemsetAsync(&b.ctrl->max_nn, 0, sizeof(int), st);
  k_max_nn<<<64, 256, 0, st>>>(s, b);
  return cudaGetLastError();
}

cudaError_t device_exclusive_scan(const int* in, int* out, int n, int* tmp, int* total, cudaStream_t st) {
  return exclusive_scan(in, out, n, tmp, total, st);
}

}  // namespace adress
