// Observables: deterministic FP64 reductions, the COM density
// profile and the thermodynamic-force iteration, and the FP64 export of centres of mass.
#include <math.h>

#include <algorithm>

#include "internal.cuh"

namespace adress {

// ---- deterministic FP64 reductions: per-block partials, then one fixed-order block ----

// Block sums of four values into part[slot].  A warp's butterfly hands half of the values to
// each half of its lanes at the first two levels, so that it takes 6 additions a lane instead of
// 20 (the FP64 pipe is the bound); the additions that reach a sum, and their order, are those of
// the plain butterfly.
__device__ __forceinline__ void block_partials(const double (&v)[4], double* part, int slot) {
  __shared__ double sm[32][4];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const bool up = lane & 16, odd = lane & 8;
  // lanes 0-15 take v[0], v[1], lanes 16-31 v[2], v[3]; then lanes with bit 3 clear the first
  double a = up ? v[2] : v[0], c = up ? v[3] : v[1];
  a += __shfl_xor_sync(0xffffffffu, up ? v[0] : v[2], 16);
  c += __shfl_xor_sync(0xffffffffu, up ? v[1] : v[3], 16);
  double r = odd ? c : a;
  r += __shfl_xor_sync(0xffffffffu, odd ? a : c, 8);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  if ((lane & 7) == 0) sm[w][lane >> 3] = r;
  __syncthreads();
  if (threadIdx.x < 4) {
    double acc = 0.0;
    for (int q = 0; q < nw; ++q) acc += sm[q][threadIdx.x];
    part[(size_t)slot * 4 + threadIdx.x] = acc;
  }
}

// Sum of the partials [nparts][4], one block.
__global__ void __launch_bounds__(1024) k_reduce_parts(const double4_32a* part, int nparts, double* out) {
  double v[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 4
  for (int p = threadIdx.x; p < nparts; p += blockDim.x) {
    const double4_32a r = part[p];
    v[0] += r.x;
    v[1] += r.y;
    v[2] += r.z;
    v[3] += r.w;
  }
  block_partials(v, out, 0);
}

template <int NA>
__global__ void __launch_bounds__(256) k_kinetic(const __grid_constant__ Sys s, Bufs b) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  double v[4] = {0.0, 0.0, 0.0, 0.0};
  if (i < s.N) {
    const double m = s.mass[i % NA];
    for (int d = 0; d < 3; ++d) {
      double u = b.v[(size_t)d * s.N + i];
      v[0] += 0.5 * m * u * u;
      v[1 + d] = m * u;
    }
  }
  block_partials(v, b.part, blockIdx.x);
}

// Centre-of-mass x in double exactly as R = sum_k m_k (x_0 + minimg(x_k - x_0)) / M, wrapped.
template <int NA>
__device__ double com_x64(const Sys& s, const Box& B, const double* x, int a) {
  const double x0 = x[a * NA];
  double acc = 0.0;
  for (int k = 0; k < NA; ++k) acc += s.mass[k] * (x0 + minimg_cmp(x[a * NA + k] - x0, B.L[0], B.halfL[0]));
  double r = acc / s.Mtot;
  r -= B.L[0] * floor(r / B.L[0]);
  if (r >= B.L[0]) r -= B.L[0];
  return r;
}

// Distance of molecule a's centre of mass (in double, from x, as the definition forms it) to
// the nearest resolution centre (the first of equal distances).
template <int NA>
__device__ double center_d64(const Sys& s, const Box& B, const Bufs& b, int a) {
  const size_t N = (size_t)s.N;
  double R[3];
  for (int d = 0; d < 3; ++d) {
    const double x0 = b.x[d * N + a * NA];
    double acc = 0.0;
    for (int k = 0; k < NA; ++k) acc += s.mass[k] * (x0 + minimg_cmp(b.x[d * N + a * NA + k] - x0, B.L[d], B.halfL[d]));
    double r = acc / s.Mtot;
    r -= B.L[d] * floor(r / B.L[d]);
    if (r >= B.L[d]) r -= B.L[d];
    R[d] = r;
  }
  double best = INFINITY;
  for (int k = 0; k < s.n_centers; ++k) {
    const double4_32a C = b.cen64[k];
    const double t0 = minimg_cmp(R[0] - C.x, B.L[0], B.halfL[0]);
    const double t1 = minimg_cmp(R[1] - C.y, B.L[1], B.halfL[1]);
    const double t2 = minimg_cmp(R[2] - C.z, B.L[2], B.halfL[2]);
    const double r = sqrt(__dadd_rn(__dadd_rn(__dmul_rn(t0, t0), __dmul_rn(t1, t1)), __dmul_rn(t2, t2)));
    if (r < best) best = r;
  }
  return best;
}

// COM histogram folded about the slab centre: bin floor(|dxc| / tf_dx), integer atomics
// (one histogram of tf_n bins per box).  The FP32 path takes |dxc| from its float mapping
// and recomputes it in double for the few molecules within 1e-4 of a bin edge, so the bin
// is the one the double value gives.  A single box counts into shared memory first.
template <int NA>
__global__ void __launch_bounds__(1024) k_density(const __grid_constant__ Sys s, Bufs b) {
  extern __shared__ unsigned hs[];
  const bool multi = s.nbox > 1;
  if (!multi) {
    for (int k = threadIdx.x; k < s.tf_n; k += blockDim.x) hs[k] = 0u;
    __syncthreads();
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) atomicAdd((unsigned long long*)b.nsamples, 1ull);
  const int cur = b.ctrl->parity;
  for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < s.M; a += gridDim.x * blockDim.x) {
    const Box& B = box_of(s, b, a);
    int k;
    if (s.fp64) {
      k = (int)floor(fabs(b.dxc64[cur][a]) / s.tf_dx);
    } else {
      const float u = fabsf(b.molf[cur][a].x) * s.f.tf_inv_dx, fr = u - floorf(u);
      k = (int)floorf(u);
      if (fr < 1e-4f || fr > 1.f - 1e-4f)
        k = (int)floor((s.n_centers > 0 ? center_d64<NA>(s, B, b, a)
                                        : fabs(minimg_cmp(com_x64<NA>(s, B, b.x, a) - B.xc, B.L[0], B.halfL[0]))) /
                       s.tf_dx);
    }
    if (k < s.tf_n) {
      if (multi) atomicAdd(&b.hist[B.tf0 + k], 1ull);
      else atomicAdd(&hs[k], 1u);
    }
  }
  if (!multi) {
    __syncthreads();
    for (int k = threadIdx.x; k < s.tf_n; k += blockDim.x)
      if (hs[k]) atomicAdd(&b.hist[k], (unsigned long long)hs[k]);
  }
}

// Thermodynamic-force iteration on the accumulated profile, one block per box (tf_n nodes):
// rho_k = counts_k / (nsamples V_k) (V_k: 2 dx Ly Lz, or the shells around the resolution
// centres), g_k = (rho_k - rho_{k-1})/dx, g_0 = 0,
// three-point moving average, tf_k -= alpha g_k on hybrid-layer nodes, then the box's
// histogram is cleared (the sample count is cleared by the launcher afterwards).
__global__ void k_tf_update(const __grid_constant__ Sys s, Bufs b, double alpha) {
  extern __shared__ double g[];
  const Box& B = s.nbox > 1 ? b.boxes[blockIdx.x] : s.bx;
  const int n = s.tf_n, o = B.tf0;
  const double ns = (double)(*b.nsamples);
  // bin volume: two slabs, or a spherical shell around each resolution centre
  auto vol = [&](int k) {
    const double dx = s.tf_dx;
    return s.n_centers > 0
               ? ns * s.n_centers * 4.0 / 3.0 * M_PI * ((k + 1.0) * (k + 1.0) * (k + 1.0) - (double)k * k * k) * dx * dx * dx
               : ns * 2.0 * dx * B.L[1] * B.L[2];
  };
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    double gk = 0.0;
    if (k > 0 && ns > 0) gk = ((double)b.hist[o + k] / vol(k) - (double)b.hist[o + k - 1] / vol(k - 1)) / s.tf_dx;
    g[k] = gk;
  }
  __syncthreads();
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    double sum = 0.0;
    int cnt = 0;
    for (int q = k - 1; q <= k + 1; ++q)
      if (q >= 0 && q < n) {
        sum += g[q];
        ++cnt;
      }
    const double dk = k * s.tf_dx;
    if (ns > 0 && dk >= B.d_at && dk <= B.d_at + B.d_hy) {
      double t = b.tf64[o + k] - alpha * sum / cnt;
      b.tf64[o + k] = t;
      b.tf32[o + k] = (float)t;
    }
  }
  __syncthreads();
  for (int k = threadIdx.x; k < n; k += blockDim.x) b.hist[o + k] = 0ull;
}

// FP64 centres of mass of the current positions (computed from x as the definition
// states) and the resolution values the force kernels use.
__global__ void k_clear_samples(long long* n) { *n = 0; }

// (Wraps and minimum images by comparing bits, and no division where the molecule's mass is a
// power of two: the same values with a fifth of the FP64 operations.)
template <int NA>
__global__ void k_export_com(const __grid_constant__ Sys s, Bufs b, double* com, double* w) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= s.M) return;
  const Box& B = box_of(s, b, a);
  const size_t N = (size_t)s.N;
  const bool pow2 = (__double_as_longlong(s.Mtot) & 0xFFFFFFFFFFFFFll) == 0 && s.Mtot > 1e-300 && s.Mtot < 1e300;
  const double inv_m = __longlong_as_double((2046ll << 52) - __double_as_longlong(s.Mtot));  // 1 / Mtot of a power of two
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const double x0 = b.x[d * N + (size_t)a * NA];
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < NA; ++k)
      acc += s.mass[k] * (x0 + minimg_bits(b.x[d * N + (size_t)a * NA + k] - x0, B.L[d], B.halfL[d]));
    double r = pow2 ? acc * inv_m : acc / s.Mtot;
    const long long bits = __double_as_longlong(r);
    if (bits < 0 || bits >= B.Lbits[d]) {  // outside [0, L)
      r -= B.L[d] * floor(r / B.L[d]);
      if (r >= B.L[d]) r -= B.L[d];
    }
    com[(size_t)d * s.M + a] = r;
  }
  if (w) {
    const int cur = b.ctrl->parity;
    w[a] = s.fp64 ? b.com64[cur][a].w : (double)__int_as_float(b.com_fx[cur][a].w);
  }
}

// ---- COM pair-distance histogram (numerator of the radial distribution function) -----------
// Every pair a < b of the same box with minimum-image distance r < nbins dr adds one to bin
// floor(r / dr) of its box.  The centres are sorted into cells at least nbins dr wide and only
// neighbouring cells are compared: at 200,000 molecules and r < 5 the all-pairs form tested 2e10
// pairs (33 ms) where 5e6 are in range.  Distances are formed in FP32 from fixed-point centres; a
// pair whose distance lies within the FP32 error of a bin edge is decided in double with
// explicitly rounded products and sums (no contraction), the operations the oracle performs, so
// bins are the oracle's.

// Cell of each centre and its place in the cell's slice.
__global__ void k_rdf_cell(const __grid_constant__ Sys s, const __grid_constant__ Bufs b, const RdfArgs q) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a >= s.M) return;
  const Box& B = box_of(s, b, a);
  const RdfGrid G = q.grids[B.index];
  unsigned X[3];
  int c[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    X[d] = (unsigned)fmin(q.com[(size_t)d * s.M + a] * B.fx_inv[d], 4294967295.0);
    c[d] = (int)(((unsigned long long)X[d] * (unsigned long long)G.nc[d]) >> 32);
  }
  const int r = G.cell0 + (c[0] * G.nc[1] + c[1]) * G.nc[2] + c[2];
  q.cell[a] = r;
  q.slot[a] = atomicAdd(&q.count[r], 1);
  q.fx[a] = make_int4((int)X[0], (int)X[1], (int)X[2], a);
}

__global__ void k_rdf_fill(int M, const RdfArgs q) {
  const int a = blockIdx.x * blockDim.x + threadIdx.x;
  if (a < M) q.sorted[q.start[q.cell[a]] + q.slot[a]] = q.fx[a];
}

// Each block takes a run of tasks, box by box (a box's counts in shared memory, added to the
// global ones when the run leaves the box).  A warp's task is a part of a cell: batches of its
// molecules, against which the lanes hold 32 candidates of the neighbour cells at a time.  Where a
// box has at least three cells each way only half the neighbour cells are visited (each pair of
// cells once), else all distinct ones, counting the pairs whose candidate comes later in the
// sorted order.  The parts are many where the cells are few (a range near half the box leaves one
// cell to some sixteen; the cell's first molecules then have the most candidates after them, so
// early and late parts alternate).  ms a call, all pairs in double / a warp per cell / now: 200,000
// molecules r < 5 32 / 0.19 / 0.18, a quarter of the shortest edge 1061 / 543 / 21, just below half
// 1610 / 16,624 / 123; 20,000: 5.6 / 0.10 / 0.08, 36 / 5.6 / 0.40, 53 / 114 / 1.1; 1000 at half the
// edge 2.5 / 1.6 / 0.10.
constexpr int kRdfThreads = 256;

// A block counts in 32 bits: after a batch a warp hands the counts on when it has tested this many
// pairs since it last did.  A batch of 32 molecules has at most 2^28 (adress_init takes fewer than
// 2^23 molecules), so the eight warps of a block never hold 2^32.  (Once in 2^20 pairs costs a
// fraction of a percent.)
constexpr unsigned kRdfHandOn = 1u << 20;
static_assert(8ll * (32 * kMaxScan + kRdfHandOn) < 1ll << 32, "counts of a block");
__device__ __noinline__ void hand_on_counts(unsigned* rh, unsigned long long* counts, int nbins) {
  for (int k = threadIdx.x & 31; k < nbins; k += 32) {
    const unsigned c = atomicExch(&rh[k], 0u);
    if (c) atomicAdd(&counts[k], (unsigned long long)c);
  }
}

__global__ void __launch_bounds__(kRdfThreads) k_rdf(const __grid_constant__ Sys s, const __grid_constant__ Bufs b, const RdfArgs q) {
  extern __shared__ unsigned rh[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int chunk = (q.ntask + gridDim.x - 1) / gridDim.x;
  int t0 = blockIdx.x * chunk;
  const int t_end = min(q.ntask, t0 + chunk);
  while (t0 < t_end) {
    // the box of the run's first task (boxes in task order)
    int lo = 0, hi = s.nbox - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (q.grids[mid].task0 <= t0) lo = mid;
      else hi = mid - 1;
    }
    const RdfGrid G = q.grids[lo];
    const Box& B = s.nbox > 1 ? b.boxes[lo] : s.bx;
    const int nx = G.nc[0], ny = G.nc[1], nz = G.nc[2];
    const int t1 = min(t_end, G.task0 + nx * ny * nz * G.parts);
    const bool half = nx >= 3 && ny >= 3 && nz >= 3;
    const float sx = B.fx_scale[0], sy = B.fx_scale[1], sz = B.fx_scale[2];
    unsigned tested = 0;
    for (int k = threadIdx.x; k < q.nbins; k += blockDim.x) rh[k] = 0u;
    __syncthreads();
    for (int t = t0 + warp; t < t1; t += kRdfThreads / 32) {
      int l = t - G.task0, part = 0;
      if (G.parts > 1) {
        const int e = l % G.parts;
        l /= G.parts;
        part = e & 1 ? G.parts - 1 - (e >> 1) : e >> 1;
      }
      const int r = G.cell0 + l, hs = q.start[r], he = q.start[r + 1], first = hs + part * q.batch;
      if (first >= he) continue;
      const int cx = l / (ny * nz), cy = (l / nz) % ny, cz = l % nz;
      // lane j < 27: neighbour cell (ox, oy, oz) = (j / 9 - 1, (j / 3) % 3 - 1, j % 3 - 1)
      int cnt = 0, start = 0;
      if (lane < 27 && (!half || lane >= 13)) {
        const int ox = lane / 9 - 1, oy = (lane / 3) % 3 - 1, oz = lane % 3 - 1;
        const bool ok = (ox >= 0 || nx >= 3) && (ox <= 0 || nx >= 2) && (oy >= 0 || ny >= 3) && (oy <= 0 || ny >= 2) &&
                        (oz >= 0 || nz >= 3) && (oz <= 0 || nz >= 2);
        if (ok) {
          const int x = (cx + ox + nx) % nx, y = (cy + oy + ny) % ny, z = (cz + oz + nz) % nz;
          const int rr = G.cell0 + (x * ny + y) * nz + z;
          start = q.start[rr];
          cnt = q.start[rr + 1] - start;
        }
      }
      int incl = cnt;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const int pre = incl - cnt, total = __shfl_sync(0xffffffffu, incl, 31);
      for (int hb = first; hb < he; hb += G.parts * q.batch) {
        const int ht = min(he, hb + q.batch);
        for (int k0 = 0; k0 < total; k0 += 32) {
          // this lane's candidate: the cells whose inclusive prefix is <= k come before its own
          const int k = k0 + lane;
          int j = 0;
#pragma unroll
          for (int step = 16; step >= 1; step >>= 1) {
            const int probe = j + step - 1;
            const int v = __shfl_sync(0xffffffffu, incl, probe < 27 ? probe : 26);
            if (probe < 27 && v <= k) j += step;
          }
          const int cc = j < 27 ? j : 26;
          const int g = __shfl_sync(0xffffffffu, start, cc) + (k - __shfl_sync(0xffffffffu, pre, cc));
          const bool in = k < total;
          const int4 D = q.sorted[in ? g : hb];
          // the batch's molecules (sorted positions) this candidate pairs with: all of them for
          // another cell of the half set, else those before it
          const int upto = !in ? hb : (half && cc != 13 ? ht : min(ht, g));
          const int most = __reduce_max_sync(0xffffffffu, upto);
          int4 Hn = __ldg(&q.sorted[hb]);
          for (int h = hb; h < most; ++h) {
            const int4 H = Hn;
            if (h + 1 < most) Hn = __ldg(&q.sorted[h + 1]);
            const float dx = (float)(int)((unsigned)H.x - (unsigned)D.x) * sx;
            const float dy = (float)(int)((unsigned)H.y - (unsigned)D.y) * sy;
            const float dz = (float)(int)((unsigned)H.z - (unsigned)D.z) * sz;
            const float r2 = dx * dx + dy * dy + dz * dz;
            if (h < upto && r2 < q.lim2) {
              float rr;
              asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(rr) : "f"(r2));
              const float u = rr * q.inv_dr, fl = floorf(u), fr = u - fl;
              int bin = (int)fl;
              if (fr < q.eps || fr > 1.f - q.eps) {
                const size_t M = (size_t)s.M;
                const double ex = minimg_cmp(q.com[H.w] - q.com[D.w], B.L[0], B.halfL[0]);
                const double ey = minimg_cmp(q.com[M + H.w] - q.com[M + D.w], B.L[1], B.halfL[1]);
                const double ez = minimg_cmp(q.com[2 * M + H.w] - q.com[2 * M + D.w], B.L[2], B.halfL[2]);
                const double e2 = __dadd_rn(__dadd_rn(__dmul_rn(ex, ex), __dmul_rn(ey, ey)), __dmul_rn(ez, ez));
                bin = (int)floor(sqrt(e2) / q.dr);
              }
              if (bin < q.nbins) atomicAdd(&rh[bin], 1u);
            }
          }
        }
        tested += (unsigned)(ht - hb) * (unsigned)total;
        if (tested >= kRdfHandOn) {
          hand_on_counts(rh, q.counts + (size_t)lo * q.nbins, q.nbins);
          tested = 0;
        }
      }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < q.nbins; k += blockDim.x)
      if (rh[k]) atomicAdd(&q.counts[(size_t)lo * q.nbins + k], (unsigned long long)rh[k]);
    __syncthreads();
    t0 = t1;
  }
}

// ---- launchers -----------------------------------------------------------------------


cudaError_t launch_energy_reduce(const Bufs& b, int nparts, cudaStream_t st) {
  k_reduce_parts<<<1, 1024, 0, st>>>((const double4_32a*)b.part, nparts, b.result);
  return cudaGetLastError();
}

cudaError_t launch_kinetic(const Sys& s, const Bufs& b, cudaStream_t st) {
  const int blocks = ceil_div(s.N, 256);
  switch (s.NA) {
    case 1: k_kinetic<1><<<blocks, 256, 0, st>>>(s, b); break;
    case 2: k_kinetic<2><<<blocks, 256, 0, st>>>(s, b); break;
    case 3: k_kinetic<3><<<blocks, 256, 0, st>>>(s, b); break;
    default: k_kinetic<4><<<blocks, 256, 0, st>>>(s, b); break;
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_energy_reduce(b, blocks, st);
}

cudaError_t launch_density(const Sys& s, const Bufs& b, int, cudaStream_t st) {
  const int blocks = std::min(ceil_div(s.M, 1024), 2 * 152);
  const size_t smem = s.nbox > 1 ? 0 : sizeof(unsigned) * std::max(1, s.tf_n);
  switch (s.NA) {
    case 1: k_density<1><<<blocks, 1024, smem, st>>>(s, b); break;
    case 2: k_density<2><<<blocks, 1024, smem, st>>>(s, b); break;
    case 3: k_density<3><<<blocks, 1024, smem, st>>>(s, b); break;
    default: k_density<4><<<blocks, 1024, smem, st>>>(s, b); break;
  }
  return cudaGetLastError();
}

cudaError_t launch_tf_update(const Sys& s, const Bufs& b, double alpha, cudaStream_t st) {
  if (s.tf_n <= 0) return cudaSuccess;
  k_tf_update<<<s.nbox, 256, sizeof(double) * s.tf_n, st>>>(s, b, alpha);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_clear_samples<<<1, 1, 0, st>>>(b.nsamples);
  return cudaGetLastError();
}

cudaError_t launch_rdf(const Sys& s, const Bufs& b, const RdfArgs& q, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(q.count, 0, sizeof(int) * q.ncell, st);
  if (e != cudaSuccess) return e;
  k_rdf_cell<<<ceil_div(s.M, 256), 256, 0, st>>>(s, b, q);
  e = device_exclusive_scan(q.count, q.start, q.ncell, (int*)b.scan_tmp, q.start + q.ncell, st);
  if (e != cudaSuccess) return e;
  k_rdf_fill<<<ceil_div(s.M, 256), 256, 0, st>>>(s.M, q);
  const int blocks = std::max(1, std::min(ceil_div(q.ntask, 2), 8 * s.n_sm));
  k_rdf<<<blocks, kRdfThreads, sizeof(unsigned) * q.nbins, st>>>(s, b, q);
  return cudaGetLastError();
}

cudaError_t launch_export_com(const Sys& s, const Bufs& b, int, double* com, double* w, cudaStream_t st) {
  const int blocks = ceil_div(s.M, 256);
  switch (s.NA) {
    case 1: k_export_com<1><<<blocks, 256, 0, st>>>(s, b, com, w); break;
    case 2: k_export_com<2><<<blocks, 256, 0, st>>>(s, b, com, w); break;
    case 3: k_export_com<3><<<blocks, 256, 0, st>>>(s, b, com, w); break;
    default: k_export_com<4><<<blocks, 256, 0, st>>>(s, b, com, w); break;
  }
  return cudaGetLastError();
}

}  // namespace adress
