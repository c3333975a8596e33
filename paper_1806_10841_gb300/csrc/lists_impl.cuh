// Neighbour search on the GPU: a linked-cell list over molecule centres of mass (the
// paper's linked-cell-list neighbour search, Sec. "Heterogeneous Spatial Domain
// Decomposition Algorithm", here on one GPU).  Cells are ranked in Morton order;
// molecules are counting-sorted by cell and each cell's members are then put in id order,
// so every list is deterministic; molecules are split into two work lists — high-resolution
// candidates (|dxc| < d_at + d_hy + skin/2) first, then coarse-grained molecules —
// and each work item gets a full Verlet list: partners within r_list when both are
// high-resolution items, within rc_cg + skin when either is coarse-grained (such a pair has
// weight 0 until the next build, so only the CG force, cut at rc_cg, acts between them;
// the lists stay symmetric).
//
// The whole build runs inside one cooperative grid (rebuild_lists): phases over all
// molecules or cells, separated by grid-wide barriers.  A step that needs no build pays only
// the decision; nothing is launched conditionally.
#pragma once
#include "internal.cuh"

namespace adress {

// Staged candidate: centre + (molecule id | high-resolution flag in bit 31).
__device__ __forceinline__ int tag_id(int id, int hr) { return (int)((unsigned)id | ((unsigned)hr << 31)); }
__device__ __forceinline__ int id_of(int w) { return w & 0x7fffffff; }

// Cell coordinate of a fixed-point coordinate X (X / 2^32 of the box edge): exact.
__device__ __forceinline__ int cell_of(unsigned int X, int nc) {
  return (int)(((unsigned long long)X * (unsigned long long)nc) >> 32);
}

// ---- grid-wide barrier -----------------------------------------------------------------
// All blocks of a cooperative launch; one 64-bit arrival counter that only grows (a launch
// finds it at a multiple of its grid).  The wait is bounded (Bufs::barrier_polls): when it gives
// up, the error word gets a timeout, Ctrl::dead is set and the block leaves the kernel; every
// later kernel with barriers leaves at once (the counters are out of step, the lists half built
// but in bounds) until the host has reported the error and reset both.  A block that passes the
// barrier all the same goes no further than the next one, where the blocks that left are missing:
// so a phase starts only when the phase before it is complete.
constexpr unsigned kPollsPerCheck = 1024;
struct GridBarrier {
  Ctrl* c;
  unsigned long long* count;
  unsigned long long target;
  const Bufs& b;
  bool first;
  // (no polls allowed: the target is out of reach)
  __device__ __forceinline__ GridBarrier(const Bufs& bufs, unsigned long long* ctr)
      : c(bufs.ctrl), count(ctr), target(bufs.barrier_polls ? 0ull : 1ull << 62), b(bufs), first(true) {}
  __device__ __forceinline__ bool sync() {
    int dead = 0;
    __syncthreads();
    if (threadIdx.x == 0) {
      // release: the block's writes (ordered before by the block barrier) are visible to whoever
      // sees the arrival; the reads below acquire.  Cheaper than full fences around the atomic.
      unsigned long long old;
      asm volatile("atom.add.release.gpu.global.u64 %0, [%1], 1;" : "=l"(old) : "l"(count) : "memory");
      if (first) target += old - old % gridDim.x;
      target += gridDim.x;
      for (unsigned n = 0;; ++n) {
        unsigned long long v;
        asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(count) : "memory");
        if ((long long)(v - target) >= 0) break;
        // (the limit is a kernel parameter: looked at at every poll it costs a step of 1000 molecules
        // in the run kernel 0.06 us of 8.1, now and then 0.02)
        if (n % kPollsPerCheck == kPollsPerCheck - 1 && n >= b.barrier_polls) {
          dead = 1;
          set_error(c, ADRESS_ERR_TIMEOUT, (int)blockIdx.x);
          atomicExch(&c->lists_err, ADRESS_ERR_TIMEOUT);
          atomicExch(&c->dead, 1);
          break;
        }
      }
    }
    first = false;
    return __syncthreads_or(dead) == 0;
  }
};

// True in warp 0 of the last block of the grid to call (each block's warp 0 calls once, after
// its block's last read of what the caller then writes); nobody waits.
__device__ __forceinline__ bool last_to_arrive(Ctrl* c) {
  unsigned old = 0;
  if (threadIdx.x == 0) {
    asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(old) : "l"(&c->arrive) : "memory");
    if (old == gridDim.x - 1) c->arrive = 0u;
  }
  return __shfl_sync(0xffffffffu, old, 0) == gridDim.x - 1;
}

// ---- rebuild decision --------------------------------------------------------------------
// After a mapping: rebuild when a centre moved more than skin/2 since the last build (it
// could have changed class or found a new partner), when the widest molecule makes
// max(rc_cg, rc_at + 2 ext) + 2 disp exceed the list cutoff, or when the host asked for it
// (the resolution region moved).  Every block folds the mapping's 2 x 32 maxima itself and
// comes to the same decision.  (All lanes of a warp call.)
// (One warp per block reads them: all blocks read the same two lines.)
struct Decision {
  int rebuild;
  int too_wide;
  int dead;  // a grid barrier gave up earlier: the block must leave
  float ext;
};
__device__ __forceinline__ Decision decide_rebuild(const Sys& s, Ctrl* c, int set, int force) {
  static_assert(kExtSlots == 32, "one slot per lane");
  __shared__ Decision sd;
  if (threadIdx.x < 32) {
    const unsigned me = __reduce_max_sync(0xffffffffu, __ldcg(&c->ext_slot[set][0][threadIdx.x]));
    const unsigned md2 = __reduce_max_sync(0xffffffffu, __ldcg(&c->ext_slot[set][1][threadIdx.x]));
    const int host = __ldcg(&c->force_rebuild), dead = __ldcg(&c->dead);
    if (threadIdx.x == 0) {
      sd.ext = sqrtf(__uint_as_float(me));
      const float md = sqrtf(__uint_as_float(md2));
      const double cut = fmax(s.rc_cg, s.rc_at + 2.0 * (double)sd.ext);
      sd.rebuild = force || host || (md > 0.5 * s.skin) || (cut + 2.0 * md > s.r_list);
      sd.too_wide = cut > s.r_list;
      sd.dead = dead;
    }
  }
  __syncthreads();
  const Decision d = sd;
  __syncthreads();  // before the next decision overwrites it
  return d;
}

// ---- block-wide sums and scans of 64-bit pairs (two 32-bit counts side by side) ------------

__device__ __forceinline__ unsigned long long warp_incl_u64(unsigned long long v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// Exclusive scan of v over the block (blockDim a multiple of 32, at most 1024); *total gets
// the block's sum.
__device__ __forceinline__ unsigned long long block_excl_u64(unsigned long long v, unsigned long long* total) {
  __shared__ unsigned long long ws[32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const unsigned long long incl = warp_incl_u64(v);
  __syncthreads();  // ws may still be read by a previous call
  if (lane == 31) ws[w] = incl;
  __syncthreads();
  const unsigned long long x = lane < nw ? ws[lane] : 0ull;
  const unsigned long long xi = warp_incl_u64(x);
  *total = __shfl_sync(0xffffffffu, xi, 31);
  return __shfl_sync(0xffffffffu, xi - x, w) + incl - v;
}

// ---- list phases -----------------------------------------------------------------------------

// Stage candidates c0 .. c0 + nc - 1 of a 27-cell neighbourhood into st[0 .. nc): lane c < 27
// holds neighbour cell c's first sorted position `start`, its offset `pre` in the candidate
// list and the inclusive prefix `incl`.  All lanes copy, 32 candidates at a time; a lane finds
// the cell of its candidate k as the number of cells whose inclusive prefix is <= k (binary
// lifting over the monotone prefixes, five shuffles).
__device__ __forceinline__ void stage_window(const Bufs& b, int lane, int incl, int pre, int start, int c0, int nc,
                                             int4* st) {
  for (int k0 = 0; k0 < nc; k0 += 32) {
    const int k = c0 + k0 + lane;
    int lo = 0;
#pragma unroll
    for (int step = 16; step >= 1; step >>= 1) {
      const int probe = lo + step - 1;
      const int v = __shfl_sync(0xffffffffu, incl, probe < 27 ? probe : 26);
      if (probe < 27 && v <= k) lo += step;
    }
    const int c = lo < 27 ? lo : 26;
    const int s0 = __shfl_sync(0xffffffffu, start, c), p0 = __shfl_sync(0xffffffffu, pre, c);
    if (k0 + lane < nc) st[k0 + lane] = b.scom[s0 + (k - p0)];
  }
  __syncwarp();
}

// Stage a whole neighbourhood (at most kMaxCand candidates): lane c copies neighbour cell c's
// members, four at a time in flight.  A quarter of the instructions of stage_window at the
// tetrahedral fluid's 2.5 molecules a cell; cells of many molecules are for stage_window.
__device__ __forceinline__ void stage_cells(const Bufs& b, int pre, int start, int cnt, int4* st) {
  for (int k = 0; __any_sync(0xffffffffu, k < cnt); k += 4) {
    int4 v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (k + e < cnt) v[e] = b.scom[start + k + e];
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (k + e < cnt) st[pre + k + e] = v[e];
  }
  __syncwarp();
}

// Neighbourhood of a cell: lane c < 27 brings neighbour cell c's slice of the sorted order
// (start, cnt; other lanes cnt = 0).
struct Neighbourhood {
  int start, cnt, incl, pre, total, n_home, home_start, home_pre;
};
__device__ __forceinline__ Neighbourhood neighbourhood(int start, int cnt, int lane) {
  Neighbourhood n;
  n.start = start;
  n.cnt = n.incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, n.incl, o);
    if (lane >= o) n.incl += t;
  }
  n.pre = n.incl - cnt;
  n.total = __shfl_sync(0xffffffffu, n.incl, 31);
  n.n_home = __shfl_sync(0xffffffffu, cnt, 13);  // the home cell is neighbour 13
  n.home_start = __shfl_sync(0xffffffffu, start, 13);
  n.home_pre = __shfl_sync(0xffffffffu, n.pre, 13);
  return n;
}
__device__ __forceinline__ int neighbour_cell(const Sys& s, const Bufs& b, int r, int lane) {
  return r < s.ncell && lane < 27 ? b.nbr_cells[(size_t)r * 27 + lane] : -1;
}
__device__ __forceinline__ void cell_slice(const Bufs& b, int rr, int& start, int& end) {
  start = end = 0;
  if (rr >= 0) {
    start = b.cell_start[rr];
    end = b.cell_start[rr + 1];
  }
}

// Two molecules H0, H1 of a warp's cell against candidate k's centre D (k < n): their neighbours
// appended to the two rows in candidate order, by ballot and popcount.  The molecules' own places
// among the candidates are k0 and k1; `two` is false when there is no second one.
struct PairRows {
  int *row0, *row1;
  int c0, c1;
};
__device__ __forceinline__ void test_two(const Sys& s, const Box& B, int4 H0, int4 H1, int k0, int k1, bool two, int4 D, int k,
                                         bool in, unsigned below, PairRows& P) {
  const float sx = B.fx_scale[0], sy = B.fx_scale[1], sz = B.fx_scale[2];
  const float x0 = (float)(int)((unsigned)H0.x - (unsigned)D.x) * sx;
  const float y0 = (float)(int)((unsigned)H0.y - (unsigned)D.y) * sy;
  const float z0 = (float)(int)((unsigned)H0.z - (unsigned)D.z) * sz;
  const float x1 = (float)(int)((unsigned)H1.x - (unsigned)D.x) * sx;
  const float y1 = (float)(int)((unsigned)H1.y - (unsigned)D.y) * sy;
  const float z1 = (float)(int)((unsigned)H1.z - (unsigned)D.z) * sz;
  const float rl2 = s.f.r_list2, rcl2 = s.f.r_cg_list2;
  const bool hit0 = in && k != k0 && x0 * x0 + y0 * y0 + z0 * z0 < ((H0.w & D.w) < 0 ? rl2 : rcl2);
  const bool hit1 = in && k != k1 && x1 * x1 + y1 * y1 + z1 * z1 < ((H1.w & D.w) < 0 ? rl2 : rcl2);
  const unsigned b0 = __ballot_sync(0xffffffffu, hit0), b1 = __ballot_sync(0xffffffffu, hit1);
  const int p0 = P.c0 + __popc(b0 & below), p1 = P.c1 + __popc(b1 & below);
  if (hit0 && p0 < s.cap) P.row0[p0] = id_of(D.w);
  if (hit1 && two && p1 < s.cap) P.row1[p1] = id_of(D.w);
  P.c0 += __popc(b0);
  P.c1 += __popc(b1);
}
// Record a finished list of c neighbours of molecule H, work item t.
__device__ __forceinline__ void close_list(const Sys& s, const Bufs& b, int4 H, int t, int c) {
  b.nn[t] = c < s.cap ? c : s.cap;
  b.com_ref[id_of(H.w)] = make_int4(H.x, H.y, H.z, 0);
  if (c > s.cap) set_error(b.ctrl, ADRESS_ERR_LIST_OVERFLOW, c);
}

// One warp, one cell: the 27 neighbour cells in the fixed (ox, oy, oz) order, their members
// (centre + id, each cell's already in id order) staged in shared memory once; each molecule
// of the cell then tests all candidates in parallel, two molecules per pass over the
// candidates, and appends its neighbours in candidate order with ballot/popc compaction.
// A cell with more than kMaxCand candidates or 32 molecules goes to the dense-cell list.
__device__ __forceinline__ void list_cell(const Sys& s, const Bufs& b, int r, int start, int cnt, int lane, int n_hr, int4* st) {
  const Box& B = s.nbox > 1 ? b.boxes[b.cell_box[r]] : s.bx;
  const Neighbourhood n = neighbourhood(start, cnt, lane);
  if (n.n_home == 0) return;
  if (n.total > kMaxCand || n.n_home > 32) {
    if (lane == 0) b.dense_cells[atomicAdd(&b.ctrl->n_dense, 1)] = r;
    return;
  }
  __syncwarp();  // the previous cell's candidates are no longer read
  stage_cells(b, n.pre, n.start, n.cnt, st);
  // work items of the home molecules: high-resolution ones first, then coarse-grained, each
  // in sorted order
  const int hw = lane < n.n_home ? st[n.home_pre + lane].w : 0;
  const unsigned hr_mask = __ballot_sync(0xffffffffu, hw < 0);
  const unsigned below = (1u << lane) - 1u;
  const int hr_below = __popc(hr_mask & below), h0 = b.cell_hr[r];
  const int my_item = hw < 0 ? h0 + hr_below : n_hr + (n.home_start - h0) + (lane - hr_below);
  if (lane < n.n_home) {
    const int a = id_of(hw);
    b.items[my_item] = a;
    b.item_of[a] = my_item;
  }
  for (int h = 0; h < n.n_home; h += 2) {
    const bool two = h + 1 < n.n_home;
    const int ka = n.home_pre + h, kb = two ? ka + 1 : ka;
    const int4 H0 = st[ka], H1 = st[kb];
    const int t0 = __shfl_sync(0xffffffffu, my_item, h), t1 = __shfl_sync(0xffffffffu, my_item, h + two);
    PairRows P{b.nbr + (size_t)t0 * s.cap, b.nbr + (size_t)t1 * s.cap, 0, 0};
    for (int k0 = 0; k0 < n.total; k0 += 32) {
      const int k = k0 + lane;
      test_two(s, B, H0, H1, ka, kb, two, st[k < n.total ? k : 0], k, k < n.total, below, P);
    }
    if (lane < 1 + two) close_list(s, b, lane ? H1 : H0, lane ? t1 : t0, lane ? P.c1 : P.c0);
  }
}

// Dense cells: kHomeParts warps per listed cell, each taking batches of 32 of its molecules
// (one per lane).  Candidates are staged in shared memory kMaxCand at a time by all lanes;
// each lane then walks the staged window for its own molecule and appends its neighbours in
// candidate order (the order of the ballot compaction in list_cell): the same lists for any
// density.  Task = (dense cell, part): part j takes the home batches j, j + kHomeParts, ...
// (Two molecules at a time against 32 candidates, as in list_cell, was slower: a build of 64,000
// water-like molecules 544 us against 386.)
constexpr int kHomeParts = 4;
__device__ __forceinline__ void list_dense_part(const Sys& s, const Bufs& b, int r, int part, int lane, int n_hr, int4* st) {
  if (part * 32 >= b.cell_start[r + 1] - b.cell_start[r]) return;
  const Box& B = s.nbox > 1 ? b.boxes[b.cell_box[r]] : s.bx;
  int start, end;
  cell_slice(b, neighbour_cell(s, b, r, lane), start, end);
  const Neighbourhood n = neighbourhood(start, end - start, lane);
  const float rl2 = s.f.r_list2, rcl2 = s.f.r_cg_list2;
  int hr_before = 0;  // high-resolution molecules of the cell before the current batch
  for (int hb = 0; hb < n.n_home; hb += 32) {
    const bool mine = hb + lane < n.n_home;
    const int kh = n.home_start + hb + (mine ? lane : 0);
    const int4 C = b.scom[kh];
    const unsigned hr_mask = __ballot_sync(0xffffffffu, mine && C.w < 0);
    const int hr_below = hr_before + __popc(hr_mask & ((1u << lane) - 1u));
    hr_before += __popc(hr_mask);
    if (((hb >> 5) % kHomeParts) != part) continue;
    const int a = id_of(C.w), h0 = b.cell_hr[r];
    const int tt = C.w < 0 ? h0 + hr_below : n_hr + (n.home_start - h0) + (hb + lane - hr_below);
    if (mine) {
      b.items[tt] = a;
      b.item_of[a] = tt;
    }
    int count = 0;
    int* row = b.nbr + (size_t)(mine ? tt : 0) * s.cap;
    for (int c0 = 0; c0 < n.total; c0 += kMaxCand) {
      const int nc = min(kMaxCand, n.total - c0);
      __syncwarp();  // the previous window is no longer read
      stage_window(b, lane, n.incl, n.pre, n.start, c0, nc, st);
      if (mine) {
#pragma unroll 4
        for (int k = 0; k < nc; ++k) {
          const int4 D = st[k];
          const int m = id_of(D.w);
          const float d0 = (float)(int)((unsigned)C.x - (unsigned)D.x) * B.fx_scale[0];
          const float d1 = (float)(int)((unsigned)C.y - (unsigned)D.y) * B.fx_scale[1];
          const float d2 = (float)(int)((unsigned)C.z - (unsigned)D.z) * B.fx_scale[2];
          if (m != a && d0 * d0 + d1 * d1 + d2 * d2 < ((C.w & D.w) < 0 ? rl2 : rcl2)) {
            if (count < s.cap) row[count] = m;
            ++count;
          }
        }
      }
    }
    if (mine) close_list(s, b, C, tt, count);
  }
}

// High-resolution candidate: decided from the mapping's distance to the region.
__device__ __forceinline__ int hr_candidate(const Sys& s, const Bufs& b, const Box& B, int cur, int a) {
  if (s.lam_uniform_on) return s.lam_uniform > 0.0 ? 1 : 0;
  if (s.fp64) return fabs(b.dxc64[cur][a]) < B.d_hr ? 1 : 0;
  return fabsf(b.molf[cur][a].x) < B.d_hr_f ? 1 : 0;
}

// ---- candidate pairs of the network CG force ---------------------------------------------------

// A molecule deep in the atomistic region at the list build: it keeps lambda = 1 until the
// next build (its centre moves by less than skin/2 before then).  thr = d_at - skin/2 - 1e-3
// of the molecule's box (as float for the FP32 path, whose distances are floats).
template <bool F64>
__device__ __forceinline__ bool deep_atomistic(const Sys& s, const Bufs& b, int cur, int a, double thr, float thr_f) {
  if (s.lam_uniform_on) return s.lam_uniform >= 1.0;
  if constexpr (F64)
    return fabs(b.dxc64[cur][a]) < thr;
  else
    return fabsf(b.molf[cur][a].x) < thr_f;
}

// Candidate pairs of the network force, built with the lists: every
// listed slot (t, q) whose molecule pair a = items[t] < m is within rc_cg + skin and is not
// made of two deep-atomistic molecules.  Until the next build every pair that needs the
// network (weight below 1, centres within rc_cg) is among them: the centres move by less
// than skin/2 each, and a pair of deep-atomistic molecules keeps weight 1.  Records (slot,
// mirror slot, a, m); four lanes per work item, one atomic per warp (the order varies between
// runs, the set does not).  A warp calls with the eight items of its lanes (t may lie past M).
template <bool F64>
__device__ __forceinline__ void net_candidates_of(const Sys& s, const Bufs& b, int cur, int t, int g) {
  const int lane = threadIdx.x & 31;
  const bool live = t < s.M;
  const int a = live ? b.items[t] : 0;
  const int n = live ? b.nn[t] : 0;
  const Box& X = box_of(s, b, a);
  // the threshold once per thread (neighbours share the box of the work item); the FP32
  // path forms it from float parameters (skin = sqrt(r_cg_list2) - rc_cg), off the FP64 pipe
  const double thr = F64 ? X.d_at - 0.5 * s.skin - 1e-3 : 0.0;
  const float thr_f = X.d_at_f - 0.5f * (sqrtf(s.f.r_cg_list2) - sqrtf(s.f.rc_cg2)) - 1e-3f;
  const bool deep_a = live && deep_atomistic<F64>(s, b, cur, a, thr, thr_f);
  const int* row = b.nbr + (size_t)(live ? t : 0) * s.cap;
  auto candidate = [&](int m) -> bool {
    if (m <= a || (deep_a && deep_atomistic<F64>(s, b, cur, m, thr, thr_f))) return false;
    if constexpr (F64) {
      const double4_32a A = b.com64[cur][a], B = b.com64[cur][m];
      return pair_r2(minimg_cmp(A.x - B.x, X.L[0], X.halfL[0]), minimg_cmp(A.y - B.y, X.L[1], X.halfL[1]),
                     minimg_cmp(A.z - B.z, X.L[2], X.halfL[2])) < s.r_cg_list2;
    } else {
      const int4 A = b.com_fx[cur][a], B = b.com_fx[cur][m];
      return pair_r2((float)(int)((unsigned)A.x - (unsigned)B.x) * X.fx_scale[0],
                     (float)(int)((unsigned)A.y - (unsigned)B.y) * X.fx_scale[1],
                     (float)(int)((unsigned)A.z - (unsigned)B.z) * X.fx_scale[2]) < s.f.r_cg_list2;
    }
  };
  unsigned long long sel = 0ull;
  int cnt = 0;
  for (int q = g, j = 0; q < n; q += 4, ++j)
    if (candidate(row[q])) {
      ++cnt;
      if (j < 64) sel |= 1ull << j;
    }
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  int base = 0;
  if (lane == 31 && incl > 0) base = atomicAdd(&b.ctrl->n_netc, incl);
  base = __shfl_sync(0xffffffffu, base, 31);
  long long p = (long long)base + (incl - cnt);
  int qx = g + 256;  // where the search for candidates beyond the mask resumes
  for (int left = cnt; left > 0; --left) {
    int q;
    if (sel) {
      q = g + 4 * (__ffsll((long long)sel) - 1);
      sel &= sel - 1;
    } else {
      for (q = qx; q < n; q += 4)
        if (candidate(row[q])) break;
      if (q >= n) break;  // not reached: the first walk counted this slot
      qx = q + 4;
    }
    if (p >= b.ncap) {  // not reached: at most one record per unordered listed pair
      set_error(b.ctrl, ADRESS_ERR_LIST_OVERFLOW, (int)p);
      break;
    }
    // the mirror slot: where a sits in m's list (the lists are symmetric)
    const int m = row[q], tb = b.item_of[m], nb = b.nn[tb];
    const int* rb = b.nbr + (size_t)tb * s.cap;
    int found = -1;
    for (int qq = 0; qq < nb; ++qq)
      if (rb[qq] == a) {
        found = qq;
        break;
      }
    if (found < 0) set_error(b.ctrl, ADRESS_ERR_STATE, a);
    b.netc[p] = make_int4(t * s.cap + q, found < 0 ? -1 : tb * s.cap + found, a, m);
    ++p;
  }
  __syncwarp();
}

// ---- the build ---------------------------------------------------------------------------------

// The lists of any system, through cells (see the head of this file).  WARPS: warps per block.
template <int WARPS>
__device__ __forceinline__ bool list_cells(const Sys& s, const Bufs& b, int cur, GridBarrier& bar) {
  __shared__ int4 stage[WARPS * kMaxCand];
  Ctrl* c = b.ctrl;
  const int gtid = blockIdx.x * blockDim.x + threadIdx.x, gsize = gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31, gwarp = gtid >> 5, nwarps = gsize >> 5;
  int4* st = stage + (threadIdx.x >> 5) * kMaxCand;
  // cell populations (low word: molecules, high word: high-resolution candidates); the
  // returned count is the molecule's place in its cell's unsorted slice
  for (int a = gtid; a < s.M; a += gsize) {
    const Box& B = box_of(s, b, a);
    const int4 C = b.com_fx[cur][a];
    const int cx = cell_of((unsigned)C.x, B.nc[0]), cy = cell_of((unsigned)C.y, B.nc[1]),
              cz = cell_of((unsigned)C.z, B.nc[2]);
    const int r = b.cell_rank[B.cell0 + (cx * B.nc[1] + cy) * B.nc[2] + cz];
    const int hr = hr_candidate(s, b, B, cur, a);
    const unsigned long long w = atomicAdd(&b.cell_count[r], hr ? 0x100000001ull : 1ull);
    b.mcell[a] = r;
    b.mslot[a] = tag_id((int)(unsigned)w, hr);
  }
  if (!bar.sync()) return false;
  // exclusive scan of the populations: each block sums and then scans its own run of cells
  const int chunk = (s.ncell + gridDim.x - 1) / gridDim.x;
  const int c0 = min(s.ncell, (int)blockIdx.x * chunk), c1 = min(s.ncell, c0 + chunk);
  {
    unsigned long long sum = 0, total;
    for (int r = c0 + threadIdx.x; r < c1; r += blockDim.x) sum += b.cell_count[r];
    block_excl_u64(sum, &total);
    if (threadIdx.x == 0) {
      b.scan_tmp[blockIdx.x] = total;
      if (blockIdx.x == 0) c->n_dense = 0;  // consumed by the previous build
    }
  }
  if (!bar.sync()) return false;
  {
    unsigned long long sum = 0, before, run, total;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += blockDim.x) sum += b.scan_tmp[k];
    block_excl_u64(sum, &before);
    run = before;
    for (int r0 = c0; r0 < c1; r0 += blockDim.x) {
      const int r = r0 + threadIdx.x;
      const unsigned long long v = r < c1 ? b.cell_count[r] : 0ull;
      const unsigned long long ex = run + block_excl_u64(v, &total);
      if (r < c1) {
        b.cell_start[r] = (int)(unsigned)ex;
        b.cell_hr[r] = (int)(unsigned)(ex >> 32);
        b.cell_count[r] = 0ull;  // for the next build
      }
      run += total;
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
      b.cell_start[s.ncell] = (int)(unsigned)run;
      b.cell_hr[s.ncell] = (int)(unsigned)(run >> 32);
    }
  }
  if (!bar.sync()) return false;
  const int n_hr = b.cell_hr[s.ncell];
  if (gtid == 0) {
    c->n_hr = n_hr;
    c->n_cg = s.M - n_hr;
  }
  for (int a = gtid; a < s.M; a += gsize) {
    const int w = b.mslot[a];
    b.fill_tmp[b.cell_start[b.mcell[a]] + id_of(w)] = tag_id(a, w < 0);
  }
  if (!bar.sync()) return false;
  // each molecule's position in its cell is the number of the cell's members with a smaller
  // id (ids are distinct), so every cell's slice is in increasing id
  for (int p = gtid; p < s.M; p += gsize) {
    const int w = b.fill_tmp[p], a = id_of(w), r = b.mcell[a];
    const int ps = b.cell_start[r], pe = b.cell_start[r + 1];
    int rank = 0;
    for (int q = ps; q < pe; ++q) rank += id_of(b.fill_tmp[q]) < a;
    const int4 C = b.com_fx[cur][a];
    b.scom[ps + rank] = make_int4(C.x, C.y, C.z, w);
  }
  if (!bar.sync()) return false;
  {
    // the next cell's slices and the one after's neighbour cells are fetched meanwhile
    int start, end;
    cell_slice(b, neighbour_cell(s, b, gwarp, lane), start, end);
    int rr = neighbour_cell(s, b, gwarp + nwarps, lane);
    for (int r = gwarp; r < s.ncell; r += nwarps) {
      const int cs = start, cn = end - start;
      cell_slice(b, rr, start, end);
      rr = neighbour_cell(s, b, r + 2 * nwarps, lane);
      list_cell(s, b, r, cs, cn, lane, n_hr, st);
    }
  }
  if (!bar.sync()) return false;
  const int n_dense = __ldcg(&c->n_dense);
  // consecutive tasks go to different blocks, so that few tasks reach every SM of the grid, and the
  // parts of a cell are n_dense tasks apart, so that the warps with parts that have nothing to do
  // (a cell of up to 32 molecules fills one of four) are not always the same ones.  Consecutive
  // tasks to consecutive warps, parts side by side: 1000 tetrahedra at density 0.5 218 us a build
  // where it takes 95 now (the whole call), 60,000 294 and 147, 16,000 water-like molecules 415 and 343.
  for (int task = (threadIdx.x >> 5) * gridDim.x + blockIdx.x; task < n_dense * kHomeParts; task += nwarps)
    list_dense_part(s, b, b.dense_cells[task % n_dense], task / n_dense, lane, n_hr, st);
  return true;
}

// All lists of the mapping `cur`, by every block of a cooperative grid; false when a barrier
// gave up (the block must leave).  No barrier after the last phase: the caller orders the
// lists before their readers, and clears Ctrl::force_rebuild after that.
template <int WARPS>
__device__ __forceinline__ bool rebuild_lists(const Sys& s, const Bufs& b, int cur, GridBarrier& bar) {
  if (!list_cells<WARPS>(s, b, cur, bar)) return false;
  if (s.cg_mode && b.netc) {
    const int lane = threadIdx.x & 31;
    const int gwarp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, nwarps = (gridDim.x * blockDim.x) >> 5;
    if (blockIdx.x == 0 && threadIdx.x == 0) b.ctrl->n_netc = 0;
    if (!bar.sync()) return false;
    for (int w = gwarp; w * 8 < s.M; w += nwarps) {
      if (s.fp64) net_candidates_of<true>(s, b, cur, w * 8 + (lane >> 2), lane & 3);
      else net_candidates_of<false>(s, b, cur, w * 8 + (lane >> 2), lane & 3);
    }
  }
  return true;
}

}  // namespace adress
