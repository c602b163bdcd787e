// mw_cluster.cuh -- the persistent engine's form for boxes that fit one
// thread-block cluster: one cluster per box runs that box's steps on its own.
//
// The steps of a small box are a chain of short phases (kick1 | list | force |
// kick2 + thermostat), each a microsecond or so of work, and a grid-wide
// barrier through L2 costs 1.1 to 1.6 us beside the wait for the slowest
// block.  Boxes of a batch do not depend on one another, so nothing
// needs a grid-wide barrier: the hardware cluster barrier orders a box's
// phases, small sums and flags travel through distributed shared memory, the
// thermostat is evaluated by every block for itself, and a box rebuilds its
// list when it has to, whatever the others do.  Clusters of a large batch are
// scheduled as SMs come free, the largest boxes first.
//
// Atoms: one per thread (n <= cluster blocks x threads), a contiguous range
// per block, so an atom's velocity, force and position stay in registers
// between kick2 and the next kick1.  Every decision (rebuild, stop) is taken
// from flags that all blocks of the cluster read alike after a barrier, so
// all of them meet at the same barriers; nothing here spins.
//
// A box that stops (overflow of a row, a grid left behind, an error anywhere)
// stops on its own step: its count of completed steps is kept in prog, and
// mid marks a step whose kick1 is done.  The host mends what can be mended
// and launches again for the rest; the last cluster to finish makes the
// engine's step count that of the slowest box.
#pragma once

#include "mw_device.cuh"

namespace mw {

constexpr int kCluMax = 16;          // blocks per cluster, at most
constexpr int kCluThreads = 512;    // two blocks share an SM (64 registers, 98 KB of leg tables each)
constexpr int kCluRows = kWAtoms * kLMax;  // leg records of a warp
constexpr int kCluWarpBytes = 2 * kCluRows * (int)sizeof(float4);
constexpr int kCluSteps = 1024;      // steps of one launch, at most (bits of rebuild_bits)

struct CluArgs {
  const int* order;       // boxes, largest first
  int* prog;              // per box: steps completed of this run
  int* mid;               // per box: 1 = kick1 of the next step is done
  unsigned* rebuild_bits; // one bit per step of this launch: some box rebuilt
  unsigned* ndone;        // clusters finished (zeroed by the host)
  unsigned long long step0;  // the engine's step count at the start of the run
  int nsteps;             // steps of the run
  int base;               // first step that rebuild_bits counts from
  int cells;              // cell offsets that a block's shared memory holds
};

__device__ __forceinline__ unsigned clu_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned clu_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// All threads of the cluster; release / acquire at cluster scope, so what any
// of them wrote (global, shared or remote shared memory) is seen by all.
__device__ __forceinline__ void clu_sync() {
  asm volatile("barrier.cluster.arrive.release;\n barrier.cluster.wait.acquire;" ::: "memory");
}
// The address of this block's shared variable p in block `rank`.
__device__ __forceinline__ unsigned clu_map(const void* p, unsigned rank) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void clu_st(unsigned a, int v) {
  asm volatile("st.shared::cluster.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void clu_st(unsigned a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}

enum : int { CLU_REBUILD = 1, CLU_STOP = 2, CLU_SEEN = 4 };  // (seen: the engine has a status)

struct CluShared {
  Box bx;               // this box, evolved alike by every block (isobaric runs)
  BoxState bs;
  Integ I;
  double sum[kCluMax][9];              // per block: E2, E3, W[6], KE
  int flag[2][kCluMax];                // per block: CLU_* of an exchange (two buffers in turn: a block may
                                       // write the next exchange's while another still reads this one's)
  float warp[kCluThreads / 32][9];  // per warp: the same sums
  int wsum[kCluThreads / 32];       // scan
  int stop;
};

// Exchange of this block's flags (number ex of the launch): every block's are
// in S.flag[ex & 1] after the next cluster barrier.  Called by all threads,
// which pass their own bits.
__device__ __forceinline__ void clu_flags(CluShared& S, int ex, int bits, unsigned rank, unsigned size) {
  int all = 0;
  if (__syncthreads_or(bits))
    all = (__syncthreads_or(bits & CLU_REBUILD) ? CLU_REBUILD : 0) | (__syncthreads_or(bits & CLU_STOP) ? CLU_STOP : 0) |
          (__syncthreads_or(bits & CLU_SEEN) ? CLU_SEEN : 0);
  if (threadIdx.x < size) clu_st(clu_map(&S.flag[ex & 1][rank], threadIdx.x), all);
}
__device__ __forceinline__ int clu_flags_all(const CluShared& S, int ex, unsigned size) {
  const int lane = threadIdx.x & 31;
  return (int)__reduce_or_sync(kFull, lane < (int)size ? (unsigned)S.flag[ex & 1][lane] : 0u);
}

// The sum over blocks of item k (FP64, the same order in every block).
__device__ __forceinline__ double clu_total(const CluShared& S, unsigned size, int k) {
  const int lane = threadIdx.x & 31;
  double v = lane < (int)size ? S.sum[lane][k] : 0.0;
#pragma unroll
  for (int o = kCluMax / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// Cell binning and neighbour rows of the box, by its cluster.  i: this
// thread's atom (on: there is one); start: shared memory for the box's cell
// offsets, then the warps' candidate staging.  Returns whether a row overflowed
// (this warp's part).
__device__ __forceinline__ bool clu_rebuild(const Dev& d, CluShared& S, float4* tab, int i, bool on, unsigned rank, unsigned size,
                                            int cells, float rl2) {
  const Box& bx = S.bx;
  constexpr int T = kCluThreads;
  const int tid = (int)threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const bool sort = sorts(S.bs);  // (as scatter_item and copyback_item)
  unsigned box = 0u;
  int c = 0, r = 0;
  if (on) {
    const uint4 q = d.q[i];
    box = q.w;
    c = cell_of(q, bx);
    r = atomicAdd(d.cell_cnt + c, 1);
  }
  clu_sync();
  // every block scans all the counts of the box for itself (a sparse box with
  // more cells than a block's shared memory holds reads the offsets back from
  // global memory, after one more barrier)
  int* start = reinterpret_cast<int*>(tab);
  const int ncb = bx.nc[0] * bx.nc[1] * bx.nc[2];
  const bool fits = ncb <= cells;
  const int per = (ncb + T - 1) / T;
  const int c0 = min(ncb, tid * per), c1 = min(ncb, c0 + per);
  int sum = 0;
  for (int k = c0; k < c1; ++k) sum += __ldcg(d.cell_cnt + bx.cell_off + k);
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) S.wsum[wid] = incl;
  __syncthreads();
  int run = bx.off + incl - sum;
  for (int w = 0; w < wid; ++w) run += S.wsum[w];
  for (int k = c0; k < c1; ++k) {
    if (fits) start[k] = run;
    if (k % (int)size == (int)rank) d.cell_start[bx.cell_off + k] = run;
    run += __ldcg(d.cell_cnt + bx.cell_off + k);
  }
  // the end of the last cell is the next box's first atom, whoever writes it
  if (rank == 0 && tid == 0) d.cell_start[bx.cell_off + ncb] = bx.off + bx.n;
  if (fits) __syncthreads();
  else clu_sync();
  if (on) {
    const int p = (fits ? start[c - bx.cell_off] : __ldcg(d.cell_start + c)) + r;
    uint4 q = d.q[i];
    if (p < bx.off || p >= bx.off + bx.n) {  // counts not cleared after an interrupted build: report, write nothing
      set_status(d.g, ST_CELLS);
      d.g->err_index = i;
    } else {
      if (sort) {
        d.tx[p] = d.x[i]; d.ty[p] = d.y[i]; d.tz[p] = d.z[i];
        d.tvx[p] = d.vx[i]; d.tvy[p] = d.vy[i]; d.tvz[p] = d.vz[i];
        d.tid[p] = d.id[i];
        d.timg[p] = d.img[i];
        q.w = (unsigned)p;
      } else {
        d.qb[i] = q;
        q.w = (unsigned)i;
      }
      d.tq[p] = q;
    }
  }
  clu_sync();
  if (on && sort) {
    d.x[i] = d.tx[i]; d.y[i] = d.ty[i]; d.z[i] = d.tz[i];
    d.vx[i] = d.tvx[i]; d.vy[i] = d.tvy[i]; d.vz[i] = d.tvz[i];
    d.id[i] = d.tid[i];
    d.img[i] = d.timg[i];
    uint4 q = d.tq[i];
    q.w = box;
    d.q[i] = q;
    d.qb[i] = q;
  }
  for (int k = (int)rank * T + tid; k < ncb; k += (int)size * T) d.cell_cnt[bx.cell_off + k] = 0;
  bool over = false;
  float4* stg = tab + wid * (kCluWarpBytes / (int)sizeof(float4));
  static_assert(kCluWarpBytes >= kNSlice * (int)sizeof(float4), "staging slices");
  const int nw = (T >> 5) * (int)size;
  const int parts = max(1, min(4, nw / ncb));
  for (int k = wid * (int)size + (int)rank; k < ncb * parts; k += nw)
    over |= neigh_cell(d, bx, stg, bx.cell_off + k / parts, rl2, k % parts, parts);
  return over;
}

template <bool kNpt>
__global__ void __launch_bounds__(kCluThreads, 2) k_cluster(const __grid_constant__ Dev d, const __grid_constant__ FParams P,
                                                               const __grid_constant__ CluArgs A) {
  extern __shared__ __align__(16) float4 clu_tab[];
  __shared__ CluShared S;
  const unsigned rank = clu_rank(), size = clu_size();
  constexpr int nwarp = kCluThreads / 32;
  const int tid = (int)threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int b = A.order[blockIdx.x / size];
  for (int k = tid; k < (int)(sizeof(Box) / 4); k += kCluThreads)
    reinterpret_cast<int*>(&S.bx)[k] = reinterpret_cast<const int*>(d.box + b)[k];
  for (int k = tid; k < (int)(sizeof(BoxState) / 4); k += kCluThreads)
    reinterpret_cast<int*>(&S.bs)[k] = reinterpret_cast<const int*>(d.bst + b)[k];
  for (int k = tid; k < (int)(sizeof(Integ) / 4); k += kCluThreads)
    reinterpret_cast<int*>(&S.I)[k] = reinterpret_cast<const int*>(d.integ)[k];
  int s = A.prog[b];
  bool mid = A.mid[b] != 0;
  int pend = s > 0 ? 1 : d.g->pend;
  // Every block of the cluster has started and has its copies: from here on
  // others store into its shared memory, and rank 0 writes the box's globals.
  clu_sync();
  const Integ& I = S.I;
  const int off = S.bx.off, n = S.bx.n;
  const int per = (n + (int)size - 1) / (int)size;  // atoms of a block
  const int i = off + (int)rank * per + tid;
  const bool on = tid < per && i < off + n;
  const int ngrp = (n + kWAtoms - 1) / kWAtoms, gper = (ngrp + (int)size - 1) / (int)size;
  float4* const ue = clu_tab + wid * (kCluWarpBytes / (int)sizeof(float4));
  float4* const aux = ue + kCluRows;
  Kick1In in{};
  if (on && !mid) in = kick1_load(d, i);
  bool stopped = false;
  int late = 0;  // flag bits that a quiet step leaves for the next exchange
  int ex = 0;  // flag exchanges so far
  if constexpr (kNpt) {
    // a grid left behind whose report another box's status covered
    bool grid = false;
    for (int k = 0; k < 3; ++k) {
      const double Ln = mid ? S.bx.L[k] : S.bx.Ln[k];
      const int nc = S.bx.nc[k];
      grid |= Ln < 2.0 * I.rlist || (nc >= 4 && Ln < nc * (double)I.rlist) || Ln >= (nc + 1) * kCellGrow * I.rlist;
    }
    if (grid && s < A.nsteps) {
      if (tid == 0) set_status(d.g, ST_GRID);
      stopped = true;
    }
  }
  while (!stopped && s < A.nsteps) {
    const int par = (int)((A.step0 + (unsigned long long)s) & 1ull);
    int bits = (S.bs.rebuild ? CLU_REBUILD : 0) | late;
    late = 0;
    if (!mid) {
      // a1, a7 first half, a8
      if (on) {
        bool moved, lost;
        kick1_apply<kNpt>(d, I, S.bx, S.bs.sig, i, b, pend, in, moved, lost);
        if (lost) {
          set_status(d.g, ST_LOST);
          d.g->err_index = i;
        }
        bits |= (moved ? CLU_REBUILD : 0) | (lost ? CLU_STOP : 0);
      }
    }
    // centres over the staged legs add their energies to the global sums
    if (rank == 0 && tid < 8) d.bst[b].ew[par][tid] = 0.0;
    if (rank == 0 && kNpt && tid < 3)  // (they read the edges there too)
      const_cast<Box*>(d.box)[b].Lq[tid] = mid ? S.bx.Lq[tid] : (float)(S.bx.Ln[tid] * 2.3283064365386963e-10);  // 2^-32
    clu_flags(S, ++ex, bits, rank, size);
    clu_sync();
    const int fl = clu_flags_all(S, ex, size);
    if (fl & CLU_STOP) break;
    if constexpr (kNpt) {
      if (!mid && tid == 0) npt_commit<LdShared>(S.bx);
      __syncthreads();
    }
    mid = true;
    // a2, a3
    if (fl & CLU_REBUILD) {
      // (max_count is not reset in this engine: it covers every row of the run)
      const bool over = clu_rebuild(d, S, clu_tab, i, on, rank, size, A.cells, P.rl2);
      if (over && lane == 0) set_status(d.g, ST_OVERFLOW);
      clu_flags(S, ++ex, over ? CLU_STOP : 0, rank, size);
      clu_sync();
      if (clu_flags_all(S, ex, size) & CLU_STOP) {  // the rows are grown and built again before this step goes on
        if (tid == 0) S.bs.rebuild = 1;
        __syncthreads();
        break;
      }
      if (tid == 0) {
        S.bs.rebuild = 0;
        S.bs.sorted = 1;
        S.bs.rebuilds += 1;
        S.bs.Lb = S.bx.L[0];
        if (rank == 0) atomicOr(A.rebuild_bits + ((s - A.base) >> 5), 1u << ((s - A.base) & 31));
      }
    }
    // a4 - a6
    float acc[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    for (int g = wid; g < gper; g += nwarp) {
      const int ic = off + ((int)rank * gper + g) * kWAtoms + lane / kG;
      bool over = false;
      force_group<false, 0, kG, 0>(d, P, ue, aux, ic, ic < off + n && (int)rank * gper + g < ngrp, acc, over);
      if (over) force_overflow_item<false>(d, P, ic, par);
      __syncwarp();
    }
    clu_sync();
    // Without a thermostat nothing of the next step needs the kinetic energy,
    // so a step between the run's first (which leaves sig = 0) and its last
    // ends here: no sums, no barrier, no end_of_step.  Its NaN check and a
    // status set elsewhere go with the next exchange.  50 steps of 512 atoms:
    // 730 -> 668 us.
    const bool quiet = !kNpt && I.kind == TH_NVE && s > 0 && s < A.nsteps - 1 && !(fl & CLU_SEEN);
    if (quiet) {
      if (tid == 0 && *(volatile int*)&d.g->status) late = CLU_SEEN;
      if (on) {
        in = kick1_load(d, i);
        if (!(kick2_energy(I, in.F, in.v) < 1e30f)) {
          set_status_nan(d.g);
          d.g->err_index = i;
          late |= CLU_STOP;
        }
      }
      mid = false;
      pend = 1;
      ++s;
      continue;
    }
    // a7 second half: the kinetic energy of v + a, and the next kick1's inputs
    float ke = 0.f;
    if (on) {
      in = kick1_load(d, i);
      ke = kick2_energy(I, in.F, in.v);
    }
    const bool nan = !(ke < 1e30f);
    if (nan) {
      set_status(d.g, ST_NAN);
      d.g->err_index = i;
    }
    const bool sums = kNpt || s == A.nsteps - 1;  // energies and virial are wanted
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ke += __shfl_xor_sync(kFull, ke, o);
    if (sums) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) acc[k] += __shfl_xor_sync(kFull, acc[k], o);
        if (lane == 0) S.warp[wid][k] = acc[k];
      }
    }
    if (lane == 0) S.warp[wid][8] = ke;
    const int st0 = tid == 0 ? *(volatile int*)&d.g->status : 0;  // an error of another box, or of the overflow path
    clu_flags(S, ++ex, (nan || st0) ? CLU_STOP : 0, rank, size);
    // this block's sums to every block: FP32 within a warp, FP64 above
    if (wid == 0) {
      double v = lane < nwarp ? (double)S.warp[lane][8] : 0.0;
#pragma unroll
      for (int o = nwarp / 2; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
      static_assert(kCluMax <= nwarp, "every lane that stores the sum has it");
      if (lane < (int)size) clu_st(clu_map(&S.sum[rank][8], lane), v);
    }
    if (sums) {
      for (int k = wid; k < 8; k += nwarp) {
        double v = lane < nwarp ? (double)S.warp[lane][k] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
        if (lane < (int)size) clu_st(clu_map(&S.sum[rank][k], lane), v);
      }
    }
    double ovt = 0.0;  // the overflow path's trace of the virial
    if (kNpt && tid == 0) ovt = __ldcg(&d.bst[b].ew[par][2]) + __ldcg(&d.bst[b].ew[par][3]) + __ldcg(&d.bst[b].ew[par][4]);
    clu_sync();
    // the thermostat halves of the step boundary, by every block for itself
    int geo = 0;
    if (wid == 0) {
      const double ke0 = clu_total(S, size, 8);
      double trw = 0.0;
      if constexpr (kNpt) trw = clu_total(S, size, 2) + clu_total(S, size, 3) + clu_total(S, size, 4);
      if (lane == 0) geo = end_of_step<kNpt, LdShared>(I, S.bx, S.bs, ke0, trw + ovt);
      if (kNpt && lane == 0 && (geo & 2)) set_status(d.g, ST_GRID);
      if (lane == 0) S.stop = geo & 2;
    }
    mid = false;
    pend = 1;
    ++s;
    const int stop = clu_flags_all(S, ex, size) & CLU_STOP;
    __syncthreads();
    stopped = stop || S.stop;
  }
  // the box's state back to global memory (rank 0), then the engine's by the
  // last cluster to finish
  if (rank != 0) return;
  const int spar = (int)((A.step0 + (unsigned long long)s - 1ull) & 1ull);
  if (s == A.nsteps && s > A.prog[b] && wid == 0) {  // the sums of the run's last step
    for (int k = 0; k < 8; ++k) {
      const double v = clu_total(S, size, k);
      if (lane == 0) S.bs.ew[spar][k] = v + __ldcg(&d.bst[b].ew[spar][k]);
    }
  }
  __syncthreads();
  for (int k = tid; k < (int)(sizeof(BoxState) / 4); k += kCluThreads)
    reinterpret_cast<int*>(d.bst + b)[k] = reinterpret_cast<const int*>(&S.bs)[k];
  if constexpr (kNpt)
    for (int k = tid; k < (int)(sizeof(Box) / 4); k += kCluThreads)
      reinterpret_cast<int*>(const_cast<Box*>(d.box) + b)[k] = reinterpret_cast<const int*>(&S.bx)[k];
  if (tid == 0) {
    A.prog[b] = s;
    A.mid[b] = mid ? 1 : 0;
  }
  __syncthreads();
  if (tid == 0) S.stop = bar_arrive(A.ndone) == (unsigned)d.nbox;
  __syncthreads();
  if (!S.stop) return;
  int least = A.nsteps, flagged = 0;
  for (int k = tid; k < d.nbox; k += kCluThreads) {
    least = min(least, __ldcg(A.prog + k));
    flagged |= __ldcg(&d.bst[k].rebuild);
  }
  least = __reduce_min_sync(kFull, least);
  if (lane == 0) S.wsum[wid] = least;
  flagged = __syncthreads_or(flagged);
  if (tid == 0) {
    for (int w = 1; w < nwarp; ++w) least = min(least, S.wsum[w]);
    int steps = 0;  // steps of this launch in which some box rebuilt
    for (int k = 0; k < kCluSteps / 32; ++k) steps += __popc(__ldcg(A.rebuild_bits + k));
    d.g->rebuild_steps += steps;
    d.g->any_rebuild = flagged ? 1 : 0;
    d.g->step = A.step0 + (unsigned long long)least;
    if (least > 0) {
      d.g->pend = 1;
      d.g->wpar = (int)((A.step0 + (unsigned long long)least - 1ull) & 1ull);
    }
  }
}

}  // namespace mw
