// mw_persistent.cuh -- persistent engine: one cooperative launch advances
// every box nsteps MD steps, with grid-wide barriers between the phases of
// mw_device.cuh (kick1 | [bin | scan | scatter | copy + neighbour list] |
// force | kick2, then the thermostats: by every block, or in larger batches by
// the last block to arrive).  All blocks are co-resident (cooperative launch), every barrier wait is bounded in wall
// time, and each barrier's counter carries the blocks' error flags, so that
// all blocks take the same decision to stop.  Data written in one phase is
// read by other blocks in a later phase of the same launch, so those reads
// are coherent loads (no ld.global.nc / __ldg anywhere in the phase bodies).
#pragma once

#include "mw_device.cuh"

namespace mw {

constexpr int kPersThreads = kFThreads;
// Co-resident blocks per SM the engine is compiled for (96 registers a
// thread): 7 or 8 (72 or 64 registers) measured slower on the two-box
// 32768-atom workload, and left to itself ptxas may take 128 (4 blocks).
constexpr int kPersBlocksPerSm = 5;

// Phase mark k of step s (block 0, thread 0; the SM clock): 0 step start,
// 1 kick1 done, 2 its barrier passed, 3 rebuild done, 4 force done, 5 its
// barrier passed, 6 kick2 done, 7 the last barrier passed (a launch's last
// step has none: block 0's arrival); on rebuild steps
// also 8 binning, 9 local scan, 10 scan offsets, 11 scatter, 12 copy-back,
// 13 neighbour lists done (each before its barrier).
__device__ __forceinline__ void phase_mark(const Dev& d, int s, int k) {
  if (d.marks && s < d.marks_cap && blockIdx.x == 0 && threadIdx.x == 0) d.marks[s * kPhaseMarks + k] = clock64();
}
constexpr unsigned long long kBarrierTimeoutNs = 2000000000ull;  // default wait limit, 2 s (mw_set_wait_limit)

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier.  Two 64-bit counters (Dev::bar, on lines of their own, zero
// at launch) serve the barriers in turn.  A block arrives with one atomic add
// on the barrier's counter (+ 2^32 when one of its threads has set the status
// since the launch began) and then reads that counter until every block's
// arrival is in it.  A counter gets its next arrivals only after every block
// has passed the other's barrier, so all blocks read the same final value,
// and its upper half is a status that all of them agree on: no last arrival
// has to publish a snapshot and open the barrier.  Barrier-only loops: 2.15 ->
// 1.12 us with 128 blocks, 2.77 -> 1.53 us with 760 (one counter, whose last
// arrival wrote a generation that the others read); arrivals without the
// returned value took 2.6 us with 760, block clusters with one arrival each
// 3.3, a polling pause of 0 to 100 ns the same.
//
// Memory order (PTX memory model, gpu scope, no fences): __syncthreads orders
// every thread's writes of the phase before thread 0's arrival, an acq_rel
// add; the waiters' acquire loads of the counter read the end of one chain of
// adds, hence synchronise with every arrival; the closing __syncthreads hands
// that order to the rest of each block.
//
// Waits are bounded by limit_ns of wall time (0: given up at once); a block
// that gives up sets ST_TIMEOUT and leaves, and so do the others in time.
constexpr int kBarStride = 16;  // 128 bytes
constexpr int kBarPrior = 1;    // beside the first counter: non-zero if the work before this launch met an error
struct GridBar {  // per block, in shared memory
  unsigned long long limit_ns;
  unsigned passed;     // barriers passed in this launch
  unsigned target[2];  // the counters' lower halves once the next barrier on each is complete, less one block each
  int stop, last;
};

__device__ __forceinline__ unsigned long long bar_add(unsigned long long* p, unsigned long long v) {
  unsigned long long old;
  asm volatile("atom.acq_rel.gpu.global.add.u64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v) : "memory");
  return old + v;
}
__device__ __forceinline__ unsigned long long bar_read(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void grid_bar_init(GridBar& B, unsigned long long limit_ns) {
  if (threadIdx.x == 0) {
    B.limit_ns = limit_ns;
    B.passed = B.target[0] = B.target[1] = 0u;
    block_error() = 0;
  }
  __syncthreads();
}

__device__ __forceinline__ unsigned long long* bar_counter(const Dev& d, const GridBar& B) {
  return d.bar + (B.passed & 1u) * kBarStride;
}

// Thread 0: this block's arrival; the counter's value after it.
__device__ __forceinline__ unsigned long long bar_arrival(const Dev& d, const GridBar& B) {
  return bar_add(bar_counter(d, B), 1ull + (block_error() ? 1ull << 32 : 0ull));
}

// Thread 0: wait until the lower half of the counter is n arrivals past its
// last barrier; v is a value read already.  Returns the number of blocks with
// an error, or -1 if this block gave up waiting; non-zero stops.
__device__ __forceinline__ int bar_complete(const Dev& d, GridBar& B, unsigned n, unsigned long long v) {
  const unsigned long long* c = bar_counter(d, B);
  const unsigned want = B.target[B.passed & 1u] + n;
  B.target[B.passed & 1u] = want;
  if ((unsigned)v != want) {
    const unsigned long long t0 = globaltimer_ns(), limit = B.limit_ns;
    while ((unsigned)(v = bar_read(c)) != want) {
      if (globaltimer_ns() - t0 >= limit) {
        set_status(d.g, ST_TIMEOUT);
        return -1;
      }
    }
  }
  B.passed += 1u;
  return (int)(v >> 32);
}

__device__ int grid_barrier(const Dev& d, GridBar& B) {
  __syncthreads();
  if (threadIdx.x == 0) B.stop = bar_complete(d, B, gridDim.x, bar_arrival(d, B));
  __syncthreads();
  return B.stop;
}

// Grid barrier whose last arriving block runs fn() (all its threads) and then
// completes the count with one add more, so that work that needs every block's
// results and that every block needs next costs no barrier of its own (fn's
// threads see the other blocks' writes through thread 0's acquire and the
// __syncthreads after it).
template <class Fn>
__device__ int grid_barrier_last(const Dev& d, GridBar& B, Fn fn) {
  __syncthreads();
  unsigned long long v = 0;
  if (threadIdx.x == 0) {
    v = bar_arrival(d, B);
    B.last = (unsigned)v == B.target[B.passed & 1u] + gridDim.x;
  }
  __syncthreads();
  if (B.last) {
    fn();
    __syncthreads();
    if (threadIdx.x == 0) v = bar_arrival(d, B);
  }
  if (threadIdx.x == 0) B.stop = bar_complete(d, B, gridDim.x + 1u, v);
  __syncthreads();
  return B.stop;
}

// The end of a launch: the last block to arrive runs fn(); the others return
// without waiting (no wait, so no limit).  The launch's end publishes fn's
// writes to whatever runs next on the stream.
template <class Fn>
__device__ void end_arrive_last(const Dev& d, GridBar& B, Fn fn) {
  __syncthreads();
  if (threadIdx.x == 0) B.last = (unsigned)bar_arrival(d, B) == B.target[B.passed & 1u] + gridDim.x;
  __syncthreads();
  if (B.last) fn();
}

// Two-level exclusive scan of the cell counts over the grid: each block scans
// a contiguous chunk of cells (local prefix + chunk total), then adds the
// totals of the chunks before it.
__device__ void scan_chunk_local(const Dev& d) {
  __shared__ int wsum[kPersThreads / 32];
  __shared__ int carry;
  const int per = (d.ncell + gridDim.x - 1) / gridDim.x;
  const int c0 = blockIdx.x * per, c1 = min(d.ncell, c0 + per);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = c0; base < c1; base += kPersThreads) {
    const int c = base + threadIdx.x;
    const int v = (c < c1) ? d.cell_cnt[c] : 0;
    int incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += t;
    }
    if (lane == 31) wsum[wid] = incl;
    __syncthreads();
    int before = carry;
    for (int w = 0; w < wid; ++w) before += wsum[w];
    if (c < c1) d.cell_start[c] = before + incl - v;
    __syncthreads();
    if (threadIdx.x == 0) {
      int tot = 0;
      for (int w = 0; w < kPersThreads / 32; ++w) tot += wsum[w];
      carry += tot;
    }
    __syncthreads();
  }
  if (threadIdx.x == 0 && blockIdx.x < d.chunk_cap) d.chunk[blockIdx.x] = carry;
}

__device__ void scan_chunk_offsets(const Dev& d) {
  __shared__ int red[kPersThreads / 32];
  const int per = (d.ncell + gridDim.x - 1) / gridDim.x;
  const int c0 = blockIdx.x * per, c1 = min(d.ncell, c0 + per);
  int part = 0;
  for (int b = threadIdx.x; b < (int)blockIdx.x; b += kPersThreads) part += d.chunk[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_down_sync(kFull, part, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = part;
  __syncthreads();
  int off = 0;
  for (int w = 0; w < kPersThreads / 32; ++w) off += red[w];
  for (int c = c0 + threadIdx.x; c < c1; c += kPersThreads) {
    d.cell_start[c] += off;
    d.cell_cnt[c] = 0;
  }
  if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) d.cell_start[d.ncell] = off + d.chunk[blockIdx.x];
  __syncthreads();
}

// The scan by every block for itself, into shared memory, for grids whose cell
// offsets fit there (at most kScanShared cells): no barrier between the counts
// and the scatter, where the two-level scan has two of 3 us each.  Block b
// also writes its share of the global offsets, for the list build after the
// next barrier.  The counts are read with L2 loads and cleared after it.
constexpr int kScanShared = (int)(sizeof(LegTable) / sizeof(int));
__device__ void scan_shared(const Dev& d, int* start) {
  __shared__ int wsum[kPersThreads / 32];
  const int tid = (int)threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int c = tid; c < d.ncell; c += kPersThreads) start[c] = __ldcg(d.cell_cnt + c);
  __syncthreads();
  const int per = (d.ncell + kPersThreads - 1) / kPersThreads | 1;  // odd: threads on different banks
  const int c0 = min(d.ncell, tid * per), c1 = min(d.ncell, c0 + per);
  int sum = 0;
  for (int c = c0; c < c1; ++c) sum += start[c];
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) wsum[wid] = incl;
  __syncthreads();
  int run = incl - sum;
  for (int w = 0; w < wid; ++w) run += wsum[w];
  for (int c = c0; c < c1; ++c) {
    const int n = start[c];
    start[c] = run;
    run += n;
  }
  __syncthreads();
  const int share = (d.ncell + (int)gridDim.x - 1) / (int)gridDim.x, s0 = (int)blockIdx.x * share;
  for (int c = s0 + tid; c < min(d.ncell, s0 + share); c += kPersThreads) d.cell_start[c] = start[c];
  if (blockIdx.x == 0 && tid == 0) d.cell_start[d.ncell] = d.N;
}

// The same two halves as separate kernels, for the per-phase engines (the
// graph's rebuild body and the host-launched rebuilds): a grid of blocks in
// place of the single block of k_scan, whose one-block pass over every cell
// took tens of microseconds at 10^5 cells.  Grid size <= chunk_cap.
__global__ void __launch_bounds__(kPersThreads) k_scan_local(Dev d) {
  if (!d.g->any_rebuild || d.g->status) return;
  scan_chunk_local(d);
}
__global__ void __launch_bounds__(kPersThreads) k_scan_offsets(Dev d) {
  if (!d.g->any_rebuild || d.g->status) return;
  scan_chunk_offsets(d);
}

// Up to this many boxes (of constant volume), every block evaluates their
// thermostats for itself from its own copies of their state, as the cluster
// form does, instead of waiting for the last block to arrive to do it (4096
// atoms: 17.5 -> 15.7 us a step, 2 x 32768: 42.6 -> 40.7).  One thread per box and a copy in each block's shared memory
// bound the number; larger batches have less to gain per step.
constexpr int kOwnBoxes = 8;

template <bool kCount, bool kNpt = false>
__global__ void __launch_bounds__(kPersThreads, kPersBlocksPerSm) k_persistent(const __grid_constant__ Dev d, const __grid_constant__ FParams P, int nsteps,
                                                                                        unsigned long long wait_ns) {
  __shared__ LegTable T;
  __shared__ GridBar B;
  __shared__ Box s_box[kNpt ? 1 : kOwnBoxes];
  __shared__ BoxState s_bst[kNpt ? 1 : kOwnBoxes];
  Global* g = d.g;
  if (d.bar[kBarPrior]) return;
  const bool own = !kNpt && d.nbox <= kOwnBoxes;
  if (own && (int)threadIdx.x < d.nbox) {
    s_box[threadIdx.x] = d.box[threadIdx.x];
    s_bst[threadIdx.x] = d.bst[threadIdx.x];
  }
  const Box* const boxes = own ? s_box : d.box;
  const BoxState* const states = own ? s_bst : d.bst;
  grid_bar_init(B, wait_ns);
  const Integ I = *d.integ;
  const unsigned long long step0 = g->step;
  int pend = g->pend;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  const int nth = gridDim.x * blockDim.x;
  const int gw = tid >> 5, nwarps = nth >> 5;
  const int nblk = (d.N + kFAtoms - 1) / kFAtoms;
  // Without a thermostat nothing of the next step needs the kinetic energy, so
  // a step between the launch's first (which leaves sig = 0) and its last ends
  // at the barrier after its forces: no kick2 phase, no tail, one barrier less
  // (200 steps of 4096 / 32768 / 97336 atoms: 20.7 -> 16.3, 33.4 -> 28.4,
  // 54.0 -> 48.5 us a step).
  bool quiet = false;
  for (int s = 0; s < nsteps; ++s) {
    const unsigned long long step = step0 + (unsigned long long)s;
    const int par = (int)(step & 1ull);
    phase_mark(d, s, 0);
    // a1 + a7 first half, a8 displacement check
    if (quiet && tid == 0) g->step = step;  // (the step before left that, and its NaN check, to this one)
    for (int i = tid; i < d.N; i += nth) kick1_atom<kNpt>(d, I, i, par, pend, boxes, states, quiet);
    pend = 1;
    phase_mark(d, s, 1);
    if constexpr (kNpt) {  // the new edges once every block has drifted with the old
      if (grid_barrier_last(d, B, [&] {
            for (int b = threadIdx.x; b < d.nbox; b += blockDim.x) npt_commit_box(d, b);
          }))
        return;
    } else {
      if (grid_barrier(d, B)) return;
    }
    phase_mark(d, s, 2);
    // a2 + a3: cell binning and neighbour list, when due (flag is stable until kick2)
    const bool listed = *(volatile int*)&g->any_rebuild != 0;
    if (listed) {
      if (tid == 0) g->max_count = 0;
      for (int i = tid; i < d.N; i += nth) bin_item(d, i);
      phase_mark(d, s, 8);
      if (grid_barrier(d, B)) return;
      const bool one = d.ncell <= kScanShared;
      int* const start = one ? reinterpret_cast<int*>(&T) : d.cell_start;
      if (one) {
        scan_shared(d, start);
        phase_mark(d, s, 9);
        phase_mark(d, s, 10);
      } else {
        scan_chunk_local(d);
        phase_mark(d, s, 9);
        if (grid_barrier(d, B)) return;
        scan_chunk_offsets(d);
        phase_mark(d, s, 10);
        if (grid_barrier(d, B)) return;
      }
      for (int i = tid; i < d.N; i += nth) scatter_item(d, i, start);
      phase_mark(d, s, 11);
      if (grid_barrier(d, B)) return;
      for (int i = tid; i < d.N; i += nth) copyback_item(d, i);
      if (one)
        for (int c = tid; c < d.ncell; c += nth) d.cell_cnt[c] = 0;
      phase_mark(d, s, 12);
      {  // the warp's candidate staging slice aliases the leg table (idle until the force phase)
        static_assert(sizeof(LegTable) >= (kPersThreads / 32) * kNSlice * sizeof(float4), "staging slices");
        float4* stg = reinterpret_cast<float4*>(&T) + (threadIdx.x >> 5) * kNSlice;
        for (int c = gw; c < d.ncell; c += nwarps) neigh_cell_warp(d, stg, c, P.rl2);
      }
      phase_mark(d, s, 13);
      if (tid == 0) g->rebuild_steps += 1;
      if (grid_barrier(d, B)) return;
    }
    phase_mark(d, s, 3);
    // a4 - a6: fused two- + three-body force, energy, virial
    if (tid == 0) g->wpar = par;
    for (int blk = blockIdx.x; blk < nblk; blk += gridDim.x) force_block<kCount>(d, P, T, blk, par);
    quiet = !kNpt && I.kind == TH_NVE && s > 0 && s < nsteps - 1;
    if (listed && blockIdx.x == 0) {  // the rebuild is consumed: every block has read the flag
      for (int k = threadIdx.x; k < d.nbox; k += blockDim.x) {
        if (box_flagged(d, k)) box_built(d, k);
        d.bst[k].rebuild = 0;
      }
      if (threadIdx.x == 0) g->any_rebuild = 0;
    }
    phase_mark(d, s, 4);
    if (grid_barrier(d, B)) return;
    phase_mark(d, s, 5);
    if (quiet) {
      phase_mark(d, s, 6);
      phase_mark(d, s, 7);
      continue;
    }
    // a7 second half: kinetic energy of v + a per box
    for (int i0 = blockIdx.x * kPersThreads; i0 < d.N; i0 += nth) {  // block-uniform
      float ke[1] = {0.f};
      int b = -1;
      ke[0] = kick2_atom(d, I, i0 + (int)threadIdx.x, b);
      box_accumulate<1>(ke, b, [&](int bb) { return &d.bst[bb].ke_acc[par]; });
    }
    phase_mark(d, s, 6);
    // the thermostat halves of every box (end of this step, start of the
    // next): by every block in its own copies, which block 0 (the launch's
    // last step: the block that runs it) writes back, or by the last block to
    // arrive, for the others
    auto tail = [&](bool write) {
      for (int b = threadIdx.x; b < d.nbox; b += blockDim.x) {
        if (!own) {
          end_of_step_box<kNpt>(d, I, b, par);
        } else {
          BoxState& st = s_bst[b];
          end_of_step<false, LdShared>(I, s_box[b], st, __ldcg(&d.bst[b].ke_acc[par]), 0.0);
          if (write) {
            BoxState& out = d.bst[b];
            out.th = st.th;
            out.th_e = st.th_e;
            out.ke_last = st.ke_last;
            out.s_endc = st.s_endc;
            out.sig = st.sig;
          }
        }
      }
      if (write && threadIdx.x == 0) {
        g->pend = 1;
        g->step = step + 1ull;
      }
    };
    if (s == nsteps - 1) {
      // nothing follows in this launch, so the other blocks leave at once and
      // the last one to arrive runs the tail
      phase_mark(d, s, 7);
      end_arrive_last(d, B, [&] { tail(true); });
      return;
    }
    if (own) {
      const int stop = grid_barrier(d, B);
      if (stop < 0) return;
      tail(blockIdx.x == 0);
      if (stop) return;
      __syncthreads();
    } else if (grid_barrier_last(d, B, [&] { tail(true); })) {
      return;
    }
    phase_mark(d, s, 7);
  }
}

}  // namespace mw
