// The particle kernel of one SLPIC-MCC step, batched over instances and
// species: gather, speed-limited kick and drift (Eqs. slpicEOMx, slpicEOMv,
// betaAbrupt), absorbing electrodes with ion-induced secondary emission
// (Sec. IV), the null-collision test of electrons against the majorant
// probability (Sec. III; one Philox2x32-10 draw keyed by (id, step)),
// in-place compaction of survivors, and the fixed-point deposit of
// w_p = beta w_j (Eq. Ansatz; with an imposed field the deposit is formed
// from the markers when read, and the step deposits nothing).
//
// Work decomposition.  Every (instance, species) segment is a sequence of
// tiles of kTile = 128 marker slots (tile k holds fill[k] markers), and every
// tile belongs to one warp: no block-wide barrier is needed to advance,
// rank, compact and store it.
//   - The CTAs split the tiles of all segments into contiguous ranges of
//     equal weight, so a CTA deposits into few segments, and deal the tiles of
//     their range to their warps in turn; with fewer tiles than warps on the
//     device every SM still gets its share.
//   - A warp's tiles pass through kPushStages shared-memory stages: lane 0
//     starts the bulk asynchronous copy (TMA, cp.async.bulk) of the next tile's
//     block while the warp advances the current one, two neighbouring slots
//     per lane and pass.  One copy per tile: seven (one per field) cost about
//     150 instructions per marker with their addresses, waits and stores, and
//     plain loads into registers, prefetched into L2, left its latency exposed
//     (5 % slower where few instructions hide it).
//   What bounds it: instruction issue under a speed limit (8e6 limited
//   electrons on 4096 cells: 129 us, 416 warp instructions per 32 markers at
//   69 % of the issue rate, DRAM at 2.2 TB/s; with a copy and an address per
//   field and the IEEE roots and quotients 179 us and 546), the memory system
//   without one (6e6 unlimited ions: 48 us with the deposit, 66 before).
//   - Of unlimited ions only the front of the block is copied: cell, offset and
//     v_x, and w_j when the step deposits.  The rare ones that need the other
//     fields (absorbed, or moved by compaction) read them then.
//   - Survivors are deposited into a shared-memory copy of the segment's
//     charge grid (integer atomics); cell, offset and v_x go back to the
//     marker's slot.  Ballots rank survivors and events (ion emissions,
//     electron collision candidates); when a marker left the tile the
//     survivors are stored compacted, in order, with all their fields.
// Collision candidates (the electrons that drew u < P0) are not scattered
// here: their states and final slots are queued per tile as 32-byte records
// and k_collide scatters them all at once, so the long, rare scattering path
// never stalls the stream and reads each candidate with one sector.
// The shared charge grid is added to global memory with integer atomics when
// the CTA moves to another segment (a CTA-wide barrier) or finishes, so the
// deposit is exact and independent of the order of the additions.
#include "device_common.cuh"
#include "slpic_internal.h"
#include "step_ops.cuh"

namespace slpic {

namespace {

struct PushShared {
  unsigned long long s_acc[ACC_COUNT];
};

// Add the CTA's shared charge grid and accumulators of segment seg to global
// memory and clear them (all threads; barriers before and after).
__device__ __forceinline__ void flush_segment(const DeviceRefs& r, int seg,
                                              unsigned long long* s_rho, PushShared& cs,
                                              bool use_smem) {
  const int inst = seg >> 1, sp = seg & 1;
  const InstDev& P = r.inst[inst];
  __syncthreads();
  if (use_smem) {
    const int nn = P.n_cells + 1;
    unsigned long long* g = P.rho_acc[sp];
    for (int k = threadIdx.x; k < nn; k += blockDim.x) {
      const unsigned long long v = s_rho[k];
      if (v) {
        atomicAdd(g + k, v);
        s_rho[k] = 0ull;
      }
    }
  }
  if (threadIdx.x < ACC_COUNT) {
    const unsigned long long v = cs.s_acc[threadIdx.x];
    if (v) {
      atomicAdd(P.acc + threadIdx.x, v);
      cs.s_acc[threadIdx.x] = 0ull;
    }
  }
  __syncthreads();
}

// Segment of tile q (q < n_tiles): the last segment starting at or before q.
__device__ __forceinline__ int segment_of(const DeviceRefs& r, unsigned int q) {
  int lo = 0, hi = r.n_inst * 2 - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (r.seg_start[mid] <= q) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// First tile whose weighted start is at or after `target`.
__device__ __forceinline__ unsigned int first_tile(const DeviceRefs& r, unsigned int target) {
  const int n_seg = r.n_inst * 2;
  if (target >= r.seg_wstart[n_seg]) return r.seg_start[n_seg];
  int lo = 0, hi = n_seg - 1;  // last segment with weighted start <= target
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (r.seg_wstart[mid] <= target) lo = mid;
    else hi = mid - 1;
  }
  const unsigned int w = (lo & 1) ? kWeightIon : kWeightElectron;
  // (a segment's weight begins with the cost of starting it)
  const unsigned int at = target - r.seg_wstart[lo], cost = r.ctrl->seg_cost;
  const unsigned int q = r.seg_start[lo] + (at > cost ? at - cost + w - 1 : 0u) / w;
  return min(q, r.seg_start[lo + 1]);
}

// A lane's two neighbouring slots of one field of a tile, as one access.
static_assert(kPerHalf == 2, "two neighbouring slots per lane and pass");
__device__ __forceinline__ void get_slots(const int32_t* p, int (&v)[2]) {
  const int2 t = *reinterpret_cast<const int2*>(p);
  v[0] = t.x;
  v[1] = t.y;
}
__device__ __forceinline__ void get_slots(const uint32_t* p, uint32_t (&v)[2]) {
  const uint2 t = *reinterpret_cast<const uint2*>(p);
  v[0] = t.x;
  v[1] = t.y;
}
__device__ __forceinline__ void get_slots(const float* p, float (&v)[2]) {
  const float2 t = *reinterpret_cast<const float2*>(p);
  v[0] = t.x;
  v[1] = t.y;
}
__device__ __forceinline__ void get_slots(const double* p, double (&v)[2]) {
  const double2 t = *reinterpret_cast<const double2*>(p);
  v[0] = t.x;
  v[1] = t.y;
}
__device__ __forceinline__ void put_slots(int32_t* p, const int (&v)[2]) {
  *reinterpret_cast<int2*>(p) = make_int2(v[0], v[1]);
}
__device__ __forceinline__ void put_slots(float* p, const float (&v)[2]) {
  *reinterpret_cast<float2*>(p) = make_float2(v[0], v[1]);
}
__device__ __forceinline__ void put_slots(double* p, const double (&v)[2]) {
  *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
}

// Start the bulk copy of a tile's first `bytes` bytes into a stage (lane 0).
__device__ __forceinline__ void load_tile(unsigned char* stage, const unsigned char* tile,
                                          uint32_t bytes, uint64_t* bar) {
  mbar_arrive_expect_tx(bar, bytes);
  bulk_load(stage, tile, bytes, bar);
}

}  // namespace

template <typename R>
__global__ void __launch_bounds__(kPushMaxWarps * 32, 1) k_push(DeviceRefs r) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ uint64_t s_bar[kPushMaxWarps][kPushStages];
  __shared__ PushShared cs;
  const int W = (int)(blockDim.x >> 5);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lanemask_lt = (1u << lane) - 1u;
  constexpr size_t kTB = tile_bytes<R>();
  unsigned char* const stages = smem_raw + (size_t)warp * kPushStages * kTB;
  unsigned long long* const s_rho =
      reinterpret_cast<unsigned long long*>(smem_raw + (size_t)W * kPushStages * kTB);
  uint64_t* const bars = s_bar[warp];

  step_kernel_entry();
  Control* ctrl = r.ctrl;
  if (*((volatile int*)&ctrl->error)) return;
  // this CTA's contiguous range of tiles (equal weight per CTA)
  const unsigned long long wt = ctrl->w_total;
  const unsigned int q0 =
      first_tile(r, (unsigned int)((unsigned long long)blockIdx.x * wt / gridDim.x));
  const unsigned int q1 =
      first_tile(r, (unsigned int)((unsigned long long)(blockIdx.x + 1) * wt / gridDim.x));
  if (q0 >= q1) return;

  for (int k = threadIdx.x; k < r.smem_nodes; k += blockDim.x) s_rho[k] = 0ull;
  if (threadIdx.x < ACC_COUNT) cs.s_acc[threadIdx.x] = 0ull;
  if (lane == 0) {
    for (int s = 0; s < kPushStages; ++s) mbar_init(&bars[s], 1);
    fence_mbar_init();
  }
  __syncthreads();
  // tiles of this warp whose copies were started, and those waited for: tile
  // number i goes through stage i % kPushStages in its round i / kPushStages
  uint32_t started = 0, arrived = 0;
  bool ok = true;  // no wait of this warp has run out

  int seg = segment_of(r, q0);
  for (unsigned int qs = q0; qs < q1; ++seg) {
    const unsigned int seg0 = r.seg_start[seg];
    const unsigned int qe = min(q1, r.seg_start[seg + 1]);
    if (qe <= qs) continue;  // an empty segment
    const uint32_t k_end = qe - seg0;
    uint32_t k = qs - seg0 + (uint32_t)warp;
    qs = qe;
    // ---- the segment's constants ------------------------------------------
    const int inst = seg >> 1, sp = seg & 1;
    const InstDev& P = r.inst[inst];
    const uint32_t cur = r.sstate[seg].cur;
    unsigned char* const buf = P.sp[sp].buf[cur];
    uint32_t* const fill = P.sp[sp].fill[cur];
    const uint32_t step = r.istate[inst].step;
    const StepConsts<R>& K = consts<R>(P);
    const R qmdt = K.qmdt[sp], vlim = K.vlim[sp], dtdx = K.dtdx, wscale = K.wscale;
    const uint32_t cand_thr = K.cand_thr, key2 = P.key2;
    const uint32_t N = (uint32_t)P.n_cells;
    const R* const Enode = node_field<R>(P);
    const bool electrons = sp == kElectron;
    const bool limited = vlim < (R)INFINITY;  // beta = 1 for an unlimited species
    // with an imposed field the deposit is formed from the markers when it is
    // read (k_deposit), so nothing is deposited here
    const bool dep = P.field_mode == 1;
    const bool use_smem = dep && P.n_cells + 1 <= r.smem_nodes;
    // (one generic pointer: with the two address spaces told apart at each
    // deposit the shared adds ran slower, 159 instead of 150 us a launch)
    unsigned long long* const rho = use_smem ? s_rho : P.rho_acc[sp];
    const uint32_t bytes = (uint32_t)tile_bytes_read<R>(limited || electrons, dep);
    uint32_t msteps = 0;  // of the warp: below 2^32 (a store has at most 2^31 slots)

    uint32_t fill_k = 0;
    if (k < k_end && ok) {
      if (lane == 0)
        load_tile(stages + started % kPushStages * kTB, buf + k * kTB, bytes,
                  &bars[started % kPushStages]);
      ++started;
      fill_k = fill[k];
    }
    for (; k < k_end && ok; k += (uint32_t)W) {
      const uint32_t n = fill_k;
      // the next tile, into the stage that the tile before this one has left
      if (k + W < k_end) {
        if (lane == 0)
          load_tile(stages + started % kPushStages * kTB, buf + (k + W) * kTB, bytes,
                    &bars[started % kPushStages]);
        ++started;
        fill_k = fill[k + W];
      }
      const uint32_t tbase = k * kTile;
      const Slot<R> tile = Markers<R>{buf}.at(k, 0);
      const Slot<R> stage = Markers<R>{stages + arrived % kPushStages * kTB}.at(0, 0);
      // ---- the tile's copy: wait (bounded) -----------------------------------
      {
        uint64_t* const bar = &bars[arrived % kPushStages];
        const uint32_t parity = arrived / kPushStages & 1u;
        if (!mbar_try_wait(bar, parity)) {
          const uint32_t limit = spin_limit(ctrl);
          uint32_t polls = 1;
          while (!mbar_try_wait(bar, parity)) {
            if (++polls > limit) {
              atomicCAS(&ctrl->error, 0, kErrTimeout);
              ok = false;
              break;
            }
          }
          if (lane == 0) {
            atomicAdd(&ctrl->spin_waits, 1u);
            atomicMax(&ctrl->spin_max, polls);
          }
        }
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        ++arrived;
      }
      uint32_t n_surv = 0, n_event = 0;
      // The lane's slots are advanced in kHalves passes of kPerHalf
      // neighbouring slots (lane l, pass h: slots (32 h + l) kPerHalf + j).
      // Ranks of survivors and events run on across the passes, in slot order.
#pragma unroll 1
      for (int i0 = 0; i0 < (int)n; i0 += kPerHalf * 32) {
        const int ib = i0 + lane * kPerHalf;
        const Slot<R> m{stage.c + ib, stage.r + ib};  // as copied
        const Slot<R> g{tile.c + ib, tile.r + ib};    // in the store
        // slots past the fill are read but never used; their cell is taken as
        // 0 so that the gather stays in range
        int cell[kPerHalf];
        R off[kPerHalf], vx[kPerHalf], vy[kPerHalf], vz[kPerHalf], wj[kPerHalf];
        uint32_t id[kPerHalf];
        bool live[kPerHalf];
        get_slots(&m.cell(), cell);
        get_slots(&m.off(), off);
        get_slots(&m.vx(), vx);
        if (limited) {
          get_slots(&m.vy(), vy);
          get_slots(&m.vz(), vz);
        }
        if (dep) get_slots(&m.wj(), wj);
        if (electrons) get_slots(&m.id(), id);
        // ---- advance the slots ---------------------------------------------
        R a[kPerHalf], b1[kPerHalf];
#pragma unroll
        for (int j = 0; j < kPerHalf; ++j) {
          live[j] = ib + j < (int)n;
          if (!live[j]) cell[j] = 0;
          // gather (linear between the cell's nodes)
          const R E0 = __ldg(Enode + cell[j]), E1 = __ldg(Enode + cell[j] + 1);
          a[j] = qmdt * (E0 + off[j] * (E1 - E0));
        }
        // speed-limited kick (leapfrog below the limit, the exact solution of
        // Eq. slpicEOMv across and above it) and drift (beta of the post-kick
        // speed); an unlimited species has beta = 1
        if (limited) {
          limited_kick_beta<R, kPerHalf>(vx, vy, vz, a, live, vlim, b1);
        } else {
#pragma unroll
          for (int j = 0; j < kPerHalf; ++j) {
            vx[j] = vx[j] + a[j];
            b1[j] = (R)1;
          }
        }
        bool alive[kPerHalf], event[kPerHalf], any_out = false;
#pragma unroll
        for (int j = 0; j < kPerHalf; ++j) {
          R o = off[j] + b1[j] * (vx[j] * dtdx);
          const R fl = r_floor(o);
          int c = cell[j] + (int)fl;
          o = o - fl;
          if (o >= (R)1) {
            o = (R)0;
            c += 1;
          }
          cell[j] = c;
          off[j] = o;
          alive[j] = live[j] && (uint32_t)c < N;
          event[j] = false;
          any_out |= live[j] && !alive[j];
        }
        // ---- candidate draws ------------------------------------------------
        if (electrons) {
#pragma unroll
          for (int j = 0; j < kPerHalf; ++j) {
            const uint2 rr = philox2x32_10(make_uint2(id[j], step), key2);
            event[j] = alive[j] && (rr.x >> 9) < cand_thr;
          }
        }
        // ---- deposit w_p = beta w_j now unless a collision may change v -------
        if (dep) {
#pragma unroll
          for (int j = 0; j < kPerHalf; ++j) {
            if (alive[j] && !event[j]) {
              const long long Q = fixed_charge(b1[j] * wj[j], wscale);
              const long long right = right_share(Q, off[j]);
              atomicAdd(rho + cell[j], (unsigned long long)(Q - right));
              atomicAdd(rho + cell[j] + 1, (unsigned long long)right);
            }
          }
        }
        const uint32_t live_so_far = min(n, (uint32_t)(i0 + kPerHalf * 32));
        uint32_t b_event[kPerHalf];
#pragma unroll
        for (int j = 0; j < kPerHalf; ++j) b_event[j] = __ballot_sync(0xFFFFFFFFu, event[j]);
        // (rank of slot j of a lane among the marked slots: those of the lanes
        // below, then the lane's own slots before j)
        auto rank_of = [&](const uint32_t (&b)[kPerHalf], int j) {
          uint32_t c = 0;
#pragma unroll
          for (int i = 0; i < kPerHalf; ++i)
            c += __popc(b[i] & (i < j ? lanemask_lt | 1u << lane : lanemask_lt));
          return c;
        };
        const bool whole =
            n_surv == (uint32_t)i0 && !__any_sync(0xFFFFFFFFu, any_out);
        if (whole) {
          // the usual pass: every marker of the tile so far stays where it is
          n_surv = live_so_far;
          if (b_event[0] | b_event[1]) {
            // (electrons: an ion's event is its absorption)
#pragma unroll
            for (int j = 0; j < kPerHalf; ++j) {
              if (event[j]) {
                const R y = limited ? vy[j] : (&m.vy())[j], z = limited ? vz[j] : (&m.vz())[j];
                put_cand(P.sp[kElectron].crec, (size_t)(tbase + n_event + rank_of(b_event, j)), cell[j], off[j], vx[j],
                         y, z, (&m.wj())[j], id[j], (uint32_t)(ib + j));
              }
            }
            n_event += __popc(b_event[0]) + __popc(b_event[1]);
          }
        } else {
          // ---- electrodes, ranks, events, compaction -------------------------
          // the fields not read above (ions: from the store)
          const Slot<R>& f = electrons ? m : g;
          if (!limited) {
            get_slots(&f.vy(), vy);
            get_slots(&f.vz(), vz);
          }
          if (!dep) get_slots(&f.wj(), wj);
          if (!electrons) get_slots(&g.id(), id);
          if (any_out) {
#pragma unroll
            for (int j = 0; j < kPerHalf; ++j) {
              if (live[j] && !alive[j])
                event[j] = absorb<R>(P, sp, cell[j] < 0 ? 0 : 1, wj[j], id[j], step, cs.s_acc,
                                     vx[j], vy[j], vz[j]);
            }
          }
          uint32_t b_alive[kPerHalf];
          const uint32_t pre_alive = n_surv, pre_event = n_event;
          __syncwarp();
#pragma unroll
          for (int j = 0; j < kPerHalf; ++j) {
            b_alive[j] = __ballot_sync(0xFFFFFFFFu, alive[j]);
            b_event[j] = __ballot_sync(0xFFFFFFFFu, event[j]);
            n_surv += __popc(b_alive[j]);
            n_event += __popc(b_event[j]);
          }
          // events: emissions to staging, candidates to the queue
#pragma unroll
          for (int j = 0; j < kPerHalf; ++j) {
            if (event[j]) {
              const uint32_t e = pre_event + rank_of(b_event, j);
              if (electrons) {
                // the candidate's slot after compaction = its rank among survivors
                const uint32_t r_a = pre_alive + rank_of(b_alive, j);
                put_cand(P.sp[kElectron].crec, tbase + e, cell[j], off[j], vx[j], vy[j], vz[j], wj[j], id[j],
                         r_a);
              } else if (dep) {
                stage_emission<R>(P, tbase + e, wj[j]);
              } else {
                stage_emission<R, false>(P, tbase + e, wj[j]);
              }
            }
          }
          if (n_surv != live_so_far) {
            // a marker of the tile has left: the survivors go to their ranks,
            // with all their fields.  Every lane holds the pass's slots in
            // registers (the barrier orders the reads before the writes), and
            // the ranks lie below the slots of the passes to come.
            __syncwarp();
#pragma unroll
            for (int j = 0; j < kPerHalf; ++j) {
              if (alive[j]) {
                const uint32_t r_a = pre_alive + rank_of(b_alive, j);
                write_marker(Slot<R>{tile.c + r_a, tile.r + r_a}, cell[j], off[j], vx[j], vy[j],
                             vz[j], wj[j], id[j]);
              }
            }
          }
        }
        if (n_surv == live_so_far && live[0]) {
          // in place: position and v_x (a lane's slot past the fill may be
          // written: it is never used)
          put_slots(&g.cell(), cell);
          put_slots(&g.off(), off);
          put_slots(&g.vx(), vx);
        }
      }
      __syncwarp();  // every lane has read the stage
      if (lane == 0) {
        fill[k] = n_surv;
        (electrons ? P.sp[kElectron].n_cand : P.sp[kIon].births)[k] = n_event;
      }
      msteps += n;
    }
    if (lane == 0 && msteps) atomicAdd(&cs.s_acc[ACC_MSTEPS], (unsigned long long)msteps);
    flush_segment(r, seg, s_rho, cs, use_smem);
  }
  // after a wait that ran out: no copy may outlive the CTA's shared memory
  if (lane == 0)
    for (; arrived < started; ++arrived)
      for (uint32_t p = 0; p < kSpinLimit; ++p)
        if (mbar_try_wait(&bars[arrived % kPushStages], arrived / kPushStages & 1u)) break;
}

// Dynamic shared memory of a CTA: the warps' stages and the charge grid.
template <typename R>
size_t push_smem(int warps, int smem_nodes) {
  return (size_t)warps * kPushStages * tile_bytes<R>() + (size_t)smem_nodes * 8;
}

template <typename R>
int push_config_t(int smem_nodes, int* warps, int* blocks_per_sm) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return (int)e;
  *warps = 0;
  *blocks_per_sm = 0;
  // the kernel may use all the dynamic shared memory a CTA can have: every
  // context's launches (of any grid size and shape) stay within that limit,
  // so no context's configuration lowers it under another's
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, k_push<R>);
  if (e != cudaSuccess) return (int)e;
  e = cudaFuncSetAttribute(k_push<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           optin - (int)fa.sharedSizeBytes);
  if (e != cudaSuccess) return (int)e;
  for (int w = kPushMaxWarps; w >= 4; w -= 4) {
    const size_t bytes = push_smem<R>(w, smem_nodes);
    if (bytes + fa.sharedSizeBytes > (size_t)optin) continue;
    int bps = 0;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, k_push<R>, w * 32, bytes);
    if (e != cudaSuccess) return (int)e;
    if (bps > 0) {
      *warps = w;
      *blocks_per_sm = bps;
      return 0;
    }
  }
  return 0;
}

template <typename R>
int push_bps_t(int warps, int smem_nodes, int* blocks_per_sm) {
  return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      blocks_per_sm, k_push<R>, warps * 32, push_smem<R>(warps, smem_nodes));
}

int push_blocks_per_sm(int fp64, int warps, int smem_nodes, int* blocks_per_sm) {
  return fp64 ? push_bps_t<double>(warps, smem_nodes, blocks_per_sm)
              : push_bps_t<float>(warps, smem_nodes, blocks_per_sm);
}

int push_config(int fp64, int smem_nodes, int* warps, int* blocks_per_sm) {
  return fp64 ? push_config_t<double>(smem_nodes, warps, blocks_per_sm)
              : push_config_t<float>(smem_nodes, warps, blocks_per_sm);
}

template <typename R>
static void launch_push_t(const DeviceRefs& r, int grid, cudaStream_t s) {
  launch_step_kernel(k_push<R>, grid, r.push_warps * 32, push_smem<R>(r.push_warps, r.smem_nodes),
                     s, r);
}

void launch_push(const DeviceRefs& r, int grid, cudaStream_t s) {
  if (r.fp64) launch_push_t<double>(r, grid, s);
  else launch_push_t<float>(r, grid, s);
}

static_assert(kTile == 32 * kPerLane, "a tile is kPerLane slots per lane of one warp");
static_assert(tile_bytes<float>() % 128 == 0 && tile_bytes<double>() % 128 == 0,
              "tiles start on 128-byte lines");

}  // namespace slpic
