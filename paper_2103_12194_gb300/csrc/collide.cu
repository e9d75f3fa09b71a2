// Monte-Carlo collisions of the null-collision candidates queued by the
// particle kernel (Sec. III and IV).  For a candidate (an electron that drew
// u < P0 this step) the process is chosen by comparing u' P0 with the
// cumulative rates n_g sigma_k(eps) beta v dt (Eq. SLPICcollisionNumber with
// beta_n = 1, whole-marker collisions); elastic collisions scatter by the
// Vahedi-Surendra angles with the recoil loss, excitation removes its
// threshold and scatters isotropically, ionization shares the excess energy
// between the primary and a born electron and creates an Ar+ at the same
// position with the same flux weight.  Each candidate, and each pair born, is
// then deposited with its new density weight (with an imposed field the
// deposit is formed from the markers when read).
//
// Work: items of consecutive tiles of one instance (electron items of
// coll_tiles[inst] tiles, then ion items of kCollIonTiles), each taken by one
// warp.  A CTA has a contiguous range of them, handed to its warps from a
// shared counter, and deposits those of one instance into a copy of its charge
// grid in shared memory: 6e5 candidates on 1311 nodes otherwise spend more
// than half of the kernel's time on global atomics to the same lines.  No
// warp waits for another.  A warp numbers the candidates of its item in (tile,
// slot) order and takes them 32 at a time, one lane each: it reads each
// candidate's record (its state and slot, one 32-byte sector in float; the
// next round's records load meanwhile), draws the process, deposits null
// collisions at once and queues the others by kind in shared memory.  The
// queues are scattered 32 at a time on one code path and run on from item to
// item, so that they are drained part full only once; only the new velocity is
// written to the candidate's slot.
//
// The births are not placed here.  Their slots and serial numbers follow the
// (tile, slot) order of their parents over the whole instance, which only the
// counts of all items give: each item leaves its number of births and, in
// order, the records of its ionizations (or where its emitted electrons are
// staged), and the next kernel (k_finish, beside the end of the step) places
// them (place_births).  Placing them here took an
// ordered look-back over the chunks and three barriers a chunk: CTAs waited
// for the slowest before them.
//
// Bound by the latency and the instructions of the scattering (log1p, expm1,
// sin and cos per elastic collision) at 24 warps per SM.  1.0e6 candidates of
// 4e6 electrons on 6340 nodes: 89 us a step with the look-back and global
// deposits, 66 now; 6.4e5 of 2e6 on 1311 nodes: 80 and 36.
#include "device_common.cuh"
#include "slpic_internal.h"
#include "step_ops.cuh"

namespace slpic {

namespace {

// Warps per CTA: one CTA per SM in float (80 registers a thread), with the
// room beside its queues for the charge grid; in double several small ones,
// which deposit to global memory (the FP64 unit is the limit there).
template <typename R>
__host__ __device__ constexpr int coll_warps() {
  return sizeof(R) == 4 ? 24 : 8;
}
constexpr int kQ = 64;  // entries of each queue (a round adds at most 32 to one below 32)

// One warp's collision queues in shared memory (structure of arrays, one
// entry per lane of a drain).  Elastic collisions keep the incident velocity;
// excitations and ionizations (rare; one queue) only the energy, and the
// candidate's record.
template <typename R>
struct CollQueues {
  uint32_t e_slot[kQ];
  int32_t e_cell[kQ];
  R e_off[kQ], e_wj[kQ], e_vx[kQ], e_vy[kQ], e_vz[kQ], e_eps[kQ], e_u2[kQ], e_u3[kQ];
  uint32_t n_slot[kQ], n_rec[kQ], n_id[kQ], n_k[kQ];
  int32_t n_cell[kQ];
  R n_off[kQ], n_wj[kQ], n_eps[kQ], n_u2[kQ], n_u3[kQ];
  uint32_t count[4];  // of the current instance: candidates, then collisions by kind
};

// Add a warp's (or CTA's) collisions of a kind to instance inst's counters.
// The last addition of ionizations sees their total: with the electrons
// emitted in the step they must fit the stores (the births are placed after
// this kernel; a step that does not fit is not committed).
__device__ __forceinline__ void add_counter(const DeviceRefs& r, int inst, int k,
                                            unsigned long long v) {
  const InstDev& P = r.inst[inst];
  const unsigned long long old = atomicAdd(P.acc + k, v);
  if (k != ACC_COLL2) return;
  const unsigned long long n = old + v, n_see = P.acc[ACC_SEE];
  const unsigned long long te = tail_slot(P.sp[kElectron], r.sstate[inst * 2]);
  const unsigned long long ti = tail_slot(P.sp[kIon], r.sstate[inst * 2 + 1]);
  if (te + n + n_see > (unsigned long long)P.sp[kElectron].cap_tiles * kTile ||
      ti + n > (unsigned long long)P.sp[kIon].cap_tiles * kTile)
    atomicCAS(&r.ctrl->error, 0, kErrCapacity);
}

// The slots of the staging that the electrons emitted by ion tiles k0 .. k1 - 1
// lie in, in order, from list[0] on (one warp; rare, kept out of line).
__device__ __noinline__ void list_emissions(const uint32_t* births, uint32_t k0, uint32_t k1,
                                            uint32_t* list) {
  const uint32_t lane = threadIdx.x & 31;
  for (uint32_t k = k0 + lane; k - lane < k1; k += 32) {
    const uint32_t n = k < k1 ? births[k] : 0u;
    uint32_t inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xFFFFFFFFu, inc, o);
      if (lane >= (uint32_t)o) inc += y;
    }
    for (uint32_t e = 0; e < n; ++e) list[inc - n + e] = k * kTile + e;
    list += __shfl_sync(0xFFFFFFFFu, inc, 31);
  }
}

}  // namespace

template <typename R>
__global__ void __launch_bounds__(coll_warps<R>() * 32, sizeof(R) == 4 ? 1 : 3)
    k_collide(DeviceRefs r) {
  extern __shared__ __align__(16) unsigned char coll_smem[];
  __shared__ unsigned long long s_acc[ACC_COUNT];
  __shared__ unsigned int s_next;
  constexpr int W = coll_warps<R>();
  step_kernel_entry();
  Control* ctrl = r.ctrl;
  const int stop = *((volatile int*)&ctrl->error);
  const unsigned int n_items = ctrl->n_coll_items;
  // (k_finish plans the next step while the births are still placed)
  if (blockIdx.x == 0)
    for (int i = threadIdx.x; i <= r.n_inst; i += blockDim.x) r.birth_start[i] = r.coll_start[i];
  const unsigned int i0 = (unsigned int)((unsigned long long)blockIdx.x * n_items / gridDim.x);
  const unsigned int i1 =
      (unsigned int)((unsigned long long)(blockIdx.x + 1) * n_items / gridDim.x);
  if (i0 >= i1) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t lanemask_lt = (1u << lane) - 1u;
  // instance of an item: the last one with coll_start <= it
  auto inst_of = [&](unsigned int it) {
    int lo = 0, hi = r.n_inst - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (r.coll_start[mid] <= it) lo = mid;
      else hi = mid - 1;
    }
    return lo;
  };
  // the CTA counts and deposits one instance's collisions in shared memory
  // (any other's go straight to global memory); the grid's copy pays when the
  // CTA has about a candidate for every two nodes
  const int tag = inst_of(i0 + (i1 - i0) / 2);
  const int tag_nodes = r.inst[tag].n_cells + 1;
  const bool use_smem = r.inst[tag].field_mode == 1 && tag_nodes <= r.coll_nodes &&
                        (i1 - i0) * (kCollTarget / 2) >= (unsigned int)tag_nodes / 2;
  unsigned long long* const s_rho =
      reinterpret_cast<unsigned long long*>(coll_smem + W * sizeof(CollQueues<R>));
  if (use_smem)
    for (int k = threadIdx.x; k < tag_nodes; k += blockDim.x) s_rho[k] = 0ull;
  if (threadIdx.x < ACC_COUNT) s_acc[threadIdx.x] = 0ull;
  if (threadIdx.x == 0) s_next = i0 + W;
  // (as one: an item of another CTA that does not fit its store may set the
  // word between two threads' reads of it)
  if (__syncthreads_or(stop)) return;

  CollQueues<R>& Q = reinterpret_cast<CollQueues<R>*>(coll_smem)[warp];
  unsigned int item = i0 + warp;
  unsigned int i_begin = 1u, i_end = 0u;  // items of the current instance
  int inst = -1;
  while (item < i1) {
    // ---- the item's instance ------------------------------------------------
    inst = inst_of(item);
    i_begin = r.coll_start[inst];
    i_end = min(i1, r.coll_start[inst + 1]);
    const InstDev& P = r.inst[inst];
    const SpeciesDev& E = P.sp[kElectron];
    const SpeciesDev& I = P.sp[kIon];
    const SpeciesState se = r.sstate[inst * 2 + kElectron];
    const uint32_t step = r.istate[inst].step;
    const uint32_t wt = r.coll_tiles[inst];
    const unsigned int e_items = (se.n_tiles + wt - 1) / wt;
    unsigned long long* const acc = inst == tag ? s_acc : P.acc;
    const Markers<R> me{E.buf[se.cur]};
    uint32_t* const list = reinterpret_cast<uint32_t*>(E.buf[se.cur ^ 1u]);
    CandRec<R>* const crec = reinterpret_cast<CandRec<R>*>(E.crec);
    const StepConsts<R>& K = consts<R>(P);
    const R kv = K.K_V[kElectron], vlim = K.vlim[kElectron], wscale = K.wscale;
    const uint32_t ctr2 = P.ctr_inst * 2u, key0 = P.key0, key1 = P.key1;
    const bool dep = P.field_mode == 1;  // imposed field: the deposit is formed when read
    unsigned long long* const rho_e = inst == tag && use_smem ? s_rho : P.rho_acc[kElectron];

    // the new velocity of slot o, and the deposit with it
    auto finish_one = [&](uint32_t o, int cell, R off, R wj, const Velocity<R>& nv) {
      const Slot<R> m = me[o];
      m.vx() = nv.vx;
      m.vy() = nv.vy;
      m.vz() = nv.vz;
      if (dep)
        deposit(rho_e, cell, off,
                fixed_charge(beta_any(nv.vx * nv.vx + nv.vy * nv.vy + nv.vz * nv.vz, vlim) * wj,
                             wscale));
    };
    uint32_t e_head = 0, e_tail = 0, n_head = 0, n_tail = 0;
    // scatter the n <= 32 oldest elastic (inelastic) entries, lane l the l-th
    auto drain_elastic = [&](uint32_t n) {
      const uint32_t i = (e_head + lane) & (kQ - 1);
      const bool on = lane < n;
      uint32_t slot = 0;
      int cell = 0;
      R off = 0, wj = 0, vx = 0, vy = 0, vz = 0, eps = 0, u2 = 0, u3 = 0;
      if (on) {
        slot = Q.e_slot[i];
        cell = Q.e_cell[i];
        off = Q.e_off[i];
        wj = Q.e_wj[i];
        vx = Q.e_vx[i];
        vy = Q.e_vy[i];
        vz = Q.e_vz[i];
        eps = Q.e_eps[i];
        u2 = Q.e_u2[i];
        u3 = Q.e_u3[i];
      }
      __syncwarp();  // the entries are read before the next round refills them
      if (on)
        finish_one(slot, cell, off, wj, scatter_elastic_any(K, kv, vx, vy, vz, eps, u2, u3));
      e_head += n;
    };
    auto drain_inelastic = [&](uint32_t n) {
      const uint32_t i = (n_head + lane) & (kQ - 1);
      const bool on = lane < n;
      uint32_t slot = 0, rec = 0, id = 0, k = 0;
      int cell = 0;
      R off = 0, wj = 0, eps = 0, u2 = 0, u3 = 0;
      if (on) {
        slot = Q.n_slot[i];
        rec = Q.n_rec[i];
        id = Q.n_id[i];
        k = Q.n_k[i];
        cell = Q.n_cell[i];
        off = Q.n_off[i];
        wj = Q.n_wj[i];
        eps = Q.n_eps[i];
        u2 = Q.n_u2[i];
        u3 = Q.n_u3[i];
      }
      __syncwarp();
      if (on) {
        Velocity<R> nv;
        if ((int)k <= P.n_exc) {
          nv = scatter_excitation<R>(K, kv, eps, (int)k, u2, u3, acc);
        } else {
          R es;
          nv = scatter_ionization<R>(P, kv, eps, u2, u3, id, step, wj, acc, &es);
          crec[rec].vx = es;  // for place_births: the secondary's energy
          if (dep) deposit_pair<R>(P, cell, off, wj, id, step, es);
        }
        finish_one(slot, cell, off, wj, nv);
      }
      n_head += n;
    };
    if (lane < 4) Q.count[lane] = 0u;
    __syncwarp();

    // ---- the instance's items that fall to this warp: one round of candidates
    // or one item's start per turn, then whatever queue is full (both, part
    // full, after the last item) ----------------------------------------------
    uint32_t total = 0, c0 = 0;      // the item's candidates, those taken
    uint32_t excl = 0, kbase = 0;    // their prefix by tile (lane j: tile j), first slot
    uint32_t births = 0, rec_n = 0;  // ionizations so far; the next round's record ...
    CandRec<R> nx = {};              // ... and its contents
    bool first = true, last = false;
    // record of candidate number e < total: the last tile whose prefix is <= e
    // (that tile has candidates), and the rank inside it
    auto locate = [&](uint32_t e) -> uint32_t {
      int j = 0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const uint32_t v = __shfl_sync(0xFFFFFFFFu, excl, j + o);
        if (v <= e) j += o;
      }
      return kbase + (uint32_t)j * kTile + e - __shfl_sync(0xFFFFFFFFu, excl, j);
    };
    auto fetch = [&](uint32_t c) {  // round c's records
      const uint32_t e = c + lane;
      rec_n = locate(e < total ? e : total - 1);
      if (e < total) nx = get_cand<R>(crec, rec_n);
    };
    do {
      if (c0 < total) {
        // ---- a round of 32 candidates, one per lane: each lane draws its
        // candidate's process; null collisions are deposited at once, the
        // others queued by kind.  Each collision's arithmetic is that of
        // collide(); the deposits and counters are integer sums, so the order
        // of the scatterings does not matter.
        const uint32_t rec = rec_n;
        const CandRec<R> cr = nx;
        const bool on = c0 + lane < total;
        c0 += 32;
        if (c0 < total) fetch(c0);
        int proc = 3, kx = 0;
        R u[4] = {0, 0, 0, 0}, eps = 0;
        if (on) {
          const R s1 = cr.vx * cr.vx + cr.vy * cr.vy + cr.vz * cr.vz;
          const R v1 = sqrt_any(s1);
          const uint4 rr = philox4x32_10(make_uint4(cr.id, step, ctr2, 0u), key0, key1);
          proc = choose_process<R>(P, vlim, v1, s1, rr, acc, u, eps, kx);
          if (proc == 3 && dep)  // null: the velocity is kept
            deposit(rho_e, cr.cell, cr.off, fixed_charge(beta_any(s1, vlim) * cr.wj, wscale));
        }
        const uint32_t be = __ballot_sync(0xFFFFFFFFu, proc == 0);
        const uint32_t bn = __ballot_sync(0xFFFFFFFFu, proc == 1 || proc == 2);
        const uint32_t bi = __ballot_sync(0xFFFFFFFFu, proc == 2);
        if (lane < 3) Q.count[1 + lane] += __popc(lane == 0 ? be : lane == 1 ? bn & ~bi : bi);
        const uint32_t slot = (rec & ~(uint32_t)(kTile - 1)) + cr.slot;
        if (proc == 0) {
          const uint32_t i = (e_tail + __popc(be & lanemask_lt)) & (kQ - 1);
          Q.e_slot[i] = slot;
          Q.e_cell[i] = cr.cell;
          Q.e_off[i] = cr.off;
          Q.e_wj[i] = cr.wj;
          Q.e_vx[i] = cr.vx;
          Q.e_vy[i] = cr.vy;
          Q.e_vz[i] = cr.vz;
          Q.e_eps[i] = eps;
          Q.e_u2[i] = u[2];
          Q.e_u3[i] = u[3];
        } else if (proc != 3) {
          const uint32_t i = (n_tail + __popc(bn & lanemask_lt)) & (kQ - 1);
          Q.n_slot[i] = slot;
          Q.n_rec[i] = rec;
          Q.n_id[i] = cr.id;
          Q.n_k[i] = (uint32_t)kx;
          Q.n_cell[i] = cr.cell;
          Q.n_off[i] = cr.off;
          Q.n_wj[i] = cr.wj;
          Q.n_eps[i] = eps;
          Q.n_u2[i] = u[2];
          Q.n_u3[i] = u[3];
          // the item's ionizations, in order
          if (proc == 2) list[kbase + births + __popc(bi & lanemask_lt)] = rec;
        }
        births += __popc(bi);
        e_tail += __popc(be);
        n_tail += __popc(bn);
        if (c0 >= total && lane == 0) r.item_births[item] = births;
      } else {
        // ---- the next item -----------------------------------------------------
        if (!first) {
          if (lane == 0) item = atomicAdd(&s_next, 1u);
          item = __shfl_sync(0xFFFFFFFFu, item, 0);
        }
        first = false;
        if (item >= i_end) {
          last = true;
        } else {
          const unsigned int local = item - i_begin;
          if (local == 0 && lane == 0) {
            // where this step's births go (k_finish moves the state on)
            const SpeciesState si = r.sstate[inst * 2 + kIon];
            BirthBase b;
            b.cur[0] = se.cur;
            b.cur[1] = si.cur;
            b.tail[0] = tail_slot(E, se);
            b.tail[1] = tail_slot(I, si);
            b.next_id[0] = se.next_id;
            b.next_id[1] = si.next_id;
            b.step = step;
            b.e_items = e_items;
            b.tiles = wt;
            r.birth_base[inst] = b;
            if (b.tail[0] + P.acc[ACC_SEE] > (unsigned long long)E.cap_tiles * kTile)
              atomicCAS(&ctrl->error, 0, kErrCapacity);
          }
          total = c0 = births = 0;
          if (local >= e_items) {
            // ions: electrons emitted at the cathode (staged by the particle kernel)
            const uint32_t k0 = (local - e_items) * kCollIonTiles;
            const uint32_t k1 = min(k0 + kCollIonTiles, r.sstate[inst * 2 + kIon].n_tiles);
            for (uint32_t k = k0 + lane; k < k1; k += 32) births += I.births[k];
            births = __reduce_add_sync(0xFFFFFFFFu, births);
            if (births)
              list_emissions(I.births, k0, k1,
                             reinterpret_cast<uint32_t*>(
                                 I.buf[r.sstate[inst * 2 + kIon].cur ^ 1u]) +
                                 (size_t)k0 * kTile);
          } else {
            // wt consecutive tiles, tile kw + j at lane j: their candidates are
            // numbered in (tile, slot) order
            const uint32_t kw = local * wt;
            const uint32_t cnt =
                (uint32_t)lane < wt && kw + lane < se.n_tiles ? E.n_cand[kw + lane] : 0u;
            excl = cnt;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, excl, o);
              if (lane >= o) excl += n;
            }
            total = __shfl_sync(0xFFFFFFFFu, excl, 31);
            excl -= cnt;
            kbase = kw * kTile;
            if (lane == 0) Q.count[0] += total;
            if (total) fetch(0);
          }
          if (total == 0 && lane == 0) r.item_births[item] = births;
        }
      }
      __syncwarp();
      const uint32_t full = last ? 1u : 32u;
      if (e_tail - e_head >= full) drain_elastic(min(e_tail - e_head, 32u));
      if (n_tail - n_head >= full) drain_inelastic(min(n_tail - n_head, 32u));
    } while (!last);
    __syncwarp();
    // the warp's candidates and collisions, counted once
    if (lane < 4 && Q.count[lane]) {
      const int a = lane ? ACC_COLL0 + lane - 1 : ACC_CAND;
      if (inst == tag) atomicAdd(&s_acc[a], (unsigned long long)Q.count[lane]);
      else add_counter(r, inst, a, Q.count[lane]);
    }
  }
  __syncthreads();
  if (threadIdx.x < ACC_COUNT && s_acc[threadIdx.x])
    add_counter(r, tag, threadIdx.x, s_acc[threadIdx.x]);
  if (use_smem) {
    unsigned long long* const g = r.inst[tag].rho_acc[kElectron];
    for (int k = threadIdx.x; k < tag_nodes; k += blockDim.x)
      if (s_rho[k]) atomicAdd(g + k, s_rho[k]);
  }
}

// Dynamic shared memory of a CTA: the queues and a charge grid of `nodes` nodes.
template <typename R>
static size_t coll_smem_bytes(int nodes) {
  return coll_warps<R>() * sizeof(CollQueues<R>) + (size_t)nodes * 8;
}

template <typename R>
static void launch_collide_t(const DeviceRefs& r, int grid, cudaStream_t s) {
  launch_step_kernel(k_collide<R>, grid, coll_warps<R>() * 32, coll_smem_bytes<R>(r.coll_nodes),
                     s, r);
}

void launch_collide(const DeviceRefs& r, int grid, cudaStream_t s) {
  if (r.fp64) launch_collide_t<double>(r, grid, s);
  else launch_collide_t<float>(r, grid, s);
}

// CTAs of the kernel that an SM holds at once (more would only make a second
// wave), and the nodes of the shared charge grid: max_nodes when it fits beside
// a float CTA's queues, else 0.
template <typename R>
static int collide_config_t(int max_nodes, int* resident, int* nodes) {
  int dev = 0, optin = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return (int)e;
  e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return (int)e;
  cudaFuncAttributes fa;
  e = cudaFuncGetAttributes(&fa, k_collide<R>);
  if (e != cudaSuccess) return (int)e;
  // the limit is the most a CTA can have, so that one context's configuration
  // never lowers it under another's
  const size_t most = (size_t)optin - fa.sharedSizeBytes;
  e = cudaFuncSetAttribute(k_collide<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)most);
  if (e != cudaSuccess) return (int)e;
  *nodes = sizeof(R) == 4 && coll_smem_bytes<R>(max_nodes) <= most ? max_nodes : 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(resident, k_collide<R>, coll_warps<R>() * 32,
                                                    coll_smem_bytes<R>(*nodes));
  if (e == cudaSuccess && *resident < 1) *resident = 1;
  return (int)e;
}

int collide_config(int fp64, int max_nodes, int* resident, int* nodes) {
  return fp64 ? collide_config_t<double>(max_nodes, resident, nodes)
              : collide_config_t<float>(max_nodes, resident, nodes);
}

static_assert(kCollMaxTiles <= 32, "per-tile counts live one per lane");
static_assert(sizeof(CollQueues<float>) % 16 == 0 && sizeof(CollQueues<double>) % 16 == 0,
              "the charge grid follows the queues");
static_assert((kTile & (kTile - 1)) == 0, "a record's tile by a mask");

}  // namespace slpic
