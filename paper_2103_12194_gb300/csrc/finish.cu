// End of a step.  k_finish updates the marker counts of every instance from
// the step's exact counters (the particle kernel compacted every tile,
// k_collide counted every birth), decides whether a store is repacked, commits
// the step's tallies and plans the next step; beside this it publishes the
// step's deposit with the sums of its net charge, block by block, and appends
// the step's births to the stores.  k_move evaluates the field of the 1D
// Poisson equation from those sums and repacks the stores that became sparse.
// With an imposed field the step deposits nothing and k_deposit forms the
// deposit from the markers when it is read.  Also: seeding, loading and reading
// markers and the Philox self-check kernel.
#include <algorithm>

#include "device_common.cuh"
#include "slpic_internal.h"
#include "step_ops.cuh"

namespace slpic {

namespace {

constexpr int kMoveThreads = 256;

// Segments a single warp plans (kPlanPerLane consecutive ones per lane; an
// instance's two segments stay in one lane).
constexpr int kPlanPerLane = 8;

__device__ __forceinline__ long long warp_incl_scan(long long v, int lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const long long y = __shfl_up_sync(0xFFFFFFFFu, v, o);
    if (lane >= o) v += y;
  }
  return v;
}

// Write the plan's totals and reset the step's counters (one thread).
__device__ __forceinline__ void plan_totals(const DeviceRefs& r, int n_seg, unsigned int start,
                                            unsigned int wstart, unsigned int move,
                                            unsigned int coll) {
  r.seg_start[n_seg] = start;
  r.seg_wstart[n_seg] = wstart;
  r.coll_start[r.n_inst] = coll;
  r.move_start[n_seg] = move;
  r.ctrl->n_tiles = start;
  r.ctrl->w_total = wstart;
  r.ctrl->n_seg = n_seg;
  r.ctrl->n_coll_items = coll;
  r.ctrl->n_move_chunks = move;
  r.ctrl->move_counter = 0;
  r.ctrl->epoch = (r.ctrl->epoch + 1u) & 0x3FFFFFFFu;
  r.ctrl->finish_done = 0;
}

// Sum over the lanes of a warp.
__device__ __forceinline__ long long warp_sum(long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, o);
  return v;
}
__device__ __forceinline__ __int128 warp_sum(__int128 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long l = __shfl_xor_sync(0xFFFFFFFFu, (unsigned long long)v, o);
    const long long h = __shfl_xor_sync(0xFFFFFFFFu, (long long)(v >> 64), o);
    v += (__int128)(((unsigned __int128)(unsigned long long)h << 64) | l);
  }
  return v;
}

// Instance of block u of the nodes of all instances.
__device__ __forceinline__ int field_inst(const DeviceRefs& r, int u) {
  int lo = 0, hi = r.n_inst - 1;  // last instance with field_start <= u
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (r.field_start[mid] <= u) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// Block `block` of the node field of instance P's last Poisson solve, by the
// kMoveThreads threads of a CTA.
//   (phi[k+1] - 2 phi[k] + phi[k-1]) = -C net_k, k = 1 .. N-1.  With D_k =
// phi[k] - phi[k-1]: D_k = D_1 - C I_k, I_k = sum_{0<j<k} net_j, and phi[N] = V
// fixes D_1 = (V + C J_N) / N, J_N = sum_{0<i<=N} I_i = sum_{0<j<N} (N - j) net_j.
// The node field is the centred difference of phi, written with these exact
// integer sums: E_k = -(D_k + D_{k+1}) / (2 dx) = -(2 D_1 - C (I_k + I_{k+1}))
// / (2 dx), one-sided at the electrodes.  k_finish has left every block's
// sums; phi is formed on demand (k_phi) when it is read.
struct FieldShared {
  long long S;     // net charge of the blocks before
  double D1;
  long long w[kMoveThreads / 32];
};
__device__ __forceinline__ void poisson_field(const InstDev& P, int block, FieldShared& sh) {
  constexpr int kPer = kFieldNodes / kMoveThreads;
  const int N = P.n_cells, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int k0 = block * kFieldNodes + t * kPer;
  long long net[kPer] = {};
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int k = k0 + j;
    if (k > 0 && k < N) net[j] = P.rho_last[kIon][k] - P.rho_last[kElectron][k];
  }
  if (warp == 0) {
    const int nb = N / kFieldNodes + 1;
    long long S = 0;
    __int128 W = 0;
    for (int b = lane; b < nb; b += 32) {
      if (b < block) S += P.pois_S[b];
      W += P.pois_W[b];
    }
    S = warp_sum(S);
    W = warp_sum(W);
    // one thread forms D_1 (FP64 is scarce on this part) and shares it
    if (lane == 0) {
      sh.S = S;
      sh.D1 = (P.V + P.pois_C * (double)W) / (double)N;
    }
  }
  long long loc = 0;
#pragma unroll
  for (int j = 0; j < kPer; ++j) loc += net[j];
  const long long inc = warp_incl_scan(loc, lane);
  if (lane == 31) sh.w[warp] = inc;
  __syncthreads();
  long long I = sh.S + inc - loc;  // I_{k0}
#pragma unroll
  for (int w = 0; w < kMoveThreads / 32; ++w)
    if (w < warp) I += sh.w[w];
  const double D1 = sh.D1, C = P.pois_C;
  const double inv2dx = 1.0 / (2.0 * P.dx);
  const double twoD1 = D1 + D1;
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int k = k0 + j;
    if (k > N) break;
    const long long I1 = I + net[j];
    double e;
    if (k == 0) e = -D1 / P.dx;  // I_1 = 0: D_1
    else if (k < N) e = -(twoD1 - C * (double)(I + I1)) * inv2dx;
    else e = -(D1 - C * (double)I) / P.dx;
    P.E64[k] = e;
    P.E32[k] = (float)e;
    I = I1;
  }
  __syncthreads();  // sh is free for the next block
}

// Tiles per electron collision item of an instance of n_tiles electron tiles:
// `room` of them hold kCollTarget candidates.  Fewer where the instance would
// not give coll_share items, but in float not below an eighth of room (a round
// of 32 candidates).
__device__ __forceinline__ unsigned int item_tiles(const DeviceRefs& r, unsigned long long room,
                                                   uint32_t n_tiles) {
  const unsigned long long share = n_tiles / r.coll_share;
  const unsigned long long most = min(room, max(share, r.fp64 ? 1ull : room / 8u));
  return (unsigned int)min(max(most, 1ull), (unsigned long long)kCollMaxTiles);
}

// Weight of starting a segment, in the particle kernel's split of `total`
// weights over its CTAs: a barrier, a flush of the charge grid and an empty
// pipeline, about as long as 16 electron tiles of a CTA.  (A CTA whose range
// held ten small gaps took far longer than the others: k_push on 32 uneven gaps
// 242 us, 201 with this; 24 or 96 instead of 48 run the same.)  No more than a
// CTA's share, which populations of few tiles are spread over.
__device__ __forceinline__ long long seg_cost(const DeviceRefs& r, long long total) {
  return min((long long)kSegCost, total / r.push_grid);
}

// The plan below by one warp (n_seg <= 32 kPlanPerLane), with shuffle scans
// and no block barrier.
__device__ void plan_next_warp(const DeviceRefs& r) {
  const int lane = threadIdx.x & 31;
  const int n_seg = r.n_inst * 2;
  long long ns[kPlanPerLane], w[kPlanPerLane], mv[kPlanPerLane], nc[kPlanPerLane / 2];
  long long s_ns = 0, s_w = 0, s_mv = 0, s_nc = 0;
#pragma unroll
  for (int j = 0; j < kPlanPerLane; ++j) {
    const int sg = lane * kPlanPerLane + j;
    ns[j] = w[j] = mv[j] = 0;
    if (sg < n_seg) {
      ns[j] = r.sstate[sg].n_tiles;
      w[j] = ns[j] * ((sg & 1) ? kWeightIon : kWeightElectron);
      const Transfer& x = r.xfer[sg];
      if (x.compact) mv[j] = ((long long)x.n_tiles_old + kMoveChunkTiles - 1) / kMoveChunkTiles;
    }
    s_ns += ns[j];
    s_w += w[j];
    s_mv += mv[j];
  }
#pragma unroll
  for (int j = 0; j < kPlanPerLane / 2; ++j) {
    const int i = lane * (kPlanPerLane / 2) + j;
    nc[j] = 0;
    if (i < r.n_inst) {
      const long long T = item_tiles(r, r.coll_room[i], r.sstate[2 * i].n_tiles);
      r.coll_tiles[i] = (unsigned int)T;
      nc[j] = ((long long)r.sstate[2 * i].n_tiles + T - 1) / T +
              ((long long)r.sstate[2 * i + 1].n_tiles + kCollIonTiles - 1) / kCollIonTiles;
    }
    s_nc += nc[j];
  }
  const long long i_ns = warp_incl_scan(s_ns, lane);
  long long i_w = warp_incl_scan(s_w, lane);
  // and the cost of every segment that is not empty
  const long long cost = seg_cost(r, __shfl_sync(0xFFFFFFFFu, i_w, 31));
  long long s_c = 0;
#pragma unroll
  for (int j = 0; j < kPlanPerLane; ++j) {
    const long long c = ns[j] ? cost : 0;
    w[j] += c;
    s_c += c;
  }
  s_w += s_c;
  i_w += warp_incl_scan(s_c, lane);
  const long long i_mv = warp_incl_scan(s_mv, lane), i_nc = warp_incl_scan(s_nc, lane);
  long long e_ns = i_ns - s_ns, e_w = i_w - s_w, e_mv = i_mv - s_mv, e_nc = i_nc - s_nc;
#pragma unroll
  for (int j = 0; j < kPlanPerLane; ++j) {
    const int sg = lane * kPlanPerLane + j;
    if (sg < n_seg) {
      r.seg_start[sg] = (unsigned int)e_ns;
      r.seg_wstart[sg] = (unsigned int)e_w;
      r.move_start[sg] = (unsigned int)e_mv;
    }
    e_ns += ns[j];
    e_w += w[j];
    e_mv += mv[j];
  }
#pragma unroll
  for (int j = 0; j < kPlanPerLane / 2; ++j) {
    const int i = lane * (kPlanPerLane / 2) + j;
    if (i < r.n_inst) r.coll_start[i] = (unsigned int)e_nc;
    e_nc += nc[j];
  }
  if (lane == 31) {
    r.ctrl->seg_cost = (unsigned int)cost;
    plan_totals(r, n_seg, (unsigned int)i_ns, (unsigned int)i_w, (unsigned int)i_mv,
                (unsigned int)i_nc);
  }
}

// Plan the next step from the tiles in use (all threads of one CTA):
// particle-kernel tiles and their weights and repacking chunks per segment and
// collision items per instance, as exclusive block scans in rounds of kFinThreads entries.
__device__ void plan_next(const DeviceRefs& r, long long* s_buf) {
  __shared__ long long s_carry[5];
  const int n_seg = r.n_inst * 2;
  if (n_seg <= 32 * kPlanPerLane) {
    if (threadIdx.x < 32) plan_next_warp(r);
    return;
  }
  const int t = threadIdx.x;
  if (t < 5) s_carry[t] = 0;
  __syncthreads();
  // the summed weights of the tiles give the cost of a segment
  for (int base = 0; base < n_seg; base += kFinThreads) {
    const int sg = base + t;
    const long long w = sg < n_seg ? (long long)r.sstate[sg].n_tiles *
                                         ((sg & 1) ? kWeightIon : kWeightElectron)
                                   : 0;
    const long long i_w = block_incl_scan<long long>(w, s_buf);
    if (t == kFinThreads - 1) s_carry[4] += i_w;
  }
  __syncthreads();
  const long long cost = seg_cost(r, s_carry[4]);
  if (t == 0) r.ctrl->seg_cost = (unsigned int)cost;
  for (int base = 0; base < n_seg; base += kFinThreads) {
    const int sg = base + t;
    long long ns = 0, w = 0, mv = 0;
    if (sg < n_seg) {
      ns = r.sstate[sg].n_tiles;
      w = ns * ((sg & 1) ? kWeightIon : kWeightElectron) + (ns ? cost : 0);
      const Transfer& x = r.xfer[sg];
      if (x.compact) mv = ((long long)x.n_tiles_old + kMoveChunkTiles - 1) / kMoveChunkTiles;
    }
    const long long i_ns = block_incl_scan<long long>(ns, s_buf);
    const long long i_w = block_incl_scan<long long>(w, s_buf);
    const long long i_mv = block_incl_scan<long long>(mv, s_buf);
    if (sg < n_seg) {
      r.seg_start[sg] = (unsigned int)(s_carry[0] + i_ns - ns);
      r.seg_wstart[sg] = (unsigned int)(s_carry[1] + i_w - w);
      r.move_start[sg] = (unsigned int)(s_carry[2] + i_mv - mv);
    }
    __syncthreads();
    if (t == kFinThreads - 1) {
      s_carry[0] += i_ns;
      s_carry[1] += i_w;
      s_carry[2] += i_mv;
    }
    __syncthreads();
  }
  for (int base = 0; base < r.n_inst; base += kFinThreads) {
    const int i = base + t;
    long long nc = 0;
    if (i < r.n_inst) {
      const long long T = item_tiles(r, r.coll_room[i], r.sstate[2 * i].n_tiles);
      r.coll_tiles[i] = (unsigned int)T;
      nc = ((long long)r.sstate[2 * i].n_tiles + T - 1) / T +
           ((long long)r.sstate[2 * i + 1].n_tiles + kCollIonTiles - 1) / kCollIonTiles;
    }
    const long long i_nc = block_incl_scan<long long>(nc, s_buf);
    if (i < r.n_inst) r.coll_start[i] = (unsigned int)(s_carry[3] + i_nc - nc);
    __syncthreads();
    if (t == kFinThreads - 1) s_carry[3] += i_nc;
    __syncthreads();
  }
  if (t == 0)
    plan_totals(r, n_seg, (unsigned int)s_carry[0], (unsigned int)s_carry[1],
                (unsigned int)s_carry[2], (unsigned int)s_carry[3]);
}

// Append the step's births to the stores, by CTA b of nb: the births of its
// share of the items, in item order (ionization electrons in (tile, slot)
// order of their parents, emitted electrons after them), one thread each.
// Every CTA sums the counts of the items before its own, so none waits.
template <typename R>
__device__ __noinline__ void place_births(const DeviceRefs& r, int b, int nb, uint32_t* s_pre,
                                          long long* s_i64) {
  const unsigned int n_items = r.birth_start[r.n_inst];
  const unsigned int per = (n_items + nb - 1) / nb;
  unsigned int i0 = (unsigned int)b * per;
  const unsigned int i1 = min(i0 + per, n_items);
  const int t = threadIdx.x;
  int inst = 0;
  {
    int lo = 0, hi = r.n_inst - 1;  // last instance with coll_start <= i0
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (r.birth_start[mid] <= i0) lo = mid;
      else hi = mid - 1;
    }
    inst = lo;
  }
  for (; i0 < i1; ++inst) {
    const unsigned int first = r.birth_start[inst], end = min(i1, r.birth_start[inst + 1]);
    if (end <= i0) continue;  // an instance without items
    const InstDev& P = r.inst[inst];
    const BirthBase B = r.birth_base[inst];
    const uint32_t wt = B.tiles;
    const uint32_t step = B.step;
    // births of the instance before item i0
    long long before;
    {
      long long n = 0;
      for (unsigned int k = first + t; k < i0; k += kFinThreads) n += r.item_births[k];
      const long long inc = block_incl_scan<long long>(n, s_i64);
      if (t == kFinThreads - 1) s_i64[0] = inc;
      __syncthreads();
      before = s_i64[0];
      __syncthreads();
    }
    const SpeciesDev& E = P.sp[kElectron];
    const Markers<R> me{E.buf[B.cur[0]]}, mi{P.sp[kIon].buf[B.cur[1]]};
    const uint32_t* list = reinterpret_cast<const uint32_t*>(E.buf[B.cur[0] ^ 1u]);
    const uint32_t* ilist = reinterpret_cast<const uint32_t*>(P.sp[kIon].buf[B.cur[1] ^ 1u]);
    const unsigned int e_items = B.e_items;
    for (; i0 < end; i0 += kFinThreads) {
      // prefixes of up to kFinThreads items
      const unsigned int m = min(end - i0, (unsigned int)kFinThreads);
      const uint32_t c = (unsigned int)t < m ? r.item_births[i0 + t] : 0u;
      const long long inc = block_incl_scan<long long>((long long)c, s_i64);
      s_pre[t] = (uint32_t)(inc - c);
      if (t == kFinThreads - 1) s_i64[0] = inc;
      __syncthreads();
      const uint32_t total = (uint32_t)s_i64[0];
      for (uint32_t n = t; n < total; n += kFinThreads) {
        // the item of birth n: the last one whose prefix is <= n
        unsigned int lo = 0, hi = m - 1;
        while (lo < hi) {
          const unsigned int mid = (lo + hi + 1) >> 1;
          if (s_pre[mid] <= n) lo = mid;
          else hi = mid - 1;
        }
        const uint32_t q = n - s_pre[lo], rank = (uint32_t)before + n;
        const unsigned int local = i0 + lo - first;
        const Slot<R> pe = me[B.tail[0] + rank];
        if (local < e_items) {
          const CandRec<R> cr = get_cand<R>(E.crec, list[local * wt * kTile + q]);
          born_pair<R>(P, pe, mi[B.tail[1] + rank], cr.cell, cr.off, cr.wj, cr.id, step, cr.vx,
                       B.next_id[0] + rank, B.next_id[1] + rank);
        } else {
          // emitted at the cathode by an ion of the item's tiles (looking for
          // the tile here, one count after the other, took k_finish from 15 to
          // 28 us on 3e7 ions that emit 10 electrons a step)
          const uint32_t o = ilist[(size_t)(local - e_items) * kCollIonTiles * kTile + q];
          write_marker(pe, 0, (R)0, (R)0, (R)0, (R)0, reinterpret_cast<const R*>(E.stage_w)[o],
                       kGenBit | ((B.next_id[0] + rank) & kSerialMask));
        }
      }
      before += total;
      __syncthreads();
    }
    i0 = end;
  }
}

// What the state CTA of an instance keeps in shared memory.
struct StateShared {
  unsigned long long acc[ACC_COUNT];
  InstState is;
  SpeciesState st[2];
  Transfer x[2];
};

// The plan of a single instance, by one thread, from what its state CTA holds.
__device__ __forceinline__ void plan_single(const DeviceRefs& r, const StateShared& sh,
                                            unsigned int room) {
  unsigned int ns = 0, w = 0, mv = 0;
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    r.seg_start[s] = ns;
    r.seg_wstart[s] = w;
    r.move_start[s] = mv;
    ns += sh.st[s].n_tiles;
    w += sh.st[s].n_tiles * (s ? kWeightIon : kWeightElectron);
    if (sh.x[s].compact) mv += (sh.x[s].n_tiles_old + kMoveChunkTiles - 1) / kMoveChunkTiles;
  }
  r.ctrl->seg_cost = 0u;
  const unsigned int T = item_tiles(r, room, sh.st[0].n_tiles);
  r.coll_tiles[0] = T;
  r.coll_start[0] = 0u;
  plan_totals(r, 2, ns, w, mv,
              (sh.st[0].n_tiles + T - 1) / T +
                  (sh.st[1].n_tiles + kCollIonTiles - 1) / kCollIonTiles);
}

// The end of a step of instance inst: counts, fills, tallies.  A chain of
// global round trips, so every load that can be is issued at the start.
// Returns the tiles that hold about kCollTarget candidates.
__device__ __forceinline__ unsigned int finish_state(const DeviceRefs& r, int inst,
                                                     StateShared& sh) {
  const int t = threadIdx.x;
  const InstDev& P = r.inst[inst];
  unsigned long long* a = P.acc;
  const long long total = t < kTallySlots ? reinterpret_cast<long long*>(P.total)[t] : 0ll;
  if (t < ACC_COUNT) {
    sh.acc[t] = a[t];
    a[t] = 0ull;
  }
  if (t == 32) sh.is = r.istate[inst];
  uint32_t tail = 0;
  if (t < 2) {
    const SpeciesState st = r.sstate[inst * 2 + t];
    sh.st[t] = st;
    tail = tail_slot(P.sp[t], st);
  }
  __syncthreads();

  // ---- marker counts and where the stores end (one thread per species) -------
  // survivors = live - absorbed; births (ionizations: an electron and an ion
  // each; emitted electrons) are appended after the last live marker
  unsigned int room = 0;
  if (t < 2) {
    const int sp = t;
    const uint32_t n_ionz = (uint32_t)sh.acc[ACC_COLL2], n_see = (uint32_t)sh.acc[ACC_SEE];
    const uint32_t absorbed =
        (uint32_t)(sh.acc[ACC_NABS + 2 * sp] + sh.acc[ACC_NABS + 2 * sp + 1]);
    const uint32_t nb = sp ? n_ionz : n_ionz + n_see;
    const SpeciesState s0 = sh.st[sp];
    const uint32_t surv = s0.n_live - absorbed;
    const uint32_t end = tail + nb;
    const uint32_t n_new = surv + nb;
    const uint32_t nt = (end + kTile - 1) / kTile;
    // repack when under 15/16 of the slots in use are live: tiles with holes
    // cost the particle kernel nearly as much as full ones, and a growing
    // avalanche leaves many (at 3/4 a 1000-step run of the benchmark ran at
    // half the rate in its last steps)
    const uint32_t compact =
        (nt > 2 && (unsigned long long)n_new * 16 < (unsigned long long)nt * kTile * 15) ? 1u : 0u;
    Transfer x;
    x.compact = compact;
    x.src = s0.cur;
    x.dst = compact ? s0.cur ^ 1u : s0.cur;
    x.n_tiles_old = nt;
    x.n_new = n_new;
    x.tail = tail;
    x.end = end;
    x.pad = 0u;
    SpeciesState s1;
    s1.cur = x.dst;
    s1.n_live = n_new;
    s1.next_id = s0.next_id + nb;
    s1.n_tiles = compact ? (n_new + kTile - 1) / kTile : nt;
    sh.x[sp] = x;
    sh.st[sp] = s1;
    r.xfer[inst * 2 + sp] = x;
    r.sstate[inst * 2 + sp] = s1;
    if (sp == kElectron) {
      // tiles that hold about kCollTarget candidates at this step's density
      const unsigned long long cand = sh.acc[ACC_CAND];
      const unsigned long long fit =
          cand ? (unsigned long long)kCollTarget * s0.n_tiles / cand
               : (unsigned long long)kCollMaxRoom;
      room = (unsigned int)min(max(fit, 1ull), (unsigned long long)kCollMaxRoom);
      r.coll_room[inst] = room;
    }
  }
  __syncthreads();
  // fills of the tail tile and the new tiles: their slots below `end` are live
  // (k_move reads them when it repacks the store)
  for (int sp = 0; sp < 2; ++sp) {
    const Transfer& x = sh.x[sp];
    if (x.end == x.tail) continue;
    uint32_t* const fill = P.sp[sp].fill[x.src];
    for (uint32_t k = x.tail / kTile + t; k < x.n_tiles_old; k += kFinThreads)
      fill[k] = min(x.end - k * (uint32_t)kTile, (uint32_t)kTile);
  }
  // ---- tallies: one thread per 8-byte slot of the record ---------------------
  if (t < kTallySlots)
    commit_tally_slot(P, t, sh.acc, sh.is.step, sh.is.n_steps_done, sh.st[0].n_live,
                      sh.st[1].n_live, sh.is.w_live, &sh.is.ion_steps, 1.0 / P.c64.wscale, total);
  __syncthreads();
  if (t == 32) {
    sh.is.step += 1u;
    sh.is.n_steps_done += 1;
    r.istate[inst] = sh.is;
  }
  return room;
}

// A block's sums of the net charge and of it weighted, from its nodes' values.
__device__ __forceinline__ void block_sums(const InstDev& P, int block, long long net, int weight,
                                           long long* s_i64, __int128* s_i128) {
  const long long S = block_incl_scan<long long>(net, s_i64);
  const __int128 W = block_incl_scan<__int128>((__int128)net * weight, s_i128);
  if (threadIdx.x == kFinThreads - 1) {
    P.pois_S[block] = S;
    P.pois_W[block] = W;
  }
}

// One block of kFieldNodes nodes of an instance: the step's deposit becomes
// the last step's, and the block leaves its sums of the net charge net_j
// (0 < j < N) for the field: S = sum net_j and W = sum (N - j) net_j.
__device__ __forceinline__ void finish_nodes(const InstDev& P, int block, long long* s_i64,
                                             __int128* s_i128) {
  const int k = block * kFieldNodes + (int)threadIdx.x, N = P.n_cells;
  long long net = 0;
  if (k <= N) {
    const long long qe = (long long)P.rho_acc[kElectron][k], qi = (long long)P.rho_acc[kIon][k];
    P.rho_last[kElectron][k] = qe;
    P.rho_last[kIon][k] = qi;
    P.rho_acc[kElectron][k] = 0ull;
    P.rho_acc[kIon][k] = 0ull;
    if (k > 0 && k < N) net = qi - qe;
  }
  block_sums(P, block, net, N - k, s_i64, s_i128);
}

}  // namespace

// mode 0: finish a step.  CTAs 0 .. n_inst - 1, one per instance, update its
// state (the last one plans the next step); the next n_field take the blocks of
// nodes of all instances in turn; the last kBirthCtas place the births.  No CTA
// waits for another, and the longest chain is that of an instance's state: 12
// us a step at 256 cells with the whole deposit and the Poisson sums in that
// CTA, 16 at 4096 and 39 at 21832; 8, 10 and 11 spread like this, births
// included.  mode 1: plan only (one CTA).
__global__ void __launch_bounds__(kFinThreads) k_finish(DeviceRefs r, int mode, int n_field) {
  __shared__ long long s_i64[32];
  __shared__ __int128 s_i128[32];
  __shared__ StateShared sh;
  __shared__ uint32_t s_pre[kFinThreads];
  __shared__ int s_flag;
  step_kernel_entry();
  Control* ctrl = r.ctrl;
  const int t = threadIdx.x;
  if (mode == 1) {
    for (int sg = t; sg < 2 * r.n_inst; sg += kFinThreads) r.xfer[sg].compact = 0;
    __syncthreads();
    plan_next(r, s_i64);
    return;
  }
  if (*((volatile int*)&ctrl->error)) return;
  int b = blockIdx.x;
  if (b >= r.n_inst) {
    b -= r.n_inst;
    if (b < n_field) {
      for (int u = b; u < r.field_start[r.n_inst]; u += n_field) {
        const int inst = field_inst(r, u);
        const InstDev& P = r.inst[inst];
        // (with an imposed field nothing was deposited: the deposit is formed
        // from the markers when it is read)
        if (P.field_mode == 1) finish_nodes(P, u - r.field_start[inst], s_i64, s_i128);
      }
    } else if (r.fp64) {
      place_births<double>(r, b - n_field, kBirthCtas, s_pre, s_i64);
    } else {
      place_births<float>(r, b - n_field, kBirthCtas, s_pre, s_i64);
    }
    return;
  }
  const unsigned int room = finish_state(r, b, sh);
  if (r.n_inst == 1) {
    if (t == 0) plan_single(r, sh, room);
    return;
  }
  // ---- the last instance plans the next step ---------------------------------
  __threadfence();
  __syncthreads();
  if (t == 0) {
    const unsigned int ticket = atomicAdd(&ctrl->finish_done, 1u);
    s_flag = ticket == (unsigned int)r.n_inst - 1u ? 1 : 0;
  }
  __syncthreads();
  if (s_flag) {
    __threadfence();
    plan_next(r, s_i64);
  }
}

// The deposit of instance inst's live markers into its last-step grids
// (zeroed by the caller): each marker adds fixed_charge(beta(|v|) w_j) at its
// position, as the step deposits it.  A step's deposit is a function of the
// markers after it, so with an imposed field it is formed here, when read,
// instead of during every step.  CTA b takes its share of the tiles of each
// species, one warp per tile, into a copy of the grid in shared memory when
// its markers outnumber the nodes (smem != 0): with every marker's two adds
// going to the same few lines of global memory 8e6 markers on 4097 nodes took
// 280 us, 87 with the copies.
constexpr int kDepositThreads = 512;
template <typename R>
__global__ void __launch_bounds__(kDepositThreads) k_deposit(DeviceRefs r, int inst, int smem) {
  extern __shared__ unsigned long long s_rho[];
  const InstDev& P = r.inst[inst];
  const StepConsts<R>& K = consts<R>(P);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nn = P.n_cells + 1;
  for (int sp = 0; sp < 2; ++sp) {
    const SpeciesState st = r.sstate[inst * 2 + sp];
    const uint32_t k0 = (uint32_t)((unsigned long long)blockIdx.x * st.n_tiles / gridDim.x);
    const uint32_t k1 = (uint32_t)((unsigned long long)(blockIdx.x + 1) * st.n_tiles / gridDim.x);
    if (k0 == k1) continue;
    const Markers<R> mk{P.sp[sp].buf[st.cur]};
    const uint32_t* const fill = P.sp[sp].fill[st.cur];
    const R vlim = K.vlim[sp];
    const bool limited = vlim < (R)INFINITY;
    unsigned long long* const g = reinterpret_cast<unsigned long long*>(P.rho_last[sp]);
    unsigned long long* const rho = smem ? s_rho : g;
    if (smem) {
      for (int k = threadIdx.x; k < nn; k += kDepositThreads) s_rho[k] = 0ull;
      __syncthreads();
    }
    for (uint32_t k = k0 + warp; k < k1; k += kDepositThreads / 32) {
      const uint32_t n = fill[k];
      for (uint32_t i = lane; i < n; i += 32) {
        const Slot<R> m = mk.at(k, i);
        R b = (R)1;
        if (limited) {
          const R vx = m.vx(), vy = m.vy(), vz = m.vz();
          b = beta_any(vx * vx + vy * vy + vz * vz, vlim);
        }
        deposit(rho, m.cell(), m.off(), fixed_charge(b * m.wj(), K.wscale));
      }
    }
    if (smem) {
      __syncthreads();
      for (int k = threadIdx.x; k < nn; k += kDepositThreads)
        if (s_rho[k]) atomicAdd(g + k, s_rho[k]);
      __syncthreads();
    }
  }
}

template <typename R>
static void launch_deposit_t(const DeviceRefs& r, int inst, int n_tiles, int n_nodes, int sms,
                             cudaStream_t s) {
  const int most = sms * 2;
  const int grid = std::max(1, std::min((n_tiles + 15) / 16, most));
  // two CTAs per SM hold a copy each while it fits
  const size_t bytes = (size_t)n_nodes * 8;
  const bool smem = bytes <= kDepositSmem && (long long)n_tiles * kTile / grid >= n_nodes;
  k_deposit<R><<<grid, kDepositThreads, smem ? bytes : 0, s>>>(r, inst, smem ? 1 : 0);
}

void launch_deposit(const DeviceRefs& r, int inst, int n_tiles, int n_nodes, int sms,
                    cudaStream_t s) {
  if (r.fp64) launch_deposit_t<double>(r, inst, n_tiles, n_nodes, sms, s);
  else launch_deposit_t<float>(r, inst, n_tiles, n_nodes, sms, s);
}

int deposit_config(int fp64) {
  return (int)(fp64 ? cudaFuncSetAttribute(k_deposit<double>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kDepositSmem)
                    : cudaFuncSetAttribute(k_deposit<float>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kDepositSmem));
}

// The potential of instance inst from its last deposit (read only when the
// field is read), block by block like the field: the blocks' sums first, then
// phi_k = k D_1 - C J_k, J_k = sum_{0<i<=k} I_i, with J at a block's first node
// k_b = sum (k_b - j) net_j = sum over the blocks before of W - (N - k_b) S.
// (By one CTA over the whole grid 4096 cells took 14 us and 21832 69.)
__global__ void __launch_bounds__(kFinThreads) k_phi_sums(DeviceRefs r, int inst) {
  __shared__ long long s_i64[32];
  __shared__ __int128 s_i128[32];
  const InstDev& P = r.inst[inst];
  const int k = blockIdx.x * kFieldNodes + (int)threadIdx.x, N = P.n_cells;
  const long long net = k > 0 && k < N ? P.rho_last[kIon][k] - P.rho_last[kElectron][k] : 0ll;
  block_sums(P, blockIdx.x, net, N - k, s_i64, s_i128);
}

__global__ void __launch_bounds__(kFinThreads) k_phi(DeviceRefs r, int inst) {
  __shared__ long long s_i64[32];
  __shared__ __int128 s_i128[32];
  __shared__ __int128 s_J;
  __shared__ long long s_S;
  __shared__ double s_D1;
  const InstDev& P = r.inst[inst];
  const int kb = blockIdx.x * kFieldNodes, k = kb + (int)threadIdx.x, N = P.n_cells;
  const long long net = k > 0 && k < N ? P.rho_last[kIon][k] - P.rho_last[kElectron][k] : 0ll;
  if (threadIdx.x < 32) {
    const int nb = N / kFieldNodes + 1;
    long long S = 0;
    __int128 W = 0, J = 0;
    for (int b = threadIdx.x; b < nb; b += 32) {
      if (b < (int)blockIdx.x) {
        S += P.pois_S[b];
        J += P.pois_W[b] - (__int128)P.pois_S[b] * (N - kb);
      }
      W += P.pois_W[b];
    }
    S = warp_sum(S);
    J = warp_sum(J);
    W = warp_sum(W);
    if (threadIdx.x == 0) {
      s_S = S;
      s_J = J;
      s_D1 = (P.V + P.pois_C * (double)W) / (double)N;
    }
  }
  const long long inc = block_incl_scan<long long>(net, s_i64);  // (ends with a barrier)
  const long long I = s_S + inc - net;                           // I_k
  // J_k = J_kb + sum_{kb<i<=k} I_i
  const __int128 J = s_J + block_incl_scan<__int128>(threadIdx.x ? (__int128)I : (__int128)0, s_i128);
  if (k > N) return;
  P.phi[k] = k == 0 ? 0.0 : k == N ? P.V : (double)k * s_D1 - P.pois_C * (double)J;
}

void launch_phi(const DeviceRefs& r, int inst, int n_cells, cudaStream_t s) {
  const int blocks = n_cells / kFieldNodes + 1;
  k_phi_sums<<<blocks, kFinThreads, 0, s>>>(r, inst);
  k_phi<<<blocks, kFinThreads, 0, s>>>(r, inst);
}

__global__ void __launch_bounds__(256) k_vacuum(double* phi, double* E64, float* E32, int N,
                                                double V, double E, float Ef) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k > N) return;
  phi[k] = V * k / N;
  E64[k] = E;
  E32[k] = Ef;
}

void launch_vacuum(const InstDev& P, double E, float E32, cudaStream_t s) {
  k_vacuum<<<P.n_cells / 256 + 1, 256, 0, s>>>(P.phi, P.E64, P.E32, P.n_cells, P.V, E, E32);
}

__global__ void __launch_bounds__(256) k_fills(uint32_t* fill, uint32_t first, uint32_t last,
                                               uint32_t end) {
  const uint32_t k = first + blockIdx.x * blockDim.x + threadIdx.x;
  if (k < last) fill[k] = min(end - k * (uint32_t)kTile, (uint32_t)kTile);
}

void launch_fills(uint32_t* fill, uint32_t first, uint32_t end, cudaStream_t s) {
  const uint32_t last = end / kTile + (end % kTile != 0);
  if (last > first) k_fills<<<(last - first + 255) / 256, 256, 0, s>>>(fill, first, last, end);
}

// Exclusive prefix of the fills by one CTA (when markers are read).
__global__ void __launch_bounds__(kFinThreads) k_prefix(const uint32_t* fill, uint32_t n,
                                                        uint32_t* prefix, uint32_t* total) {
  __shared__ long long s_i64[32];
  const uint32_t chunk = (n + kFinThreads - 1) / kFinThreads;
  const uint32_t k0 = min(threadIdx.x * chunk, n), k1 = min(k0 + chunk, n);
  long long loc = 0;
  for (uint32_t k = k0; k < k1; ++k) loc += fill[k];
  const long long inc = block_incl_scan<long long>(loc, s_i64);
  long long run = inc - loc;
  for (uint32_t k = k0; k < k1; ++k) {
    prefix[k] = (uint32_t)run;
    run += fill[k];
  }
  if (threadIdx.x == kFinThreads - 1) *total = (uint32_t)inc;
}

void launch_prefix(const uint32_t* fill, uint32_t n_tiles, uint32_t* prefix, uint32_t* total,
                   cudaStream_t s) {
  k_prefix<<<1, kFinThreads, 0, s>>>(fill, n_tiles, prefix, total);
}

void launch_finish(const DeviceRefs& r, int mode, cudaStream_t s) {
  const int n_field = std::min(r.n_field, kFieldCtas);
  const int grid = mode == 1 ? 1 : r.n_inst + n_field + kBirthCtas;
  launch_step_kernel(k_finish, grid, kFinThreads, 0, s, r, mode, n_field);
}

// ---------------------------------------------------------------------------
// Repacking of the stores k_finish marked sparse: chunks of kMoveChunkTiles
// tiles, handed out in order; each chunk's destination is the prefix of the
// fills of the tiles before it (ordered scan with decoupled look-back); the
// live markers keep their order.  The chunk also writes the fills of the
// repacked store for the tiles with its indices.
// ---------------------------------------------------------------------------
template <typename R>
__global__ void __launch_bounds__(kMoveThreads) k_move(DeviceRefs r) {
  __shared__ uint32_t s_fill[kMoveChunkTiles];
  __shared__ uint32_t s_pre[kMoveChunkTiles];
  __shared__ unsigned int s_chunk;
  __shared__ FieldShared s_field;
  constexpr int kPerLaneTiles = kMoveChunkTiles / 32;
  step_kernel_entry();
  Control* ctrl = r.ctrl;
  // (as one: a wait of another CTA that runs out may set the word between two
  // threads' reads of it, and the chunks are handed out by thread 0)
  if (__syncthreads_or(*((volatile int*)&ctrl->error))) return;
  // the field of the step's Poisson solves, a block of nodes at a time
  for (int u = blockIdx.x; u < r.n_field; u += gridDim.x) {
    const int inst = field_inst(r, u);
    if (r.inst[inst].field_mode == 1) poisson_field(r.inst[inst], u - r.field_start[inst], s_field);
  }
  const unsigned int n_chunks = ctrl->n_move_chunks;
  if (n_chunks == 0) return;
  const unsigned int epoch = ctrl->epoch;
  const int n_seg = r.n_inst * 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (;;) {
    if (threadIdx.x == 0) s_chunk = atomicAdd(&ctrl->move_counter, 1u);
    __syncthreads();
    const unsigned int c = s_chunk;
    if (c >= n_chunks) break;
    int seg = 0;
    {
      int lo = 0, hi = n_seg - 1;  // last segment with move_start <= c
      while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (r.move_start[mid] <= c) lo = mid;
        else hi = mid - 1;
      }
      seg = lo;
    }
    const Transfer& x = r.xfer[seg];
    const SpeciesDev& S = r.inst[seg >> 1].sp[seg & 1];
    const unsigned int first = r.move_start[seg];
    const uint32_t k0 = (c - first) * kMoveChunkTiles;
    for (int j = threadIdx.x; j < kMoveChunkTiles; j += kMoveThreads) {
      const uint32_t k = k0 + j;
      s_fill[j] = k < x.n_tiles_old ? S.fill[x.src][k] : 0u;
    }
    __syncthreads();
    if (warp == 0) {
      // lane l sums tiles l * kPerLaneTiles ..; scan over the lanes
      uint32_t loc = 0;
      for (int j = 0; j < kPerLaneTiles; ++j) loc += s_fill[lane * kPerLaneTiles + j];
      uint32_t inc = loc;
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(0xFFFFFFFFu, inc, o);
        if (lane >= o) inc += n;
      }
      const uint32_t agg = __shfl_sync(0xFFFFFFFFu, inc, 31);
      const uint32_t excl = chunk_lookback(r.move_scan, c, first, agg, epoch, ctrl);
      uint32_t run = excl + inc - loc;
      for (int j = 0; j < kPerLaneTiles; ++j) {
        s_pre[lane * kPerLaneTiles + j] = run;
        run += s_fill[lane * kPerLaneTiles + j];
      }
    }
    __syncthreads();
    // one warp per tile, in order of the tiles
    const Markers<R> src{S.buf[x.src]}, dst{S.buf[x.dst]};
    for (int j = warp; j < kMoveChunkTiles; j += kMoveThreads / 32) {
      const uint32_t n = s_fill[j];
      const uint32_t to = s_pre[j];
      for (uint32_t i = lane; i < n; i += 32) copy_marker(dst[to + i], src.at(k0 + j, i));
    }
    // fills of the repacked store: full tiles, the last one partial
    const uint32_t nt_new = (x.n_new + kTile - 1) / kTile;
    for (int j = threadIdx.x; j < kMoveChunkTiles; j += kMoveThreads) {
      const uint32_t k = k0 + j;
      if (k < nt_new) S.fill[x.dst][k] = min(x.n_new - k * (uint32_t)kTile, (uint32_t)kTile);
    }
    __syncthreads();
  }
}

void launch_move(const DeviceRefs& r, int grid, cudaStream_t s) {
  if (r.fp64) launch_step_kernel(k_move<double>, grid, kMoveThreads, 0, s, r);
  else launch_step_kernel(k_move<float>, grid, kMoveThreads, 0, s, r);
}

// ---------------------------------------------------------------------------
// Seeding: n markers appended at index base = n_live of the species, drawn
// from Philox with counter (id, 0xFFFFFFFF, inst * 2 + species, block).
// ---------------------------------------------------------------------------
template <typename R>
__global__ void k_seed(DeviceRefs r, int inst, int sp, uint32_t base, uint32_t first_id,
                       uint32_t n, int mode, double ekin_d, double elo_d, double lr_d,
                       double wj_d) {
  const uint32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const InstDev& P = r.inst[inst];
  const SpeciesDev& S = P.sp[sp];
  const StepConsts<R>& K = consts<R>(P);
  const Markers<R> d{S.buf[r.sstate[inst * 2 + sp].cur]};
  const R ekin = (R)ekin_d, elo = (R)elo_d, lr = (R)lr_d, wj = (R)wj_d;
  const uint32_t id = first_id + i;
  R u[4];
  uniform4<R>(philox4x32_10(make_uint4(id, kSeedStep, P.ctr_inst * 2u + (uint32_t)sp, 0u),
                            P.key0, P.key1),
              u);
  int cell = 0;
  R off = (R)0, vx = (R)0, vy = (R)0, vz = (R)0;
  const int N = P.n_cells;
  if (mode == 0) {
    off = u[0];
    const R v = r_sqrt(ekin * K.K_V[sp]);
    const R ct = u[1];
    const R st = r_sqrt(r_max((R)0, ((R)1 - ct) * ((R)1 + ct)));
    const R ph = K.two_pi * u[2];
    vx = v * ct;
    vy = v * (st * r_cos(ph));
    vz = v * (st * r_sin(ph));
  } else if (mode == 2 || mode == 3) {
    const R p = u[0] * (R)N;
    const R fl = r_floor(p);
    cell = (int)fl;
    off = p - fl;
    if (cell >= N) {
      cell = N - 1;
      off = nextafter_below_one<R>();
    }
    if (mode == 2) {
      const R e = elo * r_exp(u[1] * lr);
      isotropic(r_sqrt(e * K.K_V[sp]), u[2], u[3], K.two_pi, vx, vy, vz);
    } else {
      R g[4];
      uniform4<R>(philox4x32_10(make_uint4(id, kSeedStep, P.ctr_inst * 2u + (uint32_t)sp, 1u),
                                P.key0, P.key1),
                  g);
      // gas-temperature Maxwellian of this species
      const R sig = ekin;  // sqrt(k T / m), passed in ekin for this mode
      const R r1 = r_sqrt((R)-2 * r_log(u[1]));
      const R r2 = r_sqrt((R)-2 * r_log(u[3]));
      const R a1 = K.two_pi * u[2], a2 = K.two_pi * g[0];
      vx = sig * (r1 * r_cos(a1));
      vy = sig * (r1 * r_sin(a1));
      vz = sig * (r2 * r_cos(a2));
    }
  }
  write_marker(d[base + i], cell, off, vx, vy, vz, wj, id & kSerialMask);
}

void launch_seed(const DeviceRefs& r, int inst, int species, uint32_t base, uint32_t first_id,
                 uint32_t n, int mode, double e0, double e_lo, double lr, double wj,
                 cudaStream_t s) {
  if (n == 0) return;
  const int threads = 256;
  const unsigned int grid = (n + threads - 1) / threads;
  if (r.fp64)
    k_seed<double><<<grid, threads, 0, s>>>(r, inst, species, base, first_id, n, mode, e0, e_lo,
                                           lr, wj);
  else
    k_seed<float><<<grid, threads, 0, s>>>(r, inst, species, base, first_id, n, mode, e0, e_lo,
                                          lr, wj);
}

// Copy a caller's markers into a tiled store and check them (cell in [0, N),
// offset in [0, 1), finite velocities, non-negative weight below 2^39 charge
// units); records the smallest bad index in *bad and the fixed-point sum of
// the weights in *wsum.  One pass: each marker is read and written once, and a
// CTA adds its weights once (an add per warp to the one sum took 4e6 markers
// from 40 to 97 us).
template <typename R>
__global__ void __launch_bounds__(256) k_place(SoAT<R> src, Markers<R> dst, uint32_t n, int N,
                                               int shift, unsigned int* bad,
                                               unsigned long long* wsum) {
  const R wscale = (R)ldexp(1.0, shift);  // 2^shift, exact
  __shared__ unsigned long long s_w[8];
  unsigned long long w = 0;
  const uint32_t stride = gridDim.x * blockDim.x;
  for (uint32_t i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    const R o = src.f[0][i], x = src.f[1][i], y = src.f[2][i], z = src.f[3][i], wj = src.f[4][i];
    const int c = src.cell[i];
    // the fixed-point weight must stay below 2^39 units so that the 24-bit
    // linear split of the deposit cannot overflow 64 bits
    const bool ok = c >= 0 && c < N && o >= (R)0 && o < (R)1 && isfinite(x) && isfinite(y) &&
                    isfinite(z) && wj >= (R)0 && wj * wscale < (R)549755813888.0;
    if (!ok) atomicMin(bad, i);
    else w += (unsigned long long)fixed_charge(wj, wscale);
    write_marker(dst[i], c, o, x, y, z, wj, src.id[i]);
  }
  for (int o = 16; o > 0; o >>= 1) w += __shfl_down_sync(0xFFFFFFFFu, w, o);
  if ((threadIdx.x & 31) == 0) s_w[threadIdx.x >> 5] = w;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < 8; ++k) w += s_w[k];
    if (w) atomicAdd(wsum, w);
  }
}

template <typename R>
static void place(const void* const src[7], unsigned char* buf, uint32_t n, int N, int shift,
                  unsigned int* bad, unsigned long long* wsum, cudaStream_t s) {
  SoAT<R> a;
  a.cell = static_cast<const int32_t*>(src[0]);
  for (int k = 0; k < 5; ++k) a.f[k] = static_cast<const R*>(src[1 + k]);
  a.id = static_cast<const uint32_t*>(src[6]);
  k_place<R><<<std::min((n + 255) / 256, 4096u), 256, 0, s>>>(a, Markers<R>{buf}, n, N, shift, bad, wsum);
}

void launch_place(int fp64, const void* const src[7], unsigned char* buf, uint32_t n, int N,
                  int shift, unsigned int* bad, unsigned long long* wsum, cudaStream_t s) {
  if (n == 0) return;
  if (fp64) place<double>(src, buf, n, N, shift, bad, wsum, s);
  else place<float>(src, buf, n, N, shift, bad, wsum, s);
}

// The live markers of a tiled store, in store order, into seven arrays (one
// warp per tile).
template <typename R>
__global__ void __launch_bounds__(256) k_gather(Markers<R> src, const uint32_t* fill,
                                                const uint32_t* prefix, uint32_t n_tiles,
                                                int32_t* cell, R* off, R* vx, R* vy, R* vz,
                                                R* wj, uint32_t* id) {
  const int lane = threadIdx.x & 31;
  const uint32_t k = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (k >= n_tiles) return;
  const uint32_t n = fill[k], to = prefix[k];
  for (uint32_t i = lane; i < n; i += 32) {
    const Slot<R> m = src.at(k, i);
    const size_t o = to + i;
    cell[o] = m.cell();
    off[o] = m.off();
    vx[o] = m.vx();
    vy[o] = m.vy();
    vz[o] = m.vz();
    wj[o] = m.wj();
    id[o] = m.id();
  }
}

template <typename R>
static void gather(const unsigned char* buf, const uint32_t* fill, const uint32_t* prefix,
                   uint32_t n_tiles, void* const d[7], cudaStream_t s) {
  k_gather<R><<<(n_tiles + 7) / 8, 256, 0, s>>>(
      Markers<R>{const_cast<unsigned char*>(buf)}, fill, prefix, n_tiles,
      static_cast<int32_t*>(d[0]), static_cast<R*>(d[1]), static_cast<R*>(d[2]),
      static_cast<R*>(d[3]), static_cast<R*>(d[4]), static_cast<R*>(d[5]),
      static_cast<uint32_t*>(d[6]));
}

void launch_gather(int fp64, const unsigned char* buf, const uint32_t* fill,
                   const uint32_t* prefix, uint32_t n_tiles, void* const dst[7], cudaStream_t s) {
  if (n_tiles == 0) return;
  if (fp64) gather<double>(buf, fill, prefix, n_tiles, dst, s);
  else gather<float>(buf, fill, prefix, n_tiles, dst, s);
}

__global__ void k_philox(uint32_t k0, uint32_t k1, const uint4* ctr, uint4* out, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = philox4x32_10(ctr[i], k0, k1);
}

__global__ void k_philox2(uint32_t k, const uint2* ctr, uint2* out, long long n) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = philox2x32_10(ctr[i], k);
}

void launch_philox2(uint32_t k, const uint32_t* ctr, uint32_t* out, long long n,
                    cudaStream_t s) {
  if (n <= 0) return;
  const int threads = 256;
  const long long grid = (n + threads - 1) / threads;
  k_philox2<<<(unsigned int)grid, threads, 0, s>>>(k, reinterpret_cast<const uint2*>(ctr),
                                                   reinterpret_cast<uint2*>(out), n);
}

// Load the Philox kernel's module now (CUDA loads modules lazily, and the
// load can reserve device memory).
int philox_preload() {
  cudaFuncAttributes a;
  return (int)cudaFuncGetAttributes(&a, k_philox);
}

void launch_philox(uint32_t k0, uint32_t k1, const uint32_t* ctr, uint32_t* out, long long n,
                   cudaStream_t s) {
  if (n <= 0) return;
  const int threads = 256;
  const long long grid = (n + threads - 1) / threads;
  k_philox<<<(unsigned int)grid, threads, 0, s>>>(k0, k1, reinterpret_cast<const uint4*>(ctr),
                                                  reinterpret_cast<uint4*>(out), n);
}

}  // namespace slpic
