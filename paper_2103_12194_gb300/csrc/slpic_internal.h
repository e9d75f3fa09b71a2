// Internal device-side layout shared by the kernels and the host driver of
// libslpic.  Nothing here is part of the public ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace slpic {

constexpr int kElectron = 0;
constexpr int kIon = 1;
constexpr uint32_t kGenBit = 0x80000000u;
constexpr uint32_t kSerialMask = 0x7FFFFFFFu;
constexpr uint32_t kSeedStep = 0xFFFFFFFFu;

// Marker stores are sequences of tiles of kTile slots.  The particle kernel
// gives every tile to one warp, which advances it in kHalves passes of
// kPerHalf neighbouring slots per lane; a warp streams its tiles through
// kPushStages shared-memory stages.
constexpr int kTile = 128;
constexpr int kPerLane = kTile / 32;
constexpr int kPushMaxWarps = 20;
constexpr int kPushStages = 2;
constexpr int kHalves = 2;
constexpr int kPerHalf = kPerLane / kHalves;
// A tile is one block of memory: its seven fields in runs of kTile values, in
// the order cell, off, vx, w_j, id, vy, vz (cell and id of 4 bytes, the others
// reals).  All fields of a slot are at constant distances from one address,
// and what a step of unlimited ions reads is the front of the block (up to vx,
// or w_j when the step deposits; electrons need all): the particle kernel
// fetches a tile with one bulk copy and forms one address per tile.  With the fields in seven
// arrays of the whole store the copies and addresses took a quarter of its
// instructions.
template <typename R>
__host__ __device__ constexpr size_t tile_bytes() {
  return kTile * (8 + 5 * sizeof(R));
}
template <typename R>
__host__ __device__ constexpr size_t tile_bytes_read(bool all, bool w) {
  return all ? tile_bytes<R>() : kTile * (4 + (w ? 3 : 2) * sizeof(R));
}
// Relative cost of a tile of each species in the particle kernel's static
// split of the tiles over the CTAs.  (4 : 5, and 4 : 8 under a speed limit,
// nearer to the instruction counts, ran the same on shared-memory grids and
// 18 % slower on a grid of 21832 cells, whose ions wait for global atomics.)
constexpr unsigned int kWeightElectron = 3;
constexpr unsigned int kWeightIon = 2;
constexpr unsigned int kSegCost = 48;

// Device error word values (copied to the host status codes).
constexpr int kErrNone = 0;
constexpr int kErrCapacity = 1;
constexpr int kErrTimeout = 2;
constexpr int kErrIdWrap = 3;

// Bounded waits: polls before a wait gives up with kErrTimeout (each poll of
// an mbarrier suspends the thread for up to about a microsecond), unless the
// context sets another limit (Control::spin_limit).
constexpr uint32_t kSpinLimit = 1u << 22;

// Per-step accumulators of one instance (integer; weights in fixed point).
enum Acc : int {
  ACC_CAND = 0,
  ACC_COLL0,  // elastic
  ACC_COLL1,  // excitation
  ACC_COLL2,  // ionization
  ACC_SEE,
  ACC_NABS,        // 4 entries: [species][electrode]
  ACC_WABS = ACC_NABS + 4,
  ACC_WSEE = ACC_WABS + 4,
  ACC_WIONZ,
  ACC_WCATH,
  ACC_WCATH0,
  ACC_CLAMP,
  ACC_MAJ,
  ACC_MSTEPS,
  ACC_GWCATH0,  // yield * w_j of first-generation ions at the cathode
  ACC_COUNT
};

// Record of one step, converted (same layout as slpic_tallies).
struct TallyRec {
  long long step;
  long long n_live[2];
  double w_live[2];
  long long n_coll[3];
  long long n_candidates;
  long long n_abs[2][2];
  double w_abs[2][2];
  long long n_see;
  double w_see;
  double w_ionz;
  double w_cath_ion;
  double w_cath_ion_gen0;
  long long n_clamp;
  long long n_majorant;
  long long marker_steps;
  double w_gain_gen0;
};

// A caller's markers: one array per field, the five reals in the marker
// path's type R (float in FP32 contexts, double in FP64 contexts).
template <typename R>
struct SoAT {
  const int32_t* cell;
  const R* f[5];  // off, vx, vy, vz, w_j
  const uint32_t* id;
};

// The fields of one slot of a tiled store.
template <typename R>
struct Slot {
  int32_t* c;
  R* r;
  static constexpr int kPer4 = sizeof(R) / 4;        // 4-byte words per real
  static constexpr int kV = 3 * kTile + kTile / kPer4;  // reals from off to vy
  __host__ __device__ __forceinline__ int32_t& cell() const { return c[0]; }
  __host__ __device__ __forceinline__ R& off() const { return r[0]; }
  __host__ __device__ __forceinline__ R& vx() const { return r[kTile]; }
  __host__ __device__ __forceinline__ R& wj() const { return r[2 * kTile]; }
  __host__ __device__ __forceinline__ uint32_t& id() const {
    return reinterpret_cast<uint32_t*>(c)[kTile + 3 * kTile * kPer4];
  }
  __host__ __device__ __forceinline__ R& vy() const { return r[kV]; }
  __host__ __device__ __forceinline__ R& vz() const { return r[kV + kTile]; }
};

// A tiled store in the marker path's type.
template <typename R>
struct Markers {
  unsigned char* b;
  // slot i of tile k
  __host__ __device__ __forceinline__ Slot<R> at(size_t k, uint32_t i) const {
    unsigned char* p = b + k * tile_bytes<R>();
    return Slot<R>{reinterpret_cast<int32_t*>(p) + i, reinterpret_cast<R*>(p + kTile * 4) + i};
  }
  // slot o of the store
  __host__ __device__ __forceinline__ Slot<R> operator[](uint32_t o) const {
    return at(o / kTile, o % kTile);
  }
};

// Processes of an electron collision: elastic, up to three excitation
// levels, ionization.
constexpr int kMaxExc = 3;
constexpr int kMaxProc = kMaxExc + 2;

// One node of the FP64 cross-section table: the cumulative cross sections of
// the processes in order, and a pad.
struct alignas(64) TabNode64 {
  double s[kMaxProc];
  double pad[8 - kMaxProc];
};

// Constants of the step in the marker path's arithmetic type R; the host
// derives both sets from the same double-precision configuration.
template <typename R>
struct StepConsts {
  R qmdt[2];      // (q / m) dt per species
  R vlim[2];      // speed limit per species (+inf: beta = 1)
  R K_V[2];       // 2 e / m: speed^2 per eV, per species
  R dtdx;         // dt / dx
  R K_E;          // m_e / (2 e): eV per (m/s)^2
  R ndt;          // n_g dt
  R P0;           // null-collision majorant probability
  uint32_t cand_thr;  // a draw's top 23 bits are below it exactly when u < P0
  R vb_cap;       // cap of beta v in the majorant
  R R2;           // 2 m_e / M
  R e_ex[kMaxExc];  // excitation thresholds [eV]
  R e_io;           // ionization threshold [eV]
  R sigT_ion;     // sqrt(k T / M)
  R K_Ei;         // M / (2 e): eV per (m/s)^2 of an ion
  R gamma;        // secondary-emission yield
  R wscale;       // 2^charge_shift
  R two_pi;
  R e_lo, e_hi;   // table range [eV]
};

// Marker store of one (instance, species): a sequence of tiles of kTile
// slots; tile k holds fill[k] live markers in its first slots, in order.  The
// particle kernel compacts each tile in place (no dependence between tiles);
// births are appended after the last live marker; when the tiles become
// sparse the whole store is repacked into the other buffer.
//
// Mutable per-(instance, species) state, resident on the device.
struct SpeciesState {
  uint32_t cur;       // buffer holding the markers
  uint32_t n_tiles;   // tiles in use
  uint32_t n_live;    // live markers (sum of the fills)
  uint32_t next_id;   // next serial number
};

// Repacking of one segment at the end of a step (decided by k_finish,
// done by k_move).
struct Transfer {
  uint32_t compact;       // repack the tiles of buffer src into buffer dst
  uint32_t src, dst;
  uint32_t n_tiles_old;   // tiles to repack
  uint32_t n_new;         // live markers after the step
  uint32_t tail;          // first slot the step's births went to
  uint32_t end;           // one past the last birth
  uint32_t pad;
};

// A null-collision candidate as the particle kernel leaves it: the electron's
// state after its push and its slot in the tile after compaction (once it has
// ionized, vx holds the energy given to the secondary).  One record fills a
// 32-byte sector in float, so the collision kernel reads a candidate with one
// sector instead of one per field.
template <typename R>
struct CandRec;
template <>
struct alignas(32) CandRec<float> {
  int cell;
  float off, vx, vy, vz, wj;
  uint32_t id, slot;
};
template <>
struct alignas(16) CandRec<double> {
  int cell;
  uint32_t id;
  double off, vx, vy, vz, wj;
  uint32_t slot, pad;
};
static_assert(sizeof(CandRec<float>) == 32, "one sector per float record");

// Configuration of one species of one instance (constant during a run).
struct SpeciesDev {
  unsigned char* buf[2];  // tiled marker store (cap_tiles tiles each; see Markers)
  uint32_t* fill[2];  // [cap_tiles] live markers per tile of each buffer
  void* stage_w;      // electrons only: w_j of the electrons emitted at the cathode
                      // (at rest at x = 0), slot = ion tile * kTile + rank
  uint32_t* births;   // ions: [cap_tiles] electrons emitted by each tile in the step
  void* crec;         // electrons: [cap_tiles * kTile] CandRec<R>, the tile's
                      // null-collision candidates in slot order (during a step
                      // the buffer that is not in use holds, from an item's
                      // first slot on, the numbers of its ionizations' records,
                      // and that of the ions where its emissions are staged)
  uint32_t* n_cand;   // electrons: [cap_tiles] candidates per tile
  uint32_t cap_tiles;
  uint32_t pad;
};

// Configuration of one instance (constant during a run).
struct InstDev {
  int n_cells;
  int field_mode;
  int charge_shift;
  int tab_lo_exp2;
  int tab_log2_sub;
  int tab_nodes;      // real nodes (a padding node follows)
  uint32_t key0, key1;
  uint32_t ctr_inst;  // counter word 2 = ctr_inst * 2 + species
  uint32_t key2;      // Philox2x32 key of the null-collision draw
  int n_exc;          // excitation levels (1..kMaxExc)
  int tab_stride;     // float4s per node of the FP32 table (1, or 2 with more levels)
  int emission_model; // 0: constant gamma; 1: Eq. sey
  int emit;           // 0: tally the yield, emit no electron
  StepConsts<float> c32;
  StepConsts<double> c64;
  double dx, d, V, area, dt;
  double pois_C;      // e dx 2^-shift / (area eps0)
  const float4* table;          // FP32: cumulative cross sections per node, n_exc + 2 of them, in tab_stride float4s
  const TabNode64* table64;     // FP64: the same in double
  float* E32;                   // node field used by the FP32 push
  double* phi;                  // node potential
  double* E64;                  // node field
  long long* pois_S;            // per block of kFieldNodes nodes: net charge of the last step
  __int128* pois_W;             // and its sum weighted by N - node
  unsigned long long* rho_acc[2];  // fixed-point deposit of the current step
  long long* rho_last[2];          // deposit of the last finished step
  unsigned long long* acc;         // ACC_COUNT per-step accumulators
  TallyRec* ring;                  // per-step records
  TallyRec* total;                 // sums since the last reset
  int ring_len;
  int pad;
  SpeciesDev sp[2];
};

// Mutable per-instance counters.
struct InstState {
  uint32_t step;        // step index (Philox counter word 1)
  uint32_t pad;
  long long n_steps_done;
  unsigned long long w_seed;     // fixed-point sum of seeded electron weights
  unsigned long long w_live[2];  // fixed-point sum of live weights per species
  long long ion_steps;           // sum over the steps of the live ions after each
};

// Global state of the batched step.
struct Control {
  unsigned int epoch;        // step epoch of the look-back records
  unsigned int n_tiles;      // particle-kernel tiles this step
  unsigned int w_total;      // their summed weights
  unsigned int seg_cost;     // of which for starting a segment that is not empty
  unsigned int n_seg;        // segments = instances * 2
  unsigned int finish_done;  // CTAs of the finish kernel that completed
  int error;                 // first device error (kErr*)
  int error_inst;
  unsigned int spin_waits;   // polls that found data not yet there
  unsigned int spin_max;     // longest single wait, in polls
  unsigned int n_coll_items;
  unsigned int move_counter; // next repacking chunk to hand out
  unsigned int n_move_chunks;
  unsigned int small_bar;    // single-CTA path: arrivals at its grid barriers
  int small_stop;            // single-CTA path: a store outgrew it
  long long small_done;      // single-CTA path: steps run by the last launch
  unsigned int spin_limit;   // polls before a bounded wait gives up (0: kSpinLimit)
  int skip_cta;              // test hook: CTA + 1 of the single-CTA path that skips
  long long skip_barrier;    //   its arrival at this grid barrier (0: none)
};

// Look-back record of one chunk of an ordered scan.
struct ChunkStatus {
  unsigned int flag;  // (epoch << 2) | state; state 1 = aggregate, 2 = inclusive
  unsigned int agg;
  unsigned int incl;
  unsigned int pad;
};

// Collision items, one warp each: consecutive tiles of one instance, electron
// items of coll_tiles[inst] tiles and then ion items of kCollIonTiles (the
// electrons emitted at the cathode, rare).  coll_tiles[inst] is at
// most kCollMaxTiles: small enough that an item holds about kCollTarget
// candidates at the instance's last step's density, and, down to a round of 32
// candidates (in double, where the FP64 unit of each SM counts, down to one
// tile), that the instance gives its share of kCollPerSm items per SM
// (DeviceRefs::coll_share).
constexpr int kCollMaxTiles = 32;
constexpr int kCollIonTiles = 256;
constexpr int kCollTarget = 128;
constexpr int kCollPerSm = 16;
// (a bound of the tiles that hold that many candidates)
constexpr int kCollMaxRoom = 64 * kCollMaxTiles;
// CTAs of k_finish beside the instances' own: those that place the births, and
// at most so many for the blocks of nodes.  (4e6 electrons, 1e6 candidates:
// 184 us a step with 16 CTAs, 177 with 32, 172 with 64, 170 with 96; 21833
// nodes: 83 with 64, 84 with 96, 89 with 128.)
constexpr int kBirthCtas = 64;
constexpr int kFieldCtas = 80;
constexpr int kFieldNodes = 1024;
// Repacking chunks: tiles each.
constexpr int kMoveChunkTiles = 128;
// Single-CTA path (small.cu): at most this many tiles per store and instance
// when a step starts.
constexpr int kSmallMaxTiles = 32;

// Where a step's births go in the stores of one instance: buffers, first free
// slots, next serial numbers, step, electron items and their tiles, before the
// step's end moves the state and the plan on.
struct BirthBase {
  uint32_t cur[2], tail[2], next_id[2], step, e_items, tiles;
};

struct DeviceRefs {
  InstDev* inst;          // [n_inst]
  InstState* istate;      // [n_inst]
  SpeciesState* sstate;   // [n_inst * 2]
  Transfer* xfer;         // [n_inst * 2]
  Control* ctrl;
  unsigned int* seg_start;   // [n_seg + 1] first tile of each segment
  unsigned int* seg_wstart;  // [n_seg + 1] summed tile weights before each segment
  unsigned int* coll_start;  // [n_inst + 1] first collision item of each instance
  unsigned int* coll_tiles;  // [n_inst] tiles per electron collision item
  unsigned int* coll_room;   // [n_inst] the most its density of candidates allows
  unsigned int* move_start;  // [n_seg + 1] first repacking chunk of each segment
  uint32_t* item_births;     // [max collision items] births of each item in the step
  BirthBase* birth_base;     // [n_inst]
  unsigned int* birth_start; // [n_inst + 1] coll_start of the step whose births are placed
  int* field_start;          // [n_inst + 1] first block of nodes of each instance
  ChunkStatus* move_scan;    // [max repacking chunks]
  int n_inst;
  int smem_nodes;         // deposit grid nodes in shared memory (0: global atomics)
  int push_warps;         // warps per particle-kernel CTA
  int push_grid;          // its CTAs
  unsigned int coll_share;  // collision items an instance should give at least (see kCollPerSm)
  int coll_nodes;         // collision kernel: deposit grid nodes in shared memory (0: none)
  int fp64;               // marker path in double precision (else float)
  int n_field;            // blocks of kFieldNodes nodes of all instances
};

// Launchers (defined in the .cu files).
void launch_push(const DeviceRefs& r, int grid, cudaStream_t s);
// Particle-kernel shape for a shared-memory deposit grid of smem_nodes nodes:
// warps per CTA and resident CTAs per SM.
int push_config(int fp64, int smem_nodes, int* warps, int* blocks_per_sm);
// Resident particle-kernel CTAs per SM for `warps` warps per CTA.
int push_blocks_per_sm(int fp64, int warps, int smem_nodes, int* blocks_per_sm);
// mode 0: finish a step and plan the next; mode 1: plan only (one CTA).
void launch_finish(const DeviceRefs& r, int mode, cudaStream_t s);
void launch_move(const DeviceRefs& r, int grid, cudaStream_t s);
// Node potential of instance inst from its last deposit (Poisson mode).
void launch_phi(const DeviceRefs& r, int inst, int n_cells, cudaStream_t s);
// The vacuum field of an instance: phi = V k / N, E on every node.
void launch_vacuum(const InstDev& P, double E, float E32, cudaStream_t s);
// Fills of tiles [first, ceil(end / kTile)) of a store whose slots from
// first * kTile to end are all live.
void launch_fills(uint32_t* fill, uint32_t first, uint32_t end, cudaStream_t s);
// Markers before each of n_tiles tiles, and (*total) in all of them.
void launch_prefix(const uint32_t* fill, uint32_t n_tiles, uint32_t* prefix, uint32_t* total,
                   cudaStream_t s);
// Deposit of instance inst's live markers (n_tiles tiles of both species)
// added to its last-step grids; used with an imposed field, where the step
// itself deposits nothing.  kDepositSmem: shared memory of a CTA's charge grid.
constexpr size_t kDepositSmem = 100 * 1024;
void launch_deposit(const DeviceRefs& r, int inst, int n_tiles, int n_nodes, int sms,
                    cudaStream_t s);
int deposit_config(int fp64);
// Scatter the null-collision candidates queued by the particle kernel.
void launch_collide(const DeviceRefs& r, int grid, cudaStream_t s);
// Its resident CTAs per SM and the nodes of its shared charge grid (0: deposits
// go to global memory) in a context of grids of up to max_nodes nodes.
int collide_config(int fp64, int max_nodes, int* resident, int* nodes);
// Seeding: n markers written contiguously from slot `base` of the current
// buffer; mode 0/1/2 as SLPIC_SEED_*; for mode 3 (thermal) e0 carries the
// thermal speed sqrt(k T / m).
void launch_seed(const DeviceRefs& r, int inst, int species, uint32_t base, uint32_t first_id,
                 uint32_t n, int mode, double e0, double e_lo, double lr, double wj,
                 cudaStream_t s);
// Copy n markers of a caller's arrays on the device (field order: cell, off,
// vx, vy, vz, w_j, id) into slots 0 .. n - 1 of a tiled store, checking them:
// *bad gets the smallest index of a marker that must not be stepped, *wsum the
// fixed-point sum of the weights.
void launch_place(int fp64, const void* const src[7], unsigned char* buf, uint32_t n, int N,
                  int shift, unsigned int* bad, unsigned long long* wsum, cudaStream_t s);
// The reverse: the live markers of n_tiles tiles, in store order, into seven
// arrays (prefix: live markers before each tile).
void launch_gather(int fp64, const unsigned char* buf, const uint32_t* fill,
                   const uint32_t* prefix, uint32_t n_tiles, void* const dst[7], cudaStream_t s);
int philox_preload();
void launch_philox(uint32_t k0, uint32_t k1, const uint32_t* ctr, uint32_t* out,
                   long long n, cudaStream_t s);
void launch_philox2(uint32_t k, const uint32_t* ctr, uint32_t* out, long long n,
                    cudaStream_t s);
// Single-CTA path: shared memory for field-mode-1 grids of up to
// max_poisson_nodes nodes and resident CTAs per SM (0: does not fit); then up
// to n_steps steps of every instance (one CTA each), stopping before a step
// when a store has more than max_tiles tiles.  Steps run: Control::small_done.
int small_config(int fp64, int max_poisson_nodes, size_t* smem_bytes, int* blocks_per_sm);
int launch_small(const DeviceRefs& r, long long n_steps, int max_tiles, size_t smem_bytes,
                 cudaStream_t s);

}  // namespace slpic
