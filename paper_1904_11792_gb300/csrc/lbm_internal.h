// Host-side internals of liblbm.so: the handle and the kernel launchers each
// translation unit provides.  Not part of the public ABI (include/lbm.h).
#pragma once

#include <cuda_runtime.h>

#include <string>
#include <vector>

#include "lbm.h"
#include "lbm_device.cuh"

namespace lbm {

// Streaming modes of one time step.
enum Mode {
  MODE_AB = 0,      // A-B push: read f_a(x) from src, write f*_a to dst at x + c_a
  MODE_AA_EVEN = 1, // AA even step: read slot a at x, write f*_a to slot opp(a) at x
  MODE_AA_ODD = 2   // AA odd step: read slot opp(a) at x - c_a, write f*_a to slot a at x + c_a
};

// Where the pre-collision population a of node x lives for a given state
// layout: LOCAL = slot a at x (A-B, and AA before an even step); GATHER =
// slot opp(a) at x - c_a (AA before an odd step).
enum Layout { LAYOUT_LOCAL = 0, LAYOUT_GATHER = 1 };

size_t elem_size(int precision);
// Whether the two-kernel step updates two neighbouring nodes per thread
// (vec: option "vector").
bool node_pairs(int precision, bool vec, const Geom& g);

// Where the last stages of a diagnostics reduction run while a graph is
// captured: on a second stream, forked after the kernel that wrote the
// partials, so that the next steps need not wait for these small kernels (two
// or three single launches of a few blocks: 17 us per diagnostic step of
// 64x32x32 FP32 in the steps' own chain, 6 us beside it).  The
// caller waits for `join` (where open) before the next use of the partials and
// at the end of the capture.
struct ReduceSide {
  cudaStream_t stream;
  cudaEvent_t fork, join;
  bool open;
};

// ---- launchers (lbm_step.cu) ---------------------------------------------
// psi pass: psi[i] = psi(rho_i) for all nodes; flag |= 1 on a non-positive
// or non-finite density.
// vec: two nodes per thread with vector accesses (used when nx is even).
// dst: the destination array of an A-B step, whose slot 0 FP64 storage uses
// to hand the densities to the step's collide kernel (required before a FP64
// A-B launch_collide; nullptr otherwise).
cudaError_t launch_psi(int precision, int layout, bool vec, const Geom& g, const Phys& ph,
                       const void* f, void* psi, int* flag, cudaStream_t s, void* dst = nullptr);
// Fills the table of psi_of<double> (kPsiTab entries in device memory).
cudaError_t psi_table_launch(double2* tab, cudaStream_t s);
// fused force + collision + streaming of one step; block has at most 256
// threads (with vec, block.x counts node pairs); minb (2, 3, 4) = blocks per
// SM the register budget must allow.
cudaError_t launch_collide(int precision, int mode, int minb, bool vec, const Geom& g,
                           const Phys& ph, const void* src, void* dst, const void* psi, dim3 block,
                           cudaStream_t s);

// force + collision + streaming of an A-B step into an array with rows px
// elements apart (the first step of a run on padded rows; 4- and 2-byte
// storage, one node per thread).
cudaError_t launch_collide_padded(int precision, const Geom& g, const Phys& ph, const void* src, void* dst, int px,
                                  const void* psi, dim3 block, cudaStream_t s);

// Lattices up to this many nodes run the two kernels by default where the
// fused step applies: their populations stay in L2, and two short passes over
// all nodes at once beat a march through planes by few blocks (plain steps,
// two kernels against single pass: 64x32x32 FP32 5.57 / 7.76 us, FP16 4.85 /
// 10.6; 64x96x96 14.9 / 17.1, 14.2 / 14.8; 128x80x80 24.0 / 22.8, 18.3 / 20.2;
// 256x64x64 32.7 / 31.9, 22.8 / 22.8; 128x96x96 38.3 / 36.1, 27.6 / 26.7; MRT:
// 128x80x80 27.4 / 28.8, 256x64x64 36.6 / 38.3, 192x96x96 69.8 / 57.8).
// kFusedNodes: FP32 and the paper's collision; kFusedNodesLate: the others.
constexpr long long kFusedNodes = 5 << 17, kFusedNodesLate = 1 << 20;
// Lattices up to this many nodes launch their steps chained (lbm_launch.cuh)
// and replay longer graphs: their kernels take a few microseconds each.
constexpr long long kChainNodes = 1 << 20;
// SMs of a GB300: lattices with little work split it to reach them all.
constexpr int kSmCount = 152;

// Default collide-stream block shape of a lattice, as the block_x .. block_z
// options start from, and the shape launched where none was asked for
// (lbm_api.cu).
dim3 default_block(const Geom& g);
dim3 auto_block(const Geom& g, bool pairs, int precision);
// The register budget (minb of launch_collide) launched with where none was
// asked for.
int auto_minb(bool vec, int mode, int precision, long long N);

// force + collision + streaming with the MRT collision (lbm_mrt.cu); the
// same modes and layouts as launch_collide
cudaError_t launch_collide_mrt(int precision, int mode, bool vec, const Geom& g, const Phys& ph,
                               const void* src, void* dst, const void* psi, dim3 block, cudaStream_t s);

// ---- fused single-pass step (lbm_fused.cu) ----------------------------------
// One kernel per A-B step (psi of each tile and its ring computed in shared
// memory); 4- and 2-byte storage, nx % 64 == 0, ny % 4 == 0, nz >= 3.
bool fused_applicable(const Geom& g, int precision);
// fz: z planes per block (0: chosen from the lattice and the GPU).  diag
// (nullable): also reduce the diagnostics of the starting state in the same
// pass and append the record to the ring (or write out[0..DIAG_OUT)); the
// scratch must hold fused_diag_scratch_doubles(g, precision, fz) doubles.
struct FusedDiag {
  double rho_l, rho_v;
  double* scratch;
  size_t scratch_doubles;
  double* out;
  unsigned long long* ring_count;
  int ring_cap;
};
// stall_ns > 0 (test hook): every block also waits that long, bounded, on a
// barrier nothing completes, so the launch takes its timeout path.
// The run length and runs per group the fused step launches with for the
// requested values (0 = automatic).
cudaError_t fused_launch_shape(int precision, const Geom& g, int coll, int fz_req, int grp_req, int* fz, int* grp);
// fz: z planes per block (0 = automatic); grp: z runs per group of the
// block order (0 = automatic).
cudaError_t launch_fused(int precision, const Geom& g, const Phys& ph, const void* src, void* dst,
                         int* flag, int fz, int grp, const FusedDiag* diag, unsigned long long stall_ns,
                         cudaStream_t s, ReduceSide* side = nullptr);
size_t fused_diag_scratch_doubles(const Geom& g, int precision, int fz);

// The single-pass step for lattices that the fused step does not take (any nx
// and ny, 4- and 2-byte storage), on tiles cut at the lattice's edges;
// bitwise the two-kernel step.  TMA needs source rows that start on 16-byte
// boundaries (src_px elements apart; src 16-byte aligned, Q px ny nz
// elements): ragged_row is nx where the lattice's own rows do, else the pitch
// of a padded copy.  dst_px: row pitch of the destination, any.  fz, grp: as
// launch_fused.
// Smaller lattices keep the two kernels by default: they live in L2, where the
// two short passes are as fast or faster (plain steps, two kernels against
// single pass: FP32 150x80x80 33.7 / 36.2 us, 101x100x100 42.2 / 39.7, 180x90x90
// 53.6 / 48.9, 251x128x128 170 / 130; FP16 199x100x100 72 / 76, 251x100x100 87 /
// 87, 251x128x128 136 / 126, 503x200x200 624 / 553); so do rows of less than
// half a tile, and 2-byte storage with even nx, whose two kernels take node
// pairs (FP16 198x120x119 84 / 97, 502x112x112 157 / 173, 504x200x200 468 / 533;
// MRT 502x112x112 197 / 203, 456x256x256 949 / 915).
constexpr long long kRaggedNodes = 1 << 20, kRaggedNodesDev = 5 << 19;
constexpr int kRaggedMinNx = 32;
bool ragged_applicable(const Geom& g, int precision);
int ragged_row(const Geom& g, int precision);
cudaError_t launch_ragged(int precision, const Geom& g, const Phys& ph, const void* src, int src_px, void* dst,
                          int dst_px, int* flag, int fz, int grp, cudaStream_t s);

// ---- auxiliary kernels (lbm_aux.cu) ---------------------------------------
struct InitSpec {
  double R0, lambda, eps, phase, rho_l, rho_v, width;
  const double* prof;  // device table, or nullptr for the tanh profile
  int n;
  double d0, dd;
};
cudaError_t launch_init(int precision, const Geom& g, const Phys& ph, const InitSpec& spec,
                        void* f, cudaStream_t s);
// Canonical FP64 populations to and from a host array of 19 N doubles, through
// `work` (device), which takes as many whole planes at a time as it holds (at
// least one).  Both wait for the stream.  Copies of a few MB into host pages
// that nothing has touched yet cost more than 1 ms each whatever their size,
// so the planes of small lattices cross together (48x48x96, 19 planes of 1.8
// MB one by one: 22 ms; together: 2 ms).
cudaError_t export_populations(int precision, int layout, const Geom& g, const Phys& ph, const void* f, double* work,
                               size_t work_doubles, double* host, cudaStream_t s);
cudaError_t import_populations(int precision, int layout, const Geom& g, const Phys& ph, void* f, double* work,
                               size_t work_doubles, const double* host, cudaStream_t s);
// Doubles of `work` for a lattice of N nodes and `planes` planes: all of them
// up to 64 MiB, at least one.
inline size_t transfer_doubles(long long N, int planes) {
  const size_t cap = (size_t)8 << 20, all = (size_t)planes * N;
  return all <= cap ? all : ((size_t)N > cap ? (size_t)N : cap);
}
// rho and u = (j + F/2)/rho into four FP64 device arrays (psi must be current)
cudaError_t launch_moments(int precision, int layout, const Geom& g, const Phys& ph,
                           const void* f, const void* psi, double* rho, double* ux, double* uy,
                           double* uz, cudaStream_t s);

// Diagnostics reduction.  scratch must hold diag_scratch_doubles(g) doubles.
size_t diag_scratch_doubles(const Geom& g);
// Results: DIAG_OUT doubles, 0 mass, 1-3 momentum, 4 liquid volume (phi),
// 5 liquid count, 6 min slice area (phi), 7 min slice count, 8 its x,
// 9 max |j|/rho, 10 min rho, 11 max rho, 12 numeric ok (1/0).  A ring
// record holds them plus, at DIAG_OUT, its sequence number and, from
// DIAG_CCL, the droplet counts of a step that also ran the labelling
// (components, components >= 8 nodes, largest, guard error; -1 if it did not).
constexpr int DIAG_OUT = 13;
constexpr int DIAG_NG = 12;   // partial slots per block of the diagnostics reduction
constexpr int DIAG_CCL = 14;
constexpr int DIAG_STRIDE = 20;
// psi (nullable): also write psi of every node and raise flag on a bad
// density (the psi pass of a diagnostic step).  ring_count (nullable):
// append the record to the ring at out instead of writing out[0..12].
struct DiagExtra {
  void* dst = nullptr;          // as launch_psi (with psi)
  ReduceSide* side = nullptr;   // where the stages after the pass over the populations run
  int *labels = nullptr, *sizes = nullptr;   // also start the labelling (diag_labels)
  float thr_lo = 0.0f;
};
// The labelling part of a DiagExtra for a pass over f (writing psi, or
// nullptr), empty where the pass has no such form.
DiagExtra diag_labels(int precision, int layout, const Geom& g, const void* f, const void* psi, double threshold,
                      int* labels, int* sizes);
cudaError_t launch_diagnostics(int precision, int layout, const Geom& g, const Phys& ph,
                               const void* f, double rho_l, double rho_v, double* scratch,
                               double* out, void* psi, int* flag,
                               unsigned long long* ring_count, int ring_cap, cudaStream_t s,
                               const DiagExtra& x = {});

// Stochastic-rounding step salt (Phys::salt): set to value, or advance by one.
cudaError_t launch_salt(unsigned* salt, bool set, unsigned value, cudaStream_t s);
// The salt after n steps from the word `from` into the word `to` (the same or
// another one), after a launch that ran them.
cudaError_t launch_salt_add(const unsigned* from, unsigned* to, unsigned n, cudaStream_t s);

// Second and third stage of the diagnostics reduction from partials
// slices[row_blocks][nx][2] and blocks[nblocks][DIAG_NG] (slice_tot: 2 nx
// doubles of scratch; with many block records they are folded in place, so
// blocks is overwritten); arguments after slice_tot as launch_diagnostics.
cudaError_t launch_diag_reduce(const Geom& g, int row_blocks, int nblocks, const double* slices,
                               double* blocks, double* slice_tot, double* out,
                               unsigned long long* ring_count, int ring_cap, cudaStream_t s,
                               ReduceSide* side = nullptr);

// Connected components of the liquid mask.  labels: N ints; sizes: N ints;
// out3 (device, 4 long long): components, components with >= 8 nodes,
// largest size, error flag (a union-find guard tripped).  started: a
// diagnostics pass has started the labels (diag_labels); slots: replace the
// size of every root by its number among the roots (for launch_droplets).
cudaError_t launch_ccl(int precision, int layout, const Geom& g, const Phys& ph, const void* f,
                       double threshold, int* labels, int* sizes, long long* out3,
                       cudaStream_t s, bool started = false, bool slots = false);

// Appends the counts of the last launch_ccl (out4, device) to the newest
// ring record (fields DIAG_CCL ..).
cudaError_t launch_ccl_ring(const long long* out4, double* ring, const unsigned long long* ring_count,
                            int ring_cap, cudaStream_t s);

// Per-droplet statistics after launch_ccl with slots on the same state: cap
// records (one per root) of DROP_REC doubles [root, nodes, sum phi, sum rho,
// cos/sin sums of the angles 2 pi x/nx, 2 pi y/ny, 2 pi z/nz], and x-occupancy
// bit masks of (nx + 31)/32 words per record.  trig: nx + ny + nz entries
// filled by launch_trig.
constexpr int DROP_REC = 10;
cudaError_t launch_trig(const Geom& g, double2* trig, cudaStream_t s);
cudaError_t launch_droplets(int precision, int layout, const Geom& g, const Phys& ph, const void* f,
                            double rho_l, double rho_v, const int* labels, const int* slots, const double2* trig,
                            double* rec, unsigned* xbits, int cap, cudaStream_t s);


// ---- batched single-pass step on padded rows (lbm_fused.cu) ----------------
// One instance: geometry, physics, element offset of its array 0 in the
// padded pool (arrays 0 and 1 are Q px ny nz elements each) and its row
// pitch px (nx rounded up to batch_tma_row_align elements, 16 bytes).
struct BatchTmaInst {
  Geom g;
  Phys ph;
  long long off_f;
  int px;
};
int batch_tma_row_align(int precision);
// The launch of one step: tile width (32 or 64), instance records, blocks,
// chained launches.
struct BatchTmaPlan {
  int width, count, blocks, chain;
};
// Bytes of the device table (instance records and their tensor maps).
size_t batch_tma_table_bytes(int count);
// Encodes the tensor maps, builds the block table for tiles tile_w (32 or
// 64) nodes wide and z runs of fz planes (0: chosen) in groups of grp runs (0: all runs
// of a tile one after another), and copies it to d_table (device,
// batch_tma_table_bytes).  FP32, FP16-dev, BF16-dev.  Synchronises s.
cudaError_t batch_tma_build(int precision, int tile_w, const BatchTmaInst* insts, int count, int fz, int grp,
                            const void* pool, void* d_table, BatchTmaPlan* plan, cudaStream_t s);
// One step of every instance: padded pool arrays cur -> cur ^ 1.  salt: two
// words, of which the step reads word cur (its step number) and writes the
// other.
cudaError_t batch_tma_launch(int precision, const void* d_table, const BatchTmaPlan& plan, void* pool, int cur,
                             int* flag, unsigned* salt, cudaStream_t s);
// nsteps such steps in one cooperative launch of persistent blocks: grid
// barriers on *bar (zeroed here), per-step work tickets tickets[nsteps]
// (zeroed here); salt as batch_tma_launch (read only: the caller sets the word
// of the next launch); stall_ns > 0 is the barrier-timeout test hook.
cudaError_t batch_tma_persist_launch(int precision, const void* d_table, const BatchTmaPlan& plan, void* pool,
                                     int cur, int nsteps, unsigned* bar, unsigned* tickets, int* flag,
                                     const unsigned* salt, unsigned long long stall_ns, cudaStream_t s);

// True if LBM_ALLOC_CAP_BYTES is set and a device allocation of `bytes`
// exceeds it (out-of-memory handling without exhausting a GPU).
bool alloc_over_cap(size_t bytes);

// While a graph of steps is captured or memory for them allocated: calls that
// the runtime forbids to a thread with a capture of its own under way (on
// another stream, by the program that uses the library) do not void that
// capture.  They touch none of its streams.
struct CaptureAllowed {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  CaptureAllowed() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~CaptureAllowed() { cudaThreadExchangeStreamCaptureMode(&mode); }
};

// Device memory that an object keeps between calls although it can do without
// (planes of host transfers, padded arrays): whenever a device allocation of the library is
// refused, every Spare on the device that no call is using is freed, and the
// allocation tried again (device_alloc).  spare_alloc, spare_free and p belong to
// the call between spare_enter and spare_leave.
struct Spare {
  void* p = nullptr;
  size_t bytes = 0;
  bool busy = false;
  int device = 0;
  Spare* next = nullptr;
};
void spare_enter(Spare& s);
void spare_leave(Spare& s);
struct SpareUse {
  Spare& s;
  explicit SpareUse(Spare& spare) : s(spare) { spare_enter(s); }
  ~SpareUse() { spare_leave(s); }
};
// `bytes` in place of what s holds (nothing where they are refused; capped: also
// by LBM_ALLOC_CAP_BYTES on all that the lattices hold); frees no other Spare.
cudaError_t spare_alloc(Spare& s, size_t bytes, bool capped);
void spare_free(Spare& s);
// Room for FP64 planes of N nodes: transfer_doubles(N, planes) of them, one
// plane where that many are refused.
cudaError_t transfer_room(Spare& s, long long N, int planes, bool capped);
// cudaMalloc, tried again once the idle Spares are freed.
cudaError_t device_alloc(void** p, size_t bytes);

}  // namespace lbm

// ---- the handle -------------------------------------------------------------
struct lbm_ctx {
  lbm_config cfg;
  lbm::Geom g;
  lbm::Phys ph;
  cudaStream_t stream = nullptr;
  cudaStream_t own_stream = nullptr;
  int device = 0;

  void* state = nullptr;  // populations: A-B = two arrays, AA = one
  size_t state_bytes = 0;
  bool own_state = false;
  // two private arrays of pad_bytes each with rows padded to 16 bytes, between
  // which the steps inside a captured chunk run where the lattice's own rows are
  // not 16-byte multiples; pad_graphs: the captured graphs use them; pad_failed:
  // there was no room for them, or they were given back
  lbm::Spare pads;
  size_t pad_bytes = 0;
  bool pad_graphs = false, pad_failed = false;
  void* psi = nullptr;
  size_t psi_bytes = 0;
  bool own_psi = false;
  int cur = 0;            // A-B: index of the current array
  long long step = 0;
  bool initialized = false;
  double rho_l = 1.0, rho_v = 0.0;

  int* d_flag = nullptr;          // [0] numeric / timeout flag, [2] stochastic-rounding step salt
  double2* d_psi_tab = nullptr;   // FP64: table of psi_of<double>
  double* d_small = nullptr;      // small result buffer (diagnostics out etc.)
  double* d_scratch = nullptr;    // diagnostics partials
  lbm::Spare transfer;            // FP64 planes on their way to or from the host (kept up to 64 MiB)
  size_t scratch_doubles = 0;
  int* d_labels = nullptr;        // CCL labels and sizes (2 N ints)
  bool diag_ccl = false;          // label droplets at every in-loop diagnostic step
  double2* d_trig = nullptr;      // angles of the coordinates (lbm_droplets)
  double* d_drop = nullptr;       // droplet records and x masks (lbm_droplets)
  size_t drop_bytes = 0;

  // CUDA graphs of one chunk of steps, keyed by the A-B array they start on
  // (AA chunks always start on an even step)
  cudaGraphExec_t graph[2][2] = {{nullptr, nullptr}, {nullptr, nullptr}};   // [phase][longer chunk]
  int graph_chunk = 0;            // steps per captured chunk (the shorter one)
  long long replays = 0;          // of the shorter chunk's graphs
  bool use_graph = true;
  dim3 block{0, 0, 0};
  bool block_asked = false;       // block was given (else auto_block is launched)
  int minb = 0;                   // collide kernel register budget variant (0 = auto)
  bool vec = true;                // two nodes per thread (when nx is even)
  bool aligned = true;            // the buffers start where node pairs and groups of four may (own ones do)
  // single-pass A-B steps: -1 (until the option is set) where they apply and
  // pay, 0 never, 1 the 64-wide tiles where they apply and cut tiles where
  // they pay, 2 both where they apply
  int fused = -1;
  int fused_fz = 0;               // z planes per block of the fused step (0 = automatic)
  int fused_group = 0;            // z runs per group of its block order (0 = automatic)
  unsigned long long fused_stall_test_ns = 0;   // test hook of the fused step's timeout path

  // diagnostics inside the time loop: every diag_interval steps the psi
  // pass also reduces the diagnostics into a device ring of records
  int diag_interval = 0;
  static constexpr int kRing = 1024;
  double* d_ring = nullptr;                 // kRing * DIAG_STRIDE doubles
  unsigned long long* d_ring_count = nullptr;
  std::vector<long long> diag_steps;        // step of every record launched
  long long diag_fetched = 0;               // records already returned

  // kernel timing
  bool kernel_timing = false;
  std::vector<cudaEvent_t> ev_free;
  struct Pending {
    int k;
    cudaEvent_t a, b;
  };
  std::vector<Pending> pending;
  long long t_launches[3] = {0, 0, 0};
  double t_ms[3] = {0.0, 0.0, 0.0};
};
