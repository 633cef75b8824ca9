// Host runtime and C ABI of liblbm.so (declared in include/lbm.h): handle
// life cycle, device memory, the stream, CUDA-graph replay of the time step,
// kernel timing, checkpoints and the host side of diagnostics.
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <new>
#include <string>

#include "lbm_internal.h"

using namespace lbm;

namespace lbm {
inline bool Prec_dev(int precision) { return precision == LBM_F16DEV || precision == LBM_BF16DEV; }

// Default collide-stream block: 256 threads, as long along x (the
// contiguous axis) as the lattice allows; with two nodes per thread (nx
// even) block.x counts node pairs.
dim3 default_block(const Geom& g) {
  const int ux = g.nx % 2 == 0 ? g.nx / 2 : g.nx;
  const unsigned bx = ux >= 256 ? 256 : (ux >= 128 ? 128 : (ux >= 64 ? 64 : 32));
  return dim3(bx, 256 / bx, 1);
}

// The block a collide-stream kernel launches with where no shape was asked
// for: two warps.  These kernels hold 80 to 100 registers, so an SM takes few
// warps, and a block's place is free for the next one only when its last warp
// is done: small blocks keep more warps in flight (per collide kernel, 256 ->
// 64 threads: 512x256x256 FP16 A-B 580 -> 565 us, AA odd 707 -> 633 us with
// its larger register budget, auto_minb; 256x128x128 FP64 988 -> 981 us; per
// step: 150x80x80 FP32 37.8 -> 33.7 us, FP16 30.4 -> 25.6 us).  64 along x, 32
// where that pads the row less (150x80x80 FP32 in 64 x 1: 36.1 us), and for
// FP32 rows of whole 128s four warps (512x256x256 A-B: 767 us, 64 x 1 775).
// Lattices too small to give every SM two such blocks take one warp, and rows
// shorter than a warp are not padded to one: the block takes whole rows of
// several y and z, so a warp's lanes all hold nodes (4x49x49 FP64, whose pipe a
// warp instruction occupies for 16 clocks whatever its live lanes: 68 us per
// step in 32 x 8 blocks, 2 of 32 lanes live, 10.3 us in 4 x 8 x 1).  More rows
// than 65535 such blocks take (the limit of a grid along y) go in the default
// shape, whose blocks hold up to 8.
static dim3 small_block(const Geom& g, bool pairs, int precision) {
  const unsigned ux = pairs ? g.nx / 2 : g.nx;
  const long long units = (long long)ux * g.ny * g.nz;
  const unsigned threads = units < 64LL * 2 * kSmCount ? 32 : 64;
  if (ux >= 32) {
    if (threads == 64 && precision == LBM_F32 && ux % 128 == 0) return dim3(128, 1, 1);
    const unsigned bx = threads == 64 && (ux - 1) % 64 >= 32 ? 64 : 32;
    return dim3(bx, threads / bx, 1);
  }
  const unsigned by = std::min<unsigned>(g.ny, std::max(1u, threads / ux));
  const unsigned bz = std::min<unsigned>(std::min(g.nz, 64), std::max(1u, threads / (ux * by)));
  return dim3(ux, by, bz);
}
dim3 auto_block(const Geom& g, bool pairs, int precision) {
  const dim3 b = small_block(g, pairs, precision);
  return (g.ny + b.y - 1) / b.y > 65535 ? default_block(g) : b;
}

// Default register budget of the collide-stream kernel (as blocks of 256
// threads per SM), measured in the blocks of auto_block: 3 for the one-node
// kernel and for the AA even step's two-node kernel (local loads and stores: no
// spills at 80 registers); for the A-B step's two-node kernel 3 with 2-byte
// storage above 2^21 nodes (512x256x256 FP16: 565 us per launch against 584
// with 2; 150x80x80: 26.5 us per step against 25.6); 2 otherwise, with which
// nothing spills (AA odd step of 512x256x256, FP16: 633 us per launch, with 3
// 666; FP32: 783 against 930).
int auto_minb(bool vec, int mode, int precision, long long N) {
  if (precision == LBM_F64) return 2;   // 981 us per launch on 256x128x128 against 1009 with 3 (spills)
  if (!vec || mode == MODE_AA_EVEN) return 3;
  return mode == MODE_AB && precision != LBM_F32 && N > 2LL << 20 ? 3 : 2;
}
}  // namespace lbm

namespace {

thread_local std::string g_last_error;

int fail(int status, const std::string& msg) {
  g_last_error = msg;
  return status;
}

// The error is reported by this call alone: the runtime keeps the last one
// until it is read, and a later check of a launch (here or in the caller's
// program) would take it for its own.
int cuda_fail(cudaError_t e, const char* where) {
  (void)cudaGetLastError();
  g_last_error = std::string(where) + ": " + cudaGetErrorString(e);
  return e == cudaErrorMemoryAllocation ? LBM_ERR_OOM : LBM_ERR_CUDA;
}

#define CK(call)                                      \
  do {                                                \
    cudaError_t e_ = (call);                          \
    if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
  } while (0)

// Bytes that the lattices hold, and whether `bytes` more exceed the optional cap
// (environment LBM_ALLOC_CAP_BYTES: out-of-memory handling without exhausting a GPU).
std::atomic<size_t> g_alloc_total{0};
bool over_total_cap(size_t bytes) {
  const char* cap = std::getenv("LBM_ALLOC_CAP_BYTES");
  return cap && *cap && g_alloc_total + bytes > std::strtoull(cap, nullptr, 10);
}

std::mutex g_spare_mu;
Spare* g_spares = nullptr;   // those that hold memory

// Takes s from the list and frees its memory (under the lock).
void spare_drop(Spare& s) {
  for (Spare** at = &g_spares; *at; at = &(*at)->next)
    if (*at == &s) {
      *at = s.next;
      break;
    }
  if (s.p) cudaFree(s.p);
  g_alloc_total -= s.bytes;
  s.p = nullptr;
  s.bytes = 0;
}

// Frees the idle Spares of the current device; whether there were any.
bool spares_give_back() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return false;
  std::lock_guard<std::mutex> lock(g_spare_mu);
  bool any = false;
  for (Spare* s = g_spares; s;) {
    Spare* const next = s->next;
    if (!s->busy && s->device == dev) {
      if (!any) cudaDeviceSynchronize();   // work of earlier calls may still use them
      spare_drop(*s);
      any = true;
    }
    s = next;
  }
  return any;
}

// A lattice's device allocation, under the cap.
int dev_alloc(void** p, size_t bytes, const char* what) {
  bool capped = over_total_cap(bytes);
  if (capped && spares_give_back()) capped = over_total_cap(bytes);
  *p = nullptr;
  if (capped) return fail(LBM_ERR_OOM, std::string("allocation of ") + what + " exceeds LBM_ALLOC_CAP_BYTES");
  const cudaError_t e = device_alloc(p, bytes);
  if (e != cudaSuccess) return cuda_fail(e, what);
  g_alloc_total += bytes;
  return LBM_OK;
}

void dev_free(void* p, size_t bytes) {
  if (p) {
    cudaFree(p);
    g_alloc_total -= bytes;
  }
}

int validate(const lbm_config* c) {
  if (!c) return fail(LBM_ERR_ARG, "null config");
  if (c->nx < 3 || c->ny < 3 || c->nz < 3)
    return fail(LBM_ERR_ARG, "every lattice dimension must be >= 3");
  const long long N = (long long)c->nx * c->ny * c->nz;
  if (N > 0x7fffffffLL) return fail(LBM_ERR_ARG, "lattice has more than 2^31-1 nodes");
  if (!std::isfinite(c->tau) || !(c->tau > 0.5)) return fail(LBM_ERR_ARG, "tau must be finite and > 1/2");
  if (!std::isfinite(c->G)) return fail(LBM_ERR_ARG, "G must be finite");
  if (c->psi_form != LBM_PSI_EXP && c->psi_form != LBM_PSI_RHO) return fail(LBM_ERR_ARG, "unknown psi_form");
  if (!std::isfinite(c->rho0) || !(c->rho0 > 0.0)) return fail(LBM_ERR_ARG, "rho0 must be finite and > 0");
  if (c->precision < LBM_F64 || c->precision > LBM_BF16DEV) return fail(LBM_ERR_ARG, "unknown precision");
  if (c->pattern != LBM_AB && c->pattern != LBM_AA) return fail(LBM_ERR_ARG, "unknown pattern");
  if (!std::isfinite(c->rho_ref)) return fail(LBM_ERR_ARG, "rho_ref must be finite");
  const int bx = c->block_x, by = c->block_y, bz = c->block_z;
  if (bx < 0 || by < 0 || bz < 0) return fail(LBM_ERR_ARG, "negative block size");
  if ((bx || by || bz) && (bx == 0 || by == 0 || bz == 0 || (long long)bx * by * bz > 256 || bz > 64))
    return fail(LBM_ERR_ARG, "block shape must be all zero or have 1..256 threads (bz <= 64)");
  return LBM_OK;
}

void sizes_for(const lbm_config* c, size_t* state, size_t* psi) {
  const size_t N = (size_t)c->nx * c->ny * c->nz;
  const size_t e = elem_size(c->precision);
  const size_t arrays = c->pattern == LBM_AB ? 2 : 1;
  *state = arrays * Q * N * e;
  *psi = N * (c->precision == LBM_F64 ? 8 : 4);
}


// ---- per-handle helpers -----------------------------------------------------

void* array_ptr(lbm_ctx* h, int k) {
  const size_t one = (size_t)Q * h->g.N * elem_size(h->cfg.precision);
  return (char*)h->state + (size_t)k * one;
}

void* cur_array(lbm_ctx* h) { return h->cfg.pattern == LBM_AB ? array_ptr(h, h->cur) : h->state; }

int cur_layout(const lbm_ctx* h) {
  return (h->cfg.pattern == LBM_AA && (h->step & 1)) ? LAYOUT_GATHER : LAYOUT_LOCAL;
}

void drop_graphs(lbm_ctx* h) {
  for (auto& pair : h->graph)
    for (auto& ge : pair)
      if (ge) {
        cudaGraphExecDestroy(ge);
        ge = nullptr;
      }
  h->pad_graphs = false;
}

cudaEvent_t take_event(lbm_ctx* h) {
  if (!h->ev_free.empty()) {
    cudaEvent_t e = h->ev_free.back();
    h->ev_free.pop_back();
    return e;
  }
  cudaEvent_t e = nullptr;
  cudaEventCreate(&e);
  return e;
}

// The word of the salt pair step `step` reads: the A-B array index, or the
// step parity for AA (whose graph chunks hold an even number of steps).
int salt_word(const lbm_ctx* h, long long step, int cur) {
  return h->cfg.pattern == LBM_AA ? (int)(step & 1) : (cur & 1);
}

bool ragged_direct(const lbm_ctx* h);

// Whether steps run as the fused single pass: small lattices only when asked
// for (option "fused", or one of its launch shape or test hook).
bool fused_form(const lbm_ctx* h) {
  const long long least = h->cfg.precision == LBM_F32 && h->ph.coll == COLL_SRT ? kFusedNodes : kFusedNodesLate;
  return h->fused && h->cfg.pattern == LBM_AB && fused_applicable(h->g, h->cfg.precision) &&
         (h->fused > 0 || h->g.N > least || h->fused_fz || h->fused_group || h->fused_stall_test_ns ||
          (uintptr_t)h->state % 16);   // (TMA refuses such populations, on small lattices too)
}

// Whether node pairs move as vectors: not where the caller's buffers start at an
// address that their loads and stores (and the psi pass's of four nodes, where nx
// allows them) are not aligned to.
bool buffers_aligned(const lbm_ctx* h) {
  if (h->cfg.precision == LBM_F64) return true;   // one node at a time
  const size_t unit = h->g.nx % 4 == 0 ? 4 : 2;
  return (uintptr_t)h->state % (unit * elem_size(h->cfg.precision)) == 0 && (uintptr_t)h->psi % (unit * sizeof(float)) == 0;
}
bool vector_form(const lbm_ctx* h) { return h->vec && h->aligned; }

// The psi pass of a diagnostic step of the two kernels: with the diagnostics,
// and the droplet counts where they are on.
int enqueue_diagnostics(lbm_ctx* h, cudaStream_t s, const Geom& g, int layout, const void* src, void* dst,
                        ReduceSide* side) {
  const int prec = h->cfg.precision;
  const double thr = 0.5 * (h->rho_l + h->rho_v);
  DiagExtra x;
  if (h->diag_ccl) x = diag_labels(prec, layout, g, src, h->psi, thr, h->d_labels, h->d_labels + g.N);
  x.dst = dst;
  x.side = side;
  CK(launch_diagnostics(prec, layout, g, h->ph, src, h->rho_l, h->rho_v, h->d_scratch, h->d_ring, h->psi, h->d_flag,
                        h->d_ring_count, lbm_ctx::kRing, s, x));
  if (h->diag_ccl) {
    long long* d4 = (long long*)(h->d_small + 32);
    CK(launch_ccl(prec, layout, g, h->ph, src, thr, h->d_labels, h->d_labels + g.N, d4, s, x.labels != nullptr));
    CK(launch_ccl_ring(d4, h->d_ring, h->d_ring_count, lbm_ctx::kRing, s));
  }
  return LBM_OK;
}

// Enqueues one time step on stream s.  `phase` is the step parity (AA) or
// the index of the current array (A-B).  With timing on, each kernel is
// bracketed by events on s.  side (captures): where the diagnostics'
// reduction runs beside the following steps.
int enqueue_step(lbm_ctx* h, cudaStream_t s, long long step, int cur, bool timed, ReduceSide* side = nullptr) {
  const int prec = h->cfg.precision;
  const bool aa = h->cfg.pattern == LBM_AA;
  const int layout = (aa && (step & 1)) ? LAYOUT_GATHER : LAYOUT_LOCAL;
  const void* src = aa ? h->state : array_ptr(h, cur);
  void* dst = aa ? h->state : array_ptr(h, cur ^ 1);
  const int mode = aa ? ((step & 1) ? MODE_AA_ODD : MODE_AA_EVEN) : MODE_AB;
  cudaEvent_t e0 = nullptr, e1 = nullptr, e2 = nullptr;
  const bool diag_step = h->diag_interval > 0 && step % h->diag_interval == 0;
  const bool fused = fused_form(h);
  Geom g = h->g;
  if (h->diag_ccl) side = nullptr;   // the labelling appends to the record of its own step
  if (side && side->open && diag_step) {
    CK(cudaStreamWaitEvent(s, side->join, 0));
    side->open = false;
    g.chain = 0;   // a kernel with two predecessors
  }
  // stochastic-rounding salt: a pair of words, read and advanced by the
  // step's collision kernel; the word a step reads follows the A-B array
  // (AA: the step parity), so graph replays and eager steps agree
  Phys ph = h->ph;
  if (Prec_dev(prec) && h->ph.sr) {
    const int w = salt_word(h, step, cur);
    ph.salt = (const unsigned*)(h->d_flag + 2 + w);
    ph.salt_next = (unsigned*)(h->d_flag + 2 + (w ^ 1));
  }
  // a diagnostic step runs fused too when the scratch holds its partials
  const bool fused_diag =
      fused && diag_step && h->d_scratch && fused_diag_scratch_doubles(g, prec, h->fused_fz) <= h->scratch_doubles;
  if (fused && (!diag_step || fused_diag)) {
    // single pass: psi of each tile is computed from the staged populations
    if (timed) {
      e0 = take_event(h);
      e1 = take_event(h);
      CK(cudaEventRecord(e0, s));
    }
    if (diag_step) {
      const FusedDiag fd{h->rho_l, h->rho_v, h->d_scratch, h->scratch_doubles, h->d_ring, h->d_ring_count,
                         lbm_ctx::kRing};
      CK(launch_fused(prec, g, ph, src, dst, h->d_flag, h->fused_fz, h->fused_group, &fd,
                      h->fused_stall_test_ns, s, side));
    } else {
      CK(launch_fused(prec, g, ph, src, dst, h->d_flag, h->fused_fz, h->fused_group, nullptr, h->fused_stall_test_ns, s));
    }
    if (timed) {
      CK(cudaEventRecord(e1, s));
      h->pending.push_back({2, e0, e1});
    }
    if (diag_step && h->diag_ccl) {
      long long* d4 = (long long*)(h->d_small + 32);
      CK(launch_ccl(prec, layout, h->g, h->ph, src, 0.5 * (h->rho_l + h->rho_v), h->d_labels,
                    h->d_labels + h->g.N, d4, s));
      CK(launch_ccl_ring(d4, h->d_ring, h->d_ring_count, lbm_ctx::kRing, s));
    }
    return LBM_OK;
  }
  if (!diag_step && ragged_direct(h)) {
    if (timed) {
      e0 = take_event(h);
      e1 = take_event(h);
      CK(cudaEventRecord(e0, s));
    }
    CK(launch_ragged(prec, g, ph, src, g.nx, dst, g.nx, h->d_flag, h->fused_fz, h->fused_group, s));
    if (timed) {
      CK(cudaEventRecord(e1, s));
      h->pending.push_back({2, e0, e1});
    }
    return LBM_OK;
  }
  if (timed) {
    e0 = take_event(h);
    e1 = take_event(h);
    e2 = take_event(h);
    CK(cudaEventRecord(e0, s));
  }
  if (diag_step) {
    if (int rc = enqueue_diagnostics(h, s, g, layout, src, aa ? nullptr : dst, side)) return rc;
  } else {
    CK(launch_psi(prec, layout, vector_form(h), g, h->ph, src, h->psi, h->d_flag, s, aa ? nullptr : dst));
  }
  if (timed) CK(cudaEventRecord(e1, s));
  const bool vec = node_pairs(prec, vector_form(h), h->g);
  const int minb = h->minb ? h->minb : auto_minb(vec, mode, prec, h->g.N);
  const dim3 block = h->block_asked ? h->block : auto_block(h->g, vec, prec);
  if (h->ph.coll == COLL_MRT)
    CK(launch_collide_mrt(prec, mode, vec, g, ph, src, dst, h->psi, block, s));
  else
    CK(launch_collide(prec, mode, minb, vec, g, ph, src, dst, h->psi, block, s));
  if (timed) {
    CK(cudaEventRecord(e2, s));
    h->pending.push_back({0, e0, e1});
    h->pending.push_back({1, e1, e2});
  }
  return LBM_OK;
}

// Whether plain steps run as the ragged single pass between the lattice's own
// arrays (its rows are 16-byte multiples), and whether the steps inside a
// captured chunk run on padded copies (they are not, and there is room).
bool ragged_form(const lbm_ctx* h) {
  const bool pays = Prec_dev(h->cfg.precision) ? h->g.N > kRaggedNodesDev && h->g.nx % 2 : h->g.N > kRaggedNodes;
  return h->fused && (h->fused == 2 || (pays && h->g.nx >= kRaggedMinNx)) &&
         h->cfg.pattern == LBM_AB && ragged_applicable(h->g, h->cfg.precision);
}
bool ragged_direct(const lbm_ctx* h) {
  return ragged_form(h) && ragged_row(h->g, h->cfg.precision) == h->g.nx && ((uintptr_t)h->state & 15) == 0;
}
bool padded_form(const lbm_ctx* h) { return ragged_form(h) && !ragged_direct(h) && h->pads.p; }
void* pad_ptr(const lbm_ctx* h, int k) { return (char*)h->pads.p + k * h->pad_bytes; }

// Allocates the padded arrays where they take at most a quarter of the free
// memory; without them the steps stay on the two kernels.  Called only where
// the steps at hand replay a chunk of several, whose later ones use them.
void ensure_padded(lbm_ctx* h) {
  if (h->pads.p || h->pad_failed || !ragged_form(h) || ragged_direct(h)) return;
  const CaptureAllowed allowed;
  const size_t bytes =
      ((size_t)Q * ragged_row(h->g, h->cfg.precision) * h->g.ny * h->g.nz * elem_size(h->cfg.precision) + 255) / 256 * 256;
  size_t free_b = 0, total_b = 0;
  h->pad_failed = cudaMemGetInfo(&free_b, &total_b) != cudaSuccess || 8 * bytes > free_b ||
                  spare_alloc(h->pads, 2 * bytes, true) != cudaSuccess;
  if (h->pad_failed) (void)cudaGetLastError();
  h->pad_bytes = bytes;
}

// Step k of a captured chunk of `steps` that starts on array `phase`, on
// padded rows: the first step (the chunk's diagnostic step, if any) is the
// two-kernel one and writes its collision's result to the first padded array,
// the others are single passes between the two, the last one back into the
// lattice's own array.  20 FP32 steps on 251x112x112 with
// a diagnostic step in ten: 2843 -> 2208 us.
int enqueue_padded_step(lbm_ctx* h, cudaStream_t s, int k, int steps, int phase, ReduceSide* side) {
  const int prec = h->cfg.precision, px = ragged_row(h->g, prec);
  const Geom& g = h->g;
  Phys ph = h->ph;
  if (Prec_dev(prec) && ph.sr) {
    const int w = salt_word(h, k, phase ^ (k & 1));
    ph.salt = (const unsigned*)(h->d_flag + 2 + w);
    ph.salt_next = (unsigned*)(h->d_flag + 2 + (w ^ 1));
  }
  if (k == 0) {
    const void* src = array_ptr(h, phase);
    if (h->diag_interval > 0) {
      if (int rc = enqueue_diagnostics(h, s, g, LAYOUT_LOCAL, src, nullptr, h->diag_ccl ? nullptr : side)) return rc;
    } else {
      CK(launch_psi(prec, LAYOUT_LOCAL, vector_form(h), g, h->ph, src, h->psi, h->d_flag, s));
    }
    CK(launch_collide_padded(prec, g, ph, src, pad_ptr(h, 0), px, h->psi, auto_block(g, false, prec), s));
    return LBM_OK;
  }
  const bool last = k == steps - 1;
  CK(launch_ragged(prec, g, ph, pad_ptr(h, (k - 1) & 1), px, last ? array_ptr(h, phase ^ (steps & 1)) : pad_ptr(h, k & 1),
                   last ? g.nx : px, h->d_flag, h->fused_fz, h->fused_group, s));
  return LBM_OK;
}

int settle_timing(lbm_ctx* h) {
  if (h->pending.empty()) return LBM_OK;
  CK(cudaStreamSynchronize(h->stream));
  // events shared between consecutive kernels are returned once
  std::vector<cudaEvent_t> seen;
  for (auto& p : h->pending) {
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, p.a, p.b));
    h->t_launches[p.k] += 1;
    h->t_ms[p.k] += ms;
    seen.push_back(p.a);
    seen.push_back(p.b);
  }
  h->pending.clear();
  for (size_t i = 0; i < seen.size(); ++i) {
    bool dup = false;
    for (size_t k = 0; k < i; ++k) dup |= seen[k] == seen[i];
    for (auto e : h->ev_free) dup |= e == seen[i];
    if (!dup) h->ev_free.push_back(seen[i]);
  }
  return LBM_OK;
}

// Steps per captured graph: 2 without in-loop diagnostics; with them, the
// diagnostic interval k (2k for AA when k is odd, so every chunk starts on
// an even step).  Chunks are replayed only from steps that are multiples of
// the chunk length, so the diagnostic steps inside a chunk are fixed.
int chunk_len(const lbm_ctx* h) {
  const int k = h->diag_interval;
  if (k <= 0) return 2;
  if (h->cfg.pattern == LBM_AA && (k & 1)) return 2 * k;
  return k;
}

// Steps of the longer graph that small lattices, and plain steps on padded
// rows (whose first step is the slow one), replay while enough steps are left:
// the multiple of chunk_len() from 16 on.  A graph launch costs about
// 2.7 us between two replays (64x32x32 FP32 and 4x49x49 FP64, 2-step against
// 50- and 100-step graphs), as much as a kernel of such a step; larger
// lattices do not feel it and keep the shorter capture.  On small lattices it
// is captured once the replays it saves in a call, and those done before, come
// to twice its steps: capturing takes about 5 us a step, as much as two replays
// (a first call of 100 steps with a diagnostic step in ten took 550 us with
// the 20-step graph captured at once, 480 with the 10-step one).
int long_chunk_len(const lbm_ctx* h) {
  const int c = chunk_len(h);
  const bool longer = padded_form(h) ? h->diag_interval == 0 : h->g.chain != 0;
  return longer ? (16 + c - 1) / c * c : c;
}

// Captures `steps` consecutive steps (a multiple of chunk_len()) starting at
// array `phase` (A-B; 0 for AA) into an executable graph.  Capture runs on a private stream
// (capture is not allowed on the legacy default stream); the graph is
// launched on the handle's stream.
int capture_chunk(lbm_ctx* h, int phase, int steps, cudaGraphExec_t* exec) {
  const CaptureAllowed allowed;
  cudaStream_t cs = nullptr;
  ReduceSide side{nullptr, nullptr, nullptr, false};
  cudaGraph_t graph = nullptr;
  int rc = LBM_OK;
  cudaError_t e = cudaStreamCreateWithFlags(&cs, cudaStreamNonBlocking);
  if (e == cudaSuccess && h->diag_interval > 0) {
    e = cudaStreamCreateWithFlags(&side.stream, cudaStreamNonBlocking);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&side.fork, cudaEventDisableTiming);
    if (e == cudaSuccess) e = cudaEventCreateWithFlags(&side.join, cudaEventDisableTiming);
  }
  if (e == cudaSuccess) e = cudaStreamBeginCapture(cs, cudaStreamCaptureModeThreadLocal);
  if (e == cudaSuccess) {
    // step numbers relative to a chunk start (a multiple of chunk_len()): the same
    // parity and the same diagnostic steps as every replay
    const bool padded = padded_form(h) && steps > 1;
    h->pad_graphs |= padded;
    for (int k = 0; k < steps && rc == LBM_OK; ++k)
      rc = padded ? enqueue_padded_step(h, cs, k, steps, phase, side.join ? &side : nullptr)
                  : enqueue_step(h, cs, k, phase ^ (k & 1), false, side.join ? &side : nullptr);
    if (side.open) e = cudaStreamWaitEvent(cs, side.join, 0);
    const cudaError_t e2 = cudaStreamEndCapture(cs, &graph);
    if (e == cudaSuccess) e = e2;
  }
  if (side.join) cudaEventDestroy(side.join);
  if (side.fork) cudaEventDestroy(side.fork);
  if (side.stream) cudaStreamDestroy(side.stream);
  if (cs) cudaStreamDestroy(cs);
  if (rc != LBM_OK || e != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    (void)cudaGetLastError();   // of ending a capture that a failed launch had spoilt
    return rc != LBM_OK ? rc : cuda_fail(e, "graph capture of the steps");
  }
  e = cudaGraphInstantiate(exec, graph, 0);
  cudaGraphDestroy(graph);
  if (e != cudaSuccess) {
    *exec = nullptr;
    return cuda_fail(e, "cudaGraphInstantiate");
  }
  return LBM_OK;
}

// Diagnostics partials: room for the two-kernel reduction and, where the
// fused step applies, for the fused step's (which depends on its z runs).
int ensure_scratch(lbm_ctx* h) {
  size_t need = diag_scratch_doubles(h->g);
  if (h->fused && h->cfg.pattern == LBM_AB)
    need = std::max(need, fused_diag_scratch_doubles(h->g, h->cfg.precision, h->fused_fz));
  if (h->d_scratch && h->scratch_doubles >= need) return LBM_OK;
  if (h->d_scratch) dev_free(h->d_scratch, h->scratch_doubles * sizeof(double));
  h->d_scratch = nullptr;
  h->scratch_doubles = 0;
  int rc = dev_alloc((void**)&h->d_scratch, need * sizeof(double), "diagnostics scratch");
  if (rc == LBM_OK) h->scratch_doubles = need;
  return rc;
}

int ensure_labels(lbm_ctx* h) {
  if (h->d_labels) return LBM_OK;
  return dev_alloc((void**)&h->d_labels, (size_t)h->g.N * 2 * sizeof(int), "labels");
}

int ensure_ring(lbm_ctx* h) {
  if (h->d_ring_count) return LBM_OK;   // (allocated last)
  int rc = h->d_ring ? LBM_OK
                     : dev_alloc((void**)&h->d_ring, sizeof(double) * DIAG_STRIDE * lbm_ctx::kRing, "diagnostics ring");
  if (rc) return rc;
  rc = dev_alloc((void**)&h->d_ring_count, sizeof(unsigned long long), "ring counter");
  if (rc) return rc;
  CK(cudaMemsetAsync(h->d_ring_count, 0, sizeof(unsigned long long), h->stream));
  return LBM_OK;
}

void fill_diag(lbm_diag* out, const double* r, long long step) {
  out->step = step;
  out->mass = r[0];
  out->mom[0] = r[1];
  out->mom[1] = r[2];
  out->mom[2] = r[3];
  out->liquid_volume_w = r[4];
  out->liquid_count = (long long)r[5];
  out->min_slice_area_w = r[6];
  out->min_slice_count = (long long)r[7];
  out->min_slice_x = (int)r[8];
  out->neck_radius = std::sqrt(r[6] / 3.14159265358979323846);
  out->max_u = r[9];
  out->rho_min = r[10];
  out->rho_max = r[11];
  out->numeric_ok = (int)r[12];
  out->droplets = -1;
  out->droplets_min8 = -1;
  out->largest_droplet = -1;
}

// Room for `planes` FP64 planes on their way to or from the host (fewer where
// they exceed 64 MiB or are refused), used until end_transfer, which gives back
// what is larger than 64 MiB.
int begin_transfer(lbm_ctx* h, int planes) {
  spare_enter(h->transfer);
  const cudaError_t e = transfer_room(h->transfer, h->g.N, planes, true);
  if (e == cudaSuccess) return LBM_OK;
  spare_leave(h->transfer);
  if (e != cudaErrorMemoryAllocation) return cuda_fail(e, "transfer planes");
  return fail(LBM_ERR_OOM, over_total_cap((size_t)h->g.N * sizeof(double))
                               ? "allocation of transfer planes exceeds LBM_ALLOC_CAP_BYTES"
                               : "transfer planes: out of memory");
}
void end_transfer(lbm_ctx* h) {
  if (h->transfer.bytes > (size_t)64 << 20) spare_free(h->transfer);
  spare_leave(h->transfer);
}

size_t trig_bytes(const Geom& g) { return sizeof(double2) * ((size_t)g.nx + g.ny + g.nz); }

struct StateHeader {
  char magic[8];
  int version, precision, pattern, nx, ny, nz, cur, pad;
  long long step;
  double rho_l, rho_v;
};

}  // namespace

extern "C" {

void lbm_config_default(lbm_config* c) {
  if (!c) return;
  std::memset(c, 0, sizeof(*c));
  c->nx = c->ny = c->nz = 3;
  c->tau = 1.0;
  c->G = 0.0;
  c->psi_form = LBM_PSI_EXP;
  c->rho0 = 1.0;
  c->precision = LBM_F32;
  c->pattern = LBM_AB;
  c->rho_ref = 0.0;
}

int lbm_required_bytes(const lbm_config* cfg, size_t* state_bytes, size_t* psi_bytes) {
  int rc = validate(cfg);
  if (rc) return rc;
  size_t s, p;
  sizes_for(cfg, &s, &p);
  if (state_bytes) *state_bytes = s;
  if (psi_bytes) *psi_bytes = p;
  return LBM_OK;
}

const char* lbm_last_error(void) { return g_last_error.c_str(); }

const char* lbm_strerror(int status) {
  switch (status) {
    case LBM_OK: return "ok";
    case LBM_ERR_ARG: return "invalid argument";
    case LBM_ERR_CUDA: return "CUDA error";
    case LBM_ERR_OOM: return "out of device memory";
    case LBM_ERR_NUMERIC: return "non-positive or non-finite density";
    case LBM_ERR_TIMEOUT: return "bounded device wait timed out";
    case LBM_ERR_STATE: return "invalid state for this call";
  }
  return "unknown status";
}

int lbm_lattice(int* c, double* w) {
  for (int a = 0; a < Q; ++a) {
    if (c) {
      c[3 * a] = cx(a);
      c[3 * a + 1] = cy(a);
      c[3 * a + 2] = cz(a);
    }
    if (w) w[a] = wgt(a);
  }
  return LBM_OK;
}

void lbm_destroy(lbm_handle h) {
  if (!h) return;
  if (h->stream) cudaStreamSynchronize(h->stream);
  drop_graphs(h);
  for (auto& p : h->pending) {
    h->ev_free.push_back(p.a);
    h->ev_free.push_back(p.b);
  }
  std::vector<cudaEvent_t> uniq;
  for (auto e : h->ev_free) {
    bool dup = false;
    for (auto u : uniq) dup |= u == e;
    if (!dup) uniq.push_back(e);
  }
  for (auto e : uniq) cudaEventDestroy(e);
  if (h->own_state) dev_free(h->state, h->state_bytes);
  if (h->own_psi) dev_free(h->psi, h->psi_bytes);
  dev_free(h->d_flag, sizeof(int) * 4);
  dev_free(h->d_psi_tab, sizeof(double2) * kPsiTab);
  dev_free(h->d_small, sizeof(double) * 64);
  dev_free(h->d_scratch, h->scratch_doubles * sizeof(double));
  spare_free(h->pads);
  spare_free(h->transfer);
  dev_free(h->d_labels, (size_t)h->g.N * 2 * sizeof(int));
  dev_free(h->d_drop, h->drop_bytes);
  dev_free(h->d_trig, trig_bytes(h->g));
  dev_free(h->d_ring, sizeof(double) * DIAG_STRIDE * lbm_ctx::kRing);
  dev_free(h->d_ring_count, sizeof(unsigned long long));
  if (h->own_stream) cudaStreamDestroy(h->own_stream);
  delete h;
}

lbm_handle lbm_create_ex(const lbm_config* cfg) {
  if (validate(cfg) != LBM_OK) return nullptr;
  lbm_ctx* h = new (std::nothrow) lbm_ctx();
  if (!h) {
    fail(LBM_ERR_OOM, "host allocation failed");
    return nullptr;
  }
  h->cfg = *cfg;
  const long long N = (long long)cfg->nx * cfg->ny * cfg->nz;
  h->g = Geom{cfg->nx, cfg->ny, cfg->nz, N, N <= kChainNodes ? 1 : 0};
  // stochastic rounding is on by default for the reduced-precision forms
  h->ph = Phys{cfg->tau, cfg->G, cfg->rho0, cfg->rho_ref, cfg->psi_form,
               cfg->precision >= LBM_F16DEV ? 1 : 0, COLL_SRT, 1.19, 1.4, 1.2, 1.4, 1.98};
  h->ph.inv_rho0 = 1.0 / cfg->rho0;
  phys_finalize(h->ph, cfg->precision);
  h->block_asked = cfg->block_x && cfg->block_y && cfg->block_z;
  h->block = h->block_asked ? dim3(cfg->block_x, cfg->block_y, cfg->block_z) : default_block(h->g);
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) {
    cudaDeviceProp prop;
    e = cudaGetDeviceProperties(&prop, dev);
    if (e == cudaSuccess && !(prop.major == 10 && prop.minor == 3)) {
      fail(LBM_ERR_CUDA, "liblbm.so is built for sm_103a (GB300); device has compute capability " +
                             std::to_string(prop.major) + "." + std::to_string(prop.minor));
      delete h;
      return nullptr;
    }
  }
  if (e != cudaSuccess) {
    cuda_fail(e, "cudaGetDevice");
    delete h;
    return nullptr;
  }
  h->device = dev;
  sizes_for(cfg, &h->state_bytes, &h->psi_bytes);
  int rc = LBM_OK;
  if (cfg->stream) {
    h->stream = (cudaStream_t)cfg->stream;
  } else {
    e = cudaStreamCreateWithFlags(&h->own_stream, cudaStreamNonBlocking);
    if (e != cudaSuccess) rc = cuda_fail(e, "cudaStreamCreate");
    h->stream = h->own_stream;
  }
  if (rc == LBM_OK) {
    if (cfg->ext_state) {
      if (cfg->ext_state_bytes < h->state_bytes)
        rc = fail(LBM_ERR_ARG, "ext_state_bytes smaller than required");
      else if ((uintptr_t)cfg->ext_state % elem_size(cfg->precision))
        rc = fail(LBM_ERR_ARG, "ext_state is not aligned to its elements");
      h->state = cfg->ext_state;
    } else {
      rc = dev_alloc(&h->state, h->state_bytes, "populations");
      h->own_state = rc == LBM_OK;
    }
  }
  if (rc == LBM_OK) {
    if (cfg->ext_psi) {
      if (cfg->ext_psi_bytes < h->psi_bytes) rc = fail(LBM_ERR_ARG, "ext_psi_bytes smaller than required");
      else if ((uintptr_t)cfg->ext_psi % (cfg->precision == LBM_F64 ? 8 : 4))
        rc = fail(LBM_ERR_ARG, "ext_psi is not aligned to its elements");
      h->psi = cfg->ext_psi;
    } else {
      rc = dev_alloc(&h->psi, h->psi_bytes, "psi");
      h->own_psi = rc == LBM_OK;
    }
  }
  h->aligned = buffers_aligned(h);
  if (rc == LBM_OK) rc = dev_alloc((void**)&h->d_flag, sizeof(int) * 4, "flag");
  if (rc == LBM_OK) h->ph.salt = (const unsigned*)(h->d_flag + 2);
  if (rc == LBM_OK) rc = dev_alloc((void**)&h->d_small, sizeof(double) * 64, "results");
  // (where there is no room for the table, psi is computed by exp)
  if (rc == LBM_OK && cfg->precision == LBM_F64 && !over_total_cap(sizeof(double2) * kPsiTab) &&
      dev_alloc((void**)&h->d_psi_tab, sizeof(double2) * kPsiTab, "psi table") == LBM_OK) {
    e = psi_table_launch(h->d_psi_tab, h->stream);
    if (e != cudaSuccess) rc = cuda_fail(e, "psi table");
    h->ph.psi_tab = h->d_psi_tab;
  }
  if (rc == LBM_OK) {
    e = cudaMemsetAsync(h->d_flag, 0, sizeof(int) * 4, h->stream);
    if (e == cudaSuccess) e = cudaMemsetAsync(h->state, 0, h->state_bytes, h->stream);
    if (e == cudaSuccess) e = cudaStreamSynchronize(h->stream);
    if (e != cudaSuccess) rc = cuda_fail(e, "initial clear");
  }
  if (rc != LBM_OK) {
    std::string msg = g_last_error;
    lbm_destroy(h);
    g_last_error = msg;
    return nullptr;
  }
  return h;
}

lbm_handle lbm_create(int nx, int ny, int nz, double tau, double G, int psi_form) {
  lbm_config c;
  lbm_config_default(&c);
  c.nx = nx;
  c.ny = ny;
  c.nz = nz;
  c.tau = tau;
  c.G = G;
  c.psi_form = psi_form;
  return lbm_create_ex(&c);
}

int lbm_set_stream(lbm_handle h, void* stream) {
  if (!h) return fail(LBM_ERR_ARG, "null handle");
  CK(cudaStreamSynchronize(h->stream));
  h->stream = stream ? (cudaStream_t)stream : h->own_stream;
  if (!h->stream) {
    CK(cudaStreamCreateWithFlags(&h->own_stream, cudaStreamNonBlocking));
    h->stream = h->own_stream;
  }
  return LBM_OK;
}

int lbm_set_option(lbm_handle h, const char* key, double v) {
  if (!h || !key) return fail(LBM_ERR_ARG, "null handle or key");
  const std::string k(key);
  if (!std::isfinite(v)) return fail(LBM_ERR_ARG, "option value must be finite");
  if (k == "tau") {
    if (!(v > 0.5)) return fail(LBM_ERR_ARG, "tau must be > 1/2");
    h->ph.tau = h->cfg.tau = v;
    phys_finalize(h->ph, h->cfg.precision);
    drop_graphs(h);
  } else if (k == "G") {
    h->ph.G = h->cfg.G = v;
    phys_finalize(h->ph, h->cfg.precision);
    drop_graphs(h);
  } else if (k == "rho_l") {
    h->rho_l = v;
    drop_graphs(h);   // the in-loop diagnostics capture the densities
  } else if (k == "rho_v") {
    h->rho_v = v;
    drop_graphs(h);
  } else if (k == "graph") {
    h->use_graph = v != 0.0;
  } else if (k == "stochastic_rounding") {
    h->ph.sr = v != 0.0 ? 1 : 0;
    drop_graphs(h);
  } else if (k == "collision") {
    if (v != 0.0 && v != 1.0) return fail(LBM_ERR_ARG, "collision must be 0 (SRT) or 1 (MRT)");
    h->ph.coll = v != 0.0 ? COLL_MRT : COLL_SRT;
    drop_graphs(h);
  } else if (k == "mrt_s_e" || k == "mrt_s_eps" || k == "mrt_s_q" || k == "mrt_s_pi" || k == "mrt_s_m") {
    if (!(v > 0.0 && v < 2.0)) return fail(LBM_ERR_ARG, "MRT relaxation rates must lie in (0, 2)");
    if (k == "mrt_s_e") h->ph.s_e = v;
    if (k == "mrt_s_eps") h->ph.s_eps = v;
    if (k == "mrt_s_q") h->ph.s_q = v;
    if (k == "mrt_s_pi") h->ph.s_pi = v;
    if (k == "mrt_s_m") h->ph.s_m = v;
    phys_finalize(h->ph, h->cfg.precision);
    drop_graphs(h);
  } else if (k == "fused") {
    h->fused = v == 0.0 ? 0 : (v == 2.0 ? 2 : 1);
    drop_graphs(h);
    if (!h->fused && h->pads.p) {   // no step uses the padded arrays any more
      CK(cudaStreamSynchronize(h->stream));
      spare_free(h->pads);
    }
    h->pad_failed = false;
    if (h->diag_interval > 0) {
      int rc = ensure_scratch(h);
      if (rc) return rc;
    }
  } else if (k == "fused_stall_test") {
    if (!(v >= 0.0 && v <= 10.0)) return fail(LBM_ERR_ARG, "fused_stall_test must be in 0..10 ms");
    h->fused_stall_test_ns = (unsigned long long)(v * 1e6);
    drop_graphs(h);
  } else if (k == "fused_group") {
    const long long gr = (long long)v;
    if (gr < 0 || gr > (1LL << 20) || (double)gr != v)
      return fail(LBM_ERR_ARG, "fused_group must be a non-negative integer");
    h->fused_group = (int)gr;
    drop_graphs(h);
  } else if (k == "fused_fz") {
    const long long z = (long long)v;
    if (z < 0 || z > h->g.nz || (double)z != v) return fail(LBM_ERR_ARG, "fused_fz must be an integer in 0..nz");
    h->fused_fz = (int)z;
    drop_graphs(h);
    if (h->diag_interval > 0) {
      int rc = ensure_scratch(h);
      if (rc) return rc;
    }
  } else if (k == "vector") {
    h->vec = v != 0.0;
    drop_graphs(h);
  } else if (k == "occupancy") {
    if (v != 0.0 && v != 2.0 && v != 3.0 && v != 4.0) return fail(LBM_ERR_ARG, "occupancy must be 0 (auto), 2, 3 or 4");
    h->minb = (int)v;
    drop_graphs(h);
  } else if (k == "diag_interval") {
    const long long d = (long long)v;
    if (d < 0 || d > 1000000 || (double)d != v) return fail(LBM_ERR_ARG, "diag_interval must be an integer in 0..1e6");
    if (d > 0) {
      int rc = ensure_scratch(h);
      if (rc == LBM_OK) rc = ensure_ring(h);
      if (rc) return rc;
    }
    h->diag_interval = (int)d;
    drop_graphs(h);
  } else if (k == "diag_ccl") {
    if (v != 0.0) {
      int rc = ensure_labels(h);
      if (rc) return rc;
    }
    h->diag_ccl = v != 0.0;
    drop_graphs(h);
  } else if (k == "kernel_timing") {
    if (v != 0.0 && !h->kernel_timing) {
      int rc = settle_timing(h);
      if (rc) return rc;
      for (int c = 0; c < 3; ++c) {
        h->t_launches[c] = 0;
        h->t_ms[c] = 0.0;
      }
    }
    h->kernel_timing = v != 0.0;
  } else if (k == "block_x" || k == "block_y" || k == "block_z") {
    const long long b = (long long)v;
    if (b < 1 || b > 256 || (double)b != v) return fail(LBM_ERR_ARG, "block size must be an integer in 1..256");
    dim3 nb = h->block;
    if (k == "block_x") nb.x = (unsigned)b;
    if (k == "block_y") nb.y = (unsigned)b;
    if (k == "block_z") nb.z = (unsigned)b;
    if ((long long)nb.x * nb.y * nb.z > 256 || nb.z > 64)
      return fail(LBM_ERR_ARG, "block shape has more than 256 threads");
    h->block = nb;
    h->block_asked = true;
    drop_graphs(h);
  } else {
    return fail(LBM_ERR_ARG, "unknown option " + k);
  }
  return LBM_OK;
}

int lbm_get_option(lbm_handle h, const char* key, double* v) {
  if (!h || !key || !v) return fail(LBM_ERR_ARG, "null argument");
  const std::string k(key);
  if (k == "tau") *v = h->ph.tau;
  else if (k == "G") *v = h->ph.G;
  else if (k == "rho_l") *v = h->rho_l;
  else if (k == "rho_v") *v = h->rho_v;
  else if (k == "graph") *v = h->use_graph;
  else if (k == "diag_interval") *v = h->diag_interval;
  else if (k == "diag_ccl") *v = h->diag_ccl;
  else if (k == "occupancy")
    *v = h->minb ? h->minb
                 : auto_minb(node_pairs(h->cfg.precision, vector_form(h), h->g), h->cfg.pattern == LBM_AA ? MODE_AA_ODD : MODE_AB,
                             h->cfg.precision, h->g.N);
  else if (k == "vector") *v = vector_form(h) && (h->g.nx % 2 == 0);
  else if (k == "stochastic_rounding") *v = h->ph.sr;
  else if (k == "fused")
    *v = h->fused && h->cfg.pattern == LBM_AB && fused_applicable(h->g, h->cfg.precision);
  else if (k == "fused_fz") *v = h->fused_fz;
  else if (k == "fused_group") *v = h->fused_group;
  else if (k == "fused_fz_used" || k == "fused_group_used") {
    int fz = 0, grp = 0;
    if (fused_applicable(h->g, h->cfg.precision)) {
      const cudaError_t e = fused_launch_shape(h->cfg.precision, h->g, h->ph.coll, h->fused_fz, h->fused_group, &fz, &grp);
      if (e != cudaSuccess) return cuda_fail(e, "fused launch shape");
    }
    *v = k == "fused_fz_used" ? fz : grp;
  }
  else if (k == "fused_stall_test") *v = h->fused_stall_test_ns * 1e-6;
  else if (k == "collision") *v = h->ph.coll;
  else if (k == "mrt_s_e") *v = h->ph.s_e;
  else if (k == "mrt_s_eps") *v = h->ph.s_eps;
  else if (k == "mrt_s_q") *v = h->ph.s_q;
  else if (k == "mrt_s_pi") *v = h->ph.s_pi;
  else if (k == "mrt_s_m") *v = h->ph.s_m;
  else if (k == "kernel_timing") *v = h->kernel_timing;
  else if (k == "block_x") *v = h->block.x;
  else if (k == "block_y") *v = h->block.y;
  else if (k == "block_z") *v = h->block.z;
  else if (k == "step") *v = (double)h->step;
  else if (k == "nx") *v = h->g.nx;
  else if (k == "ny") *v = h->g.ny;
  else if (k == "nz") *v = h->g.nz;
  else if (k == "precision") *v = h->cfg.precision;
  else if (k == "pattern") *v = h->cfg.pattern;
  else return fail(LBM_ERR_ARG, "unknown option " + k);
  return LBM_OK;
}

static int init_common(lbm_handle h, const InitSpec& sp) {
  h->step = 0;
  h->cur = 0;
  CK(launch_salt((unsigned*)(h->d_flag + 2), true, 0u, h->stream));
  drop_graphs(h);   // the in-loop diagnostics capture the densities
  CK(launch_init(h->cfg.precision, h->g, h->ph, sp, array_ptr(h, 0), h->stream));
  h->initialized = true;
  return LBM_OK;
}

int lbm_init_ligament(lbm_handle h, double R0, double lambda, double eps, double phase, double rho_l,
                      double rho_v, double width) {
  if (!h) return fail(LBM_ERR_ARG, "null handle");
  for (double v : {R0, lambda, eps, phase, rho_l, rho_v, width})
    if (!std::isfinite(v)) return fail(LBM_ERR_ARG, "non-finite ligament parameter");
  if (!(rho_l > rho_v) || !(rho_v > 0.0)) return fail(LBM_ERR_ARG, "need rho_l > rho_v > 0");
  if (!(width > 0.0) || !(lambda > 0.0) || !(R0 >= 0.0)) return fail(LBM_ERR_ARG, "need width, lambda > 0, R0 >= 0");
  InitSpec sp{R0, lambda, eps, phase, rho_l, rho_v, width, nullptr, 0, 0.0, 1.0};
  h->rho_l = rho_l;
  h->rho_v = rho_v;
  return init_common(h, sp);
}

int lbm_init_profile(lbm_handle h, double R0, double lambda, double eps, double phase, const double* prof,
                     int n, double d0, double dd) {
  if (!h || !prof) return fail(LBM_ERR_ARG, "null argument");
  if (n < 2 || !(dd > 0.0) || !std::isfinite(d0) || !std::isfinite(dd) || !(lambda > 0.0))
    return fail(LBM_ERR_ARG, "need n >= 2, dd > 0, lambda > 0");
  double lo = prof[0], hi = prof[0];
  for (int k = 0; k < n; ++k) {
    if (!std::isfinite(prof[k]) || !(prof[k] > 0.0)) return fail(LBM_ERR_ARG, "profile must be finite and > 0");
    lo = prof[k] < lo ? prof[k] : lo;
    hi = prof[k] > hi ? prof[k] : hi;
  }
  double* dprof = nullptr;
  int rc = dev_alloc((void**)&dprof, sizeof(double) * n, "profile");
  if (rc) return rc;
  cudaError_t e = cudaMemcpyAsync(dprof, prof, sizeof(double) * n, cudaMemcpyHostToDevice, h->stream);
  if (e != cudaSuccess) {
    dev_free(dprof, sizeof(double) * n);
    return cuda_fail(e, "profile upload");
  }
  InitSpec sp{R0, lambda, eps, phase, hi, lo, 1.0, dprof, n, d0, dd};
  h->rho_l = hi;
  h->rho_v = lo;
  rc = init_common(h, sp);
  e = cudaStreamSynchronize(h->stream);
  dev_free(dprof, sizeof(double) * n);
  if (rc == LBM_OK && e != cudaSuccess) rc = cuda_fail(e, "init_profile");
  return rc;
}

int lbm_step(lbm_handle h, int n) {
  if (!h) return fail(LBM_ERR_ARG, "null handle");
  if (n < 0) return fail(LBM_ERR_ARG, "negative step count");
  if (!h->initialized) return fail(LBM_ERR_STATE, "lattice not initialised");
  const bool aa = h->cfg.pattern == LBM_AA;
  const SpareUse use(h->pads);
  if (h->pad_graphs && !h->pads.p) {   // given back since the last call
    drop_graphs(h);
    h->pad_failed = true;
  }
  const int base = chunk_len(h);
  const long long first = (h->step + base - 1) / base * base;   // the first step a graph may start at
  if (h->use_graph && !h->kernel_timing && base > 1 && h->step + n >= first + base) ensure_padded(h);
  const int longer = long_chunk_len(h);
  const int k = h->diag_interval;
  if (h->graph_chunk != base) {
    drop_graphs(h);
    h->graph_chunk = base;
  }
  while (n > 0) {
    if (h->use_graph && !h->kernel_timing && n >= base && h->step % base == 0) {
      const int phase = aa ? 0 : h->cur;
      const int C = n >= longer && (h->graph[phase][1] || padded_form(h) ||
                                    h->replays + n / base - n / longer >= 2 * longer)
                        ? longer
                        : base;
      h->replays += C == base;
      cudaGraphExec_t& ge = h->graph[phase][C != base];
      if (!ge) {
        int rc = capture_chunk(h, phase, C, &ge);
        if (rc) return rc;
      }
      CK(cudaGraphLaunch(ge, h->stream));
      if (k > 0)
        for (long long t = h->step; t < h->step + C; t += k) h->diag_steps.push_back(t);
      if (!aa && (C & 1)) h->cur ^= 1;
      h->step += C;
      n -= C;
    } else {
      int rc = enqueue_step(h, h->stream, h->step, h->cur, h->kernel_timing);
      if (rc) return rc;
      if (k > 0 && h->step % k == 0) h->diag_steps.push_back(h->step);
      if (!aa) h->cur ^= 1;
      h->step += 1;
      n -= 1;
    }
  }
  return LBM_OK;
}

int lbm_diag_history(lbm_handle h, lbm_diag* out, int max_records, int* count) {
  if (!h || !count || max_records < 0 || (max_records > 0 && !out)) return fail(LBM_ERR_ARG, "bad argument");
  *count = 0;
  const long long total = (long long)h->diag_steps.size();
  if (!h->d_ring || total == h->diag_fetched) {
    CK(cudaStreamSynchronize(h->stream));
    return LBM_OK;
  }
  long long first = h->diag_fetched;
  if (total - first > lbm_ctx::kRing) first = total - lbm_ctx::kRing;  // older records were overwritten
  if (total - first > max_records) first = total - max_records;
  // the records' slots are one or two runs of the ring; one wait for all
  std::vector<double> rec((size_t)(total - first) * DIAG_STRIDE);
  unsigned long long dev_total = 0;
  CK(cudaMemcpyAsync(&dev_total, h->d_ring_count, sizeof(dev_total), cudaMemcpyDeviceToHost, h->stream));
  for (long long r = first; r < total;) {
    const long long slot = r % lbm_ctx::kRing, run = std::min(total - r, (long long)lbm_ctx::kRing - slot);
    CK(cudaMemcpyAsync(&rec[(size_t)(r - first) * DIAG_STRIDE], h->d_ring + slot * DIAG_STRIDE,
                       sizeof(double) * DIAG_STRIDE * run, cudaMemcpyDeviceToHost, h->stream));
    r += run;
  }
  CK(cudaStreamSynchronize(h->stream));
  if ((long long)dev_total != total) return fail(LBM_ERR_STATE, "diagnostics ring out of step with the host log");
  int n = 0;
  for (long long r = first; r < total; ++r) {
    const double* v = &rec[(size_t)(r - first) * DIAG_STRIDE];
    fill_diag(&out[n], v, h->diag_steps[(size_t)r]);
    if (v[DIAG_CCL + 3] != 0.0) return fail(LBM_ERR_TIMEOUT, "connected-component labelling guard tripped");
    out[n].droplets = (int)v[DIAG_CCL];
    out[n].droplets_min8 = (int)v[DIAG_CCL + 1];
    out[n].largest_droplet = (long long)v[DIAG_CCL + 2];
    ++n;
  }
  h->diag_fetched = total;
  *count = n;
  return LBM_OK;
}

int lbm_sync(lbm_handle h) {
  if (!h) return fail(LBM_ERR_ARG, "null handle");
  int flag = 0;
  CK(cudaMemcpyAsync(&flag, h->d_flag, sizeof(int), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  if (flag) {
    CK(cudaMemsetAsync(h->d_flag, 0, sizeof(int), h->stream));
    CK(cudaStreamSynchronize(h->stream));
    if (flag & 2) return fail(LBM_ERR_TIMEOUT, "a staged copy of the fused step did not complete in time");
    return fail(LBM_ERR_NUMERIC, "a density became non-positive or non-finite");
  }
  return LBM_OK;
}

int lbm_moments(lbm_handle h, double* rho, double* ux, double* uy, double* uz) {
  if (!h) return fail(LBM_ERR_ARG, "null handle");
  if (!h->initialized) return fail(LBM_ERR_STATE, "lattice not initialised");
  const int layout = cur_layout(h);
  const void* f = cur_array(h);
  CK(launch_psi(h->cfg.precision, layout, vector_form(h), h->g, h->ph, f, h->psi, h->d_flag, h->stream));
  double* outs[4] = {rho, ux, uy, uz};
  int want = 0;
  for (double* o : outs) want += o != nullptr;
  int rc = begin_transfer(h, want > 0 ? want : 1);
  if (rc) return rc;
  // the requested fields together where the planes hold them, else one by one
  const long long N = h->g.N;
  double* const room = (double*)h->transfer.p;
  const bool together = h->transfer.bytes >= (size_t)want * N * sizeof(double);
  cudaError_t e = cudaSuccess;
  double* dev[4] = {nullptr, nullptr, nullptr, nullptr};
  for (int k = 0, n = 0; k < 4; ++k)
    if (outs[k]) dev[k] = room + (together ? (n++) * N : 0);
  if (together)
    e = launch_moments(h->cfg.precision, layout, h->g, h->ph, f, h->psi, dev[0], dev[1], dev[2], dev[3], h->stream);
  for (int k = 0; k < 4 && e == cudaSuccess; ++k) {
    if (!outs[k]) continue;
    if (!together)
      e = launch_moments(h->cfg.precision, layout, h->g, h->ph, f, h->psi, k == 0 ? dev[0] : nullptr,
                         k == 1 ? dev[1] : nullptr, k == 2 ? dev[2] : nullptr, k == 3 ? dev[3] : nullptr, h->stream);
    if (e == cudaSuccess) e = cudaMemcpyAsync(outs[k], dev[k], sizeof(double) * N, cudaMemcpyDeviceToHost, h->stream);
  }
  const cudaError_t e2 = cudaStreamSynchronize(h->stream);
  end_transfer(h);
  if (e == cudaSuccess) e = e2;
  return e == cudaSuccess ? LBM_OK : cuda_fail(e, "moments");
}

int lbm_diagnostics(lbm_handle h, lbm_diag* out, int want_ccl) {
  if (!h || !out) return fail(LBM_ERR_ARG, "null argument");
  if (!h->initialized) return fail(LBM_ERR_STATE, "lattice not initialised");
  int rc = ensure_scratch(h);
  if (rc) return rc;
  const int layout = cur_layout(h);
  const void* f = cur_array(h);
  const double thr = 0.5 * (h->rho_l + h->rho_v);
  DiagExtra x;
  if (want_ccl) {
    rc = ensure_labels(h);
    if (rc) return rc;
    x = diag_labels(h->cfg.precision, layout, h->g, f, nullptr, thr, h->d_labels, h->d_labels + h->g.N);
  }
  CK(launch_diagnostics(h->cfg.precision, layout, h->g, h->ph, f, h->rho_l, h->rho_v, h->d_scratch,
                        h->d_small, nullptr, nullptr, nullptr, 0, h->stream, x));
  double r[DIAG_OUT];
  long long c4[4] = {-1, -1, -1, 0};
  if (want_ccl) {
    long long* d4 = (long long*)(h->d_small + 32);
    CK(launch_ccl(h->cfg.precision, layout, h->g, h->ph, f, thr, h->d_labels, h->d_labels + h->g.N, d4, h->stream,
                  x.labels != nullptr));
    CK(cudaMemcpyAsync(c4, d4, sizeof(c4), cudaMemcpyDeviceToHost, h->stream));
  }
  CK(cudaMemcpyAsync(r, h->d_small, sizeof(r), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  if (want_ccl && c4[3]) return fail(LBM_ERR_TIMEOUT, "connected-component labelling guard tripped");
  fill_diag(out, r, h->step);
  out->droplets = (int)c4[0];
  out->droplets_min8 = (int)c4[1];
  out->largest_droplet = c4[2];
  return LBM_OK;
}

int lbm_droplets(lbm_handle h, lbm_droplet* out, int max_droplets, int* count) {
  if (!h || !count || max_droplets < 0 || (max_droplets > 0 && !out)) return fail(LBM_ERR_ARG, "bad argument");
  if (!h->initialized) return fail(LBM_ERR_STATE, "lattice not initialised");
  *count = 0;
  int rc = ensure_labels(h);
  if (rc) return rc;
  const int layout = cur_layout(h);
  const void* f = cur_array(h);
  long long* d4 = (long long*)(h->d_small + 32);
  int* L = h->d_labels;
  int* sizes = h->d_labels + h->g.N;
  if (!h->d_trig) {
    rc = dev_alloc((void**)&h->d_trig, trig_bytes(h->g), "angles");
    if (rc) return rc;
    CK(launch_trig(h->g, h->d_trig, h->stream));
  }
  CK(launch_ccl(h->cfg.precision, layout, h->g, h->ph, f, 0.5 * (h->rho_l + h->rho_v), L, sizes, d4, h->stream, false,
                true));
  long long c4[4];
  CK(cudaMemcpyAsync(c4, d4, sizeof(c4), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  if (c4[3]) return fail(LBM_ERR_TIMEOUT, "connected-component labelling guard tripped");
  const long long nd = c4[0];
  *count = (int)nd;
  if (nd == 0) return LBM_OK;
  const int words = (h->g.nx + 31) / 32;
  const size_t rec_bytes = sizeof(double) * DROP_REC * (size_t)nd;
  const size_t need = rec_bytes + sizeof(unsigned) * (size_t)words * nd;
  if (need > h->drop_bytes) {
    dev_free(h->d_drop, h->drop_bytes);
    h->d_drop = nullptr;
    h->drop_bytes = 0;
    rc = dev_alloc((void**)&h->d_drop, need, "droplet records");
    if (rc) return rc;
    h->drop_bytes = need;
  }
  double* rec = h->d_drop;
  unsigned* xbits = (unsigned*)((char*)h->d_drop + rec_bytes);
  CK(launch_droplets(h->cfg.precision, layout, h->g, h->ph, f, h->rho_l, h->rho_v, L, sizes, h->d_trig, rec, xbits,
                     (int)nd, h->stream));
  std::vector<double> hr((size_t)DROP_REC * nd);
  std::vector<unsigned> hb((size_t)words * nd);
  CK(cudaMemcpyAsync(hr.data(), rec, rec_bytes, cudaMemcpyDeviceToHost, h->stream));
  CK(cudaMemcpyAsync(hb.data(), xbits, sizeof(unsigned) * hb.size(), cudaMemcpyDeviceToHost, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  std::vector<lbm_droplet> d((size_t)nd);
  const double two_pi = 6.283185307179586476925286766559;
  const int dims[3] = {h->g.nx, h->g.ny, h->g.nz};
  for (long long k = 0; k < nd; ++k) {
    const double* r = &hr[(size_t)k * DROP_REC];
    lbm_droplet& o = d[(size_t)k];
    o.first_node = (long long)r[0];
    o.nodes = (long long)r[1];
    o.volume_w = r[2];
    o.mass = r[3];
    for (int a = 0; a < 3; ++a) {
      const double c = r[4 + 2 * a], sn = r[5 + 2 * a];
      double t = std::atan2(sn, c);
      if (t < 0.0) t += two_pi;
      double pos = t / two_pi * dims[a];
      if (pos >= dims[a]) pos -= dims[a];
      o.centroid[a] = pos;
      o.resultant[a] = std::sqrt(c * c + sn * sn) / r[1];
    }
    int xs = 0;
    for (int w = 0; w < words; ++w) xs += __builtin_popcount(hb[(size_t)k * words + w]);
    o.x_slices = xs;
    o.reserved = 0;
  }
  std::sort(d.begin(), d.end(), [](const lbm_droplet& a, const lbm_droplet& b) {
    return a.nodes != b.nodes ? a.nodes > b.nodes : a.first_node < b.first_node;
  });
  const long long n = std::min<long long>(nd, max_droplets);
  for (long long k = 0; k < n; ++k) out[k] = d[(size_t)k];
  return LBM_OK;
}

int lbm_get_populations(lbm_handle h, double* host) {
  if (!h || !host) return fail(LBM_ERR_ARG, "null argument");
  int rc = begin_transfer(h, Q);
  if (rc) return rc;
  const cudaError_t e = export_populations(h->cfg.precision, cur_layout(h), h->g, h->ph, cur_array(h),
                                           (double*)h->transfer.p, h->transfer.bytes / sizeof(double), host, h->stream);
  end_transfer(h);
  return e == cudaSuccess ? LBM_OK : cuda_fail(e, "get_populations");
}

int lbm_set_populations(lbm_handle h, const double* host) {
  if (!h || !host) return fail(LBM_ERR_ARG, "null argument");
  int rc = begin_transfer(h, Q);
  if (rc) return rc;
  const cudaError_t e = import_populations(h->cfg.precision, cur_layout(h), h->g, h->ph, cur_array(h),
                                           (double*)h->transfer.p, h->transfer.bytes / sizeof(double), host, h->stream);
  end_transfer(h);
  if (e != cudaSuccess) return cuda_fail(e, "set_populations");
  h->initialized = true;
  return LBM_OK;
}

int lbm_state_bytes(lbm_handle h, size_t* bytes) {
  if (!h || !bytes) return fail(LBM_ERR_ARG, "null argument");
  *bytes = sizeof(StateHeader) + (size_t)Q * h->g.N * elem_size(h->cfg.precision);
  return LBM_OK;
}

int lbm_save_state(lbm_handle h, void* host, size_t bytes) {
  size_t need = 0;
  int rc = lbm_state_bytes(h, &need);
  if (rc) return rc;
  if (!host || bytes < need) return fail(LBM_ERR_ARG, "buffer too small for the state");
  StateHeader hd;
  std::memset(&hd, 0, sizeof(hd));
  std::memcpy(hd.magic, "LBMD3Q19", 8);
  hd.version = 1;
  hd.precision = h->cfg.precision;
  hd.pattern = h->cfg.pattern;
  hd.nx = h->g.nx;
  hd.ny = h->g.ny;
  hd.nz = h->g.nz;
  hd.cur = 0;
  hd.step = h->step;
  hd.rho_l = h->rho_l;
  hd.rho_v = h->rho_v;
  std::memcpy(host, &hd, sizeof(hd));
  CK(cudaMemcpyAsync((char*)host + sizeof(hd), cur_array(h), need - sizeof(hd), cudaMemcpyDeviceToHost,
                     h->stream));
  CK(cudaStreamSynchronize(h->stream));
  return LBM_OK;
}

int lbm_load_state(lbm_handle h, const void* host, size_t bytes) {
  size_t need = 0;
  int rc = lbm_state_bytes(h, &need);
  if (rc) return rc;
  if (!host || bytes < need) return fail(LBM_ERR_ARG, "buffer too small for the state");
  StateHeader hd;
  std::memcpy(&hd, host, sizeof(hd));
  if (std::memcmp(hd.magic, "LBMD3Q19", 8) != 0 || hd.version != 1)
    return fail(LBM_ERR_ARG, "not a saved lattice state");
  if (hd.precision != h->cfg.precision || hd.pattern != h->cfg.pattern || hd.nx != h->g.nx || hd.ny != h->g.ny ||
      hd.nz != h->g.nz)
    return fail(LBM_ERR_ARG, "saved state has another size, precision or pattern");
  h->cur = 0;
  h->step = hd.step;
  CK(launch_salt((unsigned*)(h->d_flag + 2 + salt_word(h, h->step, h->cur)), true, (unsigned)hd.step, h->stream));
  // the in-loop diagnostics capture the densities
  if (hd.rho_l != h->rho_l || hd.rho_v != h->rho_v) drop_graphs(h);
  h->rho_l = hd.rho_l;
  h->rho_v = hd.rho_v;
  CK(cudaMemcpyAsync(array_ptr(h, 0), (const char*)host + sizeof(hd), need - sizeof(hd),
                     cudaMemcpyHostToDevice, h->stream));
  CK(cudaStreamSynchronize(h->stream));
  h->initialized = true;
  return LBM_OK;
}

int lbm_kernel_time(lbm_handle h, int k, long long* launches, double* ms) {
  if (!h || k < 0 || k > 2) return fail(LBM_ERR_ARG, "bad handle or kernel class");
  int rc = settle_timing(h);
  if (rc) return rc;
  if (launches) *launches = h->t_launches[k];
  if (ms) *ms = h->t_ms[k];
  return LBM_OK;
}

}  // extern "C"

namespace lbm {
// The allocation cap of LBM_ALLOC_CAP_BYTES for one request of `bytes`
// (the batched form's pools; the single lattice also counts what it holds).
bool alloc_over_cap(size_t bytes) {
  const char* cap = std::getenv("LBM_ALLOC_CAP_BYTES");
  return cap && *cap && bytes > std::strtoull(cap, nullptr, 10);
}

void spare_enter(Spare& s) {
  std::lock_guard<std::mutex> lock(g_spare_mu);
  s.busy = true;
}
void spare_leave(Spare& s) {
  std::lock_guard<std::mutex> lock(g_spare_mu);
  s.busy = false;
}
void spare_free(Spare& s) {
  std::lock_guard<std::mutex> lock(g_spare_mu);
  spare_drop(s);
}
cudaError_t spare_alloc(Spare& s, size_t bytes, bool capped) {
  std::lock_guard<std::mutex> lock(g_spare_mu);
  spare_drop(s);
  if (capped && over_total_cap(bytes)) return cudaErrorMemoryAllocation;
  cudaError_t e = cudaGetDevice(&s.device);
  if (e == cudaSuccess) e = cudaMalloc(&s.p, bytes);
  if (e != cudaSuccess) {
    (void)cudaGetLastError();
    s.p = nullptr;
    return e;
  }
  g_alloc_total += bytes;
  s.bytes = bytes;
  s.next = g_spares;
  g_spares = &s;
  return cudaSuccess;
}
cudaError_t transfer_room(Spare& s, long long N, int planes, bool capped) {
  const size_t all = sizeof(double) * transfer_doubles(N, planes), one = sizeof(double) * (size_t)N;
  if (s.bytes >= all) return cudaSuccess;
  cudaError_t e = spare_alloc(s, all, true);
  if (e == cudaErrorMemoryAllocation) e = spare_alloc(s, one, capped);
  if (e == cudaErrorMemoryAllocation && spares_give_back()) e = spare_alloc(s, one, capped);
  return e;
}
cudaError_t device_alloc(void** p, size_t bytes) {
  cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation && spares_give_back()) {
    (void)cudaGetLastError();
    e = cudaMalloc(p, bytes);
  }
  if (e != cudaSuccess) *p = nullptr;
  return e;
}
}  // namespace lbm
