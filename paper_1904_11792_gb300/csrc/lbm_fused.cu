// Fused time step, host side: the tensor maps of the population arrays, the
// launch shape (z-run length, runs per block-order group, blocks) and the
// launches of the kernel in lbm_fused_kernel.cuh.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstring>
#include <map>
#include <mutex>
#include <tuple>
#include <vector>

#include "lbm_fused_kernel.cuh"

namespace lbm {

namespace {

// Tile rows of the fused step for a storage precision (FusedShape<P>::TY).
int fused_tile_rows(int precision) {
  return precision == LBM_F16DEV ? FusedShape<LBM_F16DEV>::TY
                                 : (precision == LBM_BF16DEV ? FusedShape<LBM_BF16DEV>::TY : FusedShape<LBM_F32>::TY);
}

// ---- tensor maps ------------------------------------------------------------

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
  });
  return fn;
}

CUtensorMapDataType tma_type(int precision) {
  switch (precision) {
    case LBM_F64: return CU_TENSOR_MAP_DATA_TYPE_FLOAT64;
    case LBM_F32: return CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
    case LBM_F16DEV: return CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
    default: return CU_TENSOR_MAP_DATA_TYPE_BFLOAT16;
  }
}

// The 4-D view [19][nz][ny][nx] of a population array with box (bx, by, 1, 19),
// rows px elements apart (px = nx, or nx padded for the batched step).
cudaError_t make_map(CUtensorMap* tm, int precision, const Geom& g, const void* base, int bx, int by, int px = 0) {
  auto fn = encode_fn();
  if (!fn) return cudaErrorNotSupported;
  const size_t e = elem_size(precision);
  const cuuint64_t p = px > 0 ? (cuuint64_t)px : (cuuint64_t)g.nx;
  const cuuint64_t dims[4] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz, (cuuint64_t)Q};
  const cuuint64_t strides[3] = {p * e, p * g.ny * e, p * g.ny * g.nz * e};
  const cuuint32_t box[4] = {(cuuint32_t)bx, (cuuint32_t)by, 1u, (cuuint32_t)Q};
  const cuuint32_t estr[4] = {1u, 1u, 1u, 1u};
  const CUresult r = fn(tm, tma_type(precision), 4, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Tensor maps are pure host-side descriptors; they are cached per array.
cudaError_t maps_for(int precision, const Geom& g, const void* base, Maps* out) {
  static std::mutex mu;
  static std::map<std::tuple<const void*, int, int, int, int>, Maps> cache;
  const auto key = std::make_tuple(base, precision, g.nx, g.ny, g.nz);
  std::lock_guard<std::mutex> lock(mu);
  auto it = cache.find(key);
  if (it == cache.end()) {
    const int cw = 16 / (int)elem_size(precision);
    Maps m;
    const int ty = fused_tile_rows(precision);
    cudaError_t e = make_map(&m.interior, precision, g, base, TX, ty);
    if (e == cudaSuccess) e = make_map(&m.row, precision, g, base, TX, 1);
    if (e == cudaSuccess) e = make_map(&m.col, precision, g, base, cw, ty);
    if (e == cudaSuccess) e = make_map(&m.cor, precision, g, base, cw, 1);
    if (e != cudaSuccess) return e;
    it = cache.emplace(key, m).first;
  }
  *out = it->second;
  return cudaSuccess;
}

// Tile width of the ragged step, as for batches: 64 for FP32, 32 for 2-byte
// storage (fewer idle lanes at the x end).
template <int P> constexpr int kRaggedW = Prec<P>::dev ? 32 : TX;

// Predicted time of a launch with z runs of fz planes on `tiles` tiles.  Unit:
// a plane collided by one block while every slot is taken.  Both forms were
// fitted to the times of 15 to 38 run lengths on 30 (FP32) and 14 lattices of
// 0.7 to 34 M nodes.
//
// FP32 (bound by HBM): whole waves take their blocks' mean cost, where the two
// planes a run loads but does not collide count one each; the last wave what
// its blocks cost at full bandwidth, but at least 0.85 of its planes' latency;
// times 1 + fz / 50, because the longer a run, the further apart in time
// neighbouring tiles read the rows they share.  The chosen length is 2.1 %
// slower than the best one on average, at most 11 %; whole waves x (fz + 2) x
// (1 + fz / 256), the rule before, 6.5 %, at most 20 % (256x110x112: 28 planes
// 104.7 us, 10 planes 87.1 us), and on none of them more than 1.6 % faster.
double run_cost_f32(long long tiles, long long slots, int nz, int fz) {
  const long long blocks = tiles * ((nz + fz - 1) / fz), waves = blocks / slots, last = blocks - waves * slots;
  const double mean = (double)tiles * nz / blocks + 2.0;
  double cost = waves * mean;
  if (last) cost += std::max(mean * last / slots, 0.85 * (fz + 2));
  return cost * (1.0 + fz / 50.0);
}

// 2-byte storage and the MRT collision (bound by instruction issue): a small
// simulation of how the blocks run.  They start in launch order (the short last
// runs last) as slots come free, and all resident blocks progress at the same
// rate, a plane taking max(R, 0.9 slots) / slots while R blocks are resident;
// the two planes a run does not collide count h each; times 1 + fz / k.
// 2-byte storage, h = 0.8, k = 300: the chosen length is 0.8 % slower than the
// best one on average, at most 3 %; the rule before 2.6 %, at most 6 %
// (256x128x128 FP16: 15 planes 88.3 us, 29 planes 84.1 us).  FP32 with the MRT
// collision, h = 1.2, k = 100: 1.3 %, at most 3 % on ten lattices of 0.7 to 10 M
// nodes; by run_cost_f32 4.2 %, at most 12 % (576x80x83: 9 planes 121 us, 17
// planes 111 us; 256x128x128: 13 planes 119 us, 19 planes 116 us).
double run_cost_issue(long long tiles, long long slots, int nz, int fz, double h, double k) {
  struct Group {
    double left;
    long long count;
  };
  const int full = nz / fz, rem = nz - full * fz;
  Group queue[2] = {{fz + 2 * h, tiles * full}, {rem + 2 * h, rem ? tiles : 0}};
  std::vector<Group> run;
  double t = 0.0;
  long long resident = 0;
  for (int q = 0;;) {
    while (q < 2 && resident < slots) {
      const long long n = std::min(queue[q].count, slots - resident);
      if (n) run.push_back({queue[q].left, n});
      resident += n;
      queue[q].count -= n;
      if (!queue[q].count) ++q;
    }
    if (run.empty()) break;
    double step = run[0].left;
    for (const Group& g : run) step = std::min(step, g.left);
    t += step * std::max((double)resident, 0.9 * slots);
    size_t keep = 0;
    for (Group& g : run) {
      g.left -= step;
      if (g.left < 1e-9)
        resident -= g.count;
      else
        run[keep++] = g;
    }
    run.resize(keep);
  }
  return t / slots * (1.0 + fz / k);
}

// z planes per block.  Lattices with more than twice as many tiles as slots
// have many waves whatever the run: FP32 runs of 8 planes (1024x512x512, in
// groups of 4: 6.44 ms, 12-plane runs 6.99 ms), 2-byte storage by whole waves x
// (fz + 2) x (1 + fz / 2048) (1024x512x512 FP16, 27-, 32-, 48-, 64-, 86-, 128-,
// 256- and 512-plane runs take 4.598, 4.567, 4.524, 4.485, 4.506, 4.491, 4.614
// and 4.700 ms).  Others take the run length of the least predicted time, kept
// per shape (a pure function of its arguments).
template <int P>
int choose_fz(const Geom& g, int coll, long long tiles, long long slots) {
  constexpr bool dev = Prec<P>::dev;
  const bool mrt32 = !dev && coll == COLL_MRT;
  const bool many = tiles > 2 * slots;
  if (!dev && many) return std::min(g.nz, 8);
  static std::mutex mu;
  static std::map<std::tuple<long long, long long, int, bool>, int> kept;
  const auto key = std::make_tuple(tiles, slots, g.nz, mrt32);
  std::lock_guard<std::mutex> lock(mu);
  const auto it = kept.find(key);
  if (it != kept.end()) return it->second;
  int best = std::min(g.nz, 4);
  double best_cost = -1.0;
  for (int fz = best; fz <= (many ? g.nz : std::min(g.nz, 64)); ++fz) {
    const long long waves = (tiles * ((g.nz + fz - 1) / fz) + slots - 1) / slots;
    const double cost = many ? (double)waves * (fz + 2) * (1.0 + fz / 2048.0)
                        : dev   ? run_cost_issue(tiles, slots, g.nz, fz, 0.8, 300.0)
                        : mrt32 ? run_cost_issue(tiles, slots, g.nz, fz, 1.2, 100.0)
                                : run_cost_f32(tiles, slots, g.nz, fz);
    if (best_cost < 0.0 || cost < best_cost) {
      best_cost = cost;
      best = fz;
    }
  }
  if (kept.size() >= 1024) kept.clear();
  kept[key] = best;
  return best;
}

// Runs per group of the block order (a tile's y neighbours are ntx x grp
// blocks apart in the launch order; blocks of a group share the planes at
// their runs' ends).  FP32: 4 on lattices at least 8 tiles wide (512x256x256:
// 819 us against 833 us with 2; 1024x512x512: 6.42 ms, 8 take 6.53 ms), one
// on narrower ones (256x128x128 within 1 % for 1 to 4, 304x150x150 1 %
// slower with 2); 2-byte storage: one (1024x512x512 FP16 6.20 ms against 6.33
// ms in pairs).
template <int P>
int choose_grp(int ntx) {
  return !Prec<P>::dev && ntx >= 8 ? 4 : 1;
}

// Per device and storage type: the kernels' shared-memory limit is set and
// the SM count and resident blocks per SM of the step kernel are read on
// the first call with that device current (under a lock: several threads,
// or several devices, may make their first calls at once).
template <int P>
cudaError_t fused_device_info(int* slots_per_sm, int* sms) {
  using S = FusedShape<P>;
  constexpr int kMaxDev = 64;
  static std::mutex mu;
  static int slots_of[kMaxDev] = {}, sms_of[kMaxDev] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDev) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(mu);
  if (!slots_of[dev]) {
    for (const void* k : {(const void*)fused_kernel<P, false, COLL_SRT>, (const void*)fused_kernel<P, true, COLL_SRT>,
                          (const void*)fused_kernel<P, false, COLL_MRT>, (const void*)fused_kernel<P, true, COLL_MRT>})
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem);
    for (const void* k : {(const void*)bfused_kernel<P, TX>, (const void*)bpersist_kernel<P, TX>})
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::smem);
    constexpr int RW = kRaggedW<P>;
    for (const void* k :
         {(const void*)ragged_kernel<P, COLL_SRT, RW, false>, (const void*)ragged_kernel<P, COLL_SRT, RW, true>,
          (const void*)ragged_kernel<P, COLL_MRT, RW, false>, (const void*)ragged_kernel<P, COLL_MRT, RW, true>})
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FusedShape<P, RW>::smem);
    for (const void* k : {(const void*)bfused_kernel<P, 32>, (const void*)bpersist_kernel<P, 32>})
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FusedShape<P, 32>::smem);
    int n_sm = 0, slots = 0;
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&slots, fused_kernel<P, false, COLL_SRT>, S::NT, S::smem);
    if (e != cudaSuccess) return e;
    if (slots < 1) return cudaErrorInvalidConfiguration;
    sms_of[dev] = n_sm;
    slots_of[dev] = slots;
  }
  *slots_per_sm = slots_of[dev];
  *sms = sms_of[dev];
  return cudaSuccess;
}

// Grid of the fused step: z run length, runs per tile column, blocks.
template <int P>
cudaError_t fused_grid(const Geom& g, int coll, int fz_req, int grp_req, int* fz, int* nchunks, int* grp,
                       long long* blocks) {
  int slots_per_sm = 0, sms = 0;
  cudaError_t e = fused_device_info<P>(&slots_per_sm, &sms);
  if (e != cudaSuccess) return e;
  const long long tiles = (long long)(g.nx / TX) * (g.ny / FusedShape<P>::TY);
  *fz = fz_req > 0 ? std::min(fz_req, g.nz) : choose_fz<P>(g, coll, tiles, (long long)slots_per_sm * sms);
  *nchunks = (g.nz + *fz - 1) / *fz;
  *blocks = tiles * *nchunks;
  *grp = std::min(grp_req > 0 ? grp_req : choose_grp<P>(g.nx / TX), *nchunks);
  return *blocks > 0x7fffffffLL ? cudaErrorInvalidConfiguration : cudaSuccess;
}

// The steps are launched chained (Geom::chain) only where the blocks of two of
// them are resident at once.  Else the next step's first blocks take the places
// this one leaves, wherever they are, the rest comes as places fall free, and
// the SMs are unevenly loaded (192x80x68 FP32, 300 blocks on 456 places: 34.3 us
// per step chained, 30.0 plainly; 256x64x64, 448 blocks: 31.1 / 29.3).
inline int chain_steps(const Geom& g, long long blocks, long long slots) { return g.chain && 2 * blocks <= slots; }

template <int P>
cudaError_t fused_t(const Geom& g, const Phys& ph, const void* src, void* dst, int* flag, int fz_req,
                    int grp_req, const FusedDiag* diag, unsigned long long stall_ns, cudaStream_t s,
                    ReduceSide* side) {
  using S = FusedShape<P>;
  int fz = 0, nchunks = 0, grp = 0;
  long long blocks = 0;
  cudaError_t e = fused_grid<P>(g, ph.coll, fz_req, grp_req, &fz, &nchunks, &grp, &blocks);
  int slots_per_sm = 0, sms = 0;
  if (e == cudaSuccess) e = fused_device_info<P>(&slots_per_sm, &sms);
  if (e != cudaSuccess) return e;
  const int chain = chain_steps(g, blocks, (long long)slots_per_sm * sms);
  Maps m;
  e = maps_for(P, g, src, &m);
  if (e != cudaSuccess) return e;
  const int ntx = g.nx / TX;
  using T = typename Prec<P>::T;
  DirBases<T> db;
  for (int a = 0; a < Q; ++a) db.p[a] = (T*)dst + (long long)a * g.N;
  if (!diag) {
    const DiagOut none = diag_out(0.0, 0.0, nullptr, nullptr, stall_ns);
    return chain_launch(chain, ph.coll == COLL_MRT ? fused_kernel<P, false, COLL_MRT> : fused_kernel<P, false, COLL_SRT>,
                        (unsigned)blocks, S::NT, S::smem, s, m, g, ph, (T*)dst, flag, ntx, nchunks, fz, grp, none, db);
  }
  const long long row_blocks = (long long)(g.ny / S::TY) * nchunks;
  const size_t need = (size_t)row_blocks * g.nx * 2 + (size_t)blocks * DIAG_NG + (size_t)g.nx * 2;
  if (need > diag->scratch_doubles) return cudaErrorInvalidValue;
  double* slices = diag->scratch;
  double* bl = slices + (size_t)row_blocks * g.nx * 2;
  double* slice_tot = bl + (size_t)blocks * DIAG_NG;
  const DiagOut dg = diag_out(diag->rho_l, diag->rho_v, slices, bl, stall_ns);
  e = chain_launch(chain, ph.coll == COLL_MRT ? fused_kernel<P, true, COLL_MRT> : fused_kernel<P, true, COLL_SRT>,
                   (unsigned)blocks, S::NT, S::smem, s, m, g, ph, (T*)dst, flag, ntx, nchunks, fz, grp, dg, db);
  if (e != cudaSuccess) return e;
  return launch_diag_reduce(g, (int)row_blocks, (int)blocks, slices, bl, slice_tot, diag->out, diag->ring_count,
                            diag->ring_cap, s, side);
}

template <int P>
size_t fused_scratch_t(const Geom& g, int fz_req) {
  int fz = 0, nchunks = 0, grp = 0;
  long long blocks = 0;
  size_t need = 0;   // of either collision's run length
  for (int coll : {COLL_SRT, COLL_MRT}) {
    if (fused_grid<P>(g, coll, fz_req, 0, &fz, &nchunks, &grp, &blocks) != cudaSuccess) return 0;
    need = std::max(need, (size_t)(g.ny / FusedShape<P>::TY) * nchunks * g.nx * 2 + (size_t)blocks * DIAG_NG +
                              (size_t)g.nx * 2);
  }
  return need;
}

template <int P>
cudaError_t ragged_t(const Geom& g, const Phys& ph, const void* src, int src_px, void* dst, int dst_px, int* flag,
                     int fz_req, int grp_req, cudaStream_t s) {
  constexpr int W = kRaggedW<P>;
  using S = FusedShape<P, W>;
  using T = typename Prec<P>::T;
  int slots_per_sm = 0, sms = 0;
  cudaError_t e = fused_device_info<P>(&slots_per_sm, &sms);
  if (e != cudaSuccess) return e;
  const int cw = 16 / (int)sizeof(T);
  Maps m;
  e = make_map(&m.interior, P, g, src, W, S::TY, src_px);
  if (e == cudaSuccess) e = make_map(&m.row, P, g, src, W, 1, src_px);
  if (e == cudaSuccess) e = make_map(&m.col, P, g, src, cw, S::TY, src_px);
  if (e == cudaSuccess) e = make_map(&m.cor, P, g, src, cw, 1, src_px);
  if (e != cudaSuccess) return e;
  const int ntx = (g.nx + W - 1) / W;
  const long long tiles = (long long)ntx * ((g.ny + S::TY - 1) / S::TY);
  const int fz =
      fz_req > 0 ? std::min(fz_req, g.nz) : choose_fz<P>(g, ph.coll, tiles, (long long)slots_per_sm * sms);
  const int nchunks = (g.nz + fz - 1) / fz;
  if (tiles * nchunks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  const int grp = std::min(grp_req > 0 ? grp_req : choose_grp<P>(ntx), nchunks);
  const long long dstride = (long long)dst_px * g.ny * g.nz;
  DirBases<T> db;
  for (int a = 0; a < Q; ++a) db.p[a] = (T*)dst + a * dstride;
  // pairs of nodes are stored as one 2-element vector where every row starts
  // at such a vector's boundary
  const bool odd = dst_px % 2 != 0 || (uintptr_t)dst % (2 * sizeof(T)) != 0;
  const auto kernel = ph.coll == COLL_MRT
                          ? (odd ? ragged_kernel<P, COLL_MRT, W, true> : ragged_kernel<P, COLL_MRT, W, false>)
                          : (odd ? ragged_kernel<P, COLL_SRT, W, true> : ragged_kernel<P, COLL_SRT, W, false>);
  const int chain = chain_steps(g, tiles * nchunks, (long long)slots_per_sm * sms);
  return chain_launch(chain, kernel, (unsigned)(tiles * nchunks), S::NT, S::smem, s, m, g, ph, flag, ntx, nchunks, fz,
                      grp, dst_px, dstride, db);
}

}  // namespace

int ragged_row(const Geom& g, int precision) {
  const int al = 16 / (int)elem_size(precision);
  return (g.nx + al - 1) / al * al;
}

bool ragged_applicable(const Geom& g, int precision) {
  return precision != LBM_F64 && !fused_applicable(g, precision) &&
         (long long)ragged_row(g, precision) * g.ny * g.nz <= 0x7fffffffLL;
}

cudaError_t launch_ragged(int precision, const Geom& g, const Phys& ph, const void* src, int src_px, void* dst,
                          int dst_px, int* flag, int fz, int grp, cudaStream_t s) {
  if (src_px % (16 / (int)elem_size(precision)) || ((uintptr_t)src & 15)) return cudaErrorInvalidValue;
  switch (precision) {
    case LBM_F32: return ragged_t<LBM_F32>(g, ph, src, src_px, dst, dst_px, flag, fz, grp, s);
    case LBM_F16DEV: return ragged_t<LBM_F16DEV>(g, ph, src, src_px, dst, dst_px, flag, fz, grp, s);
    case LBM_BF16DEV: return ragged_t<LBM_BF16DEV>(g, ph, src, src_px, dst, dst_px, flag, fz, grp, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t fused_launch_shape(int precision, const Geom& g, int coll, int fz_req, int grp_req, int* fz, int* grp) {
  int nchunks = 0;
  long long blocks = 0;
  switch (precision) {
    case LBM_F32: return fused_grid<LBM_F32>(g, coll, fz_req, grp_req, fz, &nchunks, grp, &blocks);
    case LBM_F16DEV: return fused_grid<LBM_F16DEV>(g, coll, fz_req, grp_req, fz, &nchunks, grp, &blocks);
    case LBM_BF16DEV: return fused_grid<LBM_BF16DEV>(g, coll, fz_req, grp_req, fz, &nchunks, grp, &blocks);
  }
  return cudaErrorInvalidValue;
}

bool fused_applicable(const Geom& g, int precision) {
  return precision != LBM_F64 && g.nx % TX == 0 && g.ny % fused_tile_rows(precision) == 0 && g.nz >= 3;
}

cudaError_t launch_fused(int precision, const Geom& g, const Phys& ph, const void* src, void* dst, int* flag,
                         int fz, int grp, const FusedDiag* diag, unsigned long long stall_ns, cudaStream_t s,
                         ReduceSide* side) {
  if (!fused_applicable(g, precision)) return cudaErrorInvalidValue;
  switch (precision) {
    case LBM_F32: return fused_t<LBM_F32>(g, ph, src, dst, flag, fz, grp, diag, stall_ns, s, side);
    case LBM_F16DEV: return fused_t<LBM_F16DEV>(g, ph, src, dst, flag, fz, grp, diag, stall_ns, s, side);
    case LBM_BF16DEV: return fused_t<LBM_BF16DEV>(g, ph, src, dst, flag, fz, grp, diag, stall_ns, s, side);
  }
  return cudaErrorInvalidValue;
}

// ---- batched single-pass step on padded rows --------------------------------

namespace {

// z planes per block of a batch's tiles, one length for all instances: whole
// waves of blocks take their mean cost (the two planes a run does not collide
// count `halo` each half), the last wave what its blocks cost at full rate but
// at least `lat` of its planes' latency; times 1 + fz / k.  Fitted to the times
// of these run lengths on five sweeps of 3 to 48 ligaments (0.2 to 35 M nodes): it
// picks the best of them in FP32 and within 0.5 % in FP16.  The fixed 16 planes
// before cost 0 to 8 % (FP32) and 0 to 26 % (FP16) on the sweeps of 6 to 48 and
// twice (FP32, 28.0 / 14.4 us) to three times (FP16, 55.4 / 18.5 us) on three
// small ones.
template <int P, int W>
int choose_batch_fz(const BatchTmaInst* in, int count, long long slots) {
  constexpr bool dev = Prec<P>::dev;
  const double halo = dev ? 1.0 : 2.0, lat = dev ? 0.75 : 0.9, k = dev ? 400.0 : 160.0;
  int best = 16;
  double best_cost = -1.0;
  for (int fz : {2, 3, 4, 5, 6, 8, 10, 12, 16, 20, 24, 32, 48, 64}) {
    long long blocks = 0, planes = 0;
    for (int i = 0; i < count; ++i) {
      const Geom& g = in[i].g;
      const long long tiles =
          (long long)((g.nx + W - 1) / W) * ((g.ny + FusedShape<P, W>::TY - 1) / FusedShape<P, W>::TY);
      blocks += tiles * ((g.nz + fz - 1) / fz);
      planes += tiles * g.nz;
    }
    const long long waves = blocks / slots, last = blocks - waves * slots;
    const double mean = (double)planes / blocks + halo;
    double cost = waves * mean;
    if (last) cost += std::max(mean * last / slots, lat * (fz + 2));
    cost *= 1.0 + fz / k;
    if (best_cost < 0.0 || cost < best_cost) {
      best_cost = cost;
      best = fz;
    }
  }
  return best;
}

template <int P, int W>
cudaError_t batch_tma_build_t(const BatchTmaInst* in, int count, int fz_req, int grp_req, const void* pool,
                              void* d_table, BatchTmaPlan* plan, cudaStream_t s) {
  using S = FusedShape<P, W>;
  int slots_per_sm = 0, sms = 0;
  cudaError_t e = fused_device_info<P>(&slots_per_sm, &sms);   // the kernels' shared-memory limit
  if (e != cudaSuccess) return e;
  const size_t es = elem_size(P);
  const size_t inst_bytes = align128(sizeof(BTInst) * (size_t)count);
  std::vector<unsigned char> host(inst_bytes + sizeof(Maps) * 2 * (size_t)count);
  BTInst* ti = reinterpret_cast<BTInst*>(host.data());
  Maps* tm = reinterpret_cast<Maps*>(host.data() + inst_bytes);
  const Maps* d_maps = reinterpret_cast<const Maps*>((const unsigned char*)d_table + inst_bytes);
  const int cw = 16 / (int)es;
  if (fz_req <= 0) fz_req = choose_batch_fz<P, W>(in, count, (long long)slots_per_sm * sms);
  long long blocks = 0;
  for (int k = 0; k < count; ++k) {
    const BatchTmaInst& b = in[k];
    if (b.px % cw || b.off_f % cw || b.px < b.g.nx) return cudaErrorInvalidValue;
    BTInst& t = ti[k];
    std::memset(&t, 0, sizeof(t));
    t.g = b.g;
    plan->chain = b.g.chain;   // the same for all instances
    t.ph = b.ph;
    t.off_f = b.off_f;
    t.px = b.px;
    t.dstride = (long long)b.px * b.g.ny * b.g.nz;
    t.maps = d_maps + 2 * k;
    t.ntx = (b.g.nx + W - 1) / W;
    const int nty = (b.g.ny + S::TY - 1) / S::TY;
    t.fz = std::min(fz_req, b.g.nz);
    t.nchunks = (b.g.nz + t.fz - 1) / t.fz;
    // runs per block-order group (0: a tile's z runs one after another)
    t.grp = grp_req > 0 ? std::min(grp_req, t.nchunks) : t.nchunks;
    t.block0 = (int)blocks;
    blocks += (long long)t.ntx * nty * t.nchunks;
    for (int arr = 0; arr < 2; ++arr) {
      const void* base = (const unsigned char*)pool + (size_t)(b.off_f + (long long)arr * Q * t.dstride) * es;
      Maps& m = tm[2 * k + arr];
      e = make_map(&m.interior, P, b.g, base, W, S::TY, b.px);
      if (e == cudaSuccess) e = make_map(&m.row, P, b.g, base, W, 1, b.px);
      if (e == cudaSuccess) e = make_map(&m.col, P, b.g, base, cw, S::TY, b.px);
      if (e == cudaSuccess) e = make_map(&m.cor, P, b.g, base, cw, 1, b.px);
      if (e != cudaSuccess) return e;
    }
  }
  if (blocks > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  plan->width = W;
  plan->count = count;
  plan->blocks = (int)blocks;
  e = cudaMemcpyAsync(d_table, host.data(), host.size(), cudaMemcpyHostToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);   // the host table goes out of scope
  return e;
}

template <int P>
cudaError_t batch_tma_build_w(int tile_w, const BatchTmaInst* insts, int count, int fz, int grp, const void* pool,
                              void* d_table, BatchTmaPlan* plan, cudaStream_t s) {
  if (tile_w == 32) return batch_tma_build_t<P, 32>(insts, count, fz, grp, pool, d_table, plan, s);
  if (tile_w == TX) return batch_tma_build_t<P, TX>(insts, count, fz, grp, pool, d_table, plan, s);
  return cudaErrorInvalidValue;
}

template <int P, int W>
cudaError_t batch_tma_launch_t(const void* d_table, const BatchTmaPlan& plan, void* pool, int cur, int* flag,
                               unsigned* salt, cudaStream_t s) {
  using S = FusedShape<P, W>;
  return chain_launch(plan.chain, bfused_kernel<P, W>, plan.blocks, S::NT, S::smem, s, reinterpret_cast<const BTInst*>(d_table),
                      plan.count, (typename Prec<P>::T*)pool, cur, flag, salt);
}

template <int P>
cudaError_t batch_tma_launch_w(const void* d_table, const BatchTmaPlan& plan, void* pool, int cur, int* flag,
                               unsigned* salt, cudaStream_t s) {
  if (plan.width == 32) return batch_tma_launch_t<P, 32>(d_table, plan, pool, cur, flag, salt, s);
  if (plan.width == TX) return batch_tma_launch_t<P, TX>(d_table, plan, pool, cur, flag, salt, s);
  return cudaErrorInvalidValue;
}

template <int P, int W>
cudaError_t batch_tma_persist_t(const void* d_table, const BatchTmaPlan& plan, void* pool, int cur, int nsteps,
                                unsigned* bar, unsigned* tickets, int* flag, const unsigned* salt,
                                unsigned long long stall_ns,
                                cudaStream_t s) {
  using S = FusedShape<P, W>;
  using T = typename Prec<P>::T;
  int slots_per_sm = 0, sms = 0, per_sm = 0;
  cudaError_t e = fused_device_info<P>(&slots_per_sm, &sms);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, bpersist_kernel<P, W>, S::NT, S::smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
  int items = plan.blocks, count = plan.count;
  const int grid = std::min(items, per_sm * sms);
  e = cudaMemsetAsync(bar, 0, sizeof(unsigned), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(tickets, 0, sizeof(unsigned) * (size_t)nsteps, s);
  if (e != cudaSuccess) return e;
  const BTInst* t = reinterpret_cast<const BTInst*>(d_table);
  T* pf = (T*)pool;
  void* args[] = {(void*)&t, (void*)&count, (void*)&pf, (void*)&cur, (void*)&nsteps,
                  (void*)&items, (void*)&bar, (void*)&tickets, (void*)&flag, (void*)&salt, (void*)&stall_ns};
  return cudaLaunchCooperativeKernel((const void*)bpersist_kernel<P, W>, dim3(grid), dim3(S::NT), args, S::smem, s);
}

template <int P>
cudaError_t batch_tma_persist_w(const void* d_table, const BatchTmaPlan& plan, void* pool, int cur, int nsteps,
                                unsigned* bar, unsigned* tickets, int* flag, const unsigned* salt,
                                unsigned long long stall_ns,
                                cudaStream_t s) {
  if (plan.width == 32)
    return batch_tma_persist_t<P, 32>(d_table, plan, pool, cur, nsteps, bar, tickets, flag, salt, stall_ns, s);
  if (plan.width == TX)
    return batch_tma_persist_t<P, TX>(d_table, plan, pool, cur, nsteps, bar, tickets, flag, salt, stall_ns, s);
  return cudaErrorInvalidValue;
}

}  // namespace

size_t batch_tma_table_bytes(int count) {
  return align128(sizeof(BTInst) * (size_t)count) + sizeof(Maps) * 2 * (size_t)count;
}

int batch_tma_row_align(int precision) { return 16 / (int)elem_size(precision); }

cudaError_t batch_tma_build(int precision, int tile_w, const BatchTmaInst* insts, int count, int fz, int grp,
                            const void* pool, void* d_table, BatchTmaPlan* plan, cudaStream_t s) {
  switch (precision) {
    case LBM_F32: return batch_tma_build_w<LBM_F32>(tile_w, insts, count, fz, grp, pool, d_table, plan, s);
    case LBM_F16DEV: return batch_tma_build_w<LBM_F16DEV>(tile_w, insts, count, fz, grp, pool, d_table, plan, s);
    case LBM_BF16DEV: return batch_tma_build_w<LBM_BF16DEV>(tile_w, insts, count, fz, grp, pool, d_table, plan, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t batch_tma_launch(int precision, const void* d_table, const BatchTmaPlan& plan, void* pool, int cur,
                             int* flag, unsigned* salt, cudaStream_t s) {
  switch (precision) {
    case LBM_F32: return batch_tma_launch_w<LBM_F32>(d_table, plan, pool, cur, flag, salt, s);
    case LBM_F16DEV: return batch_tma_launch_w<LBM_F16DEV>(d_table, plan, pool, cur, flag, salt, s);
    case LBM_BF16DEV: return batch_tma_launch_w<LBM_BF16DEV>(d_table, plan, pool, cur, flag, salt, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t batch_tma_persist_launch(int precision, const void* d_table, const BatchTmaPlan& plan, void* pool,
                                     int cur, int nsteps, unsigned* bar, unsigned* tickets, int* flag,
                                     const unsigned* salt, unsigned long long stall_ns, cudaStream_t s) {
  switch (precision) {
    case LBM_F32:
      return batch_tma_persist_w<LBM_F32>(d_table, plan, pool, cur, nsteps, bar, tickets, flag, salt, stall_ns, s);
    case LBM_F16DEV:
      return batch_tma_persist_w<LBM_F16DEV>(d_table, plan, pool, cur, nsteps, bar, tickets, flag, salt, stall_ns, s);
    case LBM_BF16DEV:
      return batch_tma_persist_w<LBM_BF16DEV>(d_table, plan, pool, cur, nsteps, bar, tickets, flag, salt, stall_ns, s);
  }
  return cudaErrorInvalidValue;
}

size_t fused_diag_scratch_doubles(const Geom& g, int precision, int fz) {
  if (!fused_applicable(g, precision)) return 0;
  switch (precision) {
    case LBM_F32: return fused_scratch_t<LBM_F32>(g, fz);
    case LBM_F16DEV: return fused_scratch_t<LBM_F16DEV>(g, fz);
    case LBM_BF16DEV: return fused_scratch_t<LBM_BF16DEV>(g, fz);
  }
  return 0;
}

}  // namespace lbm
