// The two kernels of one time step (hot path), single lattice: the psi pass
// and the fused force + collision + streaming kernel (bodies in lbm_node.cuh).
//
// Memory layout: structure of arrays, plane a holds f_a of all nodes, x
// fastest, so a warp's 32 threads touch 32 consecutive x of one plane per
// load or store.  Both kernels are bound by HBM bandwidth (about 1 flop per
// byte); no tensor-core work exists on this path.
#include <type_traits>

#include "lbm_launch.cuh"
#include "lbm_node.cuh"

namespace lbm {

namespace {

// psi pass over all nodes of one lattice.
template <int P, int LAYOUT, bool CHAIN>
__global__ void __launch_bounds__(256) psi_kernel(Geom g, Phys ph, const typename Prec<P>::T* f,
                                                  typename Prec<P>::C* __restrict__ psi,
                                                  int* __restrict__ flag, double* rho_out) {
  if constexpr (CHAIN) chain_wait();
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  psi_node<P, LAYOUT, !CHAIN>(g, ph, f, psi, flag, i, rho_out);
}

// Fused force + collision + streaming.  One thread per node.  MINB is the
// number of 256-thread blocks per SM the register allocation must allow
// (4: <= 64 registers, 3: <= 80, 2: <= 128); the autotuner picks it.
template <int P, int MODE, int MINB, bool CHAIN>
__global__ void __launch_bounds__(256, MINB) collide_kernel(Geom g, Phys ph,
                                                            const typename Prec<P>::T* src,
                                                            typename Prec<P>::T* dst,
                                                            const typename Prec<P>::C* psi) {
  if constexpr (CHAIN) chain_wait();
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z * blockDim.z + threadIdx.z;
  if (x >= g.nx || y >= g.ny || z >= g.nz) return;
  advance_salt(ph);
  collide_node<P, MODE, !CHAIN>(g, ph, src, dst, psi, x, y, z);
}

// Two-node forms (x even, nx even): one thread per node pair.
template <int P, int LAYOUT, bool CHAIN>
__global__ void __launch_bounds__(256) psi_pair_kernel(Geom g, Phys ph, const typename Prec<P>::T* f,
                                                       typename Prec<P>::C* __restrict__ psi,
                                                       int* __restrict__ flag) {
  if constexpr (CHAIN) chain_wait();
  const long long i = 2 * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= g.N) return;
  psi_pair<P, LAYOUT, !CHAIN>(g, ph, f, psi, flag, i);
}

template <int P, bool CHAIN>
__global__ void __launch_bounds__(256) psi_quad_kernel(Geom g, Phys ph, const typename Prec<P>::T* f,
                                                       typename Prec<P>::C* __restrict__ psi,
                                                       int* __restrict__ flag) {
  if constexpr (CHAIN) chain_wait();
  const long long i = 4 * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  if (i >= g.N) return;
  psi_quad<P, !CHAIN>(g, ph, f, psi, flag, i);
}

// Gather layout, four nodes per thread; every thread of the last block takes
// part in the warp shuffles (those past the lattice on its last quad).
template <int P, bool CHAIN>
__global__ void __launch_bounds__(256) psi_quad_gather_kernel(Geom g, Phys ph, const typename Prec<P>::T* f,
                                                              typename Prec<P>::C* __restrict__ psi,
                                                              int* __restrict__ flag) {
  if constexpr (CHAIN) chain_wait();
  long long i = 4 * ((long long)blockIdx.x * blockDim.x + threadIdx.x);
  const bool live = i < g.N;
  if (!live) i = g.N - 4;
  psi_quad_gather<P, !CHAIN>(g, ph, f, psi, flag, i, live);
}

template <int P, int MODE, int MINB, bool CHAIN>
__global__ void __launch_bounds__(256, MINB) collide_pair_kernel(Geom g, Phys ph,
                                                                 const typename Prec<P>::T* src,
                                                                 typename Prec<P>::T* dst,
                                                                 const typename Prec<P>::C* psi) {
  if constexpr (CHAIN) chain_wait();
  const int x0 = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z * blockDim.z + threadIdx.z;
  if (x0 >= g.nx || y >= g.ny || z >= g.nz) return;
  advance_salt(ph);
  collide_pair<P, MODE, !CHAIN>(g, ph, src, dst, psi, x0, y, z);
}

// The one-node A-B kernel into an array with rows px elements apart.
template <int P, int COLL>
__global__ void __launch_bounds__(256, 3) collide_padded_kernel(Geom g, Phys ph, const typename Prec<P>::T* src,
                                                                typename Prec<P>::T* dst, int px,
                                                                const typename Prec<P>::C* psi) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  const int z = blockIdx.z * blockDim.z + threadIdx.z;
  if (x >= g.nx || y >= g.ny || z >= g.nz) return;
  advance_salt(ph);
  collide_node<P, MODE_AB, true, COLL>(g, ph, src, dst, psi, x, y, z, px);
}

template <int P>
cudaError_t collide_padded(const Geom& g, const Phys& ph, const void* src, void* dst, int px, const void* psi,
                           dim3 block, cudaStream_t s) {
  using T = typename Prec<P>::T;
  using C = typename Prec<P>::C;
  const dim3 grid((g.nx + block.x - 1) / block.x, (g.ny + block.y - 1) / block.y, (g.nz + block.z - 1) / block.z);
  if (ph.coll == COLL_MRT)
    collide_padded_kernel<P, COLL_MRT><<<grid, block, 0, s>>>(g, ph, (const T*)src, (T*)dst, px, (const C*)psi);
  else
    collide_padded_kernel<P, COLL_SRT><<<grid, block, 0, s>>>(g, ph, (const T*)src, (T*)dst, px, (const C*)psi);
  return cudaGetLastError();
}

// Threads per block of the psi pass: 128 (512x256x256 AA FP16, gather layout:
// 250 us per launch against 256 with 256), fewer (to one warp) where that leaves less
// than two blocks per SM.
int psi_threads(long long units) {
  int threads = 128;
  while (threads > 32 && units < (long long)threads * 2 * kSmCount) threads /= 2;
  return threads;
}

template <int P, bool CHAIN>
cudaError_t psi_dispatch(int layout, bool vec, const Geom& g, const Phys& ph, const void* f,
                         void* psi, int* flag, cudaStream_t s, double* rho_out) {
  using T = typename Prec<P>::T;
  using C = typename Prec<P>::C;
  if constexpr (P != LBM_F64) {
    const int threads = psi_threads(g.N / 4);
    const long long blocks = (g.N / 4 + threads - 1) / threads;
    if (vec && g.nx % 4 == 0 && layout == LAYOUT_LOCAL) {
      return chain_launch(CHAIN, psi_quad_kernel<P, CHAIN>, (unsigned)blocks, threads, 0, s, g, ph, (const T*)f, (C*)psi, flag);
    }
    // the gather layout in four-node form for 2-byte storage only (FP32:
    // 10.28 ms against 9.84 ms per AA step on 1024x512x512 with node pairs)
    if constexpr (Prec<P>::dev) {
      if (vec && g.nx % 4 == 0) {
        return chain_launch(CHAIN, psi_quad_gather_kernel<P, CHAIN>, (unsigned)blocks, threads, 0, s, g, ph, (const T*)f, (C*)psi,
                            flag);
      }
    }
  }
  const int threads = psi_threads(vec ? g.N / 2 : g.N);
  if constexpr (P != LBM_F64) if (vec) {
    const long long blocks = (g.N / 2 + threads - 1) / threads;
    if (layout == LAYOUT_LOCAL)
      return chain_launch(CHAIN, psi_pair_kernel<P, LAYOUT_LOCAL, CHAIN>, (unsigned)blocks, threads, 0, s, g, ph, (const T*)f,
                          (C*)psi, flag);
    else
      return chain_launch(CHAIN, psi_pair_kernel<P, LAYOUT_GATHER, CHAIN>, (unsigned)blocks, threads, 0, s, g, ph, (const T*)f,
                          (C*)psi, flag);
  }
  const long long blocks = (g.N + threads - 1) / threads;
  if (layout == LAYOUT_LOCAL)
    return chain_launch(CHAIN, psi_kernel<P, LAYOUT_LOCAL, CHAIN>, (unsigned)blocks, threads, 0, s, g, ph, (const T*)f, (C*)psi,
                        flag, rho_out);
  else
    return chain_launch(CHAIN, psi_kernel<P, LAYOUT_GATHER, CHAIN>, (unsigned)blocks, threads, 0, s, g, ph, (const T*)f, (C*)psi,
                        flag, rho_out);
}

template <int P, bool CHAIN, int MINB, bool VEC>
cudaError_t collide_mode(int mode, const Geom& g, const Phys& ph, const void* src, void* dst,
                         const void* psi, dim3 grid, dim3 block, cudaStream_t s) {
  using T = typename Prec<P>::T;
  using C = typename Prec<P>::C;
  const T* in = (const T*)src;
  T* out = (T*)dst;
  const C* ps = (const C*)psi;
  if constexpr (VEC) {
    switch (mode) {
      case MODE_AB: return chain_launch(CHAIN, collide_pair_kernel<P, MODE_AB, MINB, CHAIN>, grid, block, 0, s, g, ph, in, out, ps);
      case MODE_AA_EVEN: return chain_launch(CHAIN, collide_pair_kernel<P, MODE_AA_EVEN, MINB, CHAIN>, grid, block, 0, s, g, ph, in,
                                             out, ps);
      default: return chain_launch(CHAIN, collide_pair_kernel<P, MODE_AA_ODD, MINB, CHAIN>, grid, block, 0, s, g, ph, in, out, ps);
    }
  } else {
    switch (mode) {
      case MODE_AB: return chain_launch(CHAIN, collide_kernel<P, MODE_AB, MINB, CHAIN>, grid, block, 0, s, g, ph, in, out, ps);
      case MODE_AA_EVEN: return chain_launch(CHAIN, collide_kernel<P, MODE_AA_EVEN, MINB, CHAIN>, grid, block, 0, s, g, ph, in, out,
                                             ps);
      default: return chain_launch(CHAIN, collide_kernel<P, MODE_AA_ODD, MINB, CHAIN>, grid, block, 0, s, g, ph, in, out, ps);
    }
  }
}

template <int P, bool CHAIN>
cudaError_t collide_dispatch(int mode, int minb, bool vec, const Geom& g, const Phys& ph,
                             const void* src, void* dst, const void* psi, dim3 block,
                             cudaStream_t s) {
  const int ux = vec ? g.nx / 2 : g.nx;  // threads needed along x
  dim3 grid((ux + block.x - 1) / block.x, (g.ny + block.y - 1) / block.y,
            (g.nz + block.z - 1) / block.z);
  if constexpr (P != LBM_F64) if (vec) {
    switch (minb) {
      case 2: return collide_mode<P, CHAIN, 2, true>(mode, g, ph, src, dst, psi, grid, block, s);
      case 3: return collide_mode<P, CHAIN, 3, true>(mode, g, ph, src, dst, psi, grid, block, s);
      default: return collide_mode<P, CHAIN, 4, true>(mode, g, ph, src, dst, psi, grid, block, s);
    }
  }
  switch (minb) {
    case 2: return collide_mode<P, CHAIN, 2, false>(mode, g, ph, src, dst, psi, grid, block, s);
    case 3: return collide_mode<P, CHAIN, 3, false>(mode, g, ph, src, dst, psi, grid, block, s);
    default: return collide_mode<P, CHAIN, 4, false>(mode, g, ph, src, dst, psi, grid, block, s);
  }
}

}  // namespace

cudaError_t launch_psi(int precision, int layout, bool vec, const Geom& g, const Phys& ph,
                       const void* f, void* psi, int* flag, cudaStream_t s, void* dst) {
  vec = node_pairs(precision, vec, g);
  auto run = [&](auto chain) {
    constexpr bool CHAIN = decltype(chain)::value;
    switch (precision) {
      case LBM_F64: return psi_dispatch<LBM_F64, CHAIN>(layout, vec, g, ph, f, psi, flag, s, (double*)dst);
      case LBM_F32: return psi_dispatch<LBM_F32, CHAIN>(layout, vec, g, ph, f, psi, flag, s, nullptr);
      case LBM_F16DEV: return psi_dispatch<LBM_F16DEV, CHAIN>(layout, vec, g, ph, f, psi, flag, s, nullptr);
      case LBM_BF16DEV: return psi_dispatch<LBM_BF16DEV, CHAIN>(layout, vec, g, ph, f, psi, flag, s, nullptr);
    }
    return cudaErrorInvalidValue;
  };
  return g.chain ? run(std::true_type{}) : run(std::false_type{});
}

cudaError_t launch_collide(int precision, int mode, int minb, bool vec, const Geom& g,
                           const Phys& ph, const void* src, void* dst, const void* psi, dim3 block,
                           cudaStream_t s) {
  if ((long long)block.x * block.y * block.z > 256) return cudaErrorInvalidConfiguration;
  vec = node_pairs(precision, vec, g);
  auto run = [&](auto chain) {
    constexpr bool CHAIN = decltype(chain)::value;
    switch (precision) {
      case LBM_F64: return collide_dispatch<LBM_F64, CHAIN>(mode, minb, vec, g, ph, src, dst, psi, block, s);
      case LBM_F32: return collide_dispatch<LBM_F32, CHAIN>(mode, minb, vec, g, ph, src, dst, psi, block, s);
      case LBM_F16DEV: return collide_dispatch<LBM_F16DEV, CHAIN>(mode, minb, vec, g, ph, src, dst, psi, block, s);
      case LBM_BF16DEV: return collide_dispatch<LBM_BF16DEV, CHAIN>(mode, minb, vec, g, ph, src, dst, psi, block, s);
    }
    return cudaErrorInvalidValue;
  };
  return g.chain ? run(std::true_type{}) : run(std::false_type{});
}

cudaError_t launch_collide_padded(int precision, const Geom& g, const Phys& ph, const void* src, void* dst, int px,
                                  const void* psi, dim3 block, cudaStream_t s) {
  switch (precision) {
    case LBM_F32: return collide_padded<LBM_F32>(g, ph, src, dst, px, psi, block, s);
    case LBM_F16DEV: return collide_padded<LBM_F16DEV>(g, ph, src, dst, px, psi, block, s);
    case LBM_BF16DEV: return collide_padded<LBM_BF16DEV>(g, ph, src, dst, px, psi, block, s);
  }
  return cudaErrorInvalidValue;
}

// FP64 kernels take one node per thread: the FP64 pipe bounds them either way
// (256x128x128: 222 + 981 us per step with one node, 222 + 982 us with two),
// and lattices of a few warps per SM reach more SMs (4x49x49: 10.3 us per step
// against 16.5 us).
bool node_pairs(int precision, bool vec, const Geom& g) { return precision != LBM_F64 && vec && g.nx % 2 == 0; }

size_t elem_size(int precision) {
  switch (precision) {
    case LBM_F64: return 8;
    case LBM_F32: return 4;
    default: return 2;
  }
}

}  // namespace lbm
