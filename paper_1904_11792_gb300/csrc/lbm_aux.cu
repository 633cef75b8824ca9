// Kernels around the time step: ligament initial condition, canonical
// population export/import, macroscopic fields, FP64 diagnostics and the
// connected-component labelling of the liquid (droplet count).
#include <algorithm>

#include "lbm_internal.h"
#include "lbm_launch.cuh"

namespace lbm {

namespace {

template <int P>
__device__ __forceinline__ double shift_d(int a, double rho_ref) {
  return Prec<P>::dev ? (double)storage_shift<P>(a, rho_ref) : 0.0;
}

// The shift in the arithmetic's precision (the host's FP32 form).
template <int P>
__device__ __forceinline__ float shift_f(int a, const Phys& ph) {
  return Prec<P>::dev ? ph.shift_f[a == 0 ? 0 : (a <= 6 ? 1 : 2)] : 0.0f;
}

// Two stored neighbours (4- or 2-byte storage) as float2, shifted.
template <int P>
__device__ __forceinline__ void load_pair_nc(const typename Prec<P>::T* p, float sh, float2& v) {
  if constexpr (P == LBM_F32) {
    v = __ldg(reinterpret_cast<const float2*>(p));
  } else {
    if constexpr (P == LBM_F16DEV)
      v = __half22float2(__ldg(reinterpret_cast<const __half2*>(p)));
    else
      v = __bfloat1622float2(__ldg(reinterpret_cast<const __nv_bfloat162*>(p)));
    v.x += sh;
    v.y += sh;
  }
}

// DSum<float> of two lanes at once, in paired instructions.
struct DSum2 {
  float2 hi{0.0f, 0.0f}, lo{0.0f, 0.0f};
  __device__ __forceinline__ void add(float2 x) {
    float2 e;
    hi = two_sum(hi, x, e);
    lo = radd(lo, e);
  }
  __device__ __forceinline__ void add(float2 x, float2 xlo) {
    float2 e;
    hi = two_sum(hi, x, e);
    lo = radd(lo, radd(e, xlo));
  }
  __device__ __forceinline__ double value() const {
    return ((double)hi.x + (double)lo.x) + ((double)hi.y + (double)lo.y);
  }
};

__device__ __forceinline__ void coords(const Geom& g, long long i, int& x, int& y, int& z) {
  x = (int)(i % g.nx);
  const long long r = i / g.nx;
  y = (int)(r % g.ny);
  z = (int)(r / g.ny);
}

// Flat index in the storage of the pre-collision population a of node
// (x, y, z) for the given layout.
__device__ __forceinline__ long long slot_index(const Geom& g, int layout, int a, const Nbr& nb) {
  if (layout == LAYOUT_LOCAL) return (long long)a * g.N + nb.idx(0, 0, 0);
  return (long long)opp(a) * g.N + nb.idx(-cx(a), -cy(a), -cz(a));
}

// rho and j of a node in compute precision C (the same summation order as
// the collide kernel).
template <int P>
__device__ __forceinline__ void node_rho_j(const Geom& g, const Phys& ph, int layout,
                                           const typename Prec<P>::T* f, const Nbr& nb,
                                           typename Prec<P>::C& rho, typename Prec<P>::C j[3]) {
  using C = typename Prec<P>::C;
  C v[Q];
#pragma unroll
  for (int a = 0; a < Q; ++a) v[a] = Prec<P>::template load<true>(f + slot_index(g, layout, a, nb), (C)shift_d<P>(a, ph.rho_ref));
  rho = rho_of<C>(v);
  mom_of<C>(v, j[0], j[1], j[2]);
}

// ---------------------------------------------------------------------------
// Initial condition (section "Ligament set-up"): perturbed cylinder along x.
// ---------------------------------------------------------------------------
template <int P>
__global__ void init_kernel(Geom g, Phys ph, InitSpec sp, typename Prec<P>::T* f) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  int x, y, z;
  coords(g, i, x, y, z);
  const double R = sp.R0 * (1.0 + sp.eps * cos(6.283185307179586476925 * x / sp.lambda + sp.phase));
  const double dy = y - 0.5 * (g.ny - 1), dz = z - 0.5 * (g.nz - 1);
  const double d = sqrt(dy * dy + dz * dz) - R;
  double rho;
  if (sp.prof == nullptr) {
    rho = sp.rho_v + 0.5 * (sp.rho_l - sp.rho_v) * (1.0 - tanh(2.0 * d / sp.width));
  } else {
    const double s = (d - sp.d0) / sp.dd;
    if (s <= 0.0) {
      rho = sp.prof[0];
    } else if (s >= sp.n - 1) {
      rho = sp.prof[sp.n - 1];
    } else {
      const int k = (int)floor(s);
      const double t = s - k;
      rho = sp.prof[k] + t * (sp.prof[k + 1] - sp.prof[k]);
    }
  }
  using C = typename Prec<P>::C;
#pragma unroll
  for (int a = 0; a < Q; ++a)
    Prec<P>::store(f + (long long)a * g.N + i, (C)(wgt(a) * rho), (C)shift_d<P>(a, ph.rho_ref));
}

// ---------------------------------------------------------------------------
// Canonical FP64 planes a0 + blockIdx.y <-> storage.
// ---------------------------------------------------------------------------
template <int P>
__global__ void get_planes_kernel(Geom g, Phys ph, int layout, const typename Prec<P>::T* f, int a0,
                                  double* out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  const int a = a0 + blockIdx.y;
  int x, y, z;
  coords(g, i, x, y, z);
  Nbr nb;
  nb.make(g, x, y, z);
  using C = typename Prec<P>::C;
  out[(long long)blockIdx.y * g.N + i] =
      (double)Prec<P>::template load<true>(f + slot_index(g, layout, a, nb), (C)shift_d<P>(a, ph.rho_ref));
}

template <int P>
__global__ void set_planes_kernel(Geom g, Phys ph, int layout, typename Prec<P>::T* f, int a0,
                                  const double* in) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  const int a = a0 + blockIdx.y;
  int x, y, z;
  coords(g, i, x, y, z);
  Nbr nb;
  nb.make(g, x, y, z);
  using C = typename Prec<P>::C;
  Prec<P>::store(f + slot_index(g, layout, a, nb), (C)in[(long long)blockIdx.y * g.N + i],
                 (C)shift_d<P>(a, ph.rho_ref));
}

// ---------------------------------------------------------------------------
// Macroscopic fields: rho (Eq. 4) and u = (j + F/2)/rho, F from Eq. 5.
// which: 0 rho, 1..3 the velocity components.
// ---------------------------------------------------------------------------
template <int P>
__global__ void moments_kernel(Geom g, Phys ph, int layout, const typename Prec<P>::T* f,
                               const typename Prec<P>::C* psi, double* rho_o, double* ux,
                               double* uy, double* uz) {
  using C = typename Prec<P>::C;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.N) return;
  int x, y, z;
  coords(g, i, x, y, z);
  Nbr nb;
  nb.make(g, x, y, z);
  C rho, j[3];
  node_rho_j<P>(g, ph, layout, f, nb, rho, j);
  C s[3] = {0, 0, 0};
#pragma unroll
  for (int a = 1; a < Q; ++a) {
    const C p = psi[nb.idx(cx(a), cy(a), cz(a))];
    const C w = (C)wgt(a);
    s[0] += w * cx(a) * p;
    s[1] += w * cy(a) * p;
    s[2] += w * cz(a) * p;
  }
  const C gp = -(C)ph.G * psi[i];
  if (rho_o) rho_o[i] = (double)rho;
  const double r = (double)rho;
  if (ux) ux[i] = ((double)j[0] + 0.5 * (double)(gp * s[0])) / r;
  if (uy) uy[i] = ((double)j[1] + 0.5 * (double)(gp * s[1])) / r;
  if (uz) uz[i] = ((double)j[2] + 0.5 * (double)(gp * s[2])) / r;
}

// ---------------------------------------------------------------------------
// Diagnostics: deterministic two-kernel FP64 reduction.
// Block (32, 8): threadIdx.x walks x, threadIdx.y and blockIdx.y walk rows
// (y, z).  Per-thread accumulation in a fixed order, then fixed-order
// block reductions; the final kernel combines block partials in index order.
// With WRITE_PSI the partial kernel is also the psi pass of the step: it
// writes psi(rho) of every node and raises the numeric flag, so diagnostics
// on a time step cost no extra pass over the populations.
// ---------------------------------------------------------------------------
constexpr int DX = 32, DY = 8;
constexpr int NG = DIAG_NG;  // global partial slots per block
// slots: 0 mass, 1-3 momentum, 4 volume_w, 5 count, 6 max_u, 7 rho_min,
// 8 rho_max, 9 bad, 10-11 unused

// The warp's sums of eight values at once: halves of the lanes exchange halves
// of the values until each lane holds one, 9 FP64 additions instead of 40.
// Lane l returns the sum of v[l / 4].
__device__ __forceinline__ double warp_sum8(double v[8], int lane) {
#pragma unroll
  for (int o = 16, n = 4; n >= 1; o >>= 1, n >>= 1) {
    const bool hi = lane & o;
#pragma unroll
    for (int m = 0; m < n; ++m) {
      const double give = hi ? v[m] : v[m + n], keep = hi ? v[m + n] : v[m];
      v[m] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  }
  double t = v[0];
  t += __shfl_xor_sync(0xffffffffu, t, 2);
  return t + __shfl_xor_sync(0xffffffffu, t, 1);
}

// Row-blocks of the partial kernel with `per_sm` blocks per SM and gx blocks
// along x: each thread walks rows / (8 row-blocks) rows, and the per-slice
// partials (row-blocks x nx x 2 doubles) stay small.  A block ends with about
// 50 FP64 instructions per warp (warp and block sums; 70 with a tree per sum),
// which the FP64 pipe of its SM works off at 16 clocks each: with 16 blocks per
// SM that alone took 50 us, so the kernels launch 4 per SM, two waves.
int diag_row_blocks(const Geom& g, long long gx, int per_sm) {
  const long long rows = (long long)g.ny * g.nz;
  long long want = (per_sm * kSmCount + gx - 1) / gx;
  const long long cap = (2ll << 20) / (2ll * g.nx);  // slices <= 2 Mi doubles
  if (want > cap) want = cap;
  long long rb = (rows + DY - 1) / DY;
  if (rb > want) rb = want;
  if (rb < 1) rb = 1;
  return (int)rb;
}

// Each node's momentum and liquid fraction are computed in the compute
// precision (FP32 except in FP64 mode), its density as that sum plus its
// rounding error (rho_of_x); the per-thread sums over the thread's rows are
// DSum accumulators (an error-free FP32 pair, exact to FP64 level), the warp
// shuffle tree and the block sums of mass, momentum and the weighted liquid
// volume are FP64, so the totals carry no reduction error above FP64
// rounding, whatever the storage precision.  Counts, extrema and the
// numeric flag are exact in any precision.
template <int P, bool WRITE_PSI, int LAYOUT>
__global__ void __launch_bounds__(DX* DY, 2) diag_partial_kernel(Geom g, Phys ph,
                                                              const typename Prec<P>::T* f,
                                                              double rho_l, double rho_v,
                                                              double* slices, double* blocks,
                                                              typename Prec<P>::C* psi, int* flag,
                                                              double* rho_out) {
  using C = typename Prec<P>::C;
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int x = blockIdx.x * DX + tx;
  const long long rows = (long long)g.ny * g.nz;
  const C thr = (C)(0.5 * (rho_l + rho_v)), inv = (C)(1.0 / (rho_l - rho_v)), rv = (C)rho_v;
  DSum<C> s_mass, s_jx, s_jy, s_jz, s_vol;
  C umax = 0, rmin = (C)3.0e38, rmax = (C)-3.0e38;
  int cnt = 0;
  bool bad = false;
  const C s0 = (C)shift_d<P>(0, ph.rho_ref);
  const C s1 = (C)shift_d<P>(1, ph.rho_ref);
  const C s2 = (C)shift_d<P>(7, ph.rho_ref);
  if (x < g.nx) {
#pragma unroll 2
    for (long long r = (long long)blockIdx.y * DY + ty; r < rows; r += (long long)DY * gridDim.y) {
      const int i = x + g.nx * (int)r;
      C fv[Q];
      if constexpr (LAYOUT == LAYOUT_LOCAL) {
#pragma unroll
        for (int a = 0; a < Q; ++a)
          fv[a] = Prec<P>::template load<true>(f + (long long)a * g.N + i, a == 0 ? s0 : (a <= 6 ? s1 : s2));
      } else {
        Nbr nb;
        nb.make(g, x, (int)(r % g.ny), (int)(r / g.ny));
#pragma unroll
        for (int a = 0; a < Q; ++a)
          fv[a] = Prec<P>::template load<true>(f + (long long)opp(a) * g.N + nb.idx(-cx(a), -cy(a), -cz(a)),
                                a == 0 ? s0 : (a <= 6 ? s1 : s2));
      }
      C rho_lo;
      const C rho = rho_of_x(fv, rho_lo);   // rho_of bitwise, plus its rounding error
      C jx, jy, jz;
      mom_of<C>(fv, jx, jy, jz);
      if constexpr (WRITE_PSI) {
        psi[i] = psi_of<C>(rho, ph);
        if (P == LBM_F64 && rho_out) rho_out[i] = rho;
      }
      s_mass.add(rho, rho_lo);
      s_jx.add(jx);
      s_jy.add(jy);
      s_jz.add(jz);
      C phi = (rho - rv) * inv;
      phi = phi < (C)0 ? (C)0 : (phi > (C)1 ? (C)1 : phi);
      s_vol.add(phi);
      cnt += rho > thr;
      // the root and the division only where |j|/rho can reach the maximum, as
      // in diag_pair_kernel (FP64 256x128x128, in the loop: 433 -> 369 us per
      // record beyond the psi pass)
      const C j2 = xfma(jz, jz, xfma(jy, jy, xmul(jx, jx))), t = umax * rho;
      if (j2 >= (C)0.999998 * (t * t) || j2 < (C)1e-30) {
        const C u = sqrt(j2) / rho;
        umax = u > umax ? u : umax;
      }
      rmin = rho < rmin ? rho : rmin;
      rmax = rho > rmax ? rho : rmax;
      bad |= !(rho > (C)0) || !(rho <= (C)3.0e38);
    }
  }
  if constexpr (WRITE_PSI) raise_flag(bad, flag);
  // per-slice sums over the block's 8 row groups (FP64, fixed order)
  __shared__ double sh_s[2][DY][DX];
  sh_s[0][ty][tx] = s_vol.value();
  sh_s[1][ty][tx] = (double)cnt;
  // block totals: FP64 sums within each warp in a fixed order, then the 8
  // warp results in FP64 in warp order
  double v[8] = {s_mass.value(), s_jx.value(), s_jy.value(), s_jz.value(), s_vol.value(), (double)cnt, 0.0, 0.0};
  const double sum = warp_sum8(v, tx);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const C um = __shfl_down_sync(0xffffffffu, umax, o);
    const C mn = __shfl_down_sync(0xffffffffu, rmin, o);
    const C mx = __shfl_down_sync(0xffffffffu, rmax, o);
    umax = um > umax ? um : umax;
    rmin = mn < rmin ? mn : rmin;
    rmax = mx > rmax ? mx : rmax;
  }
  const int anybad = __any_sync(0xffffffffu, bad);
  __shared__ double sh_w[NG][DY];
  if (tx % 4 == 0 && tx < 24) sh_w[tx / 4][ty] = sum;
  if (tx == 0) {
    sh_w[6][ty] = (double)umax;
    sh_w[7][ty] = (double)rmin;
    sh_w[8][ty] = (double)rmax;
    sh_w[9][ty] = anybad ? 1.0 : 0.0;
  }
  __syncthreads();
  if (ty == 0 && x < g.nx) {
    double a = 0.0, b = 0.0;
    for (int k = 0; k < DY; ++k) {
      a += sh_s[0][k][tx];
      b += sh_s[1][k][tx];
    }
    slices[((long long)blockIdx.y * g.nx + x) * 2 + 0] = a;
    slices[((long long)blockIdx.y * g.nx + x) * 2 + 1] = b;
  }
  if (ty == 0 && tx < NG) {
    double r;
    if (tx < 6) {
      r = 0.0;
      for (int k = 0; k < DY; ++k) r += sh_w[tx][k];
    } else if (tx == 7) {
      r = 1e300;
      for (int k = 0; k < DY; ++k) r = fmin(r, sh_w[tx][k]);
    } else if (tx < 10) {
      r = -1e300;
      for (int k = 0; k < DY; ++k) r = fmax(r, sh_w[tx][k]);
    } else {
      r = 0.0;
    }
    blocks[((long long)blockIdx.y * gridDim.x + blockIdx.x) * NG + tx] = r;
  }
}

// The LAYOUT_LOCAL pass of FP32 and 2-byte storage on lattices with even nx:
// two nodes x, x + 1 per thread (block.x = 32 pairs), loaded as one vector per
// population, the density with its rounding error, the momentum and the sums
// in paired FP32 instructions.  The accumulators of the liquid fraction are
// per x, so they serve the slices and the total.  labels (nullable): also
// starts the component labelling (ccl_init_kernel's output with runs inside
// segments of 64 nodes; thr_lo the largest float not above the threshold), so
// that counting droplets reads the populations once.
// 256x128x128 FP32, HBM floor 48 us: 133 us one node per thread with 16 blocks
// per SM, 78 us so, the labels included.
template <int P, bool WRITE_PSI>
__global__ void __launch_bounds__(DX* DY, 2) diag_pair_kernel(Geom g, Phys ph, const typename Prec<P>::T* f,
                                                              double rho_l, double rho_v, double* slices,
                                                              double* blocks, float* psi, int* flag, int* labels,
                                                              int* sizes, float thr_lo) {
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int x = 2 * (blockIdx.x * DX + tx);
  const bool in = x < g.nx;
  const int rows = g.ny * g.nz;
  const float thr = (float)(0.5 * (rho_l + rho_v)), inv = (float)(1.0 / (rho_l - rho_v)), rv = (float)rho_v;
  DSum2 s_mass, s_jx, s_jy, s_jz, s_vol;
  float umax = 0.0f, rmin = 3.0e38f, rmax = -3.0e38f;
  int cnt[2] = {0, 0};
  bool bad = false;
  const float s0 = shift_f<P>(0, ph), s1 = shift_f<P>(1, ph), s2 = shift_f<P>(7, ph);
  // every lane of a warp walks the same rows (the labelling votes)
  for (int r = blockIdx.y * DY + ty; r < rows; r += DY * gridDim.y) {
    const int i = x + g.nx * r;
    float2 rho = make_float2(0.0f, 0.0f);
    if (in) {
      float2 fv[Q];
#pragma unroll
      for (int a = 0; a < Q; ++a) load_pair_nc<P>(f + (long long)a * g.N + i, a == 0 ? s0 : (a <= 6 ? s1 : s2), fv[a]);
      float2 lo, jx, jy, jz;
      rho = rho_of_x<float2>(fv, lo);
      mom_of<float2>(fv, jx, jy, jz);
      if constexpr (WRITE_PSI) *reinterpret_cast<float2*>(psi + i) = psi_of2(rho, ph);
      s_mass.add(rho, lo);
      s_jx.add(jx);
      s_jy.add(jy);
      s_jz.add(jz);
      float2 phi = xmul(vsub(rho, make_float2(rv, rv)), make_float2(inv, inv));
      phi.x = phi.x < 0.0f ? 0.0f : (phi.x > 1.0f ? 1.0f : phi.x);
      phi.y = phi.y < 0.0f ? 0.0f : (phi.y > 1.0f ? 1.0f : phi.y);
      s_vol.add(phi);
      cnt[0] += rho.x > thr;
      cnt[1] += rho.y > thr;
      const float2 jj = xfma(jz, jz, xfma(jy, jy, xmul(jx, jx)));
#pragma unroll
      for (int n = 0; n < 2; ++n) {
        const float r1 = n ? rho.y : rho.x, j2 = n ? jj.y : jj.x;
        // the root and the division only where |j|/rho can reach the maximum
        // (the factor covers the rounding of the test, the second bound
        // values whose squares lose digits)
        const float t = umax * r1;
        if (j2 >= 0.999998f * (t * t) || j2 < 1e-30f) {
          const float u = sqrtf(j2) / r1;
          umax = u > umax ? u : umax;
        }
        rmin = r1 < rmin ? r1 : rmin;
        rmax = r1 > rmax ? r1 : rmax;
        bad |= !(r1 > 0.0f) || !(r1 <= 3.0e38f);
      }
    }
    if (labels) {
      const bool l0 = in && rho.x > thr_lo, l1 = in && rho.y > thr_lo;
      const unsigned both = __ballot_sync(0xffffffffu, l0 && l1), second = __ballot_sync(0xffffffffu, l1);
      if (in) {
        // start of the run that reaches this pair from the left: after the last
        // pair below that is not liquid throughout
        const unsigned gap = ~both & ((1u << tx) - 1u);
        int from = 0;
        if (gap) {
          const int l = 31 - __clz(gap);
          from = 2 * l + ((second >> l) & 1 ? 1 : 2);
        }
        const int start = i - 2 * tx + from;
        *reinterpret_cast<int2*>(labels + i) = make_int2(l0 ? start : -1, l1 ? (l0 ? start : i + 1) : -1);
        *reinterpret_cast<int2*>(sizes + i) = make_int2(0, 0);
      }
    }
  }
  if constexpr (WRITE_PSI) raise_flag(bad, flag);
  __shared__ double sh_s[2][DY][2 * DX];
  const double w0 = (double)s_vol.hi.x + (double)s_vol.lo.x, w1 = (double)s_vol.hi.y + (double)s_vol.lo.y;
  sh_s[0][ty][2 * tx] = w0;
  sh_s[0][ty][2 * tx + 1] = w1;
  sh_s[1][ty][2 * tx] = (double)cnt[0];
  sh_s[1][ty][2 * tx + 1] = (double)cnt[1];
  double v[8] = {s_mass.value(), s_jx.value(), s_jy.value(), s_jz.value(), w0 + w1, (double)(cnt[0] + cnt[1]), 0.0, 0.0};
  const double sum = warp_sum8(v, tx);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float um = __shfl_down_sync(0xffffffffu, umax, o);
    const float mn = __shfl_down_sync(0xffffffffu, rmin, o);
    const float mx = __shfl_down_sync(0xffffffffu, rmax, o);
    umax = um > umax ? um : umax;
    rmin = mn < rmin ? mn : rmin;
    rmax = mx > rmax ? mx : rmax;
  }
  const int anybad = __any_sync(0xffffffffu, bad);
  __shared__ double sh_w[NG][DY];
  if (tx % 4 == 0 && tx < 24) sh_w[tx / 4][ty] = sum;
  if (tx == 0) {
    sh_w[6][ty] = (double)umax;
    sh_w[7][ty] = (double)rmin;
    sh_w[8][ty] = (double)rmax;
    sh_w[9][ty] = anybad ? 1.0 : 0.0;
  }
  __syncthreads();
  const int t = ty * DX + tx, xt = blockIdx.x * 2 * DX + t;
  if (t < 2 * DX) {
    if (xt < g.nx) {
      double a = 0.0, b = 0.0;
      for (int k = 0; k < DY; ++k) {
        a += sh_s[0][k][t];
        b += sh_s[1][k][t];
      }
      slices[((long long)blockIdx.y * g.nx + xt) * 2 + 0] = a;
      slices[((long long)blockIdx.y * g.nx + xt) * 2 + 1] = b;
    }
  } else if (t < 2 * DX + NG) {
    const int k = t - 2 * DX;
    double r = k < 6 || k > 9 ? 0.0 : (k == 7 ? 1e300 : -1e300);
    for (int w = 0; w < DY && k < 10; ++w)
      r = k < 6 ? r + sh_w[k][w] : (k == 7 ? fmin(r, sh_w[k][w]) : fmax(r, sh_w[k][w]));
    blocks[((long long)blockIdx.y * gridDim.x + blockIdx.x) * NG + k] = r;
  }
}

constexpr int FT = 256;

// Per-slice totals: one warp per slice x; lane l sums row-blocks l, l + 32,
// ... with four independent accumulators (loads in flight), then a fixed
// shuffle tree.  tot[2x] = liquid area A_w(x), tot[2x + 1] = liquid nodes.
__global__ void __launch_bounds__(256) diag_slices_kernel(Geom g, int row_blocks,
                                                         const double* slices, double* tot) {
  if (g.chain) chain_wait();
  const int lane = threadIdx.x & 31;
  const int x = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (x >= g.nx) return;
  double a[4] = {0.0, 0.0, 0.0, 0.0}, c[4] = {0.0, 0.0, 0.0, 0.0};
  int rb = lane;
  for (; rb + 96 < row_blocks; rb += 128) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      a[k] += slices[((long long)(rb + 32 * k) * g.nx + x) * 2 + 0];
      c[k] += slices[((long long)(rb + 32 * k) * g.nx + x) * 2 + 1];
    }
  }
  for (; rb < row_blocks; rb += 32) {
    a[0] += slices[((long long)rb * g.nx + x) * 2 + 0];
    c[0] += slices[((long long)rb * g.nx + x) * 2 + 1];
  }
  double sa = (a[0] + a[1]) + (a[2] + a[3]), sc = (c[0] + c[1]) + (c[2] + c[3]);
  for (int o = 16; o > 0; o >>= 1) {
    sa += __shfl_down_sync(0xffffffffu, sa, o);
    sc += __shfl_down_sync(0xffffffffu, sc, o);
  }
  if (lane == 0) {
    tot[2 * x] = sa;
    tot[2 * x + 1] = sc;
  }
}

// Writes the DIAG_OUT results to out, or, with a ring counter, to record
// slot (counter++ mod ring_cap) of the ring at out (DIAG_STRIDE doubles per
// record).
// First stage for many block partials (the fused step writes one per block):
// block j folds the records [j chunk, (j + 1) chunk) into record j chunk, in
// a fixed order, so the final kernel reads nblocks / chunk records.
__global__ void __launch_bounds__(FT) diag_blocks_kernel(int nblocks, int chunk, double* blocks) {
  __shared__ double sg[NG][FT];
  const int t = threadIdx.x;
  const long long b0 = (long long)blockIdx.x * chunk;
  const long long b1 = min((long long)nblocks, b0 + chunk);
  double acc[NG];
#pragma unroll
  for (int k = 0; k < NG; ++k) acc[k] = 0.0;
  acc[7] = 1e300;
  acc[8] = -1e300;
  for (long long b = b0 + t; b < b1; b += FT) {
#pragma unroll
    for (int k = 0; k < 6; ++k) acc[k] += blocks[b * NG + k];
    acc[6] = fmax(acc[6], blocks[b * NG + 6]);
    acc[7] = fmin(acc[7], blocks[b * NG + 7]);
    acc[8] = fmax(acc[8], blocks[b * NG + 8]);
    acc[9] = fmax(acc[9], blocks[b * NG + 9]);
  }
#pragma unroll
  for (int k = 0; k < NG; ++k) sg[k][t] = acc[k];
  __syncthreads();
  for (int s = FT / 2; s > 0; s >>= 1) {
    if (t < s) {
#pragma unroll
      for (int k = 0; k < 6; ++k) sg[k][t] += sg[k][t + s];
      sg[6][t] = fmax(sg[6][t], sg[6][t + s]);
      sg[7][t] = fmin(sg[7][t], sg[7][t + s]);
      sg[8][t] = fmax(sg[8][t], sg[8][t + s]);
      sg[9][t] = fmax(sg[9][t], sg[9][t + s]);
    }
    __syncthreads();
  }
  if (t < NG) blocks[b0 * NG + t] = t < 10 ? sg[t][0] : 0.0;
}

// Final reduction: the nblocks block records, stride records apart, and the
// slice totals.
__global__ void __launch_bounds__(FT) diag_final_kernel(Geom g, int nblocks, int stride,
                                                       const double* slice_tot, const double* blocks,
                                                       double* out, unsigned long long* ring_count,
                                                       int ring_cap) {
  __shared__ double sg[NG][FT];
  __shared__ double smin_w[FT], smin_n[FT];
  __shared__ int smin_x[FT];
  if (g.chain) chain_wait();
  const int t = threadIdx.x;
  double acc[NG];
#pragma unroll
  for (int k = 0; k < NG; ++k) acc[k] = 0.0;
  acc[7] = 1e300;
  acc[8] = -1e300;
#pragma unroll 4
  for (int b = t; b < nblocks; b += FT) {
    const double* r = blocks + (long long)b * stride * NG;
#pragma unroll
    for (int k = 0; k < 6; ++k) acc[k] += r[k];
    acc[6] = fmax(acc[6], r[6]);
    acc[7] = fmin(acc[7], r[7]);
    acc[8] = fmax(acc[8], r[8]);
    acc[9] = fmax(acc[9], r[9]);
  }
  // minima over the slice totals (first x on ties)
  double mw = 1e300, mn = 1e300;
  int mx = 0x7fffffff;
  for (int x = t; x < g.nx; x += FT) {
    const double a = slice_tot[2 * x], c = slice_tot[2 * x + 1];
    if (a < mw) mw = a;
    if (c < mn) {
      mn = c;
      mx = x;
    }
  }
#pragma unroll
  for (int k = 0; k < NG; ++k) sg[k][t] = acc[k];
  smin_w[t] = mw;
  smin_n[t] = mn;
  smin_x[t] = mx;
  __syncthreads();
  for (int s = FT / 2; s > 0; s >>= 1) {
    if (t < s) {
#pragma unroll
      for (int k = 0; k < 6; ++k) sg[k][t] += sg[k][t + s];
      sg[6][t] = fmax(sg[6][t], sg[6][t + s]);
      sg[7][t] = fmin(sg[7][t], sg[7][t + s]);
      sg[8][t] = fmax(sg[8][t], sg[8][t + s]);
      sg[9][t] = fmax(sg[9][t], sg[9][t + s]);
      smin_w[t] = fmin(smin_w[t], smin_w[t + s]);
      const double on = smin_n[t + s];
      const int ox = smin_x[t + s];
      if (on < smin_n[t] || (on == smin_n[t] && ox < smin_x[t])) {
        smin_n[t] = on;
        smin_x[t] = ox;
      }
    }
    __syncthreads();
  }
  if (t == 0) {
    if (ring_count) {
      const unsigned long long n = *ring_count;
      *ring_count = n + 1;
      out += (n % (unsigned long long)ring_cap) * DIAG_STRIDE;
      out[DIAG_OUT] = (double)n;
      out[DIAG_CCL + 0] = out[DIAG_CCL + 1] = out[DIAG_CCL + 2] = -1.0;
      out[DIAG_CCL + 3] = 0.0;
    }
    out[0] = sg[0][0];
    out[1] = sg[1][0];
    out[2] = sg[2][0];
    out[3] = sg[3][0];
    out[4] = sg[4][0];
    out[5] = sg[5][0];
    out[6] = smin_w[0];
    out[7] = smin_n[0];
    out[8] = (double)smin_x[0];
    out[9] = sg[6][0];
    out[10] = sg[7][0];
    out[11] = sg[8][0];
    out[12] = sg[9][0] > 0.0 ? 0.0 : 1.0;
  }
}

// ---------------------------------------------------------------------------
// Connected components of the liquid (rho > threshold), 6-connectivity,
// periodic: lock-free union-find on int labels.  Every label points to a
// node of smaller or equal index, so each root search and each union retry
// strictly decreases an index and ends within N iterations.  As a guard the
// loops still stop after kMaxHops steps and raise an error flag (out[3]).
// ---------------------------------------------------------------------------
constexpr long long kMaxHops = 1ll << 31;

__device__ __forceinline__ int find_root(const int* L, int i, long long& hops) {
  int p = L[i];
  while (p != i && hops < kMaxHops) {
    i = p;
    p = L[i];
    ++hops;
  }
  return i;
}

__device__ __forceinline__ void unite(int* L, int a, int b, unsigned long long* err) {
  long long hops = 0;
  while (hops < kMaxHops) {
    a = find_root(L, a, hops);
    b = find_root(L, b, hops);
    if (a == b) return;
    ++hops;
    if (a < b) {
      const int old = atomicMin(&L[b], a);
      if (old == b) return;
      b = old;
    } else {
      const int old = atomicMin(&L[a], b);
      if (old == a) return;
      a = old;
    }
  }
  atomicOr(err, 1ull);
}

// Labels to start from: -1 outside the liquid, else the first node of the run
// of liquid nodes that ends here, within the thread's segment (a warp's 32
// consecutive nodes, cut at row ends), so that only the segments' first nodes
// still have to be joined to their left neighbours.
template <int P>
__global__ void ccl_init_kernel(Geom g, Phys ph, int layout, const typename Prec<P>::T* f,
                                double thr, int* L, int* sizes) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  bool liquid = false;
  int x = 0, y, z;
  if (i < g.N) {
    coords(g, i, x, y, z);
    Nbr nb;
    nb.make(g, x, y, z);
    typename Prec<P>::C rho, j[3];
    node_rho_j<P>(g, ph, layout, f, nb, rho, j);
    liquid = (double)rho > thr;
  }
  const int lane = threadIdx.x & 31;
  const unsigned m = __ballot_sync(0xffffffffu, liquid);
  if (i >= g.N) return;
  const unsigned gap = ~m & ((1u << lane) - 1u);
  int from = gap ? 32 - __clz(gap) : 0;
  if (lane - from > x) from = lane - x;   // the row starts inside the warp
  L[i] = liquid ? (int)i - (lane - from) : -1;
  sizes[i] = 0;
}

// Joins the runs: a segment's first node to its left neighbour, every node to
// its neighbours at y + 1 and z + 1 unless the left neighbours of both are
// liquid too (they are joined to these, and make the same link).  seg: x
// segments of 64 (diag_pair_kernel) or, 0, warps of 32 nodes (ccl_init_kernel).
// A ligament of 0.8 M liquid nodes of 256x128x128: 83 us joining every node to
// three neighbours, 19 us.
__global__ void ccl_union_kernel(Geom g, int seg, int* L, unsigned long long* err) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= g.N || L[i] < 0) return;
  int x, y, z;
  coords(g, i, x, y, z);
  const int row = (int)i - x;
  const int left = x == 0 ? row + g.nx - 1 : (int)i - 1;
  const bool l = L[left] >= 0;
  const bool first = x == 0 || (seg ? x % seg == 0 : (i & 31) == 0);
  if (l && first) unite(L, (int)i, left, err);
  const int dy = (y == g.ny - 1 ? -(g.ny - 1) : 1) * g.nx;
  const int dz = (z == g.nz - 1 ? -(g.nz - 1) : 1) * g.nx * g.ny;
  // (the left pair's own link: not across the periodic face, where the pair
  // of x = nx - 1 would defer to this one in turn)
  const bool defer = l && x > 0;
  if (L[i + dy] >= 0 && !(defer && L[left + dy] >= 0)) unite(L, (int)i, (int)i + dy, err);
  if (L[i + dz] >= 0 && !(defer && L[left + dz] >= 0)) unite(L, (int)i, (int)i + dz, err);
}

// After the unions every tree is final, so pointing a node straight at its
// root (the smallest index of its component) leaves every concurrent root
// search valid.  The sizes are counted per block where its nodes share the
// root of its first liquid thread, per group of a warp otherwise: one atomic
// per node on a ligament's single root took 326 us of 256x128x128, now 15 us.
__global__ void __launch_bounds__(256) ccl_compress_kernel(Geom g, int* L, int* sizes, unsigned long long* err) {
  __shared__ int s_root, s_count;
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (threadIdx.x == 0) {
    s_root = -1;
    s_count = 0;
  }
  __syncthreads();
  int r = -1;
  if (i < g.N && L[i] >= 0) {
    long long hops = 0;
    r = find_root(L, (int)i, hops);
    if (hops >= kMaxHops) atomicOr(err, 1ull);
    L[i] = r;
    if (s_root < 0) atomicCAS(&s_root, -1, r);
  }
  __syncthreads();
  const int root = s_root;
  if (root < 0) return;   // no liquid in the block
  const unsigned group = __match_any_sync(0xffffffffu, r);
  if (r >= 0 && (threadIdx.x & 31) == __ffs(group) - 1) {
    if (r == root)
      atomicAdd(&s_count, __popc(group));
    else
      atomicAdd(&sizes[r], __popc(group));
  }
  __syncthreads();
  if (threadIdx.x == 0) atomicAdd(&sizes[root], s_count);
}

// Counts; slots (droplet statistics): each root's size is replaced by its
// record slot, the number of roots counted before it.
__global__ void __launch_bounds__(256) ccl_count_kernel(Geom g, const int* L, int* sizes, int slots,
                                                        unsigned long long* out) {
  const long long i0 = (long long)blockIdx.x * 4 * 256 + threadIdx.x;
  int l[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) l[k] = i0 + 256 * k < g.N ? L[i0 + 256 * k] : -1;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const long long i = i0 + 256 * k;
    if (l[k] != (int)i) continue;
    const int n = sizes[i];
    const unsigned long long c = atomicAdd(&out[0], 1ull);
    if (n >= 8) atomicAdd(&out[1], 1ull);
    atomicMax(&out[2], (unsigned long long)n);
    if (slots) sizes[i] = (int)c;
  }
}

// Copies the droplet counts of the CCL just run into the ring record the
// diagnostics of the same step appended (slot counter - 1).
__global__ void ccl_ring_kernel(const long long* out4, double* ring, const unsigned long long* ring_count,
                                int ring_cap) {
  const unsigned long long n = *ring_count - 1;
  double* rec = ring + (n % (unsigned long long)ring_cap) * DIAG_STRIDE;
  rec[DIAG_CCL + 0] = (double)out4[0];
  rec[DIAG_CCL + 1] = (double)out4[1];
  rec[DIAG_CCL + 2] = (double)out4[2];
  rec[DIAG_CCL + 3] = (double)out4[3];
}

// ---------------------------------------------------------------------------
// Per-droplet statistics (after launch_ccl with slots): every liquid node adds
// to its droplet's record
//   [root, nodes, sum phi, sum rho, cos/sin sums of 2 pi x/nx, y, z]
// and sets the bit of its x slice in the droplet's x-occupancy mask.  The
// FP64 sums are atomic (their order, and so the last bits, vary run to run).
// ---------------------------------------------------------------------------
// cos and sin of 2 pi c / n for the coordinates of x, then y, then z
__global__ void trig_kernel(Geom g, double2* trig) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int n = t < g.nx ? g.nx : (t < g.nx + g.ny ? g.ny : g.nz);
  if (t >= g.nx + g.ny + g.nz) return;
  const int c = t < g.nx ? t : (t < g.nx + g.ny ? t - g.nx : t - g.nx - g.ny);
  double2 v;
  sincospi(2.0 * c / n, &v.y, &v.x);
  trig[t] = v;
}

// A warp walks SEGS segments of 32 consecutive nodes and keeps the sums of
// one droplet in its lanes until it meets another (the common case: segments
// of one row lie in one droplet); segments that hold several droplets add
// node by node.  What bounds it is the FP64 pipe, 16 clocks per warp
// instruction: the angles come from a table (six FP64 sincospi per node before)
// and the warp sums run once per droplet met instead of once per segment,
// eight at a time, the count as an integer (256x128x128, a ligament of 0.8 M
// liquid nodes: 195 us, 61 us now; with a tree per value 90 us; with those, 16
// segments per warp, 78 us there, left the droplets of a broken-up state to
// too few warps: 100 us instead of 50).
template <int P, int SEGS>
__global__ void __launch_bounds__(256) droplet_stats_kernel(Geom g, Phys ph, int layout, const typename Prec<P>::T* f,
                                                            double rho_l, double rho_v, const int* L,
                                                            const int* slot_of, const double2* __restrict__ trig,
                                                            double* rec, unsigned* xbits, int words) {
  using C = typename Prec<P>::C;
  constexpr int NV = DROP_REC - 2;   // beside the root and the node count
  static_assert(NV == 8, "warp_sum8");
  const int lane = threadIdx.x & 31;
  const long long warp = (long long)blockIdx.x * (blockDim.x / 32) + threadIdx.x / 32;
  const double inv = 1.0 / (rho_l - rho_v);
  double v[NV];
#pragma unroll
  for (int m = 0; m < NV; ++m) v[m] = 0.0;
  int cur = -1, nodes = 0;   // slot whose sums the lanes hold, its nodes
  auto flush = [&]() {
    if (cur < 0) return;
    double* r = rec + (size_t)cur * DROP_REC;
    const double t = warp_sum8(v, lane);
    if (lane % 4 == 0) atomicAdd(r + 2 + lane / 4, t);
    if (lane == 1) atomicAdd(r + 1, (double)nodes);
#pragma unroll
    for (int m = 0; m < NV; ++m) v[m] = 0.0;
    nodes = 0;
  };
  int roots[SEGS];
#pragma unroll
  for (int seg = 0; seg < SEGS; ++seg) {
    const long long i = (warp * SEGS + seg) * 32 + lane;
    roots[seg] = i < g.N ? L[i] : -1;
  }
#pragma unroll 1
  for (int seg = 0; seg < SEGS; ++seg) {
    const long long i = (warp * SEGS + seg) * 32 + lane;
    int root = -1;
#pragma unroll
    for (int k = 0; k < SEGS; ++k) root = k == seg ? roots[k] : root;
    if (__ballot_sync(0xffffffffu, root >= 0) == 0) continue;
    int k = -1;
    double n[NV];
    if (root >= 0) {
      k = slot_of[root];
      if (root == (int)i) rec[(size_t)k * DROP_REC] = (double)root;
      int x, y, z;
      coords(g, i, x, y, z);
      Nbr nb;
      nb.make(g, x, y, z);
      C rc, j[3];
      node_rho_j<P>(g, ph, layout, f, nb, rc, j);
      const double rho = (double)rc;
      const double2 tx = __ldg(trig + x), ty = __ldg(trig + g.nx + y), tz = __ldg(trig + g.nx + g.ny + z);
      n[0] = fmin(fmax((rho - rho_v) * inv, 0.0), 1.0);
      n[1] = rho;
      n[2] = tx.x, n[3] = tx.y, n[4] = ty.x, n[5] = ty.y, n[6] = tz.x, n[7] = tz.y;
      unsigned* w = xbits + (size_t)k * words + (x >> 5);
      const unsigned bit = 1u << (x & 31);
      if (!(*(volatile unsigned*)w & bit)) atomicOr(w, bit);
    }
    const int kmax = __reduce_max_sync(0xffffffffu, k);
    if (__all_sync(0xffffffffu, k < 0 || k == kmax)) {
      if (kmax != cur) {
        flush();
        cur = kmax;
      }
      nodes += __popc(__ballot_sync(0xffffffffu, k >= 0));
      if (k >= 0) {
#pragma unroll
        for (int m = 0; m < NV; ++m) v[m] += n[m];
      }
    } else if (k >= 0) {
      double* r = rec + (size_t)k * DROP_REC + 1;
      atomicAdd(r, 1.0);
#pragma unroll
      for (int m = 0; m < NV; ++m) atomicAdd(r + 1 + m, n[m]);
    }
  }
  flush();
}

inline unsigned blocks_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

template <int P>
cudaError_t init_t(const Geom& g, const Phys& ph, const InitSpec& sp, void* f, cudaStream_t s) {
  init_kernel<P><<<blocks_for(g.N, 256), 256, 0, s>>>(g, ph, sp, (typename Prec<P>::T*)f);
  return cudaGetLastError();
}
template <int P>
cudaError_t get_t(int layout, const Geom& g, const Phys& ph, const void* f, int a0, int n, double* out,
                  cudaStream_t s) {
  get_planes_kernel<P><<<dim3(blocks_for(g.N, 256), n), 256, 0, s>>>(g, ph, layout, (const typename Prec<P>::T*)f, a0,
                                                                     out);
  return cudaGetLastError();
}
template <int P>
cudaError_t set_t(int layout, const Geom& g, const Phys& ph, void* f, int a0, int n, const double* in,
                  cudaStream_t s) {
  set_planes_kernel<P><<<dim3(blocks_for(g.N, 256), n), 256, 0, s>>>(g, ph, layout, (typename Prec<P>::T*)f, a0, in);
  return cudaGetLastError();
}
template <int P>
cudaError_t moments_t(int layout, const Geom& g, const Phys& ph, const void* f, const void* psi,
                      double* r, double* ux, double* uy, double* uz, cudaStream_t s) {
  moments_kernel<P><<<blocks_for(g.N, 256), 256, 0, s>>>(
      g, ph, layout, (const typename Prec<P>::T*)f, (const typename Prec<P>::C*)psi, r, ux, uy, uz);
  return cudaGetLastError();
}
// Whether the diagnostics pass takes node pairs (even nx, so that every row
// and slot starts at a pair if the arrays do).
bool diag_pairs(int precision, int layout, const Geom& g, const void* f, const void* psi) {
  return precision != LBM_F64 && layout == LAYOUT_LOCAL && g.nx % 2 == 0 && g.N <= 0x7fffffff &&
         (uintptr_t)f % (2 * elem_size(precision)) == 0 && (uintptr_t)psi % 8 == 0;
}

template <int P>
cudaError_t diag_t(int layout, const Geom& g, const Phys& ph, const void* f, double rho_l,
                   double rho_v, double* scratch, double* out, void* psi, int* flag,
                   unsigned long long* ring_count, int ring_cap, cudaStream_t s, const DiagExtra& x) {
  const bool pairs = diag_pairs(P, layout, g, f, psi);
  const int gx = pairs ? (g.nx + 2 * DX - 1) / (2 * DX) : (g.nx + DX - 1) / DX;
  const int rb = diag_row_blocks(g, gx, 4);
  double* slices = scratch;
  double* blocks = scratch + (size_t)rb * g.nx * 2;
  double* slice_tot = blocks + (size_t)gx * rb * NG;
  using T = typename Prec<P>::T;
  using C = typename Prec<P>::C;
  const dim3 grid(gx, rb), block(DX, DY);
  const T* in = (const T*)f;
  if constexpr (P != LBM_F64) {
    if (pairs && psi)
      diag_pair_kernel<P, true><<<grid, block, 0, s>>>(g, ph, in, rho_l, rho_v, slices, blocks, (float*)psi, flag,
                                                       x.labels, x.sizes, x.thr_lo);
    else if (pairs)
      diag_pair_kernel<P, false><<<grid, block, 0, s>>>(g, ph, in, rho_l, rho_v, slices, blocks, nullptr, nullptr,
                                                        x.labels, x.sizes, x.thr_lo);
  }
  double* const rho_out = P == LBM_F64 ? (double*)x.dst : nullptr;
  if (!pairs && psi) {
    if (layout == LAYOUT_LOCAL)
      diag_partial_kernel<P, true, LAYOUT_LOCAL><<<grid, block, 0, s>>>(
          g, ph, in, rho_l, rho_v, slices, blocks, (C*)psi, flag, rho_out);
    else
      diag_partial_kernel<P, true, LAYOUT_GATHER><<<grid, block, 0, s>>>(
          g, ph, in, rho_l, rho_v, slices, blocks, (C*)psi, flag, rho_out);
  } else if (!pairs) {
    if (layout == LAYOUT_LOCAL)
      diag_partial_kernel<P, false, LAYOUT_LOCAL><<<grid, block, 0, s>>>(
          g, ph, in, rho_l, rho_v, slices, blocks, nullptr, nullptr, nullptr);
    else
      diag_partial_kernel<P, false, LAYOUT_GATHER><<<grid, block, 0, s>>>(
          g, ph, in, rho_l, rho_v, slices, blocks, nullptr, nullptr, nullptr);
  }
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return launch_diag_reduce(g, rb, gx * rb, slices, blocks, slice_tot, out, ring_count, ring_cap, s, x.side);
}

template <int P>
cudaError_t ccl_init_t(int layout, const Geom& g, const Phys& ph, const void* f, double thr, int* L, int* sizes,
                       cudaStream_t s) {
  ccl_init_kernel<P><<<blocks_for(g.N, 256), 256, 0, s>>>(g, ph, layout, (const typename Prec<P>::T*)f, thr, L, sizes);
  return cudaGetLastError();
}

template <int P>
cudaError_t droplets_t(int layout, const Geom& g, const Phys& ph, const void* f, double rho_l, double rho_v,
                       const int* L, const int* slot_of, const double2* trig, double* rec, unsigned* xbits, int cap,
                       cudaStream_t s) {
  const int words = (g.nx + 31) / 32;
  cudaError_t e = cudaMemsetAsync(rec, 0, sizeof(double) * DROP_REC * (size_t)cap, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(xbits, 0, sizeof(unsigned) * words * (size_t)cap, s);
  if (e != cudaSuccess) return e;
  // four segments per warp where that leaves four blocks per SM
  const auto kernel = g.N >= 4 * 256LL * 4 * kSmCount ? droplet_stats_kernel<P, 4> : droplet_stats_kernel<P, 1>;
  const int segs = g.N >= 4 * 256LL * 4 * kSmCount ? 4 : 1;
  kernel<<<blocks_for(g.N, 256 * segs), 256, 0, s>>>(g, ph, layout, (const typename Prec<P>::T*)f, rho_l, rho_v, L,
                                                     slot_of, trig, rec, xbits, words);
  return cudaGetLastError();
}

}  // namespace

// The table of psi_of<double>: exp(-k/256) and 1 - exp(-k/256), k < kPsiTab.
__global__ void psi_table_kernel(double2* tab) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < kPsiTab) tab[k] = make_double2(exp(-k / 256.0), -expm1(-k / 256.0));
}

cudaError_t psi_table_launch(double2* tab, cudaStream_t s) {
  psi_table_kernel<<<(kPsiTab + 127) / 128, 128, 0, s>>>(tab);
  return cudaGetLastError();
}

// Stochastic-rounding step salt: set it, or write another word's value plus n.
__global__ void salt_set_kernel(unsigned* salt, unsigned value) { *salt = value; }
__global__ void salt_add_kernel(const unsigned* from, unsigned* to, unsigned n) { *to = *from + n; }

cudaError_t launch_salt(unsigned* salt, bool set, unsigned value, cudaStream_t s) {
  if (!set) return launch_salt_add(salt, salt, 1u, s);
  salt_set_kernel<<<1, 1, 0, s>>>(salt, value);
  return cudaGetLastError();
}

cudaError_t launch_salt_add(const unsigned* from, unsigned* to, unsigned n, cudaStream_t s) {
  salt_add_kernel<<<1, 1, 0, s>>>(from, to, n);
  return cudaGetLastError();
}

cudaError_t launch_diag_reduce(const Geom& g, int row_blocks, int nblocks, const double* slices,
                               double* blocks, double* slice_tot, double* out,
                               unsigned long long* ring_count, int ring_cap, cudaStream_t s, ReduceSide* side) {
  cudaError_t e = cudaSuccess;
  int chain = g.chain;
  if (side) {
    e = cudaEventRecord(side->fork, s);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(side->stream, side->fork, 0);
    if (e != cudaSuccess) return e;
    s = side->stream;
    chain = 0;
  }
  e = chain_launch(chain, diag_slices_kernel, (g.nx + 7) / 8, 256, 0, s, g, row_blocks, slices, slice_tot);
  // many records (one per block of the fused step): a parallel first stage
  // folds runs of kChunk records in place (a single block reading 131072
  // records of the 1024x512x512 lattice took 0.44 ms)
  constexpr int kChunk = 256;
  int stride = 1, n = nblocks;
  if (e == cudaSuccess && nblocks > 4 * kChunk) {
    n = (nblocks + kChunk - 1) / kChunk;
    diag_blocks_kernel<<<n, FT, 0, s>>>(nblocks, kChunk, blocks);
    e = cudaGetLastError();
    stride = kChunk;
  }
  if (e == cudaSuccess)
    e = chain_launch(chain, diag_final_kernel, 1, FT, 0, s, g, n, stride, slice_tot, blocks, out, ring_count, ring_cap);
  if (e == cudaSuccess && side) {
    e = cudaEventRecord(side->join, s);
    side->open = true;
  }
  return e;
}

cudaError_t launch_ccl_ring(const long long* out4, double* ring, const unsigned long long* ring_count,
                            int ring_cap, cudaStream_t s) {
  ccl_ring_kernel<<<1, 1, 0, s>>>(out4, ring, ring_count, ring_cap);
  return cudaGetLastError();
}

cudaError_t launch_droplets(int precision, int layout, const Geom& g, const Phys& ph, const void* f,
                            double rho_l, double rho_v, const int* labels, const int* slots, const double2* trig,
                            double* rec, unsigned* xbits, int cap, cudaStream_t s) {
  switch (precision) {
    case LBM_F64: return droplets_t<LBM_F64>(layout, g, ph, f, rho_l, rho_v, labels, slots, trig, rec, xbits, cap, s);
    case LBM_F32: return droplets_t<LBM_F32>(layout, g, ph, f, rho_l, rho_v, labels, slots, trig, rec, xbits, cap, s);
    case LBM_F16DEV:
      return droplets_t<LBM_F16DEV>(layout, g, ph, f, rho_l, rho_v, labels, slots, trig, rec, xbits, cap, s);
    case LBM_BF16DEV:
      return droplets_t<LBM_BF16DEV>(layout, g, ph, f, rho_l, rho_v, labels, slots, trig, rec, xbits, cap, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_trig(const Geom& g, double2* trig, cudaStream_t s) {
  trig_kernel<<<blocks_for((long long)g.nx + g.ny + g.nz, 128), 128, 0, s>>>(g, trig);
  return cudaGetLastError();
}

cudaError_t launch_init(int precision, const Geom& g, const Phys& ph, const InitSpec& spec, void* f,
                        cudaStream_t s) {
  switch (precision) {
    case LBM_F64: return init_t<LBM_F64>(g, ph, spec, f, s);
    case LBM_F32: return init_t<LBM_F32>(g, ph, spec, f, s);
    case LBM_F16DEV: return init_t<LBM_F16DEV>(g, ph, spec, f, s);
    case LBM_BF16DEV: return init_t<LBM_BF16DEV>(g, ph, spec, f, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_get_planes(int precision, int layout, const Geom& g, const Phys& ph, const void* f,
                              int a0, int n, double* out, cudaStream_t s) {
  switch (precision) {
    case LBM_F64: return get_t<LBM_F64>(layout, g, ph, f, a0, n, out, s);
    case LBM_F32: return get_t<LBM_F32>(layout, g, ph, f, a0, n, out, s);
    case LBM_F16DEV: return get_t<LBM_F16DEV>(layout, g, ph, f, a0, n, out, s);
    case LBM_BF16DEV: return get_t<LBM_BF16DEV>(layout, g, ph, f, a0, n, out, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_set_planes(int precision, int layout, const Geom& g, const Phys& ph, void* f, int a0,
                              int n, const double* in, cudaStream_t s) {
  switch (precision) {
    case LBM_F64: return set_t<LBM_F64>(layout, g, ph, f, a0, n, in, s);
    case LBM_F32: return set_t<LBM_F32>(layout, g, ph, f, a0, n, in, s);
    case LBM_F16DEV: return set_t<LBM_F16DEV>(layout, g, ph, f, a0, n, in, s);
    case LBM_BF16DEV: return set_t<LBM_BF16DEV>(layout, g, ph, f, a0, n, in, s);
  }
  return cudaErrorInvalidValue;
}

cudaError_t export_populations(int precision, int layout, const Geom& g, const Phys& ph, const void* f, double* work,
                               size_t work_doubles, double* host, cudaStream_t s) {
  const int per = (int)std::min<size_t>(Q, work_doubles / g.N);
  cudaError_t e = per < 1 ? cudaErrorInvalidValue : cudaSuccess;
  for (int a = 0; a < Q && e == cudaSuccess; a += per) {
    const int n = std::min(per, Q - a);
    e = launch_get_planes(precision, layout, g, ph, f, a, n, work, s);
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(host + (size_t)a * g.N, work, sizeof(double) * n * g.N, cudaMemcpyDeviceToHost, s);
  }
  const cudaError_t e2 = cudaStreamSynchronize(s);
  return e != cudaSuccess ? e : e2;
}

cudaError_t import_populations(int precision, int layout, const Geom& g, const Phys& ph, void* f, double* work,
                               size_t work_doubles, const double* host, cudaStream_t s) {
  const int per = (int)std::min<size_t>(Q, work_doubles / g.N);
  cudaError_t e = per < 1 ? cudaErrorInvalidValue : cudaSuccess;
  for (int a = 0; a < Q && e == cudaSuccess; a += per) {
    const int n = std::min(per, Q - a);
    e = cudaMemcpyAsync(work, host + (size_t)a * g.N, sizeof(double) * n * g.N, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = launch_set_planes(precision, layout, g, ph, f, a, n, work, s);
  }
  const cudaError_t e2 = cudaStreamSynchronize(s);
  return e != cudaSuccess ? e : e2;
}

cudaError_t launch_moments(int precision, int layout, const Geom& g, const Phys& ph, const void* f,
                           const void* psi, double* rho, double* ux, double* uy, double* uz,
                           cudaStream_t s) {
  switch (precision) {
    case LBM_F64: return moments_t<LBM_F64>(layout, g, ph, f, psi, rho, ux, uy, uz, s);
    case LBM_F32: return moments_t<LBM_F32>(layout, g, ph, f, psi, rho, ux, uy, uz, s);
    case LBM_F16DEV: return moments_t<LBM_F16DEV>(layout, g, ph, f, psi, rho, ux, uy, uz, s);
    case LBM_BF16DEV: return moments_t<LBM_BF16DEV>(layout, g, ph, f, psi, rho, ux, uy, uz, s);
  }
  return cudaErrorInvalidValue;
}

// (room for 16 row blocks per SM; the kernels use 4)
size_t diag_scratch_doubles(const Geom& g) {
  const int gx = (g.nx + DX - 1) / DX;
  const int rb = diag_row_blocks(g, gx, 16);
  return (size_t)rb * g.nx * 2 + (size_t)gx * rb * NG + (size_t)g.nx * 2;
}

cudaError_t launch_diagnostics(int precision, int layout, const Geom& g, const Phys& ph, const void* f,
                               double rho_l, double rho_v, double* scratch, double* out, void* psi,
                               int* flag, unsigned long long* ring_count, int ring_cap,
                               cudaStream_t s, const DiagExtra& x) {
  switch (precision) {
    case LBM_F64:
      return diag_t<LBM_F64>(layout, g, ph, f, rho_l, rho_v, scratch, out, psi, flag, ring_count, ring_cap, s, x);
    case LBM_F32:
      return diag_t<LBM_F32>(layout, g, ph, f, rho_l, rho_v, scratch, out, psi, flag, ring_count, ring_cap, s, x);
    case LBM_F16DEV:
      return diag_t<LBM_F16DEV>(layout, g, ph, f, rho_l, rho_v, scratch, out, psi, flag, ring_count, ring_cap, s, x);
    case LBM_BF16DEV:
      return diag_t<LBM_BF16DEV>(layout, g, ph, f, rho_l, rho_v, scratch, out, psi, flag, ring_count, ring_cap, s, x);
  }
  return cudaErrorInvalidValue;
}

DiagExtra diag_labels(int precision, int layout, const Geom& g, const void* f, const void* psi, double threshold,
                      int* labels, int* sizes) {
  DiagExtra x;
  if (!diag_pairs(precision, layout, g, f, psi)) return x;
  x.labels = labels;
  x.sizes = sizes;
  // rho > threshold for a float rho is rho > the largest float not above it
  x.thr_lo = (float)threshold;
  if ((double)x.thr_lo > threshold) x.thr_lo = nextafterf(x.thr_lo, -INFINITY);
  return x;
}

cudaError_t launch_ccl(int precision, int layout, const Geom& g, const Phys& ph, const void* f,
                       double threshold, int* labels, int* sizes, long long* out3, cudaStream_t s, bool started,
                       bool slots) {
  cudaError_t e = cudaMemsetAsync(out3, 0, 4 * sizeof(long long), s);
  if (e == cudaSuccess && !started) {
    switch (precision) {
      case LBM_F64: e = ccl_init_t<LBM_F64>(layout, g, ph, f, threshold, labels, sizes, s); break;
      case LBM_F32: e = ccl_init_t<LBM_F32>(layout, g, ph, f, threshold, labels, sizes, s); break;
      case LBM_F16DEV: e = ccl_init_t<LBM_F16DEV>(layout, g, ph, f, threshold, labels, sizes, s); break;
      case LBM_BF16DEV: e = ccl_init_t<LBM_BF16DEV>(layout, g, ph, f, threshold, labels, sizes, s); break;
      default: e = cudaErrorInvalidValue;
    }
  }
  if (e != cudaSuccess) return e;
  const unsigned nb = blocks_for(g.N, 256);
  unsigned long long* out = (unsigned long long*)out3;
  ccl_union_kernel<<<nb, 256, 0, s>>>(g, started ? 2 * DX : 0, labels, out + 3);
  ccl_compress_kernel<<<nb, 256, 0, s>>>(g, labels, sizes, out + 3);
  ccl_count_kernel<<<blocks_for(g.N, 4 * 256), 256, 0, s>>>(g, labels, sizes, slots ? 1 : 0, out);
  return cudaGetLastError();
}

}  // namespace lbm
