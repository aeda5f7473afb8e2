// Helper kernels around the fused step: state encode/decode (public layout <-> storage), the
// 16-bit scale search, the standalone and final conservation reductions, and the two-component
// phase-field update (Eq. ACeq) with the capillary force.
#pragma once

#include <type_traits>

#include "lattice.cuh"
#include "tma.cuh"

namespace lbf {

// arithmetic of the layout conversions: FP64 when either side is FP64, else FP32 - A - u u and N + u u are
// then one FMA, which rounds the exact value once, as the FP64 evaluation followed by the conversion did
// up to its double rounding. They are copies by nature: with FP64 arithmetic on every site the FP64 pipe
// (2 operations a clock per SM) held them to 23 G sites/s (256^3 FP32: 0.72 ms a pass where the 1.34 GB
// take 0.21 ms).
template <class A, class B>
struct ConvertIn {
  using type = typename std::conditional<std::is_same<A, double>::value || std::is_same<B, double>::value, double, float>::type;
};

// public [10][stride] (site i of the chunk) -> internal state at site0 + i, in dst and, if given, dst2
template <class Tin, class S>
__global__ void k_encode(const Tin* __restrict__ src, long long stride, long long site0, long long count,
                         S* __restrict__ dst, S* __restrict__ dst2, long long N, Scales sc) {
  using C = typename ConvertIn<Tin, S>::type;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    C v[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) v[k] = static_cast<C>(src[k * stride + i]);
    const C ux = v[1], uy = v[2], uz = v[3];
    v[4] = fma(-ux, ux, v[4]);
    v[5] = fma(-uy, uy, v[5]);
    v[6] = fma(-uz, uz, v[6]);
    v[7] = fma(-ux, uy, v[7]);
    v[8] = fma(-ux, uz, v[8]);
    v[9] = fma(-uy, uz, v[9]);
    const long long s = site0 + i;
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      const int g = k == 0 ? 0 : (k < 4 ? 1 : 2);
      if constexpr (Codec<S>::scaled) {
        const float x = static_cast<float>(v[k] * C(sc.enc[g]));
        Codec<S>::store(dst + k * N + s, x);
        if (dst2 != nullptr) Codec<S>::store(dst2 + k * N + s, x);
      } else {
        dst[k * N + s] = static_cast<S>(v[k]);
        if (dst2 != nullptr) dst2[k * N + s] = static_cast<S>(v[k]);
      }
    }
  }
}

// internal state at site0 + i -> public [10][stride]
template <class S, class Tout>
__global__ void k_decode(const S* __restrict__ src, long long N, long long site0, long long count,
                         Tout* __restrict__ dst, long long stride, Scales sc) {
  using C = typename ConvertIn<S, Tout>::type;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    const long long s = site0 + i;
    C v[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      const int g = k == 0 ? 0 : (k < 4 ? 1 : 2);
      if constexpr (Codec<S>::scaled)
        v[k] = static_cast<C>(Codec<S>::load(src + k * N + s)) * C(sc.dec[g]);
      else
        v[k] = static_cast<C>(src[k * N + s]);
    }
    const C ux = v[1], uy = v[2], uz = v[3];
    v[4] = fma(ux, ux, v[4]);
    v[5] = fma(uy, uy, v[5]);
    v[6] = fma(uz, uz, v[6]);
    v[7] = fma(ux, uy, v[7]);
    v[8] = fma(ux, uz, v[8]);
    v[9] = fma(uy, uz, v[9]);
#pragma unroll
    for (int k = 0; k < 10; ++k) dst[k * stride + i] = static_cast<Tout>(v[k]);
  }
}

// max |p*|, |u|, |A - u u| of a public chunk, as float bit patterns (non-negative floats order
// like their bits), into out[0..2] (atomicMax)
template <class Tin>
__global__ void k_absmax(const Tin* __restrict__ src, long long stride, long long count, unsigned* out) {
  float m[3] = {0.f, 0.f, 0.f};
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < count;
       i += (long long)gridDim.x * blockDim.x) {
    Tin v[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) v[k] = src[k * stride + i];
    const Tin ux = v[1], uy = v[2], uz = v[3];
    m[0] = fmaxf(m[0], (float)fabs(v[0]));
    m[1] = fmaxf(m[1], (float)fmax(fabs(ux), fmax(fabs(uy), fabs(uz))));
    const Tin n[6] = {fma(-ux, ux, v[4]), fma(-uy, uy, v[5]), fma(-uz, uz, v[6]),
                      fma(-ux, uy, v[7]), fma(-ux, uz, v[8]), fma(-uy, uz, v[9])};
#pragma unroll
    for (int k = 0; k < 6; ++k) m[2] = fmaxf(m[2], (float)fabs(n[k]));
  }
  for (int k = 0; k < 3; ++k) {
    float x = m[k];
    for (int o = 16; o > 0; o >>= 1) x = fmaxf(x, __shfl_xor_sync(0xffffffffu, x, o));
    if ((threadIdx.x & 31) == 0) atomicMax(out + k, __float_as_uint(x));
  }
}

// conservation sums of a state over fluid sites, one FP64 partial (8 doubles) per block
template <class S>
__global__ void k_reduce_state(const S* __restrict__ st, long long N, const uint8_t* __restrict__ mask,
                               const void* phi, bool phi_double, Scales sc, double* partials) {
  double acc[6] = {0, 0, 0, 0, 0, 0};
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N;
       s += (long long)gridDim.x * blockDim.x) {
    if (mask != nullptr && mask[s]) continue;
    double v[4];
    if constexpr (Codec<S>::scaled) {
      v[0] = static_cast<double>(Codec<S>::load(st + s)) * sc.dec[0];
      for (int k = 1; k < 4; ++k) v[k] = static_cast<double>(Codec<S>::load(st + k * N + s)) * sc.dec[1];
    } else {
      for (int k = 0; k < 4; ++k) v[k] = static_cast<double>(st[k * N + s]);
    }
    acc[0] += v[0];
    acc[1] += v[1];
    acc[2] += v[2];
    acc[3] += v[3];
    if (phi != nullptr)
      acc[4] += phi_double ? static_cast<const double*>(phi)[s] : static_cast<double>(static_cast<const float*>(phi)[s]);
    acc[5] += v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
  }
  __shared__ double sh[32][6];
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int k = 0; k < 6; ++k) {
    double x = acc[k];
    for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if (lane == 0) sh[wid][k] = x;
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    double s = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) s += sh[w][threadIdx.x];
    partials[blockIdx.x * 8 + threadIdx.x] = s;
  }
}

// deterministic sum of nblocks partials (one block of 256 threads, fixed order)
__global__ void k_reduce_final(const double* __restrict__ partials, long long nblocks, double* out) {
  __shared__ double sh[256][6];
  double acc[6] = {0, 0, 0, 0, 0, 0};
  for (long long b = threadIdx.x; b < nblocks; b += blockDim.x)
    for (int k = 0; k < 6; ++k) acc[k] += partials[b * 8 + k];
  for (int k = 0; k < 6; ++k) sh[threadIdx.x][k] = acc[k];
  __syncthreads();
  for (int step = 128; step > 0; step >>= 1) {
    if ((int)threadIdx.x < step)
      for (int k = 0; k < 6; ++k) sh[threadIdx.x][k] += sh[threadIdx.x + step][k];
    __syncthreads();
  }
  if (threadIdx.x < 6) out[threadIdx.x] = sh[0][threadIdx.x];
}

// ---------------------------------------------------------------------------------------------
// Two-component coupling (Sec. 2): D3Q27-weight stencils,
//   grad psi = 3 sum_i w_i c_i psi(x + c_i),  lap psi = 6 sum_i w_i (psi(x + c_i) - psi(x)),
//   div V = 3 sum_i w_i c_i . V(x + c_i)
// Allen-Cahn FTCS in flux form: phi' = phi - div(phi u) + D lap phi - lambda div(G),
// G = phi (1 - phi) n, n = grad phi / max(|grad phi|, 1e-12), lambda = 4 D / W.
//
// The D3Q27 weights are products of one-dimensional weights, w_i = a(c_x) a(c_y) a(c_z) with
// a(0) = 2/3 and a(+-1) = 1/6, so every stencil above separates into three-point filters along
// the axes: the smoothing A f = a(0) f(0) + a(1) (f(-1) + f(+1)) and the difference
// D f = (f(+1) - f(-1)) / 6, e.g. sum_i w_i c_i,x psi(x + c_i) = D_x A_y A_z psi and
// sum_i w_i psi(x + c_i) = A_x A_y A_z psi. The Laplacian is assembled from second differences
// only, with L = A - I = (1/6) [1, -2, 1]:
//   sum_i w_i (psi(x + c_i) - psi(x)) = L_x A_y psi + L_y psi + A_x A_y L_z psi,
// so that, as in the flux form, every term vanishes exactly on a constant field: the rounded
// weights 2/3 and 1/6 do not sum to exactly one, and "smoothed minus centre" would leak a
// systematic change of sum(phi) into every step. The kernels march along z with the same x-y tiles as
// the fused step (32 columns of which 30 are outputs, BY + 2 rows): every thread keeps three planes
// of its own column in registers and applies the z filters there, one shared-memory plane holds the
// z-filtered values, and the outputs apply the x-y filters from it. What bounds them is latency (128^3: one
// wave of CTAs, 6 per SM, marching 17 planes): the plane's shared memory is double, so a plane has one
// barrier.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
struct PhaseParams {
  int nx, ny, nz;
  long long N;
  double D, lambda, beta, kappa;
  double body[3];    // body force per unit volume (part of F^b)
  double accel[3];   // body acceleration a: F^b also holds rho(phi) a
  double rho_l, drho;  // rho(phi) = rho_l + phi drho
  const uint8_t* mask;  // solid sites (phi frozen, u = 0 there) or null
  Scales sc;
  int zchunk;
};

constexpr int kPhaseRows = 8;  // output rows per CTA of the phase-field kernels

template <class T>
struct PhaseTile {
  static constexpr int ROWS = kPhaseRows + 2;
  static constexpr int SITES = ROWS * 32;
  static constexpr T A0 = T(2) / T(3), A1 = T(1) / T(6);
  // A_x A_y f and the two first differences D_x A_y f, D_y A_x f of the staged plane at site p
  __device__ __forceinline__ static T axay(const T* f) {
    const T r0 = A0 * f[0] + A1 * (f[-1] + f[1]);
    const T rm = A0 * f[-32] + A1 * (f[-33] + f[-31]);
    const T rp = A0 * f[32] + A1 * (f[31] + f[33]);
    return A0 * r0 + A1 * (rm + rp);
  }
  __device__ __forceinline__ static T dxay(const T* f) {
    return A1 * (A0 * (f[1] - f[-1]) + A1 * ((f[-31] - f[-33]) + (f[33] - f[31])));
  }
  __device__ __forceinline__ static T dyax(const T* f) {
    return A1 * (A0 * (f[32] - f[-32]) + A1 * ((f[31] - f[-33]) + (f[33] - f[-31])));
  }
  // L_x A_y f + L_y f: the in-plane part of the Laplacian sum, zero on a constant field
  __device__ __forceinline__ static T lap_xy(const T* f) {
    const T am = A0 * f[-1] + A1 * (f[-33] + f[31]);
    const T a0 = A0 * f[0] + A1 * (f[-32] + f[32]);
    const T ap = A0 * f[1] + A1 * (f[-31] + f[33]);
    return A1 * ((am - a0) + (ap - a0)) + A1 * ((f[-32] - f[0]) + (f[32] - f[0]));
  }
};

// this thread's column of a phase-field kernel tile and its output flag
struct PhaseColumn {
  long long col;  // site index within a plane (periodically wrapped)
  bool out;
  int z0, z1;
  __device__ __forceinline__ PhaseColumn(const PhaseParams& p) {
    const int gx = int(blockIdx.x) * 30 - 1 + int(threadIdx.x);
    const int gy = int(blockIdx.y) * kPhaseRows - 1 + int(threadIdx.y);
    const int sx = ((gx % p.nx) + p.nx) % p.nx, sy = ((gy % p.ny) + p.ny) % p.ny;
    col = (long long)sy * p.nx + sx;
    out = threadIdx.y >= 1 && threadIdx.y <= kPhaseRows && threadIdx.x >= 1 && threadIdx.x <= 30 && gx < p.nx &&
          gy < p.ny;
    z0 = int(blockIdx.z) * p.zchunk;
    z1 = min(p.nz, z0 + p.zchunk);
  }
};

// phi_new from phi, u (decoded from the state) and G, all at time n:
//   phi' = phi - 3 sum_i w_i c_i . V(x + c_i) + 6 D sum_i w_i (phi(x + c_i) - phi(x)),
//   V = phi u + lambda G
// The flux and its average along z are written with their roundings (fma, mul_rn): left to the compiler, the planes
// before a chunk's first and those of its loop were contracted differently, so phi depended on where chunks begin; by
// the last bit, but the direction grad phi / |grad phi| turns that into up to 6e-5 of phi in 50 steps of a droplet.
// With walls, u is taken as 0 at solid sites and phi is not advanced there (it keeps its value),
// so a wall in contact with one bulk phase exchanges no phi.
template <class S, class T>
__global__ void __launch_bounds__(PhaseTile<T>::SITES, sizeof(T) == 4 ? 6 : 1)
    k_phase_advance(const S* st, const T* phi, const T* G, T* phi_new, PhaseParams p) {
  using PT = PhaseTile<T>;
  grid_wait();  // then plain, coherent loads (no __restrict__): the predecessor may still have been writing
  __shared__ T sm[2][5][PT::SITES];  // phi, L_z phi, A_z V_x, A_z V_y, D_z V_z of the current plane
  const PhaseColumn c(p);
  const int me = threadIdx.y * 32 + threadIdx.x;
  const long long N = p.N, plane = (long long)p.nx * p.ny;
  const T lam = T(p.lambda), dif6 = T(6) * T(p.D);
  // planes z-1, z, z+1 of this column: phi and V
  T f[3], vx[3], vy[3], vz[3];
  struct Raw {  // stored values of a plane
    T ph, ux, uy, uz, gx, gy, gz;
  };
  auto fetch = [&](int zp, Raw& r) {
    const long long s = (long long)wrap(zp, p.nz) * plane + c.col;  // zp in [-1, nz]
    r.ph = phi[s];
    if constexpr (Codec<S>::scaled) {
      r.ux = T(Codec<S>::load(st + N + s) * p.sc.dec[1]);
      r.uy = T(Codec<S>::load(st + 2 * N + s) * p.sc.dec[1]);
      r.uz = T(Codec<S>::load(st + 3 * N + s) * p.sc.dec[1]);
    } else {
      r.ux = st[N + s];
      r.uy = st[2 * N + s];
      r.uz = st[3 * N + s];
    }
    r.gx = G[s];
    r.gy = G[N + s];
    r.gz = G[2 * N + s];
    if (p.mask != nullptr && p.mask[s]) r.ux = r.uy = r.uz = T(0);
  };
  auto take = [&](int k, const Raw& r) {
    f[k] = r.ph;
    vx[k] = fma(lam, r.gx, mul_rn(r.ph, r.ux));
    vy[k] = fma(lam, r.gy, mul_rn(r.ph, r.uy));
    vz[k] = fma(lam, r.gz, mul_rn(r.ph, r.uz));
  };
  Raw r0, r1;
  fetch(c.z0 - 1, r0);
  fetch(c.z0, r1);
  take(0, r0);
  fetch(c.z0 + 1, r0);
  take(1, r1);
  for (int z = c.z0; z < c.z1; ++z) {
    take(2, r0);
    if (z + 2 <= c.z1) fetch(z + 2, r0);  // in flight during this plane
    T(*const b)[PT::SITES] = sm[(z - c.z0) & 1];
    b[0][me] = f[1];
    b[1][me] = PT::A1 * ((f[0] - f[1]) + (f[2] - f[1]));
    b[2][me] = fma(PT::A0, vx[1], mul_rn(PT::A1, vx[0] + vx[2]));
    b[3][me] = fma(PT::A0, vy[1], mul_rn(PT::A1, vy[0] + vy[2]));
    b[4][me] = PT::A1 * (vz[2] - vz[0]);
    __syncthreads();
    if (c.out) {
      const T div = PT::dxay(b[2] + me) + PT::dyax(b[3] + me) + PT::axay(b[4] + me);
      const T lap = PT::lap_xy(b[0] + me) + PT::axay(b[1] + me);
      const long long s = (long long)z * plane + c.col;
      phi_new[s] = (p.mask != nullptr && p.mask[s]) ? f[1] : f[1] - T(3) * div + dif6 * lap;
    }
    f[0] = f[1];
    f[1] = f[2];
    vx[0] = vx[1];
    vx[1] = vx[2];
    vy[0] = vy[1];
    vy[1] = vy[2];
    vz[0] = vz[1];
    vz[1] = vz[2];
  }
}

// force F = mu grad phi + F^b and compression flux G from phi (time n+1):
//   grad phi = 3 (D_x A_y A_z, D_y A_x A_z, D_z A_x A_y) phi, lap phi = 6 (A_x A_y A_z phi - phi),
//   mu = 4 beta phi (phi - 1)(phi - 1/2) - kappa lap phi,  F^b = body + rho(phi) a.
// With a density contrast grad phi is also written (gphi, else null): the fused step forms the
// pressure and viscous-gradient forces from it and the raw moments of the new state.
template <class T>
__global__ void __launch_bounds__(PhaseTile<T>::SITES, sizeof(T) == 4 ? 6 : 1)
    k_phase_forces(const T* phi, T* F, T* G, T* gphi, PhaseParams p) {
  using PT = PhaseTile<T>;
  grid_wait();  // then plain, coherent loads, as above
  __shared__ T sm[2][4][PT::SITES];  // A_z phi, D_z phi, phi, L_z phi of the current plane
  const PhaseColumn c(p);
  const int me = threadIdx.y * 32 + threadIdx.x;
  const long long N = p.N, plane = (long long)p.nx * p.ny;
  const T beta4 = T(4) * T(p.beta), kappa = T(p.kappa);
  const T b0 = T(p.body[0]), b1 = T(p.body[1]), b2 = T(p.body[2]);
  const T a0 = T(p.accel[0]), a1 = T(p.accel[1]), a2 = T(p.accel[2]);
  const T rl = T(p.rho_l), dr = T(p.drho);
  auto fetch = [&](int zp) { return phi[(long long)wrap(zp, p.nz) * plane + c.col]; };  // zp in [-1, nz]
  T f0 = fetch(c.z0 - 1), f1 = fetch(c.z0), f2, n0 = fetch(c.z0 + 1), n1 = T(0), n2 = T(0);
  if (c.z0 + 2 <= c.z1) n1 = fetch(c.z0 + 2);
  if (c.z0 + 3 <= c.z1) n2 = fetch(c.z0 + 3);
  for (int z = c.z0; z < c.z1; ++z) {
    f2 = n0;
    n0 = n1;
    n1 = n2;
    if (z + 4 <= c.z1) n2 = fetch(z + 4);
    T(*const b)[PT::SITES] = sm[(z - c.z0) & 1];
    b[0][me] = PT::A0 * f1 + PT::A1 * (f0 + f2);
    b[1][me] = PT::A1 * (f2 - f0);
    b[2][me] = f1;
    b[3][me] = PT::A1 * ((f0 - f1) + (f2 - f1));
    __syncthreads();
    if (c.out) {
      const T gx = T(3) * PT::dxay(b[0] + me), gy = T(3) * PT::dyax(b[0] + me), gz = T(3) * PT::axay(b[1] + me);
      const T lap = T(6) * (PT::lap_xy(b[2] + me) + PT::axay(b[3] + me));
      const T mu = beta4 * f1 * (f1 - T(1)) * (f1 - T(0.5)) - kappa * lap;
      const long long s = (long long)z * plane + c.col;
      const T rho = rl + f1 * dr;
      F[s] = mu * gx + (b0 + rho * a0);
      F[N + s] = mu * gy + (b1 + rho * a1);
      F[2 * N + s] = mu * gz + (b2 + rho * a2);
      if (gphi != nullptr) {
        gphi[s] = gx;
        gphi[N + s] = gy;
        gphi[2 * N + s] = gz;
      }
      // phi (1 - phi) / max(|grad phi|, 1e-12)
      const T g2 = gx * gx + gy * gy + gz * gz;
      const T cc = f1 * (T(1) - f1) * rsqrt(g2 > T(1e-24) ? g2 : T(1e-24));
      G[s] = cc * gx;
      G[N + s] = cc * gy;
      G[2 * N + s] = cc * gz;
    }
    f0 = f1;
    f1 = f2;
  }
}

// Force of the initial state with a density contrast: F += F^p + F^nu from the stored p* and
// N = A - u u (internal layout, FP32/FP64 storage), with grad rho = (rho_h - rho_l) grad phi:
//   F^p = -p* cs2 grad rho,  F^nu = -(nu omega / cs2) N . grad rho,  nu = nu(phi), omega = 1/(nu/cs2 + 1/2)
template <class S, class T>
__global__ void k_contrast_init(const S* __restrict__ st, const T* __restrict__ phi, const T* __restrict__ gphi,
                                T* __restrict__ F, long long N, double drho, double nu_l, double dnu) {
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
    const T g0 = T(drho) * gphi[s], g1 = T(drho) * gphi[N + s], g2 = T(drho) * gphi[2 * N + s];
    const T p3 = T(st[s]) * (T(1) / T(3));
    const T nxx = T(st[4 * N + s]), nyy = T(st[5 * N + s]), nzz = T(st[6 * N + s]);
    const T nxy = T(st[7 * N + s]), nxz = T(st[8 * N + s]), nyz = T(st[9 * N + s]);
    const T nu = T(nu_l) + phi[s] * T(dnu);
    const T cnu = T(-3) * nu / (T(3) * nu + T(0.5));
    F[s] += -p3 * g0 + cnu * (nxx * g0 + nxy * g1 + nxz * g2);
    F[N + s] += -p3 * g1 + cnu * (nxy * g0 + nyy * g1 + nyz * g2);
    F[2 * N + s] += -p3 * g2 + cnu * (nxz * g0 + nyz * g1 + nzz * g2);
  }
}

}  // namespace lbf
