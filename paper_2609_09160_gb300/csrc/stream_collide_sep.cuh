// Fused pull-stream-and-collide step by axis-separated partial sums.
//
// Same method as k_stream_collide (Sec. 2, Eq. (pullLLB) followed by Eq. (corr)), evaluated without
// ever forming the Q populations. The post-collision population of a site is a polynomial in the
// direction, f_c / w_c = q0 + b.c + c.e.c (D3Q27h: up to second degree per axis), and the lattice
// weights are sums of products of one-axis weights:
//   D3Q27   216 w = [1 4 1]_x [1 4 1]_y [1 4 1]_z
//   D3Q19   36 w  = c_z = 0: [1 2 1]_x [1 2 1]_y + 8 at the centre;  c_z = +-1: the cross
//                   [1 0 1]_x + [1 0 1]_y + 2 at the centre.
// So the sum over directions of one Hermite moment is three one-axis sums, and along one axis only
// two numbers of a site ever reach a neighbour: p = A + B + C, what its polynomial A + B c + C c^2
// sends to x + 1, and m = A - B + C, what it sends to x - 1. With S = p(x-1) + m(x+1) and
// D = p(x-1) - m(x+1) the one-axis moments of order 0, 1, 2 are w0 A + S, D and S.
//
// Work decomposition (GB300: 152 SMs, 228 KB shared memory per SM):
//   * a CTA owns XO x TY output columns (XO = 32 VX: VX = 2 neighbouring sites per thread, whose
//     arithmetic is the packed FP32x2 of sm_100 and later, VX = 1 in FP64) and marches along z;
//     warp w < TY + 2 holds row w; rows 0 and TY + 1, the y halo, have no outputs, and their warps
//     issue the loads and form the two x halo columns;
//   * plane s: every thread forms the 10 coefficients of its sites, the x sums come from warp
//     shuffles (the edge lanes take their outer neighbour from the x halo, which is formed one plane
//     ahead and leaves its p and m in shared memory), the y values p, m go to shared memory
//     (10 values per site on D3Q19, where the population ring holds 16 in up to three planes);
//   * after the plane's only barrier the output rows take p(y-1), m(y+1) and have the in-plane
//     moments of the plane for c_z = +1, 0, -1, which they add to the outputs of planes s+1, s, s-1
//     held in registers: plane s - 1 is complete and is corrected (Eq. corr) and stored.
// Halfway bounce-back (MASK): a solid site sends nothing, and a fluid site adds its own opposite
// population for every direction it would pull from a solid site (a bit mask per site, built once).
// Tiles without any solid site in reach run the code without it.
//
// Rows arrive by TMA, one box of 10 fields x XO columns per row, so that the periodic wrap in y and z
// costs nothing; the halo columns are loaded into registers one plane ahead. The last tile of a row
// is moved left to end at nx - 1. Rows that are not whole 16-byte units, or shorter than a tile, are
// loaded into registers one plane ahead as well.
//
// What bounds it (one GB300; us a step, steps without sums; "before" is the faster of the two population-ring kernels):
//   D3Q19 FP32 512^3 2024 -> 1895, 256^3 280 -> 248, 128^3 52 -> 37, 32^3 12.4 -> 4.5; D3Q27 FP32 512^3 2523 -> 2071,
//   256^3 354 -> 270; D3Q27h FP32 512^3 3923 -> 3283, 256^3 535 -> 425; D3Q19 FP64 32^3 75.9 -> 29.5, 256^3 7668 -> 6968.
//   By name only (16-bit storage and two components keep the ring kernels' values): D3Q19 FP16 512^3 with its sums 2043 ->
//   1448, D3Q27 FP16 2500 -> 1973, droplet 128^3 116 -> 107.
//   Thread instructions per site: D3Q19 FP32 188 (421 before), FP16 245, D3Q27 FP32 305 (600), D3Q27h 460
//   (970). FP32 moves DRAM at 5.6 TB/s of 6.7 (reads 1.03x the state); 16-bit storage and the D3Q27 lattices
//   are bound by the latency of the two halves of a plane's work with 8 to 16 warps per SM (shared-memory
//   pipe 40-66% busy, issue 45-55%; top stalls barrier and fixed latency).
// Why this split:
//   * two rows per warp (RP = 2): a row pair exchanges p and m in registers, which halves the shared-memory
//     exchange; D3Q19 FP16 84 -> 92 with 12 warps of 168 registers instead of 16 of 110. The D3Q27 lattices
//     keep 18 values per site in flight and spill or lose warps with two rows (FP16 74 -> 64).
//   * loads two to four planes ahead (STAGES): FP16 80 / 92 / 96 / 98 at 3 / 4 / 5 / 6 stages; FP32 keeps one
//     CTA per SM with 5 stages of 8 rows (72) over two of 6 rows with 4 (67).
//   * outputs leave as TMA boxes from the stage rows just read: 62.6 -> 68.6 (FP32 256^3) against per-thread
//     stores, which queue in front of the other warps' shared-memory accesses.
//   * two components (TWO, by name): the forces and phase field of the source and of the output sites are loaded as
//     pairs one plane ahead: droplet 128^3 72 -> 56 us a launch against scalar loads (83 before), layered
//     contrast flow 205 -> 175; 8 warps of 126 registers, two CTAs per SM (6 warps 118, here 115 us a step).
//   * rows 0 and TY + 1 and the halo columns on two warps of their own: the warp that carried both took
//     2100 of the 2120 cycles of a plane while the output rows took 1500.

#pragma once

#include "stream_collide.cuh"

namespace lbf {

// ---- VX neighbouring sites per thread ---------------------------------------------------------
template <class T, int VX>
struct PackOf {
  using type = T;
};
template <>
struct PackOf<float, 2> {
  using type = float2;
};
template <class V>
__device__ __forceinline__ V v_set(typename std::conditional<std::is_same<V, double>::value, double, float>::type s) {
  if constexpr (std::is_same<V, float2>::value)
    return make_float2(s, s);
  else
    return V(s);
}
__device__ __forceinline__ float2 v_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 v_mul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 v_fma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 v_sub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
// c - a b
__device__ __forceinline__ float2 v_nfma(float2 a, float2 b, float2 c) { return __ffma2_rn(make_float2(-a.x, -a.y), b, c); }
template <class T>
__device__ __forceinline__ T v_add(T a, T b) { return a + b; }
template <class T>
__device__ __forceinline__ T v_mul(T a, T b) { return a * b; }
template <class T>
__device__ __forceinline__ T v_fma(T a, T b, T c) { return fma(a, b, c); }
template <class T>
__device__ __forceinline__ T v_sub(T a, T b) { return a - b; }
template <class T>
__device__ __forceinline__ T v_nfma(T a, T b, T c) { return fma(-a, b, c); }

template <class V>
struct PairSD {
  V S, D;
};
// p(x-1) + m(x+1) and p(x-1) - m(x+1) along x; the edge lanes take their outer neighbour h from the halo
// (left, right), or, with AROUND, where a row is one tile long, by a shuffle that wraps around
template <bool AROUND>
struct Edge {
  int lane;
  bool left, right;
  __device__ __forceinline__ float from_left(float v) const {
    return AROUND ? __shfl_sync(0xffffffffu, v, (lane + 31) & 31) : __shfl_up_sync(0xffffffffu, v, 1);
  }
  __device__ __forceinline__ float from_right(float v) const {
    return AROUND ? __shfl_sync(0xffffffffu, v, (lane + 1) & 31) : __shfl_down_sync(0xffffffffu, v, 1);
  }
  __device__ __forceinline__ double from_left(double v) const {
    return AROUND ? __shfl_sync(0xffffffffu, v, (lane + 31) & 31) : __shfl_up_sync(0xffffffffu, v, 1);
  }
  __device__ __forceinline__ double from_right(double v) const {
    return AROUND ? __shfl_sync(0xffffffffu, v, (lane + 1) & 31) : __shfl_down_sync(0xffffffffu, v, 1);
  }
};
template <class E>
__device__ __forceinline__ PairSD<float2> x_sums(float2 p, float2 m, float h, const E& e) {
  float l = e.from_left(p.y), r = e.from_right(m.x);
  if (e.left) l = h;
  if (e.right) r = h;
  return {make_float2(l + m.y, p.x + r), make_float2(l - m.y, p.x - r)};
}
template <class E>
__device__ __forceinline__ PairSD<double> x_sums(double p, double m, double h, const E& e) {
  double l = e.from_left(p), r = e.from_right(m);
  if (e.left) l = h;
  if (e.right) r = h;
  return {l + r, l - r};
}

// ---- tile -------------------------------------------------------------------------------------
template <class L>
struct SepCount {
  // p (and m) values per site along x, and along y
  static constexpr int NE = L::Q == 19 ? 5 : (L::HIGH ? 9 : 7);
  static constexpr int NY = L::Q == 19 ? 5 : 9;
};

template <class L, class S, int VX, int TY, int RP>
struct SepTile {
  using T = typename ComputeOf<S>::type;
  static constexpr int XO = 32 * VX;             // output columns
  static constexpr int ROWS = TY + 2;
  static constexpr int PAIRS = TY / RP;          // warps with outputs, RP rows each
  static constexpr int WARPS = PAIRS + 2;        // and one for the y halo rows, one for loads and x halo
  static constexpr int THREADS = 32 * WARPS;
  static constexpr size_t ROWB = size_t(10) * XO * sizeof(S);  // one row of all fields
  static constexpr size_t STAGEB = ROWS * ROWB;
  static_assert(ROWB % 128 == 0, "TMA destinations start on 128-byte boundaries");
  static constexpr int NE = SepCount<L>::NE, NY = SepCount<L>::NY;
  static constexpr int NEP = (NE + 3) / 4 * 4;   // padded to 16-byte groups
  static constexpr size_t HXB = size_t(2) * 2 * ROWS * NEP * sizeof(T);
  static constexpr size_t YB = size_t(2) * 2 * NY * PAIRS * XO * sizeof(T);
  static_assert(ROWS <= (VX == 2 ? 32 : 16), "the x-halo warp holds both columns of every row");
  static_assert(TY % RP == 0 && RP <= 2, "rows per warp");
};

// bounce-back parts of the outputs, from the front half of a plane's work to the back half: in the
// row's stage where that holds 10 compute-type values per site, else in a buffer of their own
template <class S>
constexpr bool sep_cor_in_stage() {
  return sizeof(S) == sizeof(typename ComputeOf<S>::type);
}
template <class L, class S, int VX, int TY, int RP, int STAGES, bool MASK>
constexpr size_t sep_smem_bytes() {
  using G = SepTile<L, S, VX, TY, RP>;
  const size_t need = 128 + STAGES * G::STAGEB + G::HXB + G::YB +
                      (MASK && !sep_cor_in_stage<S>() ? size_t(TY) * 10 * G::XO * sizeof(typename G::T) : 0);
  return need;
}

// Tile of a kernel: TY output rows, RP of them per warp, and the CTAs per SM asked of the register
// allocator; STAGES planes of TMA stages in shared memory: the plane in use, the one before, whose rows
// hold outputs on their way out, and the others on their way in (as the decimal number STAGES TY RP MINB).
struct SepConfig {
  int stages, ty, rp, minb;
};
#ifndef LBF_SEP_CFG_Q19
#define LBF_SEP_CFG_Q19 50821
#endif
#ifndef LBF_SEP_CFG_Q19_16
#define LBF_SEP_CFG_Q19_16 60822
#endif
#ifndef LBF_SEP_CFG_Q27
#define LBF_SEP_CFG_Q27 50412
#endif
#ifndef LBF_SEP_CFG_Q27_16
#define LBF_SEP_CFG_Q27_16 50612
#endif
#ifndef LBF_SEP_CFG_Q27H
#define LBF_SEP_CFG_Q27H 50611
#endif
#ifndef LBF_SEP_CFG_Q27H_16
#define LBF_SEP_CFG_Q27H_16 50612
#endif
#ifndef LBF_SEP_CFG_F64
#define LBF_SEP_CFG_F64 40212
#endif
#ifndef LBF_SEP_CFG_SMALL
#define LBF_SEP_CFG_SMALL 40412
#endif
#ifndef LBF_SEP_CFG_TWO
#define LBF_SEP_CFG_TWO 40612
#endif
constexpr SepConfig sep_config(int Q, int bytes, bool high, bool small, bool two = false) {
  const int c = two          ? LBF_SEP_CFG_TWO
                : bytes == 8 ? LBF_SEP_CFG_F64
                : small      ? LBF_SEP_CFG_SMALL
                : Q == 19    ? (bytes == 4 ? LBF_SEP_CFG_Q19 : LBF_SEP_CFG_Q19_16)
                : high       ? (bytes == 4 ? LBF_SEP_CFG_Q27H : LBF_SEP_CFG_Q27H_16)
                             : (bytes == 4 ? LBF_SEP_CFG_Q27 : LBF_SEP_CFG_Q27_16);
  return SepConfig{c / 10000, c / 100 % 100, c / 10 % 10, c % 10};
}
constexpr int sep_vx(int bytes) { return bytes == 8 ? 1 : 2; }

// ---- stores of VX neighbouring sites ------------------------------------------------------------
template <class S, bool RN>
__device__ __forceinline__ void st_pair(S* p, float2 v, float enc, uint32_t& r0, uint32_t& r1) {
  if constexpr (std::is_same<S, float>::value) {
    *reinterpret_cast<float2*>(p) = v;
  } else {
    const float2 w = v_mul(v, make_float2(enc, enc));
    if constexpr (std::is_same<S, __half>::value) {
      if constexpr (RN) {
        *reinterpret_cast<__half2*>(p) = __floats2half2_rn(w.x, w.y);
      } else {
        r0 = lcg_next(r0);
        r1 = lcg_next(r1);
        uint32_t d;
        asm("cvt.rz.f16x2.f32 %0, %1, %2;" : "=r"(d) : "f"(__uint_as_float(__float_as_uint(w.y) + (r1 >> 19))),
            "f"(__uint_as_float(__float_as_uint(w.x) + (r0 >> 19))));
        *reinterpret_cast<uint32_t*>(p) = d;
      }
    } else {
      if constexpr (RN) {
        *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(w.x, w.y);
      } else {
        r0 = lcg_next(r0);
        r1 = lcg_next(r1);
        const uint32_t lo = __float_as_uint(w.x) + (r0 >> 16), hi = __float_as_uint(w.y) + (r1 >> 16);
        *reinterpret_cast<uint32_t*>(p) = __byte_perm(lo, hi, 0x7632);
      }
    }
  }
}

// VX neighbouring stored values as compute-type values, undecoded
template <class S>
__device__ __forceinline__ float2 ld_pair(const S* p) {
  if constexpr (std::is_same<S, float>::value)
    return *reinterpret_cast<const float2*>(p);
  else if constexpr (std::is_same<S, __half>::value)
    return __half22float2(*reinterpret_cast<const __half2*>(p));
  else
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
}

// ---- coefficients -------------------------------------------------------------------------------
// f_c / w_c = q0 + b.c + exx cx^2 + ... + exy cx cy + ... from the moments, F = 2 rho h the force (rho = 1)
// and k1 = 1 - omega (times the decode factor of N; F / rho in the place of F with two components): with
// P2 = u u + k1 N + u h + h u,
//   q0 = p* - (3/2) tr P2, b = 3 (u + h), e_aa = (9/2) P2_aa, e_ab = 9 P2_ab.
// Every constant is exact in FP32: p* and u pass through a step with a factor of one, and a factor 1/3
// rounded here would grow by 3e-8 a step.
template <class V>
struct SepCoef {
  V q0, bx, by, bz, exx, eyy, ezz, exy, exz, eyz;
};
template <class T, class V>
__device__ __forceinline__ SepCoef<V> sep_coef(const V (&m)[10], const V (&F)[3], V k1) {
  const V k9 = v_mul(k1, v_set<V>(T(9))), three = v_set<V>(T(3)), nine = v_set<V>(T(9));
  const V f15 = v_set<V>(T(1.5)), f45 = v_set<V>(T(4.5));
  const V ux = m[1], uy = m[2], uz = m[3];
  const V gx = v_mul(F[0], f45), gy = v_mul(F[1], f45), gz = v_mul(F[2], f45);  // 9 h
  SepCoef<V> c;
  const V pxx = v_fma(ux, v_add(ux, F[0]), v_mul(k1, m[4]));
  const V pyy = v_fma(uy, v_add(uy, F[1]), v_mul(k1, m[5]));
  const V pzz = v_fma(uz, v_add(uz, F[2]), v_mul(k1, m[6]));
  c.q0 = v_fma(v_add(v_add(pxx, pyy), pzz), v_set<V>(T(-1.5)), m[0]);
  c.exx = v_mul(pxx, f45);
  c.eyy = v_mul(pyy, f45);
  c.ezz = v_mul(pzz, f45);
  const V ty = v_fma(uy, nine, gy), tz = v_fma(uz, nine, gz);  // 9 (u + h)
  c.exy = v_fma(ux, ty, v_fma(uy, gx, v_mul(k9, m[7])));
  c.exz = v_fma(ux, tz, v_fma(uz, gx, v_mul(k9, m[8])));
  c.eyz = v_fma(uy, tz, v_fma(uz, gy, v_mul(k9, m[9])));
  c.bx = v_fma(ux, three, v_mul(F[0], f15));
  c.by = v_fma(uy, three, v_mul(F[1], f15));
  c.bz = v_fma(uz, three, v_mul(F[2], f15));
  return c;
}

// D3Q27h: f_c / w_c = p* + phi_x phi_y phi_z - 1 + (Guo and closure terms), phi_a(c) = 1 + 3 c u_a +
// 4.5 (c^2 - 1/3) u_a^2 (see full_populations). As a polynomial in (cx, cy) with coefficients (i, j),
// i, j <= 2, at fixed c_z:  f = p* - 1 + A_ij zA(c_z) + B_ij zB(c_z) + C_ij zC(c_z) with
//   zA = phi_z + h_z phi_z' + keep Nzz phi_z''/2,  zB = phi_z,  zC = phi_z',
//   A = phi_x phi_y,  B = (h_x phi_x' + keep Nxx phi_x''/2) phi_y + phi_x (same in y) + keep Nxy phi_x' phi_y',
//   C = keep (Nxz phi_x' phi_y + Nyz phi_x phi_y').
// A_00 and zA are 1 + small: the small parts a00, za keep the constant term free of cancellation,
// A_00 zA - 1 = a00 + (1 + a00) za.
template <class V>
struct SepFull {
  V p, A[9], a00, B[9], C[9];
  V za[3], zb[3], zc[3];  // c_z = +1, -1, 0: zA - 1, zB, zC
};
template <class T, class V>
__device__ __forceinline__ void sep_full(const V (&m)[10], const V (&F)[3], T keep, SepFull<V>& r) {
  const V kk = v_set<V>(keep), half = v_set<V>(T(0.5)), three = v_set<V>(T(3));
  V ph[2][3], dl[2][3], s[2][3];  // x, y: phi, phi', and h phi' + keep N phi''/2 by powers of c
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const V u = m[1 + a], h = v_mul(F[a], half), n = v_mul(kk, m[4 + a]);
    const V u2 = v_mul(u, u);
    ph[a][1] = v_mul(u, three);
    ph[a][2] = v_mul(u2, v_set<V>(T(4.5)));
    dl[a][0] = v_mul(u, v_set<V>(T(-3)));
    dl[a][1] = three;
    dl[a][2] = v_mul(u, v_set<V>(T(9)));
    s[a][0] = v_fma(n, v_set<V>(T(-1.5)), v_mul(h, dl[a][0]));
    s[a][1] = v_mul(h, three);
    s[a][2] = v_fma(n, v_set<V>(T(4.5)), v_mul(h, dl[a][2]));
    ph[a][0] = v_mul(u2, v_set<V>(T(-1.5)));  // phi_0 - 1 for now
  }
  r.p = m[0];
  r.a00 = v_fma(ph[0][0], ph[1][0], v_add(ph[0][0], ph[1][0]));
  ph[0][0] = v_add(ph[0][0], v_set<V>(T(1)));
  ph[1][0] = v_add(ph[1][0], v_set<V>(T(1)));
  const V nxy = v_mul(kk, m[7]), nxz = v_mul(kk, m[8]), nyz = v_mul(kk, m[9]);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const V dxy = v_mul(nxy, dl[0][i]), dxz = v_mul(nxz, dl[0][i]), pyz = v_mul(nyz, ph[0][i]);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      r.A[3 * i + j] = v_mul(ph[0][i], ph[1][j]);
      r.B[3 * i + j] = v_fma(s[0][i], ph[1][j], v_fma(ph[0][i], s[1][j], v_mul(dxy, dl[1][j])));
      r.C[3 * i + j] = v_fma(dxz, ph[1][j], v_mul(pyz, dl[1][j]));
    }
  }
  const V uz = m[3], hz = v_mul(F[2], half), nz = v_mul(kk, m[6]);
  const V u2 = v_mul(uz, uz);
  const V e = v_mul(u2, three), l = v_mul(uz, three), six = v_mul(uz, v_set<V>(T(6)));
  const V ps[3] = {v_add(e, l), v_sub(e, l), v_mul(u2, v_set<V>(T(-1.5)))};
  r.zc[0] = v_add(six, three);
  r.zc[1] = v_sub(six, three);
  r.zc[2] = v_mul(uz, v_set<V>(T(-3)));
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    r.za[k] = v_fma(nz, v_set<V>(k == 2 ? T(-1.5) : T(3)), v_fma(hz, r.zc[k], ps[k]));
    r.zb[k] = v_add(ps[k], v_set<V>(T(1)));
  }
}

// ---- the kernel -----------------------------------------------------------------------------------
// barrier of the whole CTA from different places of the code (the roles have loops of their own)
template <int THREADS>
__device__ __forceinline__ void cta_barrier() {
  asm volatile("barrier.cta.sync 1, %0;" ::"n"(THREADS) : "memory");
}

template <class L, class S, bool SMALL, bool TMA, bool MASK, bool FF, bool RN, int TWO = 0>
__global__ void __launch_bounds__(32 * (sep_config(L::Q, int(sizeof(S)), L::HIGH, SMALL, TWO != 0).ty /
                                            sep_config(L::Q, int(sizeof(S)), L::HIGH, SMALL, TWO != 0).rp + 2),
                                  sep_config(L::Q, int(sizeof(S)), L::HIGH, SMALL, TWO != 0).minb)
    k_stream_collide_sep(const FwdParams a, const __grid_constant__ CUtensorMap trow,
                         const __grid_constant__ CUtensorMap ttile, const __grid_constant__ CUtensorMap tout) {
  constexpr SepConfig CFG = sep_config(L::Q, int(sizeof(S)), L::HIGH, SMALL, TWO != 0);
  constexpr int VX = sep_vx(int(sizeof(S))), TY = CFG.ty, RP = CFG.rp, STAGES = CFG.stages;
  using G = SepTile<L, S, VX, TY, RP>;
  using T = typename ComputeOf<S>::type;
  using V = typename PackOf<T, VX>::type;
  constexpr int XO = G::XO, ROWS = G::ROWS, PAIRS = G::PAIRS, NE = G::NE, NEP = G::NEP, NY = G::NY;
  constexpr bool Q19 = L::Q == 19;

  extern __shared__ __align__(128) unsigned char smem_raw[];
  unsigned char* sbase = smem_raw + ((128u - (smem_u32(smem_raw) & 127u)) & 127u);
  unsigned char* stage0 = sbase;                                       // STAGES x STAGEB
  T* hx = reinterpret_cast<T*>(sbase + STAGES * G::STAGEB);            // [2 planes][2 sides][ROWS][NEP]
  T* yv = hx + G::HXB / sizeof(T);                                     // [2 planes][p, m][NY][PAIRS][XO]
  T* corb = yv + G::YB / sizeof(T);                                    // [TY][10][XO] (MASK, where needed)
  __shared__ __align__(8) uint64_t bars[STAGES];
  __shared__ volatile int gave_up[2];
  // with two rows a thread adds up to 192 pairs in a chunk: in FP32 its sums go to FP64 every 32 planes, after at
  // most 64 additions (a uniform flow's sums over 96 planes: 8e-7 off instead of 2.3e-6). With one row the chunks
  // are of at most 64 planes
  constexpr bool PARTS = RP == 2 && std::is_same<T, float>::value;
  __shared__ double parts[PARTS ? G::WARPS * 6 : 1];  // a warp's sums so far

  // an overlapped launch is alive while its predecessor writes: everything but the wall tables is read by plain,
  // coherent loads (no __restrict__, no __ldg), which stay behind grid_wait()
  const S* src = static_cast<const S*>(a.src);
  S* dst = static_cast<S*>(a.dst);
  const T* ffield = static_cast<const T*>(a.force_field);

  const int lane = threadIdx.x, warp = __shfl_sync(0xffffffffu, int(threadIdx.y), 0);  // warp-uniform
  const int nx = a.nx, ny = a.ny;
  const long long N = a.N, plane = (long long)nx * ny;
  const int xb = blockIdx.x * XO;
  const int x0 = TMA ? min(xb, nx - XO) : xb;
  // output rows of this launch: yrows rows from a.y_begin, taken mod ny (y0 may exceed ny)
  const int yrows = a.y_rows > 0 ? a.y_rows : ny, ybl = blockIdx.y * TY, y0 = (a.y_begin + ybl) % ny;
  const int z0 = blockIdx.z * a.zchunk;
  const int z1 = min(a.nz, z0 + a.zchunk);
  const int planes = z1 - z0 + 2;  // z0 - 1 .. z1, numbered 0 .. planes - 1
  // rows of one tile (the tile's other edge is its x halo): the shuffles wrap around and nobody forms halo
  // columns. Where lattices that small run: the short tile, and FP64 (32^3 FP64 33.1 -> 29.3 us a step); the
  // indexed shuffles cost the large FP32 tile 2-3%
  constexpr bool AROUND = SMALL || VX == 1;
  const bool one_tile = AROUND && nx == XO;
  const Edge<AROUND> edge = {lane, lane == 0 && !one_tile, lane == 31 && !one_tile};
  const bool dirty = MASK && a.tile_dirty[((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] != 0;

  T keep = T(1) - pick<T>(a.omega, a.omega_f);
  if constexpr (Codec<S>::scaled) keep *= a.sc.dec[2];  // N is used in storage units
  const T Fu0 = pick<T>(a.force[0], a.force_f[0]), Fu1 = pick<T>(a.force[1], a.force_f[1]),
          Fu2 = pick<T>(a.force[2], a.force_f[2]);
  const V zero = v_set<V>(T(0));

  auto pack = [](T v0, T v1) -> V {
    if constexpr (VX == 2)
      return make_float2(v0, v1);
    else
      return v0;
  };
  auto row_of = [&](int r) {  // lattice row of ring row r
    const int gy = y0 - 1 + r;
    return ((gy % ny) + ny) % ny;
  };
  auto stage_row = [&](int ip, int r) { return stage0 + (ip % STAGES) * G::STAGEB + r * G::ROWB; };
  // halo columns: side 0 = left (p), 1 = right (m), written one plane ahead, read by the edge lanes
  auto hx_at = [&](int ip, int side, int r) { return hx + ((ip & 1) * 2 + side) * ROWS * NEP + r * NEP; };

  constexpr bool AHEAD = FF || MASK || TWO != 0;  // the rows too load something into registers one plane ahead

  // ---- what a thread reads of one plane, for its row's sites or for the halo columns --------------
  struct Site {
    int row;        // ring row
    int o0, o1;     // offsets of the two sites within a plane
    bool needed;    // the row is read by some output
  };
  // what is loaded into registers one plane ahead besides the x-halo values: per-site force, wall links
  constexpr bool SITEF = FF || TWO != 0;  // a force of its own at every site
  static_assert(TWO == 0 || (!FF && std::is_same<S, T>::value && !L::HIGH), "two components: FP32 or FP64 storage, no force field");
  struct Extra {
    T f0[SITEF ? 3 : 1], f1[SITEF ? 3 : 1];
    T p0, p1;  // two components: phi^n
    uint32_t l0, l1;
  };
  auto fetch_values = [&](const Site& t, int ip, S (&v0)[10], S (&v1)[10]) {
    if (!t.needed) return;
    const S* b = src + (long long)wrap(z0 - 1 + ip, a.nz) * plane;
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      v0[k] = b[k * N + t.o0];
      if constexpr (VX == 2) v1[k] = b[k * N + t.o1];
    }
  };
  auto fetch_extra = [&](const Site& t, int ip, Extra& r) {
    if (!t.needed) return;
    const long long zoff = (long long)wrap(z0 - 1 + ip, a.nz) * plane;
    if constexpr (FF) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        r.f0[k] = ffield[k * N + zoff + t.o0];
        if constexpr (VX == 2) r.f1[k] = ffield[k * N + zoff + t.o1];
      }
    }
    if constexpr (TWO != 0) {
      const T* Fo = static_cast<const T*>(a.F_old) + zoff;
      const T* po = static_cast<const T*>(a.phi_old) + zoff;
      // the library's own arrays: 8-byte aligned pairs where the rows hold whole 16-byte units (TMA)
      if (TMA && VX == 2 && t.o1 == t.o0 + 1) {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const float2 q = *reinterpret_cast<const float2*>(Fo + k * N + t.o0);
          r.f0[k] = q.x, r.f1[k] = q.y;
        }
        const float2 q = *reinterpret_cast<const float2*>(po + t.o0);
        r.p0 = q.x, r.p1 = q.y;
      } else {
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          r.f0[k] = Fo[k * N + t.o0];
          if constexpr (VX == 2) r.f1[k] = Fo[k * N + t.o1];
        }
        r.p0 = po[t.o0];
        if constexpr (VX == 2) r.p1 = po[t.o1];
      }
    }
    if constexpr (MASK) {
      if (dirty) {
        r.l0 = __ldg(a.links + zoff + t.o0);
        if constexpr (VX == 2) r.l1 = __ldg(a.links + zoff + t.o1);
      }
    }
  };
  auto decode = [&](V (&m)[10]) {
    if constexpr (Codec<S>::scaled) {
      m[0] = v_mul(m[0], v_set<V>(a.sc.dec[0]));
#pragma unroll
      for (int k = 1; k < 4; ++k) m[k] = v_mul(m[k], v_set<V>(a.sc.dec[1]));
    }
  };
  auto take = [&](const Site& t, const S (&v0)[10], const S (&v1)[10], V (&m)[10]) {
#pragma unroll
    for (int k = 0; k < 10; ++k)
      m[k] = t.needed ? pack(static_cast<T>(v0[k]), VX == 2 ? static_cast<T>(v1[k]) : T(0)) : zero;
  };
  // two components: rho(phi) = rho_l + phi drho, nu(phi) = nu_l + phi dnu, 1 - omega = 1 - 1 / (3 nu + 1/2)
  const T rho_l = pick<T>(a.rho_l, a.rho_l_f), drho = pick<T>(a.rho_h - a.rho_l, a.drho_f);
  const T nu_l = pick<T>(a.nu_l, a.nu_l_f), dnu = pick<T>(a.nu_h - a.nu_l, a.dnu_f);
  const T rrho_l = TWO != 0 ? T(1) / rho_l : T(1), keep_l = TWO != 0 ? T(1) - T(1) / (T(3) * nu_l + T(0.5)) : T(0);
  auto each = [&](V v, auto f) -> V {
    if constexpr (VX == 2)
      return make_float2(f(v.x), f(v.y));
    else
      return f(v);
  };
  auto rrho_of = [&](V phi) -> V {  // 1 / rho
    if constexpr (TWO == 2)
      return each(phi, [&](T p) { return T(1) / (rho_l + p * drho); });
    else
      return v_set<V>(rrho_l);
  };
  auto keep_of = [&](const Extra& r) -> V {
    if constexpr (TWO != 0) {
      if (dnu == T(0)) return v_set<V>(keep_l);
      return each(pack(r.p0, VX == 2 ? r.p1 : T(0)), [&](T p) { return T(1) - T(1) / (T(3) * (nu_l + p * dnu) + T(0.5)); });
    } else {
      return v_set<V>(keep);
    }
  };
  // the force at the sites (two components: F / rho, as it enters the collision)
  auto force_of = [&](const Extra& r, V (&F)[3]) {
    if constexpr (TWO != 0) {
      const V rr = rrho_of(pack(r.p0, VX == 2 ? r.p1 : T(0)));
#pragma unroll
      for (int k = 0; k < 3; ++k) F[k] = v_mul(pack(r.f0[k], VX == 2 ? r.f1[k] : T(0)), rr);
    } else if constexpr (FF) {
      F[0] = pack(Fu0 + r.f0[0], VX == 2 ? Fu0 + r.f1[0] : T(0));
      F[1] = pack(Fu1 + r.f0[1], VX == 2 ? Fu1 + r.f1[1] : T(0));
      F[2] = pack(Fu2 + r.f0[2], VX == 2 ? Fu2 + r.f1[2] : T(0));
    } else {
      F[0] = v_set<V>(Fu0), F[1] = v_set<V>(Fu1), F[2] = v_set<V>(Fu2);
    }
  };
  auto silence = [&](SepCoef<V>& c, const Extra& r) {  // solid sites send nothing
    if constexpr (MASK) {
      const bool s0 = (r.l0 >> 31) != 0u, s1 = VX == 2 && (r.l1 >> 31) != 0u;
      if (dirty && __any_sync(0xffffffffu, s0 || s1)) {
        V* f = &c.q0;
#pragma unroll
        for (int k = 0; k < 10; ++k) {
          if constexpr (VX == 2) {
            f[k].x = s0 ? 0.0f : f[k].x;
            f[k].y = s1 ? 0.0f : f[k].y;
          } else {
            f[k] = s0 ? T(0) : f[k];
          }
        }
      }
    }
  };
  // f[3 i + j]: coefficient of cx^i cy^j of the full-basis polynomial at c_z = +1, -1, 0 (k)
  auto full_at = [&](const SepFull<V>& c, int k, V (&f)[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      const V bc = v_fma(c.B[i], c.zb[k], v_mul(c.C[i], c.zc[k]));
      if (i == 0)
        f[i] = v_add(v_add(v_fma(c.A[0], c.za[k], c.a00), c.p), bc);
      else
        f[i] = v_fma(c.A[i], c.za[k], v_add(c.A[i], bc));
    }
  };

  // ---- x-halo columns of plane ip ------------------------------------------------------------------
  auto halo_columns = [&](const Site& t, bool live, int ip, const S (&v0)[10], const S (&v1)[10], const Extra& r) {
    V m[10];
    take(t, v0, v1, m);
    decode(m);
    V F[3];
    force_of(r, F);
    V P[NE], M[NE];
    if constexpr (!L::HIGH) {
      SepCoef<V> c = sep_coef<T, V>(m, F, keep_of(r));
      silence(c, r);
      const V az = v_add(c.q0, c.ezz);
      const V tp = v_add(v_add(az, c.bz), c.exx), tm = v_add(v_sub(az, c.bz), c.exx), t0 = v_add(c.q0, c.exx);
      const V xp = v_add(c.bx, c.exz), xm = v_sub(c.bx, c.exz);
      auto set = [&](int e, V A, V B) { P[e] = v_add(A, B), M[e] = v_sub(A, B); };
      if constexpr (Q19) {
        set(0, tp, xp);
        set(1, tm, xm);
        set(2, t0, c.bx);
        set(3, c.by, c.exy);
        P[4] = M[4] = c.eyy;
      } else {
        set(0, tp, xp);
        set(1, v_add(c.by, c.eyz), c.exy);
        set(2, tm, xm);
        set(3, v_sub(c.by, c.eyz), c.exy);
        set(4, t0, c.bx);
        set(5, c.by, c.exy);
        P[6] = M[6] = c.eyy;
      }
    } else {
      SepFull<V> c;
      sep_full<T, V>(m, F, keep, c);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        V f[9];
        full_at(c, k, f);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const V q = v_add(f[j], f[6 + j]);
          P[3 * k + j] = v_add(q, f[3 + j]);
          M[3 * k + j] = v_sub(q, f[3 + j]);
        }
      }
    }
    if (live) {
      if constexpr (VX == 2) {
        T *l = hx_at(ip, 0, t.row), *q = hx_at(ip, 1, t.row);
#pragma unroll
        for (int e = 0; e < NE; ++e) l[e] = P[e].x, q[e] = M[e].y;
      } else {
        T* l = hx_at(ip, lane < 16 ? 0 : 1, t.row);
#pragma unroll
        for (int e = 0; e < NE; ++e) l[e] = lane < 16 ? P[e] : M[e];
      }
    }
  };

  // ---- a row's sites of plane ip: x sums, p and m along y, and the in-plane parts of its own ------
  struct RowIn {
    Site t;
    Extra e;
  };
  auto row_in = [&](int row) {
    RowIn r;
    const int gx = x0 + VX * lane;
    r.t.row = row;
    r.t.o0 = row_of(row) * nx + (TMA ? gx : gx % nx);
    r.t.o1 = TMA ? r.t.o0 + 1 : row_of(row) * nx + (gx + 1) % nx;
    r.t.needed = ybl - 1 + row <= yrows;
    r.e.l0 = r.e.l1 = 0u;
    return r;
  };
  auto fetch = [&](RowIn& r, int ip) {
    if constexpr (AHEAD) fetch_extra(r.t, ip, r.e);
  };
  // without TMA: every thread copies its own sites into the stage (cp.async, 4 or 8 bytes each) as many
  // planes ahead as TMA would, and waits for its own copies only
  auto copy_row = [&](const RowIn& r, int ip) {
    if constexpr (!TMA) {
      if (ip < planes && r.t.needed) {
        const S* b = src + (long long)wrap(z0 - 1 + ip, a.nz) * plane;
        const uint32_t d = smem_u32(stage_row(ip, r.t.row)) + uint32_t(VX * lane * int(sizeof(S)));
        auto cp = [](uint32_t to, const void* from, auto bytes) {
          asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(to), "l"(from), "n"(decltype(bytes)::value) : "memory");
        };
#pragma unroll
        for (int k = 0; k < 10; ++k) {
          const S* f = b + k * N;
          const uint32_t t = d + uint32_t(k * XO * int(sizeof(S)));
          if constexpr (sizeof(S) == 8) {
            cp(t, f + r.t.o0, std::integral_constant<int, 8>{});
          } else if constexpr (sizeof(S) == 4) {
            cp(t, f + r.t.o0, std::integral_constant<int, 4>{});
            cp(t + 4, f + r.t.o1, std::integral_constant<int, 4>{});
          } else {
            cp(t, f + r.t.o0, std::integral_constant<int, 4>{});  // nx is even: o1 = o0 + 1, o0 even
          }
        }
      }
    }
  };
  auto copies_done = [&]() {  // one group per plane: the next plane's copies have landed
    if constexpr (!TMA) asm volatile("cp.async.wait_group %0;" ::"n"(STAGES - 2) : "memory");
  };
  auto copies_group = [&]() {
    if constexpr (!TMA) asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto cor_at = [&](int ip, int row) {  // this thread's 10 values, XO apart
    T* b = sep_cor_in_stage<S>() ? reinterpret_cast<T*>(stage_row(ip, row)) : corb + (row - 1) * 10 * XO;
    return reinterpret_cast<V*>(b + VX * lane);
  };
  // outputs: this row has some (its walls then count)
  auto row_front = [&](const RowIn& in, int ip, bool outputs, V (&F)[3], V (&yp)[NY], V (&ym)[NY], V (&own)[9]) {
    const int row = in.t.row;
    V m[10];
    const S* const q = reinterpret_cast<const S*>(stage_row(ip, row)) + VX * lane;
    LBF_CHECK(a.flags, VX * lane + VX <= XO && row < ROWS);
#pragma unroll
    for (int k = 0; k < 10; ++k) {
      if constexpr (VX == 2)
        m[k] = ld_pair<S>(q + k * XO);
      else
        m[k] = q[k * XO];
    }
    decode(m);
    force_of(in.e, F);
    T he[NEP];  // the outer neighbours of the edge lanes
    {
      const T* h = hx_at(ip, lane < 16 ? 0 : 1, row);
      if constexpr (std::is_same<T, float>::value) {
#pragma unroll
        for (int e = 0; e < NEP; e += 4) {
          const float4 q = *reinterpret_cast<const float4*>(h + e);
          he[e] = q.x, he[e + 1] = q.y, he[e + 2] = q.z, he[e + 3] = q.w;
        }
      } else {
#pragma unroll
        for (int e = 0; e < NE; ++e) he[e] = h[e];
      }
    }
    // p, m of the polynomial A + B c + C c^2 along y
    auto put_y = [&](int e, V A, V B, V C) {
      const V t = v_add(A, C);
      yp[e] = v_add(t, B);
      ym[e] = v_sub(t, B);
    };
    const V two = v_set<V>(T(2)), four = v_set<V>(T(4));
    if constexpr (!L::HIGH) {
      SepCoef<V> c = sep_coef<T, V>(m, F, keep_of(in.e));
      silence(c, in.e);
      if constexpr (MASK) {
        if (dirty && outputs) {
          V cor[10];
#pragma unroll
          for (int k = 0; k < 10; ++k) cor[k] = zero;
          const uint32_t l0 = in.e.l0, l1 = in.e.l1;
          if (__any_sync(0xffffffffu, ((l0 | l1) & 0x7fffffffu) != 0u)) {
            // bit q: x - c_q is solid, so f_q(x) is the site's own f_opp(q)
            static_for<L::Q>([&](auto qc) {
              constexpr int q = decltype(qc)::value, o = L::opp(q);
              if constexpr (q < o) {
                constexpr int cx = L::cx(q), cy = L::cy(q), cz = L::cz(q);
                V s = c.q0, d = zero;
                if constexpr (cx != 0) s = v_add(s, c.exx), d = cx > 0 ? v_add(d, c.bx) : v_sub(d, c.bx);
                if constexpr (cy != 0) s = v_add(s, c.eyy), d = cy > 0 ? v_add(d, c.by) : v_sub(d, c.by);
                if constexpr (cz != 0) s = v_add(s, c.ezz), d = cz > 0 ? v_add(d, c.bz) : v_sub(d, c.bz);
                if constexpr (cx * cy != 0) s = cx * cy > 0 ? v_add(s, c.exy) : v_sub(s, c.exy);
                if constexpr (cx * cz != 0) s = cx * cz > 0 ? v_add(s, c.exz) : v_sub(s, c.exz);
                if constexpr (cy * cz != 0) s = cy * cz > 0 ? v_add(s, c.eyz) : v_sub(s, c.eyz);
                const V fq = v_add(s, d), fo = v_sub(s, d);
                V gq, go;  // what the site gets back along q and along o
                if constexpr (VX == 2) {
                  gq = make_float2((l0 >> q) & 1u ? fo.x : 0.0f, (l1 >> q) & 1u ? fo.y : 0.0f);
                  go = make_float2((l0 >> o) & 1u ? fq.x : 0.0f, (l1 >> o) & 1u ? fq.y : 0.0f);
                } else {
                  gq = (l0 >> q) & 1u ? fo : T(0);
                  go = (l0 >> o) & 1u ? fq : T(0);
                }
                // weight in the units of the sums: D3Q19 2, 1; D3Q27 16, 4, 1
                constexpr int n = cx * cx + cy * cy + cz * cz;
                constexpr T w = T(Q19 ? (n == 1 ? 2 : 1) : (n == 1 ? 16 : (n == 2 ? 4 : 1)));
                const V es = v_mul(v_add(gq, go), v_set<V>(w)), ed = v_mul(v_sub(gq, go), v_set<V>(w));
                auto add = [&](int k, int sign, V v) {
                  if (sign > 0) cor[k] = v_add(cor[k], v);
                  if (sign < 0) cor[k] = v_sub(cor[k], v);
                };
                add(0, 1, es);
                add(1, cx, ed);
                add(2, cy, ed);
                add(3, cz, ed);
                add(4, cx * cx, es);
                add(5, cy * cy, es);
                add(6, cz * cz, es);
                add(7, cx * cy, es);
                add(8, cx * cz, es);
                add(9, cy * cz, es);
              }
            });
          }
          V* const b = cor_at(ip, row);
#pragma unroll
          for (int k = 0; k < 10; ++k) b[k * 32] = cor[k];
          if constexpr (TMA) fence_proxy_async_smem();  // the stage is refilled by TMA later
        }
      }
      const V az = v_add(c.q0, c.ezz);
      const V ap = v_add(az, c.bz), am = v_sub(az, c.bz);
      const V xp = v_add(c.bx, c.exz), xm = v_sub(c.bx, c.exz);
      const V wp = v_add(c.by, c.eyz), wm = v_sub(c.by, c.eyz);
      const V tp = v_add(ap, c.exx), tm = v_add(am, c.exx), t0 = v_add(c.q0, c.exx);
      if constexpr (Q19) {
        const PairSD<V> P = x_sums(v_add(tp, xp), v_sub(tp, xp), he[0], edge);
        put_y(0, ap, wp, c.eyy);
        own[0] = v_fma(ap, two, P.S);
        own[1] = P.D;
        own[2] = P.S;
        const PairSD<V> M = x_sums(v_add(tm, xm), v_sub(tm, xm), he[1], edge);
        put_y(1, am, wm, c.eyy);
        own[3] = v_fma(am, two, M.S);
        own[4] = M.D;
        own[5] = M.S;
        const PairSD<V> Z0 = x_sums(v_add(t0, c.bx), v_sub(t0, c.bx), he[2], edge);
        const PairSD<V> Z1 = x_sums(v_add(c.by, c.exy), v_sub(c.by, c.exy), he[3], edge);
        const PairSD<V> Z2 = x_sums(c.eyy, c.eyy, he[4], edge);
        const V X0 = v_fma(c.q0, two, Z0.S), X1 = v_fma(c.by, two, Z1.S), X2 = v_fma(c.eyy, two, Z2.S);
        put_y(2, X0, X1, X2);
        put_y(3, Z0.D, Z1.D, Z2.D);
        put_y(4, Z0.S, Z1.S, Z2.S);
        own[6] = v_fma(X0, two, v_mul(c.q0, v_set<V>(T(8))));
        own[7] = v_mul(Z0.D, two);
        own[8] = v_mul(Z0.S, two);
      } else {
        const PairSD<V> Q2 = x_sums(c.eyy, c.eyy, he[6], edge);
        const V X2 = v_fma(c.eyy, four, Q2.S);
        auto part = [&](int k, V A, V B, V Y, V t) {  // constant, cx and cy coefficients, A + exx
          const PairSD<V> Q0 = x_sums(v_add(t, B), v_sub(t, B), he[2 * k], edge);
          const PairSD<V> Q1 = x_sums(v_add(Y, c.exy), v_sub(Y, c.exy), he[2 * k + 1], edge);
          const V X0 = v_fma(A, four, Q0.S), X1 = v_fma(Y, four, Q1.S);
          put_y(3 * k, X0, X1, X2);
          put_y(3 * k + 1, Q0.D, Q1.D, Q2.D);
          put_y(3 * k + 2, Q0.S, Q1.S, Q2.S);
          own[3 * k] = v_mul(X0, four);
          own[3 * k + 1] = v_mul(Q0.D, four);
          own[3 * k + 2] = v_mul(Q0.S, four);
        };
        part(0, ap, xp, wp, tp);
        part(1, am, xm, wm, tm);
        part(2, c.q0, c.bx, c.by, t0);
      }
    } else {
      SepFull<V> c;
      sep_full<T, V>(m, F, keep, c);
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        V f[9], X[3];
        full_at(c, k, f);
        PairSD<V> q[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const V t = v_add(f[j], f[6 + j]);
          q[j] = x_sums(v_add(t, f[3 + j]), v_sub(t, f[3 + j]), he[3 * k + j], edge);
          X[j] = v_fma(f[j], four, q[j].S);
        }
        put_y(3 * k, X[0], X[1], X[2]);
        put_y(3 * k + 1, q[0].D, q[1].D, q[2].D);
        put_y(3 * k + 2, q[0].S, q[1].S, q[2].S);
        own[3 * k] = v_mul(X[0], four);
        own[3 * k + 1] = v_mul(q[0].D, four);
        own[3 * k + 2] = v_mul(q[0].S, four);
      }
    }
  };
  // exchanged value e of output warp w: slot [0][e][w] is the p of the row below its rows, [1][e][w] the
  // m of the row above them
  T* const yme = yv + VX * lane;
  auto y_at = [&](int ip, int pm, int e, int w) {
    LBF_CHECK(a.flags, w >= 0 && w < PAIRS);
    return reinterpret_cast<V*>(yme + (((ip & 1) * 2 + pm) * NY + e) * (PAIRS * XO) + w * XO);
  };

  T red[6] = {T(0), T(0), T(0), T(0), T(0), T(0)};
  if (PARTS && lane < 6) parts[warp * 6 + lane] = 0.0;
  __syncwarp();
  auto warp_sum = [](T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return static_cast<double>(v);
  };
  grid_wait();  // nothing above touches what an earlier kernel writes
  if (warp == PAIRS) {
    // ---- the y halo rows: p of the one below the tile, m of the one above it ------------------------
    RowIn in[2] = {row_in(0), row_in(ROWS - 1)};
    if constexpr (AHEAD) fetch(in[0], 0), fetch(in[1], 0);
    for (int p = 0; p < STAGES - 1; ++p) {
      copy_row(in[0], p), copy_row(in[1], p);
      copies_group();
    }
    cta_barrier<G::THREADS>();
    for (int it = 0; it < planes && !gave_up[(it - 1) & 1]; ++it) {
      copies_done();
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        V F[3], P[NY], M[NY], own[9];
        row_front(in[r], it, false, F, P, M, own);
#pragma unroll
        for (int e = 0; e < NY; ++e) *y_at(it, r, e, r == 0 ? 0 : PAIRS - 1) = r == 0 ? P[e] : M[e];
      }
      if constexpr (AHEAD) {
        if (it + 1 < planes) fetch(in[0], it + 1), fetch(in[1], it + 1);
      }
      // into the stage of plane it - 1, which this thread has read (its outputs never go there)
      copy_row(in[0], it - 1 + STAGES), copy_row(in[1], it - 1 + STAGES);
      copies_group();
      cta_barrier<G::THREADS>();
    }
  } else if (warp == PAIRS + 1) {
    // ---- issues the TMA loads, waits for them, and forms the x-halo columns one plane ahead ----------
    const int hr = VX == 2 ? lane : (lane & 15);
    Site ht;
    ht.row = min(hr, ROWS - 1);
    const int cl = (x0 + nx - 1) % nx, cr = (x0 + XO) % nx;
    ht.o0 = row_of(ht.row) * nx + (VX == 2 || lane < 16 ? cl : cr);
    ht.o1 = row_of(ht.row) * nx + cr;
    ht.needed = ybl - 1 + ht.row <= yrows;
    S hraw0[10], hraw1[10];
    Extra hext;
    hext.l0 = hext.l1 = 0u;
    auto hfetch = [&](int ip) {
      fetch_values(ht, ip, hraw0, hraw1);
      if constexpr (AHEAD) fetch_extra(ht, ip, hext);
    };
    const int rows = min(ROWS, yrows + 2 - ybl), rs = row_of(min(lane, ROWS - 1));
    // all rows at once where they are consecutive in the lattice, else (y wrap, last rows) one by one:
    // a copy costs its issuing warp about 80 cycles
    const bool whole = y0 >= 1 && y0 + TY + 1 <= ny && rows == ROWS;
    auto issue = [&](int ip) {
      if (ip >= planes) return;
      const int zs = wrap(z0 - 1 + ip, a.nz);
      uint64_t* const bar = &bars[ip % STAGES];
      if (lane == 0) {
        LBF_CHECK(a.flags, (smem_u32(stage_row(ip, 0)) & 127u) == 0u && (x0 * int(sizeof(S))) % 16 == 0 && x0 >= 0 && x0 + XO <= nx);
        mbar_arrive_expect_tx(bar, uint32_t(G::ROWB) * uint32_t(rows));
        if (whole) tma_load_4d(stage_row(ip, 0), &ttile, bar, x0, 0, y0 - 1, zs);
      }
      __syncwarp();
      if (!whole && lane < rows) tma_load_4d(stage_row(ip, lane), &trow, bar, x0, 0, rs, zs);
      __syncwarp();
    };
    if (lane == 0) {
      gave_up[0] = gave_up[1] = 0;
      if constexpr (TMA) {
        prefetch_tensormap(whole ? &ttile : &trow);
        prefetch_tensormap(&tout);
        for (int s = 0; s < STAGES; ++s) mbar_init(&bars[s], 1);
        fence_mbar_init();
      }
    }
    __syncwarp();
    if constexpr (TMA) {
      for (int s = 0; s < STAGES - 1; ++s) issue(s);
    }
    if (!one_tile) hfetch(0);
    int lost = -1;  // the plane whose wait gave up
    for (int it = -1; it < planes; ++it) {
      const int ip = it + 1;
      if (ip < planes) {
        if (!one_tile) {
          halo_columns(ht, hr < ROWS, ip, hraw0, hraw1, hext);
          if (ip + 1 < planes) hfetch(ip + 1);
        }
        if (TMA && !mbar_wait_bounded(&bars[ip % STAGES], uint32_t(ip / STAGES) & 1u, kWaitPolls)) {
          atomicOr(a.flags, 2u);
          lost = ip;
          gave_up[it & 1] = 1;
        }
      }
      cta_barrier<G::THREADS>();  // passes the plane's arrival on to every row
      if (gave_up[it & 1]) break;  // written before this barrier, rewritten after the next one
      // every row has read its part of plane it - 1 and its outputs have left that stage
      if (TMA && it >= 0) issue(it - 1 + STAGES);
    }
    if constexpr (TMA) {
      // after an abandoned wait, let the copies still in flight land before the CTA exits (bounded)
      if (lost >= 0)
        for (int ip = lost; ip < min(planes, max(lost - 1, 0) + STAGES - 1); ++ip)
          mbar_wait_bounded(&bars[ip % STAGES], uint32_t(ip / STAGES) & 1u, kWaitPolls);
    }
  } else {
    // ---- the output rows ---------------------------------------------------------------------------
    const int gx = x0 + VX * lane;
    // outputs in flight, in the units of the summed weights: the plane below the current one (all but
    // its c_z = -1 part; rzz equals jz there without walls) and u**, what the current plane sends to the
    // next (c_z = +1)
    struct Flight {
      V a0, jx, jy, jz, rxx, ryy, rzz, rxy, rxz, ryz;
      V u00, u10, u01, u20, u02, u11;
      V hx, hy, hz;      // half force of the plane below (FF)
      V n0[TWO != 0 ? 3 : 1], np[1], ng[TWO == 2 ? 3 : 1];  // two components: F^{n+1}, phi^{n+1}, grad phi^{n+1} there
      bool sol0, sol1;   // its solid flags
    };
    RowIn in[RP];
    Flight fl[RP];
    int gy[RP];
#pragma unroll
    for (int r = 0; r < RP; ++r) {
      in[r] = row_in(1 + warp * RP + r);
      gy[r] = row_of(1 + warp * RP + r);
      Flight& f = fl[r];
      f.a0 = f.jx = f.jy = f.jz = f.rxx = f.ryy = f.rzz = f.rxy = f.rxz = f.ryz = zero;
      f.u00 = f.u10 = f.u01 = f.u20 = f.u02 = f.u11 = f.hx = f.hy = f.hz = zero;
      f.sol0 = f.sol1 = false;
      if constexpr (AHEAD) fetch(in[r], 0);
    }
    // two components: the correction's inputs of plane ip, loaded when it is taken in, used a plane later
    auto fetch_new = [&](const RowIn& r, Flight& f, int ip) {
      if constexpr (TWO != 0) {
        if (!r.t.needed) return;
        const long long zoff = (long long)wrap(z0 - 1 + ip, a.nz) * plane;
        const T* Fn = static_cast<const T*>(a.F_new) + zoff;  // rewritten (TWO = 2) only at the site's own output
        const T* pn = static_cast<const T*>(a.phi_new) + zoff;
        auto two_of = [&](const T* q) -> V {
          if constexpr (VX == 2 && TMA)
            return *reinterpret_cast<const float2*>(q + r.t.o0);
          else
            return pack(q[r.t.o0], VX == 2 ? q[r.t.o1] : T(0));
        };
#pragma unroll
        for (int k = 0; k < 3; ++k) f.n0[k] = two_of(Fn + k * N);
        f.np[0] = two_of(pn);
        if constexpr (TWO == 2) {
          const T* gp = static_cast<const T*>(a.grad_phi) + zoff;
#pragma unroll
          for (int k = 0; k < 3; ++k) f.ng[k] = two_of(gp + k * N);
        }
      }
    };
    bool bad = false;
    // whole rows of fluid sites leave as one TMA box from the stage rows the warp has just read
    for (int p = 0; p < STAGES - 1; ++p) {
#pragma unroll
      for (int r = 0; r < RP; ++r) copy_row(in[r], p);
      copies_group();
    }
    const bool by_tma = TMA && !dirty && x0 == xb && ybl + warp * RP + RP <= yrows && gy[RP - 1] == gy[0] + RP - 1;
    cta_barrier<G::THREADS>();
    int it = 0;
    do {
      const int part = PARTS ? min(planes, it + 32) : planes;
      for (; it < part && !gave_up[(it - 1) & 1]; ++it) {
        V F[RP][3], own[RP][9];
        V pin[RP > 1 ? NY : 1], min_[RP > 1 ? NY : 1];  // p of the lower, m of the upper of two rows
        bool s0[RP], s1[RP];
        copies_done();
  #pragma unroll
        for (int r = 0; r < RP; ++r) {
          V P[NY], M[NY];
          row_front(in[r], it, true, F[r], P, M, own[r]);
          if (r == 0 && warp > 0) {
  #pragma unroll
            for (int e = 0; e < NY; ++e) *y_at(it, 1, e, warp - 1) = M[e];
          }
          if (r == RP - 1 && warp < PAIRS - 1) {
  #pragma unroll
            for (int e = 0; e < NY; ++e) *y_at(it, 0, e, warp + 1) = P[e];
          }
          if constexpr (RP > 1) {
  #pragma unroll
            for (int e = 0; e < NY; ++e) {
              if (r == 0) pin[e] = P[e];
              else min_[e] = M[e];
            }
          }
          s0[r] = MASK && (in[r].e.l0 >> 31) != 0u;
          s1[r] = MASK && (in[r].e.l1 >> 31) != 0u;
          if constexpr (AHEAD) {
            if (it + 1 < planes) fetch(in[r], it + 1);
          }
          // c_z = -1 part of the plane below, as far as it needs no neighbour row
          Flight& f = fl[r];
          f.rzz = v_add(MASK ? f.rzz : f.jz, own[r][3]);
          f.a0 = v_add(f.a0, own[r][3]);
          f.jz = v_sub(f.jz, own[r][3]);
          f.jx = v_add(f.jx, own[r][4]);
          f.rxz = v_sub(f.rxz, own[r][4]);
          f.rxx = v_add(f.rxx, own[r][5]);
        }
        if constexpr (TMA) {
          bulk_wait_group_read0();  // the last outputs have left their stage
        } else {
  #pragma unroll
          for (int r = 0; r < RP; ++r) copy_row(in[r], it - 1 + STAGES);  // into the stage of plane it - 1
          copies_group();
        }
        cta_barrier<G::THREADS>();
  #pragma unroll
        for (int r = 0; r < RP; ++r) {
          Flight& f = fl[r];
          const int row = in[r].t.row;
          auto y_sums = [&](int e) -> PairSD<V> {
            const V l = r == 0 ? *y_at(it, 0, e, warp) : pin[RP > 1 ? e : 0];
            const V h = r == RP - 1 ? *y_at(it, 1, e, warp) : min_[RP > 1 ? e : 0];
            return {v_add(l, h), v_sub(l, h)};
          };
          {
            const PairSD<V> q = y_sums(Q19 ? 1 : 3);
            f.a0 = v_add(f.a0, q.S);
            f.jz = v_sub(f.jz, q.S);
            f.rzz = v_add(f.rzz, q.S);
            f.ryy = v_add(f.ryy, q.S);
            f.jy = v_add(f.jy, q.D);
            f.ryz = v_sub(f.ryz, q.D);
            if constexpr (!Q19) {
              const PairSD<V> q1 = y_sums(4);
              f.jx = v_add(f.jx, q1.S);
              f.rxz = v_sub(f.rxz, q1.S);
              f.rxy = v_add(f.rxy, q1.D);
              f.rxx = v_add(f.rxx, y_sums(5).S);
            }
          }
          if (it >= 2) {
            const int z = z0 + it - 2;
            // the sums are in units of the smallest weight, 1/36 or 1/216. In FP32 p* and u, which accumulate over
            // the steps, take that factor in two parts (rounded, and what it lacks): rounded once, it would scale
            // them by 1 + 7e-9 in every step (20 steps: error of u 9.1e-8 against 1.5e-7 with rounded weights). In
            // FP64 it is rounded once, as the weights are in any FP64 code that adds up populations: 50 steps are
            // 2.3e-15 off 80-bit arithmetic (the 30-column kernel 2.4e-15). In two parts they would be 3.2e-16 off
            // that, but 25 times further from FP64 code with rounded weights, whose common factor they would lack
            constexpr T sc = Q19 ? T(1) / T(36) : T(1) / T(216);
            constexpr T lack = T((Q19 ? 1.0 / 36.0 : 1.0 / 216.0) - double(sc));
            const V vs = v_set<V>(sc), vl = v_set<V>(lack);
            auto scaled = [&](V v) -> V {
              if constexpr (std::is_same<T, double>::value)
                return v_mul(v, vs);
              else
                return v_fma(v, vs, v_mul(v, vl));
            };
            const V b0 = scaled(f.a0);
            const bool own_row = ybl + warp * RP + r < yrows;
            const bool w0 = own_row && gx >= xb && gx < nx && !f.sol0;
            const bool w1 = VX == 2 && own_row && gx >= xb && gx + 1 < nx && !f.sol1;
            const long long zc = (long long)z * plane + in[r].t.o0;
            V hx_, hy_, hz_;
            if constexpr (TWO != 0) {
              V Fn[3] = {f.n0[0], f.n0[1], f.n0[2]};
              if constexpr (TWO == 2) {
                // density contrast (Sec. 2 force split): the force of the new state adds to F^s + F^b
                //   F^p = -p* cs2 grad rho and F^nu = -(nu omega / cs2) a*_neq . grad rho,
                // with p* = a*0 and a*_neq = a*2 - a*1 a*1 the raw moments just streamed in
                const V jx_ = scaled(f.jx), jy_ = scaled(f.jy), jz_ = scaled(f.jz);
                const V dr = v_set<V>(drho), gr0 = v_mul(f.ng[0], dr), gr1 = v_mul(f.ng[1], dr), gr2 = v_mul(f.ng[2], dr);
                const V p3 = v_mul(b0, v_set<V>(T(1) / T(3)));
                const V qxx = v_nfma(jx_, jx_, v_sub(v_mul(f.rxx, vs), p3));
                const V qyy = v_nfma(jy_, jy_, v_sub(v_mul(f.ryy, vs), p3));
                const V qzz = v_nfma(jz_, jz_, v_sub(v_mul(f.rzz, vs), p3));
                const V qxy = v_nfma(jx_, jy_, v_mul(f.rxy, vs)), qxz = v_nfma(jx_, jz_, v_mul(f.rxz, vs));
                const V qyz = v_nfma(jy_, jz_, v_mul(f.ryz, vs));
                const V cnu = each(f.np[0], [&](T p) {
                  const T nu = nu_l + p * dnu;
                  return T(-3) * nu / (T(3) * nu + T(0.5));
                });
                Fn[0] = v_add(Fn[0], v_nfma(p3, gr0, v_mul(cnu, v_fma(qxx, gr0, v_fma(qxy, gr1, v_mul(qxz, gr2))))));
                Fn[1] = v_add(Fn[1], v_nfma(p3, gr1, v_mul(cnu, v_fma(qxy, gr0, v_fma(qyy, gr1, v_mul(qyz, gr2))))));
                Fn[2] = v_add(Fn[2], v_nfma(p3, gr2, v_mul(cnu, v_fma(qxz, gr0, v_fma(qyz, gr1, v_mul(qzz, gr2))))));
                T* Fw = static_cast<T*>(a.F_new) + (long long)z * plane;
  #pragma unroll
                for (int k = 0; k < 3; ++k) {
                  if constexpr (VX == 2) {
                    if (w0) Fw[k * N + in[r].t.o0] = Fn[k].x;
                    if (w1) Fw[k * N + in[r].t.o1] = Fn[k].y;
                  } else {
                    if (w0) Fw[k * N + in[r].t.o0] = Fn[k];
                  }
                }
              }
              const V hr = v_mul(rrho_of(f.np[0]), v_set<V>(T(0.5)));
              hx_ = v_mul(Fn[0], hr), hy_ = v_mul(Fn[1], hr), hz_ = v_mul(Fn[2], hr);
            } else if constexpr (FF)
              hx_ = f.hx, hy_ = f.hy, hz_ = f.hz;
            else
              hx_ = v_set<V>(T(0.5) * Fu0), hy_ = v_set<V>(T(0.5) * Fu1), hz_ = v_set<V>(T(0.5) * Fu2);
            // Eq. (corr), rho = 1: u = a1 + h with h = F/2, a2 = (sum c c f - cs2 a0 delta) + u h + h u, so
            // N = a2 - u u = (sum c c f - cs2 a0 delta) - a1 a1 + h h
            const V vx = scaled(f.jx), vy = scaled(f.jy), vz = scaled(f.jz);
            const V ux = v_add(vx, hx_), uy = v_add(vy, hy_), uz = v_add(vz, hz_);
            const V third = v_set<V>(T(-1) / T(3));
            const V nxx = v_nfma(vx, vx, v_fma(f.rxx, vs, v_fma(b0, third, v_mul(hx_, hx_))));
            const V nyy = v_nfma(vy, vy, v_fma(f.ryy, vs, v_fma(b0, third, v_mul(hy_, hy_))));
            const V nzz = v_nfma(vz, vz, v_fma(f.rzz, vs, v_fma(b0, third, v_mul(hz_, hz_))));
            const V nxy = v_nfma(vx, vy, v_fma(f.rxy, vs, v_mul(hx_, hy_)));
            const V nxz = v_nfma(vx, vz, v_fma(f.rxz, vs, v_mul(hx_, hz_)));
            const V nyz = v_nfma(vy, vz, v_fma(f.ryz, vs, v_mul(hy_, hz_)));
            const V uu = v_fma(ux, ux, v_fma(uy, uy, v_mul(uz, uz)));
            LBF_CHECK(a.flags, !(w0 || w1) || (z >= 0 && z < a.nz && in[r].t.o0 >= 0 && in[r].t.o0 < plane && zc + 9 * N < 10 * N));
            S* d0 = dst + zc;
            const T um = T(a.umax2);
            if constexpr (VX == 2) {
              uint32_t r0 = 0u, r1 = 0u;
              if constexpr (Codec<S>::scaled && !RN) {
                r0 = fmix32(uint32_t(zc) ^ a.salt);
                r1 = fmix32(uint32_t(zc + 1) ^ a.salt);
              }
              if (by_tma) {
                S* o = reinterpret_cast<S*>(stage_row(it, row)) + VX * lane;
                st_pair<S, RN>(o, b0, a.sc.enc[0], r0, r1);
                st_pair<S, RN>(o + XO, ux, a.sc.enc[1], r0, r1);
                st_pair<S, RN>(o + 2 * XO, uy, a.sc.enc[1], r0, r1);
                st_pair<S, RN>(o + 3 * XO, uz, a.sc.enc[1], r0, r1);
                st_pair<S, true>(o + 4 * XO, nxx, a.sc.enc[2], r0, r1);
                st_pair<S, true>(o + 5 * XO, nyy, a.sc.enc[2], r0, r1);
                st_pair<S, true>(o + 6 * XO, nzz, a.sc.enc[2], r0, r1);
                st_pair<S, true>(o + 7 * XO, nxy, a.sc.enc[2], r0, r1);
                st_pair<S, true>(o + 8 * XO, nxz, a.sc.enc[2], r0, r1);
                st_pair<S, true>(o + 9 * XO, nyz, a.sc.enc[2], r0, r1);
                fence_proxy_async_smem();
                __syncwarp();
                if (r == RP - 1 && lane == 0) {
                  tma_store_4d(&tout, stage_row(it, row - r), x0, 0, gy[0], z);
                  bulk_commit_group();
                }
              } else if (TMA && w0 && w1) {
                st_pair<S, RN>(d0, b0, a.sc.enc[0], r0, r1);
                st_pair<S, RN>(d0 + N, ux, a.sc.enc[1], r0, r1);
                st_pair<S, RN>(d0 + 2 * N, uy, a.sc.enc[1], r0, r1);
                st_pair<S, RN>(d0 + 3 * N, uz, a.sc.enc[1], r0, r1);
                st_pair<S, true>(d0 + 4 * N, nxx, a.sc.enc[2], r0, r1);
                st_pair<S, true>(d0 + 5 * N, nyy, a.sc.enc[2], r0, r1);
                st_pair<S, true>(d0 + 6 * N, nzz, a.sc.enc[2], r0, r1);
                st_pair<S, true>(d0 + 7 * N, nxy, a.sc.enc[2], r0, r1);
                st_pair<S, true>(d0 + 8 * N, nxz, a.sc.enc[2], r0, r1);
                st_pair<S, true>(d0 + 9 * N, nyz, a.sc.enc[2], r0, r1);
              } else if (!TMA || MASK) {
                auto put = [&](int at, uint32_t& rr, float p_, float x_, float y_, float z_, float xx, float yy, float zz,
                               float xy, float xz, float yz) {
                  S* d = d0 + at;
                  st_field<S, RN>(d, 0, p_, a.sc.enc[0], rr);
                  st_field<S, RN>(d + N, 0, x_, a.sc.enc[1], rr);
                  st_field<S, RN>(d + 2 * N, 0, y_, a.sc.enc[1], rr);
                  st_field<S, RN>(d + 3 * N, 0, z_, a.sc.enc[1], rr);
                  st_field<S, true>(d + 4 * N, 0, xx, a.sc.enc[2], rr);
                  st_field<S, true>(d + 5 * N, 0, yy, a.sc.enc[2], rr);
                  st_field<S, true>(d + 6 * N, 0, zz, a.sc.enc[2], rr);
                  st_field<S, true>(d + 7 * N, 0, xy, a.sc.enc[2], rr);
                  st_field<S, true>(d + 8 * N, 0, xz, a.sc.enc[2], rr);
                  st_field<S, true>(d + 9 * N, 0, yz, a.sc.enc[2], rr);
                };
                if (w0) put(0, r0, b0.x, ux.x, uy.x, uz.x, nxx.x, nyy.x, nzz.x, nxy.x, nxz.x, nyz.x);
                if (w1) put(1, r1, b0.y, ux.y, uy.y, uz.y, nxx.y, nyy.y, nzz.y, nxy.y, nxz.y, nyz.y);
              }
              bad = bad || (w0 && !(uu.x <= um)) || (w1 && !(uu.y <= um));
              if (a.partials != nullptr) {
                red[0] += (w0 ? b0.x : 0.0f) + (w1 ? b0.y : 0.0f);
                red[1] += (w0 ? ux.x : 0.0f) + (w1 ? ux.y : 0.0f);
                red[2] += (w0 ? uy.x : 0.0f) + (w1 ? uy.y : 0.0f);
                red[3] += (w0 ? uz.x : 0.0f) + (w1 ? uz.y : 0.0f);
                if constexpr (TWO != 0) red[4] += (w0 ? f.np[0].x : 0.0f) + (w1 ? f.np[0].y : 0.0f);
                red[5] += (w0 ? uu.x : 0.0f) + (w1 ? uu.y : 0.0f);
              }
            } else if (w0) {
              d0[0] = b0;
              d0[N] = ux;
              d0[2 * N] = uy;
              d0[3 * N] = uz;
              d0[4 * N] = nxx;
              d0[5 * N] = nyy;
              d0[6 * N] = nzz;
              d0[7 * N] = nxy;
              d0[8 * N] = nxz;
              d0[9 * N] = nyz;
              bad = bad || !(uu <= um);
              red[0] += b0;
              red[1] += ux;
              red[2] += uy;
              red[3] += uz;
              if constexpr (TWO != 0) red[4] += f.np[0];
              red[5] += uu;
            }
          }
          fetch_new(in[r], f, it);
          // this plane becomes the one in flight: c_z = +1 of the plane below plus its own c_z = 0 part
          auto mid = [&](V u, V v) { return Q19 ? v_add(u, v) : v_fma(v, v_set<V>(T(4)), u); };
          {
            const PairSD<V> q0 = y_sums(Q19 ? 2 : 6), q1 = y_sums(Q19 ? 3 : 7);
            f.a0 = mid(f.u00, v_add(own[r][6], q0.S));
            f.ryy = mid(f.u02, q0.S);
            f.jy = mid(f.u01, q0.D);
            f.jx = mid(f.u10, v_add(own[r][7], q1.S));
            f.rxy = Q19 ? q1.D : mid(f.u11, q1.D);
            f.rxx = mid(f.u20, v_add(own[r][8], y_sums(Q19 ? 4 : 8).S));
          }
          f.jz = f.u00;
          f.rxz = f.u10;
          f.ryz = f.u01;
          if constexpr (MASK) {
            f.rzz = f.u00;
            if (dirty) {
              const V* const b = cor_at(it, row);
              f.a0 = v_add(f.a0, b[0]);
              f.jx = v_add(f.jx, b[32]);
              f.jy = v_add(f.jy, b[2 * 32]);
              f.jz = v_add(f.jz, b[3 * 32]);
              f.rxx = v_add(f.rxx, b[4 * 32]);
              f.ryy = v_add(f.ryy, b[5 * 32]);
              f.rzz = v_add(f.rzz, b[6 * 32]);
              f.rxy = v_add(f.rxy, b[7 * 32]);
              f.rxz = v_add(f.rxz, b[8 * 32]);
              f.ryz = v_add(f.ryz, b[9 * 32]);
            }
            f.sol0 = s0[r];
            f.sol1 = s1[r];
          }
          if constexpr (FF) {
            const V half = v_set<V>(T(0.5));
            f.hx = v_mul(F[r][0], half), f.hy = v_mul(F[r][1], half), f.hz = v_mul(F[r][2], half);
          }
          {
            const PairSD<V> q = y_sums(0);
            f.u00 = v_add(own[r][0], q.S);
            f.u02 = q.S;
            f.u01 = q.D;
            if constexpr (Q19) {
              f.u10 = own[r][1];
              f.u20 = own[r][2];
            } else {
              const PairSD<V> q1 = y_sums(1);
              f.u10 = v_add(own[r][1], q1.S);
              f.u11 = q1.D;
              f.u20 = v_add(own[r][2], y_sums(2).S);
            }
          }
        }
      }
      if constexpr (PARTS) {
        if (a.partials != nullptr) {
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            const double v = warp_sum(red[k]);
            if (lane == 0) parts[warp * 6 + k] += v;
            red[k] = T(0);
          }
        }
      }
    } while (PARTS && it < planes && !gave_up[(it - 1) & 1]);
    if constexpr (TMA) bulk_wait_group0();
    else asm volatile("cp.async.wait_all;" ::: "memory");
    if (bad) atomicOr(a.flags, 1u);
  }
  __syncthreads();
  grid_release();

  if (a.partials != nullptr) {
    // warp sums (of some planes) in the compute type, the others in FP64, in a fixed order
    double* red_s = PARTS ? parts : reinterpret_cast<double*>(sbase);
    const int tid = warp * 32 + lane;
    if constexpr (!PARTS) {
#pragma unroll
      for (int k = 0; k < 6; ++k) {
        const double v = warp_sum(red[k]);
        if (lane == 0) red_s[warp * 6 + k] = v;
      }
      __syncthreads();
    }
    const long long nb = (long long)gridDim.x * gridDim.y * gridDim.z;
    if (tid < 6) {
      double s = 0.0;
      for (int r = 0; r < G::WARPS; ++r) s += red_s[r * 6 + tid];
      const long long b = a.block_base + ((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
      a.partials[b * 8 + tid] = s;
    }
    __shared__ bool last;
    __threadfence();
    __syncthreads();
    const long long nall = a.final_blocks > 0 ? a.final_blocks : a.block_base + nb;  // partials to add
    if (tid == 0) last = atomicAdd(a.counter, 1u) == (unsigned)(a.final_blocks > 0 ? nall - 1 : nb - 1);
    __syncthreads();
    if (last) {
      __threadfence();
      constexpr int NT = G::THREADS;
      sum_partials<NT>(a.partials, nall, reinterpret_cast<double*>(sbase), a.sums, tid);
      if (tid == 0) *a.counter = 0u;
    }
  }
}

// one block per tile of the step: dirty when a solid site lies in its outputs' reach (the tile and one
// site around it, periodic). The last tile of a row covers both placements: ending at nx - 1 (the TMA
// kernel) and starting at a multiple of xo (the direct one)
static __global__ void k_tile_dirty(const uint8_t* __restrict__ mask, int nx, int ny, int nz, int xo, int ty, int zchunk,
                                    bool shift, uint8_t* __restrict__ out) {
  const int xb = int(blockIdx.x) * xo, x0 = shift ? min(xb, nx - xo) : xb;
  const int y0 = blockIdx.y * ty, z0 = blockIdx.z * zchunk, z1 = min(nz, z0 + zchunk);
  const int wx = xb - x0 + xo + 2, wy = ty + 2, wz = z1 - z0 + 2;
  int any = 0;
  for (int i = threadIdx.x; i < wx * wy * wz && !any; i += blockDim.x) {
    const int x = ((x0 - 1 + i % wx) % nx + nx) % nx, y = ((y0 - 1 + (i / wx) % wy) % ny + ny) % ny;
    const int z = ((z0 - 1 + i / (wx * wy)) % nz + nz) % nz;
    any |= mask[((long long)z * ny + y) * nx + x] != 0;
  }
  any = __syncthreads_or(any);
  if (threadIdx.x == 0) out[((long long)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = any ? 1 : 0;
}

// Per site: bit q set when x - c_q is solid (the directions along which a fluid site gets its own
// population back), bit 31 when the site itself is solid.
template <class L>
__global__ void k_wall_links(const uint8_t* __restrict__ mask, int nx, int ny, int nz, uint32_t* __restrict__ links) {
  const long long N = (long long)nx * ny * nz, plane = (long long)nx * ny;
  for (long long s = blockIdx.x * (long long)blockDim.x + threadIdx.x; s < N; s += (long long)gridDim.x * blockDim.x) {
    const int z = int(s / plane), y = int((s % plane) / nx), x = int(s % nx);
    uint32_t bits = mask[s] != 0 ? 0x80000000u : 0u;
    static_for<L::Q>([&](auto qc) {
      constexpr int q = decltype(qc)::value;
      if constexpr (q != rest_index<L>()) {
        const int xs = wrap(x - L::cx(q), nx), ys = wrap(y - L::cy(q), ny), zs = wrap(z - L::cz(q), nz);
        if (mask[zs * plane + (long long)ys * nx + xs] != 0) bits |= 1u << q;
      }
    });
    // a solid site needs no links: it sends nothing and is not written
    links[s] = (bits >> 31) != 0u ? 0x80000000u : bits;
  }
}

}  // namespace lbf
