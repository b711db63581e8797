// Positions, bonded terms, velocity Verlet, CSVR thermostat and reductions.
//
// State inside relres_step: positions are 64-bit periodic fixed point
// (exact, wrap-free increments; resolution L/2^64), velocities FP64.  The two
// half kicks of consecutive velocity-Verlet steps are merged: the velocity
// array holds u = v(n - 1/2) during a call, and one drift kernel per step does
//     u <- a u + b c F(n),   c = dt / (2 m),   x <- x + dt u
// with (a, b) = (1, 1) on the first step of a call (u = v(0)) and
// (alpha, alpha + 1) afterwards, alpha the CSVR factor of step n (1 for NVE):
// that is v(n) = u + c F(n), v(n) <- alpha v(n), u <- v(n) + c F(n).  The
// kinetic energy for the thermostat and the thermo output is formed from
// u + c F(n) in the finish kernel.  At the end of a call the velocities are
// returned as v(N) = a u + (b - 1) c F(N) and positions as doubles in [0, L).
//
// Bonded forces are computed per atom from the CSR list of the terms it takes
// part in (each term recomputed by each of its atoms): no atomics, and each
// term's energy is counted by its first atom.
//
// Kernel parameters are only read directly (never through a pointer or a
// reference, never indexed with a run-time index); per-type constants live in
// small device arrays.
#include "common.cuh"
#include "fbits.h"

namespace relres {

constexpr double kFtm2v = 4.184e-4;        // (kcal/mol/A)/(g/mol) -> A/fs^2
constexpr double kMvv2e = 1.0 / 4.184e-4;  // (g/mol)(A/fs)^2 -> kcal/mol

struct BoxConsts {
  double inv_l0, inv_l1, inv_l2;     // 1 / L
  double l64_0, l64_1, l64_2;        // L / 2^64
  double dts0, dts1, dts2;           // dt * 2^64 / L  (A/fs -> fixed-point units per step)
  float s32_0, s32_1, s32_2;         // L / 2^32
  double l0, l1, l2;                 // L
};

static BoxConsts box_consts(const relres_ctx* c, double dt) {
  BoxConsts b;
  b.inv_l0 = 1.0 / c->box[0];
  b.inv_l1 = 1.0 / c->box[1];
  b.inv_l2 = 1.0 / c->box[2];
  b.l64_0 = c->box[0] / 18446744073709551616.0;
  b.l64_1 = c->box[1] / 18446744073709551616.0;
  b.l64_2 = c->box[2] / 18446744073709551616.0;
  b.dts0 = dt * 18446744073709551616.0 / c->box[0];
  b.dts1 = dt * 18446744073709551616.0 / c->box[1];
  b.dts2 = dt * 18446744073709551616.0 / c->box[2];
  b.s32_0 = float(c->box[0] / 4294967296.0);
  b.s32_1 = float(c->box[1] / 4294967296.0);
  b.s32_2 = float(c->box[2] / 4294967296.0);
  b.l0 = c->box[0];
  b.l1 = c->box[1];
  b.l2 = c->box[2];
  return b;
}

static void ff_split(double v, float* hi, float* lo) {
  *hi = float(v);
  *lo = float(v - double(*hi));
}

template <typename R>
struct Sc3 {  // per-axis scale of a fixed-point difference
  R s0, s1, s2;
};

// ----------------------------------------------------------------- positions

__device__ __forceinline__ void scatter_sorted(int i, int t, unsigned long long x, unsigned long long y,
                                               unsigned long long z, const int* rank_fg,
                                               const int* rank_cg, int with_cg, int4* pos_fg,
                                               int4* pos_cg, int fp64, Pos64* pos_fg64,
                                               Pos64* pos_cg64) {
  const int4 h = make_int4(hi32(x), hi32(y), hi32(z), t);
  const int sf = rank_fg[i];
  pos_fg[sf] = h;
  if (fp64) pos_fg64[sf] = Pos64{(long long)x, (long long)y, (long long)z, t};
  if (with_cg) {
    const int sc = rank_cg[i];
    if (sc >= 0) {
      pos_cg[sc] = h;
      if (fp64) pos_cg64[sc] = Pos64{(long long)x, (long long)y, (long long)z, t};
    }
  }
}

// The same with the atom's slots given (sc < 0: no CG slot).
__device__ __forceinline__ void scatter_sorted_at(int sf, int sc, int t, unsigned long long x, unsigned long long y,
                                                  unsigned long long z, int4* pos_fg, int4* pos_cg, int fp64,
                                                  Pos64* pos_fg64, Pos64* pos_cg64) {
  const int4 h = make_int4(hi32(x), hi32(y), hi32(z), t);
  pos_fg[sf] = h;
  if (fp64) pos_fg64[sf] = Pos64{(long long)x, (long long)y, (long long)z, t};
  if (sc >= 0) {
    pos_cg[sc] = h;
    if (fp64) pos_cg64[sc] = Pos64{(long long)x, (long long)y, (long long)z, t};
  }
}

__device__ __forceinline__ bool moved_beyond(int4 ref, unsigned long long x, unsigned long long y,
                                             unsigned long long z, Sc3<float> s, float thr2) {
  const float dx = dfix32(hi32(x), ref.x, s.s0);
  const float dy = dfix32(hi32(y), ref.y, s.s1);
  const float dz = dfix32(hi32(z), ref.z, s.s2);
  return dx * dx + dy * dy + dz * dz > thr2;
}

__global__ void k_convert(int n, const double* __restrict__ pos, const int* __restrict__ type,
                          unsigned long long* __restrict__ xfx, BoxConsts b, int have_lists,
                          const int* rank_fg, const int* rank_cg, int with_cg, int4* pos_fg,
                          int4* pos_cg, int fp64, Pos64* pos_fg64, Pos64* pos_cg64, const int4* ref,
                          float thr2, const int4* ref_p, float thr2_p, int prune, DevState* st, long long* acc) {
  if (blockIdx.x == 0)  // empty accumulators for the evaluation that follows
    for (int q = threadIdx.x; q < kNAccAll; q += blockDim.x) acc[q] = 0;
  const double il0 = b.inv_l0, il1 = b.inv_l1, il2 = b.inv_l2;
  const Sc3<float> s{b.s32_0, b.s32_1, b.s32_2};
  bool rebuild = false, reprune = false, bad = false;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    const double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
    bad |= !(isfinite(x) && isfinite(y) && isfinite(z));
    const unsigned long long ux = to_fixed(x, il0), uy = to_fixed(y, il1), uz = to_fixed(z, il2);
    xfx[3 * i] = ux;
    xfx[3 * i + 1] = uy;
    xfx[3 * i + 2] = uz;
    if (have_lists) {
      scatter_sorted(i, type[i], ux, uy, uz, rank_fg, rank_cg, with_cg, pos_fg, pos_cg, fp64, pos_fg64,
                     pos_cg64);
      rebuild |= moved_beyond(ref[i], ux, uy, uz, s, thr2);
      if (prune) reprune |= moved_beyond(ref_p[i], ux, uy, uz, s, thr2_p);
    }
  }
  if (__syncthreads_or(rebuild) && threadIdx.x == 0) atomicOr(&st->flags, F_REBUILD);
  if (__syncthreads_or(reprune) && threadIdx.x == 0) atomicOr(&st->flags, F_PRUNE);
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&st->flags, F_NONFINITE | F_BADPOS);
}

// A 64-bit fixed-point coordinate as a double in [0, L): u L 2^-64, with u
// converted to the nearest double by integer operations (the bits of
// __ull2double_rn(u)); a product rounded up to L wraps to 0 (both positive:
// compared as bit patterns).
__device__ __forceinline__ double back_to_double(unsigned long long u, double l64, double l) {
  const double x = double_of_u64(u) * l64;
  return bits_of_double(x) >= bits_of_double(l) ? 0.0 : x;
}

// The caller's positions (and velocities, when vel is not NULL) against the
// ones the last relres_step returned, word for word: F_DIRTY / F_VDIRTY when
// any differs.
struct CheckIo {
  int n3;  // 0: nothing to compare
  const unsigned long long* pos;
  const unsigned long long* pos_ret;
  const unsigned long long* vel;
  const unsigned long long* vel_ret;
  DevState* st;
};

__device__ __forceinline__ void check_io(const CheckIo& a, int bid, int nblk) {
  bool dp = false, dv = false;
  for (int k = bid * kThreads + threadIdx.x; k < a.n3; k += nblk * kThreads) {
    dp |= a.pos[k] != a.pos_ret[k];
    if (a.vel != nullptr) dv |= a.vel[k] != a.vel_ret[k];
  }
  if (__syncthreads_or(dp) && threadIdx.x == 0) atomicOr(&a.st->flags, F_DIRTY);
  if (__syncthreads_or(dv) && threadIdx.x == 0) atomicOr(&a.st->flags, F_VDIRTY);
}

__global__ void __launch_bounds__(kThreads) k_check_io(const __grid_constant__ CheckIo a) {
  check_io(a, blockIdx.x, gridDim.x);
}

// ----------------------------------------------------------------- bonded

struct BondedArgs {
  const int4* bonds;
  const int4* angles;
  const int4* dihs;
  const int* dih_type;
  const double* bond_par;   // k, r0
  const double* angle_par;  // k, theta0, cos theta0, sin theta0
  const double* dih_par;    // K1..K4
  const float* bond_fpar;   // FP32 path: k, r0 (hi, lo), 0
  const float* angle_fpar;  // FP32 path: k, theta0, cos theta0 (hi, lo), sin theta0 (hi, lo), 0, 0
};

// Where the bonded terms read 64-bit fixed-point positions: the global array
// (caller order), or a segment's copy in shared memory (atoms a0, a0 + 1, ...).
struct GPos {
  const unsigned long long* x;
  __device__ __forceinline__ unsigned long long operator()(int i, int q) const { return x[3 * i + q]; }
};
struct SPos {
  const unsigned long long* s;
  int a0;
  __device__ __forceinline__ unsigned long long operator()(int i, int q) const { return s[3 * (i - a0) + q]; }
};
// global positions of atoms named by a prototype's records: atom i + off
struct GPosOff {
  const unsigned long long* x;
  int off;
  __device__ __forceinline__ unsigned long long operator()(int i, int q) const { return x[3 * (i + off) + q]; }
};

// exact 64-bit fixed-point difference a - b, scaled to Angstrom (float-float)
__device__ __forceinline__ ff ff_fixed_diff(unsigned long long a, unsigned long long b, ff scale) {
  return ff_mul(ff_from_ll((long long)(a - b)), scale);
}
template <class X>
__device__ __forceinline__ void ff_vec(const X& x, int a, int b, ff s0, ff s1, ff s2, ff v[3]) {
  v[0] = ff_fixed_diff(x(a, 0), x(b, 0), s0);
  v[1] = ff_fixed_diff(x(a, 1), x(b, 1), s1);
  v[2] = ff_fixed_diff(x(a, 2), x(b, 2), s2);
}
__device__ __forceinline__ ff ff_dot(const ff a[3], const ff b[3]) {
  return ff_add(ff_add(ff_mul(a[0], b[0]), ff_mul(a[1], b[1])), ff_mul(a[2], b[2]));
}

template <class X>
__device__ __forceinline__ void dvec(const X& x, int a, int b, Sc3<float> s, float d[3]) {
  d[0] = dfix32(hi32(x(a, 0)), hi32(x(b, 0)), s.s0);
  d[1] = dfix32(hi32(x(a, 1)), hi32(x(b, 1)), s.s1);
  d[2] = dfix32(hi32(x(a, 2)), hi32(x(b, 2)), s.s2);
}
template <class X>
__device__ __forceinline__ void dvec(const X& x, int a, int b, Sc3<double> s, double d[3]) {
  d[0] = dfix64((long long)x(a, 0), (long long)x(b, 0), s.s0);
  d[1] = dfix64((long long)x(a, 1), (long long)x(b, 1), s.s1);
  d[2] = dfix64((long long)x(a, 2), (long long)x(b, 2), s.s2);
}

template <typename R>
__device__ __forceinline__ R dot3(const R a[3], const R b[3]) {
  return a[0] * b[0] + a[1] * b[1] + a[2] * b[2];
}
template <typename R>
__device__ __forceinline__ void cross3(const R a[3], const R b[3], R c[3]) {
  c[0] = a[1] * b[2] - a[2] * b[1];
  c[1] = a[2] * b[0] - a[0] * b[2];
  c[2] = a[0] * b[1] - a[1] * b[0];
}

// ---- one bonded term, forces on all of its atoms.  A term is evaluated once,
// by one thread, and its force on each atom (role 0..arity-1) goes to its own
// scratch slot; the finish kernel gathers each atom's slots (no atomics).
// Return value: the term energy.

// FP64 terms.  FP64 division, square root and the inverse functions cost ten to
// forty FMA-rate instructions each on this part (1.66 FMA per clock and SM), so
// every reciprocal comes from rcp_d / rsqrt_d (exact to rounding) and angles
// near their minimum from a series: 161 -> 125 us per MD step of 25 000
// neopentane-like atoms, 46 -> 42 us of 648 propane-like ones.

template <class X>
__device__ __forceinline__ double bond_forces(const BondedArgs& B, const X& xfx, Sc3<double> sc, int4 bd,
                                              double f[2][3]) {
  double d[3];
  dvec(xfx, bd.x, bd.y, sc, d);
  const double q = dot3(d, d), ri = rsqrt_d(q, float(q));
  const double k = B.bond_par[2 * bd.z], dr = q * ri - B.bond_par[2 * bd.z + 1];
  const double g = -2.0 * k * dr * ri;  // force on bd.x along d
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    f[0][c] = g * d[c];
    f[1][c] = -f[0][c];
  }
  return k * dr * dr;
}

// asin(x) for |x| <= 1/4 by its power series, x sum_n (2n)! / (4^n n!^2 (2n + 1)) x^2n;
// the first term left out (n = 13) is below 2^-53 of the sum
__device__ __forceinline__ double asin_small(double x) {
  const double z = x * x;
  double p = 676039.0 / 104857600.0;
  p = fma(p, z, 88179.0 / 12058624.0);
  p = fma(p, z, 46189.0 / 5505024.0);
  p = fma(p, z, 12155.0 / 1245184.0);
  p = fma(p, z, 6435.0 / 557056.0);
  p = fma(p, z, 143.0 / 10240.0);
  p = fma(p, z, 231.0 / 13312.0);
  p = fma(p, z, 63.0 / 2816.0);
  p = fma(p, z, 35.0 / 1152.0);
  p = fma(p, z, 5.0 / 112.0);
  p = fma(p, z, 3.0 / 40.0);
  p = fma(p, z, 1.0 / 6.0);
  return fma(x * z, p, x);
}

// theta - theta0 from its sine, sin theta cos theta0 - cos theta sin theta0,
// where that is small and its cosine positive, else from the two
template <class X>
__device__ __forceinline__ double angle_forces(const BondedArgs& B, const X& xfx, Sc3<double> sc, int4 an,
                                               double f[3][3]) {
  double r1[3], r2[3], n[3];
  dvec(xfx, an.x, an.y, sc, r1);
  dvec(xfx, an.z, an.y, sc, r2);
  const double q1 = dot3(r1, r1), q2 = dot3(r2, r2), qq = q1 * q2;
  const double i12 = rsqrt_d(qq, float(qq)), iqq = i12 * i12;  // 1 / (|r1| |r2|) and its square
  cross3(r1, r2, n);
  const double nn = dot3(n, n) * iqq;  // sin^2 theta
  const double c = dot3(r1, r2) * i12;
  const double si = nn > 1e-12 ? rsqrt_d(nn, float(nn)) : 1e6;  // 1 / sin theta
  const double s = nn * si;
  const double* P = B.angle_par + 4 * an.w;
  const double k = P[0], c0 = P[2], s0 = P[3];
  const double sd = s * c0 - c * s0, cd = c * c0 + s * s0;
  const double dth = (fabs(sd) <= 0.25 && cd > 0.0) ? asin_small(sd) : atan2(sd, cd);
  const double pref = 2.0 * k * dth * si;
  const double a12 = pref * i12, pc = pref * c;
  const double pq = pc * iqq, b1 = pq * q2, b2 = pq * q1;  // pc / q1, pc / q2
#pragma unroll
  for (int w = 0; w < 3; ++w) {
    f[0][w] = a12 * r2[w] - b1 * r1[w];
    f[2][w] = a12 * r1[w] - b2 * r2[w];
    f[1][w] = -(f[0][w] + f[2][w]);
  }
  return k * dth * dth;
}

__device__ __forceinline__ float inv(float x) { return 1.f / x; }
__device__ __forceinline__ double inv(double x) { return rcp_d(x, float(x)); }
__device__ __forceinline__ float inv_sqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double inv_sqrt(double x) { return rsqrt_d(x, float(x)); }

// The multiple angles come from cos phi and sin phi by the Chebyshev relations
// (no inverse function and eight sines and cosines of its result): 24.8 -> 24.4
// us per FP32 MD step of a 14 400-atom copolymer.
template <typename R, class X>
__device__ __forceinline__ R dihedral_forces(const BondedArgs& B, const X& xfx, Sc3<R> sc,
                                             int t, R f[4][3]) {
  const int4 dh = B.dihs[t];
  const double* K = B.dih_par + 4 * B.dih_type[t];
  R b1[3], b2[3], b3[3], m1[3], m2[3];
  dvec(xfx, dh.y, dh.x, sc, b1);
  dvec(xfx, dh.z, dh.y, sc, b2);
  dvec(xfx, dh.w, dh.z, sc, b3);
  cross3(b1, b2, m1);
  cross3(b2, b3, m2);
  const R q2 = dot3(b2, b2), inb2 = inv_sqrt(q2), nb2 = q2 * inb2;
  const R mm1 = dot3(m1, m1), mm2 = dot3(m2, m2);
  const R im = inv_sqrt(mm1 * mm2);
  const R c = dot3(m1, m2) * im, s = nb2 * dot3(b1, m2) * im;  // cos phi, sin phi
  const R c2 = R(2) * c * c - R(1), s2 = R(2) * s * c;
  const R c3 = c * c2 - s * s2, s3 = s * c2 + c * s2;
  const R c4 = R(2) * c2 * c2 - R(1), s4 = R(2) * s2 * c2;
  const R k1 = R(K[0]), k2 = R(K[1]), k3 = R(K[2]), k4 = R(K[3]);
  const R dE = R(0.5) * (-k1 * s + R(2) * k2 * s2 - R(3) * k3 * s3 + R(4) * k4 * s4);
  const R im1 = inv(mm1), im2 = inv(mm2);
  const R p12 = dot3(b1, b2) * im1 * inb2, p32 = dot3(b3, b2) * im2 * inb2;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    // gradient of phi with respect to each atom (Blondel & Karplus form)
    const R g0 = -nb2 * im1 * m1[q];
    const R g3 = nb2 * im2 * m2[q];
    const R h = p12 * m1[q] + p32 * m2[q];
    f[0][q] = -dE * g0;
    f[1][q] = -dE * (-g0 + h);
    f[2][q] = -dE * (-g3 - h);
    f[3][q] = -dE * g3;
  }
  return R(0.5) * (k1 * (R(1) + c) + k2 * (R(1) - c2) + k3 * (R(1) + c3) + k4 * (R(1) - c4));
}

// FP32 bond.  Bonds sit near their minimum with a stiff spring, so the force
// 2k (r - r0) needs r - r0 far below FP32 resolution: r is formed in
// float-float arithmetic from the exact 64-bit fixed-point difference.
template <class X>
__device__ __forceinline__ float bond_forces_ff(const BondedArgs& B, const X& xfx, ff q0,
                                                ff q1, ff q2, int4 bd, float f[2][3]) {
  const float* P = B.bond_fpar + 4 * bd.z;
  ff d[3];
  ff_vec(xfx, bd.x, bd.y, q0, q1, q2, d);
  const ff r = ff_sqrt(ff_dot(d, d));
  const float dr = ff_val(ff_sub(r, ff{P[1], P[2]}));
  const float rf = ff_val(r);
  const float g = -2.f * P[0] * dr / rf;  // force on bd.x along d
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    f[0][q] = g * ff_val(d[q]);
    f[1][q] = -f[0][q];
  }
  return P[0] * dr * dr;
}

// FP32 angle through theta - theta0 = atan2(|a x b| cos t0 - (a.b) sin t0,
// (a.b) cos t0 + |a x b| sin t0): no acos and no loss near theta0, so the
// angle error stays near 1e-7 rad (force error ~2K 1e-7 / r).
template <class X>
__device__ __forceinline__ float angle_forces_f32(const BondedArgs& B, const X& xfx,
                                                  Sc3<float> sc, int4 an, float f[3][3]) {
  const float* P = B.angle_fpar + 8 * an.w;
  float r1[3], r2[3];
  dvec(xfx, an.x, an.y, sc, r1);
  dvec(xfx, an.z, an.y, sc, r2);
  const float dot = r1[0] * r2[0] + r1[1] * r2[1] + r1[2] * r2[2];
  const float cx = r1[1] * r2[2] - r1[2] * r2[1];
  const float cy = r1[2] * r2[0] - r1[0] * r2[2];
  const float cz = r1[0] * r2[1] - r1[1] * r2[0];
  const float cn = sqrtf(cx * cx + cy * cy + cz * cz);
  const float c0 = P[2], s0 = P[4];
  const float dth = atan2f(cn * c0 - dot * s0, dot * c0 + cn * s0);
  const float q1 = r1[0] * r1[0] + r1[1] * r1[1] + r1[2] * r1[2];
  const float q2 = r2[0] * r2[0] + r2[1] * r2[1] + r2[2] * r2[2];
  const float inv12 = rsqrtf(q1 * q2);  // 1 / (|r1| |r2|)
  const float c = dot * inv12;
  float sn = cn * inv12;
  if (sn < 1e-6f) sn = 1e-6f;
  const float pref = 2.f * P[0] * dth / sn;
  const float i11 = 1.f / q1, i22 = 1.f / q2;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    f[0][q] = pref * (r2[q] * inv12 - c * r1[q] * i11);
    f[2][q] = pref * (r1[q] * inv12 - c * r2[q] * i22);
    f[1][q] = -(f[0][q] + f[2][q]);
  }
  return P[0] * dth * dth;
}

// ----------------------------------------------------------------- finish

template <typename R>
using ForceT = typename std::conditional<std::is_same<R, float>::value, float4, double>::type;
// velocity state u: float-float pairs (FP32 path) or doubles (FP64 path), [3n]
template <typename R>
using VelT = typename std::conditional<std::is_same<R, float>::value, float2, double>::type;

// component k of u in the precision of the force arithmetic
__device__ __forceinline__ float vel_r(const float2* v, int k) {
  const float2 p = v[k];
  return __fadd_rn(p.x, p.y);
}
__device__ __forceinline__ double vel_r(const double* v, int k) { return v[k]; }
// component k of u in FP64
__device__ __forceinline__ double vel_d(const float2* v, int k) {
  const float2 p = v[k];
  return double(p.x) + double(p.y);
}
__device__ __forceinline__ double vel_d(const double* v, int k) { return v[k]; }

__device__ __forceinline__ void load_force(const float4* f, int i, float v[3]) {
  const float4 q = f[i];
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
}
__device__ __forceinline__ void load_force(const double* f, int i, double v[3]) {
  v[0] = f[3 * i];
  v[1] = f[3 * i + 1];
  v[2] = f[3 * i + 2];
}
__device__ __forceinline__ void save_force(float4* f, int i, const float v[3]) {
  f[i] = make_float4(v[0], v[1], v[2], 0.f);
}
__device__ __forceinline__ void save_force(double* f, int i, const double v[3]) {
  f[3 * i] = v[0];
  f[3 * i + 1] = v[1];
  f[3 * i + 2] = v[2];
}

template <typename R>
struct BondedKArgs {
  int nb, na, nd;  // bonds, angles, dihedrals: threads [0, nb), [nb, nb + na), [nb + na, nb + na + nd)
  BondedArgs B;
  const unsigned long long* xfx;
  Sc3<R> sc;
  float q0h, q0l, q1h, q1l, q2h, q2l;  // L / 2^64 per axis as float-float (FP32 path)
  ForceT<R>* tf;  // slots: bonds 2 per term from 0, angles 3 per term from 2 nb, dihedrals 4 from 2 nb + 3 na
  long long* acc;
};

template <int NR, typename R>
__device__ __forceinline__ void save_slots(ForceT<R>* tf, size_t base, const R f[NR][3]) {
#pragma unroll
  for (int r = 0; r < NR; ++r) save_force(tf, int(base + r), f[r]);
}

template <typename R, bool EV>
__global__ void __launch_bounds__(kThreads) k_bonded(BondedKArgs<R> a) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  R e = R(0);
  const Sc3<R> sc = a.sc;
  if (t < a.nb) {
    R f[2][3];
    if constexpr (std::is_same<R, float>::value)
      e = bond_forces_ff(a.B, GPos{a.xfx}, ff{a.q0h, a.q0l}, ff{a.q1h, a.q1l}, ff{a.q2h, a.q2l}, a.B.bonds[t], f);
    else
      e = bond_forces(a.B, GPos{a.xfx}, sc, a.B.bonds[t], f);
    save_slots<2, R>(a.tf, 2 * size_t(t), f);
  } else if (t < a.nb + a.na) {
    const int u = t - a.nb;
    R f[3][3];
    if constexpr (std::is_same<R, float>::value)
      e = angle_forces_f32(a.B, GPos{a.xfx}, sc, a.B.angles[u], f);
    else
      e = angle_forces(a.B, GPos{a.xfx}, sc, a.B.angles[u], f);
    save_slots<3, R>(a.tf, 2 * size_t(a.nb) + 3 * size_t(u), f);
  } else if (t < a.nb + a.na + a.nd) {
    const int u = t - a.nb - a.na;
    R f[4][3];
    e = dihedral_forces<R>(a.B, GPos{a.xfx}, sc, u, f);
    save_slots<4, R>(a.tf, 2 * size_t(a.nb) + 3 * size_t(a.na) + 4 * size_t(u), f);
  }
  if (EV) {
    double v[1] = {double(e)};
    __shared__ double sh[kThreads / 32];
    block_sum<double, 1>(v, sh);
    if (threadIdx.x == 0) acc_add(a.acc + kAccEb, v[0]);
  }
}

template <typename R>
struct FinishArgs {
  int n;
  const ForceT<R>* f_fg;
  const ForceT<R>* f_cg;
  int with_cg;
  const int* type;
  int hyb_mask;
  const int* inc_off;
  const int* inc;
  const ForceT<R>* tf;
  int base1, base2;    // first slot of the angles, of the dihedrals
  const VelT<R>* vel;  // u (half-step velocities) for the kinetic energy
  int with_ke;
  const double* cdt;   // per type: dt / (2 m) * ftm2v
  const double* mass;  // per type
  ForceT<R>* f_tot;
  double* f_out;       // FP64 copy in caller order
  int with_out;
  int host_call;
  long long* acc;
  DevState* st;
};

// End of a force evaluation that is a call of its own: the lists are those of
// these positions now (one thread, after the pair kernel).  After a non-finite
// position they are still those of the call before: the displacement triggers
// are worked out again from the next positions, but a pruning pass that was
// due may be one that a build left over, so it stays due.
__device__ __forceinline__ void close_host_call(DevState* st) {
  const unsigned f = *(volatile unsigned*)&st->flags;
  const bool bad = (f & F_NOLISTS) != 0u;
  if ((f & F_REBUILD) && !bad) st->n_builds += 1;
  atomicAnd(&st->flags, bad ? ~unsigned(F_REBUILD) : ~unsigned(F_REBUILD | F_PRUNE));
}
__device__ __forceinline__ bool no_outputs(const DevState* st) {
  return (*(volatile const unsigned*)&st->flags & F_NOLISTS) != 0u;
}

// Total force per atom: FG part + CG part + the slots of its bonded terms;
// kinetic energy of u + c F for the thermostat.
template <typename R>
__global__ void __launch_bounds__(kThreads) k_finish(FinishArgs<R> a) {
  R ke = R(0);
  bool bad = false;
  const bool with_out = a.with_out && !(a.host_call && no_outputs(a.st));
  if (a.host_call && blockIdx.x == 0 && threadIdx.x == 0) close_host_call(a.st);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < a.n) {
    const int t = a.type[i];
    R f[3];
    load_force(a.f_fg, i, f);
    if (a.with_cg && ((a.hyb_mask >> t) & 1)) {
      R g[3];
      load_force(a.f_cg, i, g);
      f[0] += g[0];
      f[1] += g[1];
      f[2] += g[2];
    }
    const int k1 = a.inc_off[i + 1];
    for (int k = a.inc_off[i]; k < k1; ++k) {
      const int item = a.inc[k];
      const int kind = (item >> 30) & 3, role = (item >> 28) & 3, term = item & 0x0fffffff;
      const int slot = kind == 0 ? 2 * term + role
                                 : (kind == 1 ? a.base1 + 3 * term + role : a.base2 + 4 * term + role);
      R g[3];
      load_force(a.tf, slot, g);
      f[0] += g[0];
      f[1] += g[1];
      f[2] += g[2];
    }
    bad = !(isfinite(f[0]) && isfinite(f[1]) && isfinite(f[2]));
    save_force(a.f_tot, i, f);
    if (with_out) {
      a.f_out[3 * i] = double(f[0]);
      a.f_out[3 * i + 1] = double(f[1]);
      a.f_out[3 * i + 2] = double(f[2]);
    }
    if (a.with_ke) {
      const R c = R(a.cdt[t]);
      R v2 = R(0);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const R v = vel_r(a.vel, 3 * i + q) + c * f[q];
        v2 += v * v;
      }
      ke = R(0.5 * a.mass[t] * kMvv2e) * v2;
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&a.st->flags, F_NONFINITE);
  if (a.with_ke) {
    double v[1] = {double(ke)};
    __shared__ double sh[kThreads / 32];
    block_sum<double, 1>(v, sh);
    if (threadIdx.x == 0) acc_add(a.acc + kAccKe, v[0]);
  }
}

// ---- fused bonded terms + force sum, one block per segment of whole molecules
// (at most kSegAtoms atoms that no bonded term crosses).  The block evaluates
// its segment's terms into shared-memory slots (one per atom of a term), then
// each thread sums one atom's pair forces and slots: the same arithmetic as
// k_bonded + k_finish without the global slot array.

template <typename R>
struct SegArgs {
  const int* seg;  // [n_seg][kSegRec]: atoms [a0, a1), the prototype's term ranges, its first atom
  BondedArgs B;
  const unsigned long long* xfx;
  Sc3<R> sc;
  float q0h, q0l, q1h, q1l, q2h, q2l;
  const ForceT<R>* f_fg;
  const ForceT<R>* f_cg;
  int with_cg;
  const int* type;
  int hyb_mask;
  const int* inc_off;
  const int* inc;
  const VelT<R>* vel;
  int with_ke;
  const double* cdt;
  const double* mass;
  ForceT<R>* f_tot;
  double* f_out;
  int with_out;
  int host_call;
  long long* acc;
  DevState* st;
};

template <typename R, bool EV>
__global__ void __launch_bounds__(kThreads) k_finish_seg(SegArgs<R> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  ForceT<R>* slot = reinterpret_cast<ForceT<R>*>(smem_raw);
  const int* g = a.seg + kSegRec * blockIdx.x;
  const int a0 = g[0], a1 = g[1], b0 = g[2], b1 = g[3], g0 = g[4], g1 = g[5], d0 = g[6], d1 = g[7], base = g[8];
  const int nb = b1 - b0, na = g1 - g0, nd = d1 - d0;
  const int base_a = 2 * nb, base_d = base_a + 3 * na;
  const Sc3<R> sc = a.sc;
  // the terms are the prototype's (atoms from `base`): shifted onto this segment
  const GPosOff xg{a.xfx, a0 - base};
  const bool with_out = a.with_out && !(a.host_call && no_outputs(a.st));
  if (a.host_call && blockIdx.x == 0 && threadIdx.x == 0) close_host_call(a.st);
  R e = R(0);
  for (int q = threadIdx.x; q < nb + na + nd; q += blockDim.x) {
    if (q < nb) {
      R f[2][3];
      if constexpr (std::is_same<R, float>::value)
        e += bond_forces_ff(a.B, xg, ff{a.q0h, a.q0l}, ff{a.q1h, a.q1l}, ff{a.q2h, a.q2l}, a.B.bonds[b0 + q], f);
      else
        e += bond_forces(a.B, xg, sc, a.B.bonds[b0 + q], f);
      save_slots<2, R>(slot, 2 * size_t(q), f);
    } else if (q < nb + na) {
      const int u = q - nb;
      R f[3][3];
      if constexpr (std::is_same<R, float>::value)
        e += angle_forces_f32(a.B, xg, sc, a.B.angles[g0 + u], f);
      else
        e += angle_forces(a.B, xg, sc, a.B.angles[g0 + u], f);
      save_slots<3, R>(slot, base_a + 3 * size_t(u), f);
    } else {
      const int u = q - nb - na;
      R f[4][3];
      e += dihedral_forces<R>(a.B, xg, sc, d0 + u, f);
      save_slots<4, R>(slot, base_d + 4 * size_t(u), f);
    }
  }
  if (EV) {
    double v[1] = {double(e)};
    __shared__ double sh_e[kThreads / 32];
    block_sum<double, 1>(v, sh_e);
    if (threadIdx.x == 0) acc_add(a.acc + kAccEb, v[0]);
  }
  __syncthreads();
  R ke = R(0);
  bool bad = false;
  const int i = a0 + threadIdx.x;
  if (i < a1) {
    const int t = a.type[i];
    R f[3];
    load_force(a.f_fg, i, f);
    if (a.with_cg && ((a.hyb_mask >> t) & 1)) {
      R h[3];
      load_force(a.f_cg, i, h);
      f[0] += h[0];
      f[1] += h[1];
      f[2] += h[2];
    }
    const int ip = base + threadIdx.x;  // the prototype's atom: its incident terms
    const int k1 = a.inc_off[ip + 1];
    for (int k = a.inc_off[ip]; k < k1; ++k) {
      const int item = a.inc[k];
      const int kind = (item >> 30) & 3, role = (item >> 28) & 3, term = item & 0x0fffffff;
      const int s = kind == 0 ? 2 * (term - b0) + role
                              : (kind == 1 ? base_a + 3 * (term - g0) + role : base_d + 4 * (term - d0) + role);
      R h[3];
      load_force(slot, s, h);
      f[0] += h[0];
      f[1] += h[1];
      f[2] += h[2];
    }
    bad = !(isfinite(f[0]) && isfinite(f[1]) && isfinite(f[2]));
    save_force(a.f_tot, i, f);
    if (with_out) {
      a.f_out[3 * i] = double(f[0]);
      a.f_out[3 * i + 1] = double(f[1]);
      a.f_out[3 * i + 2] = double(f[2]);
    }
    if (a.with_ke) {
      const R c = R(a.cdt[t]);
      R v2 = R(0);
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const R v = vel_r(a.vel, 3 * i + q) + c * f[q];
        v2 += v * v;
      }
      ke = R(0.5 * a.mass[t] * kMvv2e) * v2;
    }
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&a.st->flags, F_NONFINITE);
  if (a.with_ke) {
    double v[1] = {double(ke)};
    __shared__ double sh_k[kThreads / 32];
    block_sum<double, 1>(v, sh_k);
    if (threadIdx.x == 0) acc_add(a.acc + kAccKe, v[0]);
  }
}

// ----------------------------------------------------------------- drift

template <typename R>
struct DriftArgs {
  int n;
  VelT<R>* vel;  // u, updated
  unsigned long long* xfx;
  const ForceT<R>* f_tot;
  const int* type;
  const double* cdt;
  const float2* cdt_ff;        // FP32 path
  double dts0, dts1, dts2;
  float dts0h, dts0l, dts1h, dts1l, dts2h, dts2l;  // FP32 path: dts as float-float
  Sc3<float> s32;
  const int* rank_fg;
  const int* rank_cg;
  int with_cg;
  int4* pos_fg;
  int4* pos_cg;
  int fp64;
  Pos64* pos_fg64;
  Pos64* pos_cg64;
  const int4* ref;
  float thr2;
  const int4* ref_p;  // positions at the last pruning pass (read if prune)
  float thr2_p;
  int prune;
  int thermo_every;
  DevState* st;
};

// The inputs of one atom's drift that the force sum of the step does not
// write (the drift kernel loads them before waiting for that kernel).
template <typename R>
struct DriftIn {
  int t, sf, sc;
  VelT<R> v[3];
  unsigned long long x0[3];
  int4 ref, ref_p;
};

template <typename R>
__device__ __forceinline__ void drift_load(const DriftArgs<R>& a, int i, DriftIn<R>& in) {
  in.t = a.type[i];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    in.v[q] = a.vel[3 * i + q];
    in.x0[q] = a.xfx[3 * i + q];
  }
  in.sf = a.rank_fg[i];
  in.sc = a.with_cg ? a.rank_cg[i] : -1;
  in.ref = a.ref[i];
  in.ref_p = a.prune ? a.ref_p[i] : make_int4(0, 0, 0, 0);
}

// One atom of the drift: u <- a u + b c F, x <- x + dt u, the sorted copies
// of x, and the two displacement triggers.  Returns the new position in x.
// Every load of the atom is issued before its first store, so that no load
// waits behind a store to memory the compiler cannot tell apart from it.
template <typename R>
__device__ __forceinline__ void drift_rest(const DriftArgs<R>& a, int i, const DriftIn<R>& in,
                                           unsigned long long x[3], bool& rebuild, bool& reprune) {
  const int t = in.t;
  R f[3];
  load_force(a.f_tot, i, f);
  const VelT<R>* v = in.v;
  const unsigned long long* x0 = in.x0;
  const int sf = in.sf, sc = in.sc;
  const int4 ref = in.ref, ref_p = in.ref_p;
  VelT<R> un[3];
  if constexpr (std::is_same<R, float>::value) {
    // float-float: u <- a u + b c F and the increment u dt 2^64 / L, with no
    // FP64 instruction (FP64 runs at a small fraction of the FP32 rate here)
    const ff ca{a.st->a_hi, a.st->a_lo}, cb{a.st->b_hi, a.st->b_lo};
    const float2 cc = a.cdt_ff[t];
    const ff bc = ff_mul(cb, ff{cc.x, cc.y});
    const ff dts[3] = {ff{a.dts0h, a.dts0l}, ff{a.dts1h, a.dts1l}, ff{a.dts2h, a.dts2l}};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const ff u = ff_add(ff_mul(ca, ff{v[q].x, v[q].y}), ff_mul_f(bc, f[q]));
      un[q] = make_float2(u.hi, u.lo);
      x[q] = x0[q] + (unsigned long long)ff2ll(ff_mul(u, dts[q]));
    }
  } else {
    const double ca = a.st->a, cb = a.st->b;
    const R bc = R(cb * a.cdt[t]);
    const double dts[3] = {a.dts0, a.dts1, a.dts2};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      // the kick increment in the force's precision, accumulated in FP64
      const double u = fma(ca, v[q], double(bc * f[q]));
      un[q] = u;
      x[q] = x0[q] + (unsigned long long)__double2ll_rn(u * dts[q]);
    }
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    a.vel[3 * i + q] = un[q];
    a.xfx[3 * i + q] = x[q];
  }
  scatter_sorted_at(sf, sc, t, x[0], x[1], x[2], a.pos_fg, a.pos_cg, a.fp64, a.pos_fg64, a.pos_cg64);
  rebuild = moved_beyond(ref, x[0], x[1], x[2], a.s32, a.thr2);
  if (a.prune) reprune = moved_beyond(ref_p, x[0], x[1], x[2], a.s32, a.thr2_p);
}

template <typename R>
__device__ __forceinline__ void drift_atom(const DriftArgs<R>& a, int i, unsigned long long x[3], bool& rebuild,
                                           bool& reprune) {
  DriftIn<R> in;
  drift_load(a, i, in);
  drift_rest(a, i, in, x, rebuild, reprune);
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_drift(DriftArgs<R> a) {
  if (blockIdx.x == 0 && threadIdx.x == 0)
    a.st->ev = a.thermo_every > 0 && ((a.st->local_step + 1) % a.thermo_every) == 0;
  bool rebuild = false, reprune = false;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < a.n) {
    unsigned long long x[3];
    drift_atom(a, i, x, rebuild, reprune);
  }
  if (__syncthreads_or(rebuild) && threadIdx.x == 0) atomicOr(&a.st->flags, F_REBUILD);
  if (__syncthreads_or(reprune) && threadIdx.x == 0) atomicOr(&a.st->flags, F_PRUNE);
}

// ---- drift + bonded terms, one block per segment of whole molecules: the
// block drifts its atoms (same arithmetic as k_drift), keeps their new
// positions in shared memory, evaluates the segment's bonded terms from there
// into shared-memory slots (same arithmetic as k_finish_seg) and writes each
// atom's bonded force (its slots summed in incident-term order).  The bonded
// forces of the new positions are thus ready before the pair kernel runs, and
// k_sum only adds the three parts.

template <typename R>
struct DriftSegArgs {
  DriftArgs<R> d;
  const int* seg;  // [n_seg][kSegRec]: atoms [a0, a1), the prototype's term ranges, its first atom
  BondedArgs B;
  Sc3<R> sc;
  float q0h, q0l, q1h, q1l, q2h, q2l;
  const int* inc_off;
  const int* inc;
  ForceT<R>* f_bond;  // caller order
  long long* acc;
  int seg_atoms;  // atoms of the largest segment
};

// shared memory of a segment's positions (the term slots follow, 16-byte aligned)
__host__ __device__ __forceinline__ size_t seg_pos_bytes(int atoms) {
  return (sizeof(unsigned long long) * 3 * size_t(atoms) + 15) / 16 * 16;
}

// The work of block `bid` (segment bid) of one system's drift launch.
template <typename R, bool EV>
__device__ __forceinline__ void drift_seg_block(const DriftSegArgs<R>& a, int bid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  unsigned long long* sx = reinterpret_cast<unsigned long long*>(smem_raw);  // [seg_atoms][3], then the term slots
  ForceT<R>* slot = reinterpret_cast<ForceT<R>*>(smem_raw + seg_pos_bytes(a.seg_atoms));
  const int* g = a.seg + kSegRec * bid;
  const int a0 = g[0], a1 = g[1], b0 = g[2], b1 = g[3], g0 = g[4], g1 = g[5], d0 = g[6], d1 = g[7], base = g[8];
  const int nb = b1 - b0, na = g1 - g0, nd = d1 - d0;
  const int base_a = 2 * nb, base_d = base_a + 3 * na;
  const int i = a0 + threadIdx.x;
  const int ip = base + threadIdx.x;  // the prototype's atom (its incident terms)
  // loads that do not depend on the drift, issued before it: the records of
  // this thread's first two bond/angle terms and its atom's incident-term range
  const int q0 = threadIdx.x, q1 = threadIdx.x + blockDim.x;
  const int4 rec0 = q0 < nb ? a.B.bonds[b0 + q0] : (q0 < nb + na ? a.B.angles[g0 + q0 - nb] : make_int4(0, 0, 0, 0));
  const int4 rec1 = q1 < nb ? a.B.bonds[b0 + q1] : (q1 < nb + na ? a.B.angles[g0 + q1 - nb] : make_int4(0, 0, 0, 0));
  const int e0 = i < a1 ? a.inc_off[ip] : 0, e1 = i < a1 ? a.inc_off[ip + 1] : 0;
  DriftIn<R> in;
  if (i < a1) drift_load(a.d, i, in);
  // launched as a programmatic dependent of the force sum: everything above
  // was written before that kernel started; the total force, the thermostat
  // factor and the step counter are read after it has finished
  grid_dependency_wait();
  if (bid == 0 && threadIdx.x == 0)
    a.d.st->ev = a.d.thermo_every > 0 && ((a.d.st->local_step + 1) % a.d.thermo_every) == 0;
  bool rebuild = false, reprune = false;
  if (i < a1) {
    unsigned long long x[3];
    drift_rest(a.d, i, in, x, rebuild, reprune);
#pragma unroll
    for (int q = 0; q < 3; ++q) sx[3 * threadIdx.x + q] = x[q];
  }
  if (__any_sync(0xffffffffu, rebuild || reprune)) {
    const unsigned f = (__any_sync(0xffffffffu, rebuild) ? F_REBUILD : 0u) | (__any_sync(0xffffffffu, reprune) ? F_PRUNE : 0u);
    if ((threadIdx.x & 31) == 0) atomicOr(&a.d.st->flags, f);
  }
  __syncthreads();
  // bonded terms of the segment from the new positions (the records name the
  // prototype's atoms, base .. base + a1 - a0 - 1: the same local indices)
  const SPos xs{sx, base};
  const Sc3<R> sc = a.sc;
  R e = R(0);
  for (int q = threadIdx.x, r = 0; q < nb + na + nd; q += blockDim.x, ++r) {
    if (q < nb) {
      const int4 rc = r == 0 ? rec0 : (r == 1 ? rec1 : a.B.bonds[b0 + q]);
      R f[2][3];
      if constexpr (std::is_same<R, float>::value)
        e += bond_forces_ff(a.B, xs, ff{a.q0h, a.q0l}, ff{a.q1h, a.q1l}, ff{a.q2h, a.q2l}, rc, f);
      else
        e += bond_forces(a.B, xs, sc, rc, f);
      save_slots<2, R>(slot, 2 * size_t(q), f);
    } else if (q < nb + na) {
      const int u = q - nb;
      const int4 rc = r == 0 ? rec0 : (r == 1 ? rec1 : a.B.angles[g0 + u]);
      R f[3][3];
      if constexpr (std::is_same<R, float>::value)
        e += angle_forces_f32(a.B, xs, sc, rc, f);
      else
        e += angle_forces(a.B, xs, sc, rc, f);
      save_slots<3, R>(slot, base_a + 3 * size_t(u), f);
    } else {
      const int u = q - nb - na;
      R f[4][3];
      e += dihedral_forces<R>(a.B, xs, sc, d0 + u, f);
      save_slots<4, R>(slot, base_d + 4 * size_t(u), f);
    }
  }
  if (EV) {
    double v[1] = {double(e)};
    __shared__ double sh_e[kThreads / 32];
    block_sum<double, 1>(v, sh_e);
    if (threadIdx.x == 0) acc_add(a.acc + kAccEb, v[0]);
  }
  __syncthreads();
  if (i < a1) {
    R f[3] = {R(0), R(0), R(0)};
    for (int k = e0; k < e1; ++k) {
      const int item = a.inc[k];
      const int kind = (item >> 30) & 3, role = (item >> 28) & 3, term = item & 0x0fffffff;
      const int s = kind == 0 ? 2 * (term - b0) + role
                              : (kind == 1 ? base_a + 3 * (term - g0) + role : base_d + 4 * (term - d0) + role);
      R h[3];
      load_force(slot, s, h);
      f[0] += h[0];
      f[1] += h[1];
      f[2] += h[2];
    }
    save_force(a.f_bond, i, f);
  }
}

template <typename R, bool EV>
__global__ void __launch_bounds__(kSegAtoms, std::is_same<R, float>::value ? 5 * kThreads / kSegAtoms : 1)
    k_drift_seg(DriftSegArgs<R> a) {
  drift_seg_block<R, EV>(a, blockIdx.x);
}

// Batches: one launch over the segments of every replica (see k_pair_batch).
template <typename R, bool EV>
__global__ void __launch_bounds__(kSegAtoms, std::is_same<R, float>::value ? 5 * kThreads / kSegAtoms : 1)
    k_drift_seg_batch(const DriftSegArgs<R>* __restrict__ args, const int* __restrict__ off, int nrep) {
  const int r = batch_replica(off, nrep, blockIdx.x);
  drift_seg_block<R, EV>(args[r], int(blockIdx.x) - off[r]);
}

// ----------------------------------------------------------------- thermostat

// splitmix64 (Steele, Lea & Flood 2014) as a counter-based generator: the
// (c+1)-th output of the sequence started at `key`.
__device__ __forceinline__ unsigned long long mix64(unsigned long long key, unsigned long long c) {
  unsigned long long z = key + (c + 1ull) * 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__device__ __forceinline__ double uniform01(unsigned long long key, unsigned long long& c) {
  // (0, 1]: top 53 bits plus one ulp
  return (double(mix64(key, c++) >> 11) + 1.0) * 1.1102230246251565e-16;
}
__device__ double gauss(unsigned long long key, unsigned long long& c) {
  const double u1 = uniform01(key, c), u2 = uniform01(key, c);
  return sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
}
// Bussi-Donadio-Parrinello (2007) velocity rescaling.  The two random
// numbers of step `step` (a normal deviate r1 and a chi-square deviate s with
// n_f - 1 degrees of freedom, drawn as twice a gamma(n_f/2 - 1/2) deviate by
// Marsaglia & Tsang (2000): d = shape - 1/3, k = 1 / sqrt(9 d), from the host)
// depend only on the seed and the step, so a block of steps has them drawn
// in parallel ahead of time.  Four lanes of a warp share a step: the normal
// deviates of r1 and of the gamma deviate's first trial and the logarithm of
// its acceptance test are formed side by side (counters 0-1, 2-3 and 4 of the
// step), each lane ends with both numbers, and a rejected trial (one in a
// thousand and less) goes on serially.
__device__ void csvr_draws(double d, double k, unsigned long long seed, unsigned long long step, double& r1,
                           double& s) {
  const int lane = threadIdx.x & 31, j = lane & 3, base = lane & ~3;
  const unsigned long long c0 = step << 20;
  unsigned long long c = c0 + (j == 0 ? 0 : (j == 1 ? 2 : 4));
  const double u1 = uniform01(seed, c), u2 = uniform01(seed, c);
  const double lu = log(u1);
  const double g = sqrt(-2.0 * lu) * cos(6.283185307179586 * u2);
  r1 = __shfl_sync(0xffffffffu, g, base);
  double x = __shfl_sync(0xffffffffu, g, base + 1);
  double lt = __shfl_sync(0xffffffffu, lu, base + 2);
  c = c0 + 4;
  for (int it = 0; it < 1000; ++it) {
    if (it > 0) x = gauss(seed, c);
    double v = 1.0 + k * x;
    if (v <= 0.0) continue;
    v = v * v * v;
    if (it > 0)
      lt = log(uniform01(seed, c));
    else
      ++c;
    if (lt < 0.5 * x * x + d - d * v + d * log(v)) {
      s = 2.0 * (d * v);
      return;
    }
  }
  s = 2.0 * d;
}
// With e = exp(-dt / tau) (computed once per call on the host) the rescaled
// kinetic energy is K' = e K + A + B sqrt(K), where A and B hold the random
// numbers and the target; they are formed with the draws, so the end of a step
// (one thread, on the critical path of every step) is left with alpha = sqrt(K' / K) = sqrt(e + (A / sqrt K + B) / sqrt K).
__device__ __forceinline__ double csvr_alpha(double ke, double e, double ca, double cb) {
  const float kf = float(ke);
  if (kf > 1e-30f && kf < 1e30f) {
    const double rk = rsqrt_d(ke, kf);
    const double x = fma(fma(ca, rk, cb), rk, e);
    if (x > 1e-30) return x * rsqrt_d(x, float(x));
    return sqrt(x);
  }
  return sqrt(e + (ca + cb * sqrt(ke)) / ke);
}

// Start of a block of steps: the rollback snapshot of positions, velocity
// state, forces and DevState, and beside it (the first blocks) the thermostat
// terms (A, B) of the steps st->step + k, k < count, 32 steps to a block.  6.2
// us at 140 000 atoms (9.8 with one thread a step for the draws; 18 as four
// copies and a launch).
struct BlockStart {
  const unsigned long long* src[3];
  unsigned long long* dst[3];
  long long words[3];  // 8-byte words
  const DevState* st;
  DevState* snap;
  double gd, gk;         // gamma deviate (csvr_draws)
  double scale_a, scale_b;  // A = scale_a (r1^2 + s), B = scale_b r1
  unsigned long long seed;
  int count;   // 0: no thermostat
  int ndraw;   // blocks that draw (at least one: it copies DevState)
  double* draws;
};

__device__ __forceinline__ void copy_words64(unsigned long long* dst, const unsigned long long* src, long long n,
                                             long long first, long long stride) {
  if (((reinterpret_cast<size_t>(src) | reinterpret_cast<size_t>(dst)) & 15) == 0) {
    const ulonglong2* s2 = reinterpret_cast<const ulonglong2*>(src);
    ulonglong2* d2 = reinterpret_cast<ulonglong2*>(dst);
    for (long long k = first; k < n / 2; k += stride) d2[k] = s2[k];
    if ((n & 1) && first == 0) dst[n - 1] = src[n - 1];
  } else {
    for (long long k = first; k < n; k += stride) dst[k] = src[k];
  }
}

constexpr int kDrawSteps = 32;  // steps per drawing block, four lanes each

__device__ __forceinline__ void block_start(const BlockStart& a, int bid, int nblk) {
  if (bid < a.ndraw) {
    constexpr int kWords = int(sizeof(DevState) / 8);
    static_assert(sizeof(DevState) % 8 == 0 && 4 * kDrawSteps <= kThreads, "whole words, one block");
    if (bid == 0)
      for (int w = threadIdx.x; w < kWords; w += kThreads)
        reinterpret_cast<unsigned long long*>(a.snap)[w] = reinterpret_cast<const unsigned long long*>(a.st)[w];
    const int k = kDrawSteps * bid + int(threadIdx.x >> 2);
    if (a.count == 0 || threadIdx.x >= 4 * kDrawSteps) return;  // whole warps
    double r1, s;
    csvr_draws(a.gd, a.gk, a.seed, a.st->step + (unsigned long long)k, r1, s);
    if (k >= a.count || (threadIdx.x & 3) != 0) return;
    a.draws[2 * k] = a.scale_a * (r1 * r1 + s);
    a.draws[2 * k + 1] = 2.0 * r1 * a.scale_b;
    return;
  }
  const long long first = (long long)(bid - a.ndraw) * kThreads + threadIdx.x,
                  stride = (long long)(nblk - a.ndraw) * kThreads;
#pragma unroll
  for (int q = 0; q < 3; ++q) copy_words64(a.dst[q], a.src[q], a.words[q], first, stride);
}

__global__ void __launch_bounds__(kThreads) k_block_start(const __grid_constant__ BlockStart a) {
  block_start(a, blockIdx.x, gridDim.x);
}
__global__ void __launch_bounds__(kThreads) k_block_start_batch(const BlockStart* __restrict__ args) {
  block_start(args[blockIdx.x], blockIdx.y, gridDim.y);
}

// total of an accumulator and the finer one beside it
__device__ __forceinline__ double acc_value(long long hi, long long fine) {
  return (double(hi) + double(fine) / kFixFine) / kFix;
}

// End of a step (one thread): thermostat factor from the kinetic energy,
// thermo row on energy steps, counters, and the accumulators cleared for the
// next step.  ca, cb: this step's thermostat terms (k_block_start).  The accumulators are read
// through volatile loads (other blocks of the calling kernel added to them).
__device__ void end_of_step(volatile long long* acc, const StepParams& sp, DevState* st, double ca, double cb) {
  const bool ev = st->ev != 0;
  const double ke = double(acc[kAccKe]) / kFix;
  double alpha = 1.0;
  if (sp.t_target > 0.0 && ke > 0.0) alpha = csvr_alpha(ke, sp.csvr_e, ca, cb);
  st->alpha = alpha;
  st->a = alpha;
  st->b = alpha + 1.0;
  st->a_hi = float(alpha);
  st->a_lo = float(alpha - double(st->a_hi));
  st->b_hi = float(alpha + 1.0);
  st->b_lo = float((alpha + 1.0) - double(st->b_hi));
  double* thermo = sp.thermo;
  if (ev && sp.thermo_every > 0) {
    double* row = thermo + (size_t)st->thermo_row * RELRES_THERMO_COLS;
    row[0] = acc_value(acc[kAccFg], acc[kNAcc + kAccFg]);
    row[1] = acc_value(acc[kAccCg], acc[kNAcc + kAccCg]);
    row[2] = double(acc[kAccEb]) / kFix;
    row[3] = ke * alpha * alpha;
#pragma unroll
    for (int q = 1; q < kNQ; ++q)
      row[3 + q] = acc_value(acc[kAccFg + q] + acc[kAccCg + q], acc[kNAcc + kAccFg + q] + acc[kNAcc + kAccCg + q]);
    st->thermo_row += 1;
  }
#pragma unroll
  for (int q = 0; q < (ev ? kNAccAll : kNAcc); ++q) acc[q] = 0;
  st->local_step += 1;
  st->step += 1;
  if (st->flags & F_REBUILD) {
    st->n_builds += 1;
    st->flags &= ~F_REBUILD;
  }
  st->flags &= ~F_PRUNE;  // a pruning pass ran this step if it was set
}

__global__ void k_thermo(long long* acc, StepParams sp, DevState* st, const double* draw) {
  end_of_step(acc, sp, st, sp.t_target > 0.0 ? draw[0] : 0.0, sp.t_target > 0.0 ? draw[1] : 0.0);
}

// ---- end of a step with bonded forces from k_drift_seg: per atom the total
// force F = F_FG + F_CG + F_bonded and the kinetic energy of u + c F; the last
// block to finish (a ticket counter after a memory fence) runs the thermostat
// and the step bookkeeping of k_thermo, so the step needs no separate launch.

template <typename R>
struct SumArgs {
  int n;
  const ForceT<R>* f_fg;
  const ForceT<R>* f_cg;
  int with_cg;
  const ForceT<R>* f_bond;
  const int* type;
  int hyb_mask;
  const VelT<R>* vel;
  const double* cdt;
  const float2* cdt_ff;
  const double* mass;
  const float* kec;
  ForceT<R>* f_tot;
  long long* acc;
  DevState* st;
  StepParams sp;
  const double* draw;
};

// The inputs of one atom of the force sum.
template <typename R>
struct SumIn {
  int t;
  R f[3], h[3], b[3];
  VelT<R> v[3];
};

template <typename R>
__device__ __forceinline__ void sum_load(const SumArgs<R>& a, int i, SumIn<R>& in) {
  in.t = a.type[i];
  load_force(a.f_fg, i, in.f);
  // the CG part is zero for ordinary atoms (never written): loaded without
  // waiting for the type, added only for hybrids
  if (a.with_cg) load_force(a.f_cg, i, in.h);
  load_force(a.f_bond, i, in.b);
#pragma unroll
  for (int q = 0; q < 3; ++q) in.v[q] = a.vel[3 * i + q];
}

// F = F_FG + F_CG + F_bonded of one atom, stored; returns the kinetic energy
// of u + c F.
template <typename R>
__device__ __forceinline__ R sum_atom(const SumArgs<R>& a, int i, SumIn<R>& in, bool& bad) {
  const int t = in.t;
  R* f = in.f;
  if (a.with_cg && ((a.hyb_mask >> t) & 1)) {
    f[0] += in.h[0];
    f[1] += in.h[1];
    f[2] += in.h[2];
  }
  f[0] += in.b[0];
  f[1] += in.b[1];
  f[2] += in.b[2];
  bad |= !(isfinite(f[0]) && isfinite(f[1]) && isfinite(f[2]));
  save_force(a.f_tot, i, f);
  R c, kc;
  if constexpr (std::is_same<R, float>::value) {
    c = a.cdt_ff[t].x;
    kc = a.kec[t];
  } else {
    c = a.cdt[t];
    kc = 0.5 * a.mass[t] * kMvv2e;
  }
  R v2 = R(0);
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const R v = vel_r(&in.v[q], 0) + c * f[q];
    v2 += v * v;
  }
  return kc * v2;
}

// grid-stride over the nblk blocks of one system (a few blocks per SM), one
// kinetic-energy atomic and one ticket per block; step k of the block of
// steps (its thermostat draws)
template <typename R>
__device__ __forceinline__ void sum_block(const SumArgs<R>& a, int bid, int nblk, int k) {
  // this step's thermostat draws, read early (the last block uses them)
  double ca = 0.0, cb = 0.0;
  if (threadIdx.x == 0 && a.sp.t_target > 0.0) {
    ca = a.draw[2 * k];
    cb = a.draw[2 * k + 1];
  }
  // launched as a programmatic dependent of the pair kernel: wait for its
  // forces, then let the next drift launch (its early loads read nothing that
  // this kernel or the pair kernel writes after this point)
  grid_dependency_wait();
  grid_dependents_launch();
  R ke = R(0);  // a few atoms per thread
  bool bad = false;
  const int stride = nblk * blockDim.x;
  int i = bid * blockDim.x + threadIdx.x;
  for (; i + stride < a.n; i += 2 * stride) {  // two atoms in flight: both loaded before either store
    SumIn<R> in0, in1;
    sum_load(a, i, in0);
    sum_load(a, i + stride, in1);
    const R k0 = sum_atom(a, i, in0, bad);
    const R k1 = sum_atom(a, i + stride, in1, bad);
    ke += k0 + k1;
  }
  if (i < a.n) {
    SumIn<R> in;
    sum_load(a, i, in);
    ke += sum_atom(a, i, in, bad);
  }
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(&a.st->flags, F_NONFINITE);
  double v[1] = {double(ke)};
  __shared__ double sh_k[kThreads / 32];
  block_sum<double, 1>(v, sh_k);
  if (threadIdx.x == 0) {
    acc_add(a.acc + kAccKe, v[0]);
    __threadfence();
    const unsigned ticket = atomicAdd(&a.st->done_blocks, 1u);
    if (ticket == unsigned(nblk - 1)) {
      __threadfence();
      a.st->done_blocks = 0u;
      end_of_step(a.acc, a.sp, a.st, ca, cb);
    }
  }
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_sum(SumArgs<R> a, int k) {
  sum_block<R>(a, blockIdx.x, gridDim.x, k);
}

// Batches: one launch over every replica (see k_pair_batch); replica r's
// blocks count their own tickets, so its last block runs its thermostat.
template <typename R>
__global__ void __launch_bounds__(kThreads) k_sum_batch(const SumArgs<R>* __restrict__ args,
                                                        const int* __restrict__ off, int nrep, int k) {
  const int r = batch_replica(off, nrep, blockIdx.x);
  sum_block<R>(args[r], int(blockIdx.x) - off[r], off[r + 1] - off[r], k);
}

// The state to the host's pinned copy, written by a kernel: a copy of these
// few words as a transfer of its own starts 5 us behind the kernel before it,
// this one follows like any launch.
__device__ __forceinline__ void post_state(const DevState* st, DevState* host) {
  for (int w = threadIdx.x; w < int(sizeof(DevState) / 8); w += 32)
    reinterpret_cast<unsigned long long*>(host)[w] = reinterpret_cast<const unsigned long long*>(st)[w];
}

// Energies and virial of relres_compute (one warp: lane 0 the energies, lanes
// 1-6 the virial), the accumulators cleared, and the state to the host.
__global__ void __launch_bounds__(32) k_reduce_out(long long* acc, double* energy, int with_e, double* virial,
                                                   int with_w, const DevState* st, DevState* host) {
  if (no_outputs(st)) with_e = with_w = 0;
  const int q = threadIdx.x;
  if (q == 0 && with_e) {
    const double efg = acc_value(acc[kAccFg], acc[kNAcc + kAccFg]), ecg = acc_value(acc[kAccCg], acc[kNAcc + kAccCg]);
    const double eb = double(acc[kAccEb]) / kFix;
    energy[0] = efg;
    energy[1] = ecg;
    energy[2] = eb;
    energy[3] = efg + ecg + eb;
  }
  if (q >= 1 && q < kNQ && with_w)
    virial[q - 1] =
        acc_value(acc[kAccFg + q] + acc[kAccCg + q], acc[kNAcc + kAccFg + q] + acc[kNAcc + kAccCg + q]);
  __syncwarp();
  for (int k = q; k < kNAccAll; k += 32) acc[k] = 0;
  post_state(st, host);
}

// Start of a relres_step call: the state (with the flags of k_check_io) to the
// host's pinned copy, then the call's step and thermo-row counters, empty
// accumulators, those flags cleared for the next call, and (unless the call
// continues the velocity state of the last one) the factors of the first drift
// for velocities read from the caller, u = v: a = b = 1.  One warp.
struct CallStart {
  DevState* st;
  DevState* host;
  long long* acc;
  int try_u;  // the velocity state continues if the arrays are the ones returned last
};

__device__ __forceinline__ void call_start(const CallStart& a) {
  post_state(a.st, a.host);
  for (int q = threadIdx.x; q < kNAccAll; q += 32) a.acc[q] = 0;
  __syncwarp();
  if (threadIdx.x != 0) return;
  DevState* const st = a.st;
  if (!a.try_u || (st->flags & (F_DIRTY | F_VDIRTY)) != 0u) {
    st->a = 1.0;
    st->b = 1.0;
    st->a_hi = 1.f;
    st->a_lo = 0.f;
    st->b_hi = 1.f;
    st->b_lo = 0.f;
  }
  st->local_step = 0;
  st->thermo_row = 0;
  st->ev = 0;
  st->flags &= ~unsigned(F_DIRTY | F_VDIRTY);
}

__global__ void __launch_bounds__(32) k_call_start(const __grid_constant__ CallStart a) { call_start(a); }

__global__ void k_flags_and(DevState* st, unsigned keep) { atomicAnd(&st->flags, keep); }
__global__ void k_flags_or(DevState* st, unsigned set) { atomicOr(&st->flags, set); }

__global__ void __launch_bounds__(32) k_post_state(const DevState* st, DevState* host) { post_state(st, host); }

// end of a call that refreshed the lists, and the state to the host
__global__ void __launch_bounds__(32) k_close_call(DevState* st, DevState* host) {
  if (threadIdx.x == 0) close_host_call(st);
  __syncwarp();
  post_state(st, host);
}

// FP32 path: caller's FP64 velocities -> float-float state
__global__ void k_vel_in(int n3, const double* __restrict__ vel, float2* __restrict__ uff) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n3; k += gridDim.x * blockDim.x) {
    const double v = vel[k];
    const float hi = float(v);
    uff[k] = make_float2(hi, float(v - double(hi)));
  }
}

// force component q of atom i (k = 3 i + q)
__device__ __forceinline__ float force_component(const float4* f, int i, int q, int) {
  return reinterpret_cast<const float*>(f + i)[q];
}
__device__ __forceinline__ double force_component(const double* f, int, int, int k) { return f[k]; }

// End of a call: positions and velocities to the caller, and copies of both.
// One component per thread, so that every array is read and written in whole
// lines: 7.4 us at 140 000 atoms (9.3 with an atom per thread), 37 us at a
// million, 60 % of the copy rate.
struct FinishMd {
  int n3;
  const DevState* st;
  const void* vel_u;  // VelT<R>
  const void* f_tot;  // ForceT<R>
  const int* type;
  const double* cdt;
  const float2* cdt_ff;
  const unsigned long long* xfx;
  BoxConsts b;
  double* vel_out;
  double* pos_out;
  double* pos_ret;
  double* vel_ret;
};

template <typename R>
__device__ __forceinline__ void finish_md(const FinishMd& a, int bid, int nblk) {
  const VelT<R>* vel_u = static_cast<const VelT<R>*>(a.vel_u);  // FP64: also written (vel_out)
  const ForceT<R>* __restrict__ f_tot = static_cast<const ForceT<R>*>(a.f_tot);
  const int* __restrict__ type = a.type;
  const unsigned long long* __restrict__ xfx = a.xfx;
  double* const vel_out = a.vel_out;
  double* const vel_ret = a.vel_ret;
  double* __restrict__ const pos_out = a.pos_out;
  double* __restrict__ const pos_ret = a.pos_ret;
  const ff ca{a.st->a_hi, a.st->a_lo}, cb1 = ff_add(ff{a.st->b_hi, a.st->b_lo}, ff{-1.f, 0.f});
  const double da = a.st->a, db1 = a.st->b - 1.0;
  for (int k = bid * kThreads + threadIdx.x; k < a.n3; k += nblk * kThreads) {
    const int i = k / 3, q = k - 3 * i;
    const int t = type[i];
    const R f = force_component(f_tot, i, q, k);
    const unsigned long long ux = xfx[k];
    double v;
    if constexpr (std::is_same<R, float>::value) {
      // v = a u + (b - 1) c F in float-float, returned as the double nearest
      // to hi + lo: the parts converted exactly with integer operations, one
      // FP64 addition
      const float2 cc = a.cdt_ff[t];
      const ff cbc = ff_mul(cb1, ff{cc.x, cc.y});
      const float2 u = vel_u[k];
      const ff w = ff_add(ff_mul(ca, ff{u.x, u.y}), ff_mul_f(cbc, f));
      v = double_of_float(w.hi) + double_of_float(w.lo);
    } else {
      v = fma(da, vel_d(vel_u, k), double(R(db1 * a.cdt[t]) * f));
    }
    const double x = q == 0 ? back_to_double(ux, a.b.l64_0, a.b.l0)
                            : (q == 1 ? back_to_double(ux, a.b.l64_1, a.b.l1) : back_to_double(ux, a.b.l64_2, a.b.l2));
    vel_out[k] = v;
    if (vel_ret) vel_ret[k] = v;
    pos_out[k] = x;
    if (pos_ret) pos_ret[k] = x;
  }
}

template <typename R>
__global__ void __launch_bounds__(kThreads) k_finish_md(const __grid_constant__ FinishMd a) {
  finish_md<R>(a, blockIdx.x, gridDim.x);
}

// Batches: the three kernels at a call's boundaries for every replica at once
// (blockIdx.x: no limit on their number in practice), from a table filled at
// the start of the call.
struct CallArgs {
  CheckIo check;
  CallStart start;
  FinishMd finish;
  int fp64;
};
__global__ void __launch_bounds__(kThreads) k_check_io_batch(const CallArgs* __restrict__ t) {
  check_io(t[blockIdx.x].check, blockIdx.y, gridDim.y);
}
__global__ void __launch_bounds__(32) k_call_start_batch(const CallArgs* __restrict__ t) {
  call_start(t[blockIdx.x].start);
}
__global__ void __launch_bounds__(32) k_post_state_batch(const CallArgs* __restrict__ t) {
  post_state(t[blockIdx.x].start.st, t[blockIdx.x].start.host);
}
__global__ void __launch_bounds__(kThreads) k_finish_md_batch(const CallArgs* __restrict__ t) {
  const CallArgs& a = t[blockIdx.x];
  if (a.fp64)
    finish_md<double>(a.finish, blockIdx.y, gridDim.y);
  else
    finish_md<float>(a.finish, blockIdx.y, gridDim.y);
}

// ----------------------------------------------------------------- launchers

static int grid_for(int n) {
  const int b = (n + kThreads - 1) / kThreads;
  return b < 1 ? 1 : (b > 152 * 16 ? 152 * 16 : b);
}

static float trigger_thr2(const relres_ctx* c) {
  double skin = c->prm.skin;
  if (c->has_cg && c->n_h > 0 && c->skin_cg < skin) skin = c->skin_cg;
  const double h = 0.5 * skin;
  return float(h * h);
}

// pruning trigger: half the pruning margin
static float prune_thr2(const relres_ctx* c) {
  const double h = 0.5 * c->prune_delta;
  return float(h * h);
}

static Sc3<float> s32_of(const relres_ctx* c) {
  return Sc3<float>{float(c->box[0] / 4294967296.0), float(c->box[1] / 4294967296.0),
                    float(c->box[2] / 4294967296.0)};
}

cudaError_t upload_type_consts(relres_ctx* c, double dt) {
  if (c->consts_dt == dt) return cudaSuccess;  // already there (reset by relres_set_topology)
  std::vector<float2> cff(size_t(c->n_types));
  std::vector<float> kec(size_t(c->n_types));
  for (int k = 0; k < c->n_types; ++k) {
    c->h_cdt[k] = 0.5 * dt / c->mass_by_type[k] * kFtm2v;
    float hi, lo;
    ff_split(c->h_cdt[k], &hi, &lo);
    cff[size_t(k)] = make_float2(hi, lo);
    kec[size_t(k)] = float(0.5 * c->mass_by_type[k] * kMvv2e);
  }
  cudaError_t e = cudaMemcpyAsync(c->d_cdt, c->h_cdt.data(), sizeof(double) * c->n_types, cudaMemcpyHostToDevice,
                                  c->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(c->d_cdt_ff, cff.data(), sizeof(float2) * c->n_types, cudaMemcpyHostToDevice, c->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(c->d_kec, kec.data(), sizeof(float) * c->n_types, cudaMemcpyHostToDevice, c->stream);
  // the host vectors must outlive the copies
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e == cudaSuccess) c->consts_dt = dt;
  return e;
}

cudaError_t launch_vel_in(relres_ctx* c, const double* d_vel) {
  if (c->fp64) return cudaSuccess;
  const int n3 = 3 * c->n;
  k_vel_in<<<std::max(1, std::min((n3 + kThreads - 1) / kThreads, 152 * 8)), kThreads, 0, c->stream>>>(
      n3, d_vel, c->d_uff);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

static Pos64* p64(relres_ctx* c, Pos64* p) { return c->fp64 ? p : static_cast<Pos64*>(c->d_dummy); }

cudaError_t launch_convert(relres_ctx* c, const double* d_pos) {
  const BoxConsts b = box_consts(c, 0.0);
  k_convert<<<grid_for(c->n), kThreads, 0, c->stream>>>(
      c->n, d_pos, c->d_type, c->d_xfx, b, c->have_lists ? 1 : 0, c->d_rank_fg, c->d_rank_cg,
      (c->has_cg && c->n_h > 0) ? 1 : 0, c->d_pos_fg, c->d_pos_cg, c->fp64 ? 1 : 0, p64(c, c->d_pos_fg64),
      p64(c, c->d_pos_cg64), c->d_ref, trigger_thr2(c), c->prune_on ? c->d_ref_p : c->d_ref, prune_thr2(c),
      c->prune_on ? 1 : 0, c->d_state, c->d_acc);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

static CheckIo check_args(relres_ctx* c, const StepParams& sp, const double* d_pos, const double* d_vel) {
  auto words = [](const double* p) { return reinterpret_cast<const unsigned long long*>(p); };
  return CheckIo{sp.cached ? 3 * c->n : 0, words(d_pos), words(c->d_pos_ret), sp.try_u ? words(d_vel) : nullptr,
                 words(c->d_vel_ret), c->d_state};
}
static CallStart start_args(relres_ctx* c, const StepParams& sp) {
  return CallStart{c->d_state, c->h_state, c->d_acc, sp.try_u ? 1 : 0};
}
static FinishMd finish_args(relres_ctx* c, double* d_pos, double* d_vel) {
  return FinishMd{3 * c->n, c->d_state, vel_state(c, d_vel), c->d_f_tot, c->d_type, c->d_cdt, c->d_cdt_ff, c->d_xfx,
                  box_consts(c, 0.0), d_vel, d_pos, c->d_pos_ret, c->fp64 ? nullptr : c->d_vel_ret};
}

cudaError_t launch_check_io(relres_ctx* c, const StepParams& sp, const double* d_pos, const double* d_vel) {
  k_check_io<<<std::max(1, std::min((3 * c->n + kThreads - 1) / kThreads, 152 * 8)), kThreads, 0, c->stream>>>(
      check_args(c, sp, d_pos, d_vel));
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t launch_call_start(relres_ctx* c, const StepParams& sp) {
  k_call_start<<<1, 32, 0, c->stream>>>(start_args(c, sp));
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

size_t call_table_bytes(int nrep) { return sizeof(CallArgs) * size_t(nrep); }

void fill_call_table(relres_ctx* const* cs, int nrep, const StepParams* sp, double* const* d_pos,
                     double* const* d_vel, void* host) {
  CallArgs* const t = static_cast<CallArgs*>(host);
  for (int r = 0; r < nrep; ++r) {
    t[r].check = check_args(cs[r], sp[r], d_pos[r], d_vel[r]);
    t[r].start = start_args(cs[r], sp[r]);
    t[r].finish = finish_args(cs[r], d_pos[r], d_vel[r]);
    t[r].fp64 = cs[r]->fp64 ? 1 : 0;
  }
}

cudaError_t launch_call_batch(cudaStream_t s, const void* table, relres_ctx* const* cs, int nrep, CallPhase phase) {
  const CallArgs* const t = static_cast<const CallArgs*>(table);
  int most = 1;
  for (int r = 0; r < nrep; ++r) most = std::max(most, cs[r]->n);
  // a component per thread of the largest replica, at most 16 blocks per SM in all
  const int nx = std::max(1, std::min((3 * most + kThreads - 1) / kThreads, 152 * 16 / nrep));
  if (phase == kCallCheck) k_check_io_batch<<<dim3(nrep, nx), kThreads, 0, s>>>(t);
  if (phase == kCallStart) k_call_start_batch<<<nrep, 32, 0, s>>>(t);
  if (phase == kCallStatus) k_post_state_batch<<<nrep, 32, 0, s>>>(t);
  if (phase == kCallFinish) k_finish_md_batch<<<dim3(nrep, nx), kThreads, 0, s>>>(t);
  for (int r = 0; r < nrep; ++r) RELRES_LAUNCHED(cs[r]);
  return cudaGetLastError();
}

static BondedArgs bonded_args(const relres_ctx* c) {
  return BondedArgs{c->d_bonds,     c->d_angles,    c->d_dihs,     c->d_dih_type, c->d_bond_par,
                    c->d_angle_par, c->d_dih_par,   c->d_bond_fpar, c->d_angle_fpar};
}


template <typename R>
static cudaError_t launch_bonded_t(relres_ctx* c, bool ev) {
  const int nt = c->n_bonds + c->n_angles + c->n_dih;
  if (nt == 0) return cudaSuccess;
  const double k = std::is_same<R, float>::value ? 4294967296.0 : 18446744073709551616.0;
  BondedKArgs<R> a{};
  a.nb = c->n_bonds;
  a.na = c->n_angles;
  a.nd = c->n_dih;
  a.B = bonded_args(c);
  a.xfx = c->d_xfx;
  a.sc = Sc3<R>{R(c->box[0] / k), R(c->box[1] / k), R(c->box[2] / k)};
  ff_split(c->box[0] / 18446744073709551616.0, &a.q0h, &a.q0l);
  ff_split(c->box[1] / 18446744073709551616.0, &a.q1h, &a.q1l);
  ff_split(c->box[2] / 18446744073709551616.0, &a.q2h, &a.q2l);
  a.tf = static_cast<ForceT<R>*>(c->d_tf);
  a.acc = c->d_acc;
  const int nblk = (nt + kThreads - 1) / kThreads;
  if (ev)
    k_bonded<R, true><<<nblk, kThreads, 0, c->stream>>>(a);
  else
    k_bonded<R, false><<<nblk, kThreads, 0, c->stream>>>(a);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

template <typename R>
static cudaError_t launch_finish_t(relres_ctx* c, double* d_forces_out, const double* vel, bool host_call) {
  const int with_cg = (c->has_cg && c->n_h > 0) ? 1 : 0;
  FinishArgs<R> a{c->n,
                  static_cast<const ForceT<R>*>(c->d_f_fg),
                  static_cast<const ForceT<R>*>(c->d_f_cg),
                  with_cg,
                  c->d_type,
                  c->hyb_mask,
                  c->d_inc_off,
                  c->d_inc,
                  static_cast<const ForceT<R>*>(c->d_tf),
                  2 * c->n_bonds,
                  2 * c->n_bonds + 3 * c->n_angles,
                  vel ? static_cast<const VelT<R>*>(vel_state(c, const_cast<double*>(vel)))
                      : static_cast<const VelT<R>*>(c->d_dummy),
                  vel ? 1 : 0,
                  c->d_cdt,
                  c->d_mass,
                  static_cast<ForceT<R>*>(c->d_f_tot),
                  d_forces_out ? d_forces_out : static_cast<double*>(c->d_dummy),
                  d_forces_out ? 1 : 0,
                  host_call ? 1 : 0,
                  c->d_acc,
                  c->d_state};
  k_finish<R><<<(c->n + kThreads - 1) / kThreads, kThreads, 0, c->stream>>>(a);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

template <typename R>
static cudaError_t launch_finish_seg_t(relres_ctx* c, bool ev, double* d_forces_out, const double* vel,
                                       bool host_call) {
  const double k = std::is_same<R, float>::value ? 4294967296.0 : 18446744073709551616.0;
  SegArgs<R> a{};
  a.seg = c->d_seg;
  a.B = bonded_args(c);
  a.xfx = c->d_xfx;
  a.sc = Sc3<R>{R(c->box[0] / k), R(c->box[1] / k), R(c->box[2] / k)};
  ff_split(c->box[0] / 18446744073709551616.0, &a.q0h, &a.q0l);
  ff_split(c->box[1] / 18446744073709551616.0, &a.q1h, &a.q1l);
  ff_split(c->box[2] / 18446744073709551616.0, &a.q2h, &a.q2l);
  a.f_fg = static_cast<const ForceT<R>*>(c->d_f_fg);
  a.f_cg = static_cast<const ForceT<R>*>(c->d_f_cg);
  a.with_cg = (c->has_cg && c->n_h > 0) ? 1 : 0;
  a.type = c->d_type;
  a.hyb_mask = c->hyb_mask;
  a.inc_off = c->d_inc_off;
  a.inc = c->d_inc;
  a.vel = vel ? static_cast<const VelT<R>*>(vel_state(c, const_cast<double*>(vel)))
              : static_cast<const VelT<R>*>(c->d_dummy);
  a.with_ke = vel ? 1 : 0;
  a.cdt = c->d_cdt;
  a.mass = c->d_mass;
  a.f_tot = static_cast<ForceT<R>*>(c->d_f_tot);
  a.f_out = d_forces_out ? d_forces_out : static_cast<double*>(c->d_dummy);
  a.with_out = d_forces_out ? 1 : 0;
  a.host_call = host_call ? 1 : 0;
  a.acc = c->d_acc;
  a.st = c->d_state;
  const size_t smem = size_t(c->seg_slots) * (std::is_same<R, float>::value ? 16 : 24);
  if (ev)
    k_finish_seg<R, true><<<c->n_seg, c->seg_block, smem, c->stream>>>(a);
  else
    k_finish_seg<R, false><<<c->n_seg, c->seg_block, smem, c->stream>>>(a);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t launch_finish(relres_ctx* c, bool ev, double* d_forces_out, const double* d_vel, bool host_call) {
  if (c->seg_ok && c->use_seg)
    return c->fp64 ? launch_finish_seg_t<double>(c, ev, d_forces_out, d_vel, host_call)
                   : launch_finish_seg_t<float>(c, ev, d_forces_out, d_vel, host_call);
  if (c->fp64) {
    const cudaError_t e = launch_bonded_t<double>(c, ev);
    return e != cudaSuccess ? e : launch_finish_t<double>(c, d_forces_out, d_vel, host_call);
  }
  const cudaError_t e = launch_bonded_t<float>(c, ev);
  return e != cudaSuccess ? e : launch_finish_t<float>(c, d_forces_out, d_vel, host_call);
}

cudaError_t launch_reduce_out(relres_ctx* c, double* d_energy, double* d_virial) {
  double* dd = static_cast<double*>(c->d_dummy);
  k_reduce_out<<<1, 32, 0, c->stream>>>(c->d_acc, d_energy ? d_energy : dd, d_energy ? 1 : 0,
                                        d_virial ? d_virial : dd, d_virial ? 1 : 0, c->d_state, c->h_state);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

static int block_start_draws(int count) { return std::max(1, (count + kDrawSteps - 1) / kDrawSteps); }
// blocks of a snapshot of n atoms: 8 words of each array per thread
static int block_start_copies(int n) { return std::max(1, std::min((3 * n / 8 + kThreads - 1) / kThreads, 152 * 8)); }

static BlockStart block_start_args(relres_ctx* c, const StepParams& sp, double* d_vel, int count) {
  BlockStart a{};
  const long long n3 = 3LL * c->n;
  a.src[0] = c->d_xfx;
  a.dst[0] = c->d_snap_x;
  a.src[1] = static_cast<const unsigned long long*>(vel_state(c, d_vel));
  a.dst[1] = reinterpret_cast<unsigned long long*>(c->d_snap_v);
  a.src[2] = static_cast<const unsigned long long*>(c->d_f_tot);
  a.dst[2] = static_cast<unsigned long long*>(c->d_snap_f);
  a.words[0] = a.words[1] = n3;
  a.words[2] = c->fp64 ? n3 : 2LL * c->n;
  a.st = c->d_state;
  a.snap = c->d_snap_state;
  const double unit = sp.kt / sp.n_f;
  a.gd = 0.5 * (sp.n_f - 1.0) - 1.0 / 3.0;
  a.gk = 1.0 / std::sqrt(9.0 * a.gd);
  a.scale_a = (1.0 - sp.csvr_e) * unit;
  a.scale_b = std::sqrt(sp.csvr_e * (1.0 - sp.csvr_e) * unit);
  a.seed = sp.seed;
  a.count = sp.t_target > 0.0 ? count : 0;
  a.ndraw = block_start_draws(count);
  a.draws = c->d_draws;
  return a;
}

cudaError_t launch_block_start(relres_ctx* c, const StepParams& sp, double* d_vel, int count) {
  k_block_start<<<block_start_draws(count) + block_start_copies(c->n), kThreads, 0, c->stream>>>(block_start_args(c, sp, d_vel, count));
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t prepare_block_start_batch(const std::vector<relres_ctx*>& cs, const std::vector<StepParams>& sp,
                                      double* const* d_vel, int count, BatchLaunch* b) {
  std::vector<BlockStart> args(cs.size());
  int copies = 1;
  for (size_t r = 0; r < cs.size(); ++r) {
    args[r] = block_start_args(cs[r], sp[r], d_vel[r], count);
    copies = std::max(copies, std::min(block_start_copies(cs[r]->n), 16));
  }
  b->nblk = block_start_draws(count) + copies;
  return upload_batch(b, args.data(), sizeof(BlockStart) * args.size(), {0, int(cs.size())});
}

cudaError_t launch_block_start_batch(cudaStream_t s, const BatchLaunch& b, int nrep) {
  k_block_start_batch<<<dim3(nrep, b.nblk), kThreads, 0, s>>>(static_cast<const BlockStart*>(b.d_args));
  return cudaGetLastError();
}

template <typename R>
static DriftArgs<R> drift_args(relres_ctx* c, const StepParams& sp, double* d_vel) {
  const bool cg = c->has_cg && c->n_h > 0;
  const BoxConsts b = box_consts(c, sp.dt);
  float h[6];
  ff_split(b.dts0, &h[0], &h[1]);
  ff_split(b.dts1, &h[2], &h[3]);
  ff_split(b.dts2, &h[4], &h[5]);
  return DriftArgs<R>{c->n,
                      static_cast<VelT<R>*>(vel_state(c, d_vel)),
                      c->d_xfx,
                      static_cast<const ForceT<R>*>(c->d_f_tot),
                      c->d_type,
                      c->d_cdt,
                      c->d_cdt_ff,
                      b.dts0,
                      b.dts1,
                      b.dts2,
                      h[0],
                      h[1],
                      h[2],
                      h[3],
                      h[4],
                      h[5],
                      s32_of(c),
                      c->d_rank_fg,
                      c->d_rank_cg,
                      cg ? 1 : 0,
                      c->d_pos_fg,
                      c->d_pos_cg,
                      c->fp64 ? 1 : 0,
                      p64(c, c->d_pos_fg64),
                      p64(c, c->d_pos_cg64),
                      c->d_ref,
                      trigger_thr2(c),
                      c->prune_on ? c->d_ref_p : c->d_ref,
                      prune_thr2(c),
                      c->prune_on ? 1 : 0,
                      sp.thermo_every,
                      c->d_state};
}

template <typename R>
static DriftSegArgs<R> drift_seg_args(relres_ctx* c, const StepParams& sp, double* d_vel) {
  const double k = std::is_same<R, float>::value ? 4294967296.0 : 18446744073709551616.0;
  DriftSegArgs<R> a{};
  a.d = drift_args<R>(c, sp, d_vel);
  a.seg = c->d_seg;
  a.B = bonded_args(c);
  a.sc = Sc3<R>{R(c->box[0] / k), R(c->box[1] / k), R(c->box[2] / k)};
  ff_split(c->box[0] / 18446744073709551616.0, &a.q0h, &a.q0l);
  ff_split(c->box[1] / 18446744073709551616.0, &a.q1h, &a.q1l);
  ff_split(c->box[2] / 18446744073709551616.0, &a.q2h, &a.q2l);
  a.inc_off = c->d_inc_off;
  a.inc = c->d_inc;
  a.f_bond = static_cast<ForceT<R>*>(c->d_f_bond);
  a.acc = c->d_acc;
  a.seg_atoms = c->seg_atoms;
  return a;
}

template <typename R>
static size_t drift_seg_smem(const relres_ctx* c) {
  return seg_pos_bytes(c->seg_atoms) + size_t(c->seg_slots) * (std::is_same<R, float>::value ? 16 : 24);
}

template <typename R>
static cudaError_t launch_drift_t(relres_ctx* c, const StepParams& sp, double* d_vel, bool ev, bool after_sum) {
  if (step_segments(c)) {
    const DriftSegArgs<R> a = drift_seg_args<R>(c, sp, d_vel);
    const size_t smem = drift_seg_smem<R>(c);
    // after the force sum of the previous step: overlap its tail
    const bool pdl = after_sum && pdl_ok(c);
    const cudaError_t e = ev ? launch_pdl(pdl, k_drift_seg<R, true>, c->n_seg, c->seg_block, smem, c->stream, a)
                             : launch_pdl(pdl, k_drift_seg<R, false>, c->n_seg, c->seg_block, smem, c->stream, a);
    if (e != cudaSuccess) return e;
  } else {
    k_drift<R><<<(c->n + kThreads - 1) / kThreads, kThreads, 0, c->stream>>>(drift_args<R>(c, sp, d_vel));
  }
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t launch_drift(relres_ctx* c, const StepParams& sp, double* d_vel, bool ev, bool after_sum) {
  return c->fp64 ? launch_drift_t<double>(c, sp, d_vel, ev, after_sum)
                 : launch_drift_t<float>(c, sp, d_vel, ev, after_sum);
}

// blocks of the force sum: one wave of resident blocks (56 registers a
// thread: four blocks per SM); batches give each replica the same blocks, so
// its kinetic-energy partial sums, and with them its trajectory, are the same
// bits as stepping it alone
static int sum_blocks(const relres_ctx* c) { return std::max(1, std::min((c->n + kThreads - 1) / kThreads, 152 * 4)); }

template <typename R>
static SumArgs<R> sum_args(relres_ctx* c, const StepParams& sp, const double* d_vel) {
  SumArgs<R> a{};
  a.n = c->n;
  a.f_fg = static_cast<const ForceT<R>*>(c->d_f_fg);
  a.f_cg = static_cast<const ForceT<R>*>(c->d_f_cg);
  a.with_cg = (c->has_cg && c->n_h > 0) ? 1 : 0;
  a.f_bond = static_cast<const ForceT<R>*>(c->d_f_bond);
  a.type = c->d_type;
  a.hyb_mask = c->hyb_mask;
  a.vel = static_cast<const VelT<R>*>(vel_state(c, const_cast<double*>(d_vel)));
  a.cdt = c->d_cdt;
  a.cdt_ff = c->d_cdt_ff;
  a.mass = c->d_mass;
  a.kec = c->d_kec;
  a.f_tot = static_cast<ForceT<R>*>(c->d_f_tot);
  a.acc = c->d_acc;
  a.st = c->d_state;
  a.sp = sp;
  if (a.sp.thermo == nullptr) {
    a.sp.thermo = static_cast<double*>(c->d_dummy);
    a.sp.thermo_every = 0;
  }
  a.draw = c->d_draws;
  return a;
}

template <typename R>
static cudaError_t launch_sum_t(relres_ctx* c, const StepParams& sp, int k, const double* d_vel) {
  const SumArgs<R> a = sum_args<R>(c, sp, d_vel);
  // after the pair kernel: overlap its tail
  const cudaError_t e = launch_pdl(pdl_ok(c), k_sum<R>, sum_blocks(c), kThreads, 0, c->stream, a, k);
  if (e != cudaSuccess) return e;
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t launch_end_of_step(relres_ctx* c, const StepParams& sp, int k, bool ev, double* d_vel) {
  if (step_segments(c))
    return c->fp64 ? launch_sum_t<double>(c, sp, k, d_vel) : launch_sum_t<float>(c, sp, k, d_vel);
  cudaError_t e = launch_finish(c, ev, nullptr, d_vel, false);
  return e != cudaSuccess ? e : launch_thermo(c, sp, k);
}

cudaError_t launch_thermo(relres_ctx* c, const StepParams& sp, int k) {
  StepParams q = sp;
  if (q.thermo == nullptr) {
    q.thermo = static_cast<double*>(c->d_dummy);
    q.thermo_every = 0;
  }
  k_thermo<<<1, 1, 0, c->stream>>>(c->d_acc, q, c->d_state, c->d_draws + 2 * k);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t launch_post_state(relres_ctx* c) {
  k_post_state<<<1, 32, 0, c->stream>>>(c->d_state, c->h_state);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t launch_flags_and(relres_ctx* c, unsigned keep) {
  k_flags_and<<<1, 1, 0, c->stream>>>(c->d_state, keep);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t launch_flags_or(relres_ctx* c, unsigned set) {
  k_flags_or<<<1, 1, 0, c->stream>>>(c->d_state, set);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

cudaError_t launch_close_call(relres_ctx* c) {
  k_close_call<<<1, 32, 0, c->stream>>>(c->d_state, c->h_state);
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

// ---- batches (relres_batch_step): argument tables of every replica
template <typename R>
static cudaError_t prepare_drift_batch_t(const std::vector<relres_ctx*>& cs, const std::vector<StepParams>& sp,
                                         double* const* d_vel, BatchLaunch* b) {
  std::vector<DriftSegArgs<R>> args(cs.size());
  std::vector<int> off(cs.size() + 1, 0);
  size_t smem = 0;
  int threads = 32;
  for (size_t r = 0; r < cs.size(); ++r) {
    args[r] = drift_seg_args<R>(cs[r], sp[r], d_vel[r]);
    off[r + 1] = off[r] + cs[r]->n_seg;
    smem = std::max(smem, drift_seg_smem<R>(cs[r]));
    threads = std::max(threads, cs[r]->seg_block);
  }
  b->nblk = off.back();
  b->threads = threads;
  b->smem = smem;
  return upload_batch(b, args.data(), sizeof(DriftSegArgs<R>) * args.size(), off);
}

cudaError_t prepare_drift_batch(const std::vector<relres_ctx*>& cs, const std::vector<StepParams>& sp,
                                double* const* d_vel, BatchLaunch* b) {
  return cs[0]->fp64 ? prepare_drift_batch_t<double>(cs, sp, d_vel, b) : prepare_drift_batch_t<float>(cs, sp, d_vel, b);
}

template <typename R>
static void launch_drift_batch_t(cudaStream_t s, bool ev, const BatchLaunch& b, int nrep) {
  const auto* args = static_cast<const DriftSegArgs<R>*>(b.d_args);
  if (ev)
    k_drift_seg_batch<R, true><<<b.nblk, b.threads, b.smem, s>>>(args, b.d_off, nrep);
  else
    k_drift_seg_batch<R, false><<<b.nblk, b.threads, b.smem, s>>>(args, b.d_off, nrep);
}

cudaError_t launch_drift_batch(cudaStream_t s, bool fp64, bool ev, const BatchLaunch& b, int nrep) {
  if (b.nblk == 0) return cudaSuccess;
  if (fp64)
    launch_drift_batch_t<double>(s, ev, b, nrep);
  else
    launch_drift_batch_t<float>(s, ev, b, nrep);
  return cudaGetLastError();
}

template <typename R>
static cudaError_t prepare_sum_batch_t(const std::vector<relres_ctx*>& cs, const std::vector<StepParams>& sp,
                                       double* const* d_vel, BatchLaunch* b) {
  std::vector<SumArgs<R>> args(cs.size());
  std::vector<int> off(cs.size() + 1, 0);
  for (size_t r = 0; r < cs.size(); ++r) {
    args[r] = sum_args<R>(cs[r], sp[r], d_vel[r]);
    off[r + 1] = off[r] + sum_blocks(cs[r]);
  }
  b->nblk = off.back();
  b->smem = 0;
  return upload_batch(b, args.data(), sizeof(SumArgs<R>) * args.size(), off);
}

cudaError_t prepare_sum_batch(const std::vector<relres_ctx*>& cs, const std::vector<StepParams>& sp,
                              double* const* d_vel, BatchLaunch* b) {
  return cs[0]->fp64 ? prepare_sum_batch_t<double>(cs, sp, d_vel, b) : prepare_sum_batch_t<float>(cs, sp, d_vel, b);
}

cudaError_t launch_sum_batch(cudaStream_t s, bool fp64, int k, const BatchLaunch& b, int nrep) {
  if (b.nblk == 0) return cudaSuccess;
  if (fp64)
    k_sum_batch<double><<<b.nblk, kThreads, 0, s>>>(static_cast<const SumArgs<double>*>(b.d_args), b.d_off, nrep, k);
  else
    k_sum_batch<float><<<b.nblk, kThreads, 0, s>>>(static_cast<const SumArgs<float>*>(b.d_args), b.d_off, nrep, k);
  return cudaGetLastError();
}

cudaError_t launch_write_back(relres_ctx* c, double* d_pos, double* d_vel) {
  if (c->fp64)
    k_finish_md<double><<<(3 * c->n + kThreads - 1) / kThreads, kThreads, 0, c->stream>>>(finish_args(c, d_pos, d_vel));
  else
    k_finish_md<float><<<(3 * c->n + kThreads - 1) / kThreads, kThreads, 0, c->stream>>>(finish_args(c, d_pos, d_vel));
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

}  // namespace relres
