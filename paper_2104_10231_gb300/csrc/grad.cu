// Backward pass of the RelRes pair interaction (the differentiable form of
// Eq. 20, Section 2.5): gradients of a scalar L(E, F) of the pair energy E
// and the pair forces F with respect to the positions and to the LJ
// parameters, given gE = dL/dE and g_i = dL/dF_i.
//
// Every smoothing coefficient (Eq. 17, Eq. 18) and shift (Eq. 19) is linear
// in the potential, so for each type pair and each part of the exact FG/CG
// split  u~ = C12 phi12(r) - C6 phi6(r)  with C12 = 4 eps sig^12,
// C6 = 4 eps sig^6 and phik the same construction applied to r^-k
// (BasisTab).  Hence
//   dL/dC12 = gE S12 + T12,   dL/dC6 = -(gE S6 + T6),
//   S_k = sum over pairs of phik(r),  T_k = sum_i g_i . sum_j (-phik'(r) rhat_ij),
//   dL/dx_i = gE sum_j u~'(r) rhat_ij - sum_j h_ij (g_i - g_j),
//   h_ij = u~''(r) rhat rhat^T + (u~'(r)/r) (I - rhat rhat^T)
// (the second term is the Hessian-vector product of E with g).  The C2
// smoothing of the paper makes u~'' well defined in every region.
//
// One launch walks both lists (CG blocks first) like the force kernel; the
// lists are those of the last force evaluation (nothing of the forward pass
// is stored besides them).  Per-type-pair sums are kept per thread (the atom's
// own type is fixed, the partner's type selects the accumulator), added per warp
// and pair of types, per block, and to FP64 totals with atomics.
#include "common.cuh"

namespace relres {

template <typename R>
using GVec = typename std::conditional<std::is_same<R, float>::value, float4, double>::type;
template <typename R>
using GPos = typename std::conditional<std::is_same<R, float>::value, int4, Pos64>::type;

__device__ __forceinline__ void ld3(const float4* a, int i, float v[3]) {
  const float4 q = a[i];
  v[0] = q.x;
  v[1] = q.y;
  v[2] = q.z;
}
__device__ __forceinline__ void ld3(const double* a, int i, double v[3]) {
  v[0] = a[3 * i];
  v[1] = a[3 * i + 1];
  v[2] = a[3 * i + 2];
}
__device__ __forceinline__ void st3(float4* a, int i, const float v[3]) { a[i] = make_float4(v[0], v[1], v[2], 0.f); }
__device__ __forceinline__ void st3(double* a, int i, const double v[3]) {
  a[3 * i] = v[0];
  a[3 * i + 1] = v[1];
  a[3 * i + 2] = v[2];
}
__device__ __forceinline__ int gtype(const int4& p) { return p.w; }
__device__ __forceinline__ int gtype(const Pos64& p) { return int(p.t); }

// f, f', f'' of the quartic Eq. 16 at d
template <typename R>
__device__ __forceinline__ void poly3(const R (&g)[5], R d, R& f, R& f1, R& f2) {
  f = (((g[4] * d + g[3]) * d + g[2]) * d + g[1]) * d + g[0];
  f1 = ((R(4) * g[4] * d + R(3) * g[3]) * d + R(2) * g[2]) * d + g[1];
  f2 = (R(12) * g[4] * d + R(6) * g[3]) * d + R(2) * g[2];
}

// One pair: difference vector, r, and the powers 1/r, r^-2, r^-12, r^-6.
template <typename R>
struct PairGeo {
  R d[3], r2, r, ri, r2i, v[2];
};

// phi, phi', phi'' of both bases (b = 0: r^-12, b = 1: r^-6) for one part.
template <typename R, bool CG>
__device__ __forceinline__ void basis(const BasisTab<R>& T, const PairGeo<R>& G, R (&p)[2], R (&p1)[2], R (&p2)[2]) {
  const R r = G.r, ri = G.ri, r2i = G.r2i;
  const R (&v)[2] = G.v;
  const R kk[2] = {R(12), R(6)};
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    if (!CG) {
      if (r < T.rsm) {
        p[b] = v[b] - T.fg_sh[b];
        p1[b] = -kk[b] * v[b] * ri;
        p2[b] = kk[b] * (kk[b] + R(1)) * v[b] * r2i;
      } else {
        poly3<R>(T.fg[b], r - T.rsm, p[b], p1[b], p2[b]);
        p[b] -= T.fg_sh[b];
      }
    } else {
      if (r < T.rsm) {
        p[b] = T.on[b][0] - T.gam[b];
        p1[b] = R(0);
        p2[b] = R(0);
      } else if (r < T.rsp) {
        poly3<R>(T.on[b], r - T.rsm, p[b], p1[b], p2[b]);
        p[b] -= T.gam[b];
      } else if (r < T.rcm) {
        p[b] = v[b] - T.gam[b];
        p1[b] = -kk[b] * v[b] * ri;
        p2[b] = kk[b] * (kk[b] + R(1)) * v[b] * r2i;
      } else {
        poly3<R>(T.off[b], r - T.rcm, p[b], p1[b], p2[b]);
        p[b] -= T.gam[b];
      }
    }
  }
}

template <typename R>
struct GradWalk {
  int nslots;
  const GPos<R>* pos;
  const int* nbr;
  const int* cnt;
  const int* perm;
  const GVec<R>* g;  // dL/dF in this list's slot order
  GVec<R>* gx;       // dL/dx of this list's part, caller order
};

template <typename R>
struct GradLaunch {
  int nblk_cg;
  GradWalk<R> fg, cg;
  const BasisTab<R>* tab;
  int nt;
  R sx, sy, sz;
  float sxl, syl, szl;  // FP32: lo parts of L / 2^32
  R g_energy;
  double* gc;  // [nt*nt][4]: dL/dC12_FG, dL/dC6_FG, dL/dC12_CG, dL/dC6_CG
  const unsigned* flags;  // F_NOLISTS: no walk
};

constexpr int kGradThreads = 128;

// a coordinate difference as hi + lo: the integer difference is hi + lo exactly,
// the scale's two parts leave 2^-47 of it
struct Split {
  float hi, lo;
};
__device__ __forceinline__ Split split_diff(int a, int b, float s, float sl) {
  const int d = int(unsigned(a) - unsigned(b));
  const float h = __int2float_rn(d), l = __int2float_rn(d - __float2int_rn(h));
  const float p = __fmul_rn(h, s);
  return Split{p, fmaf(l, s, fmaf(h, sl, fmaf(h, s, -p)))};
}
// The geometry of one pair.  FP32: the second derivative goes as r^-14, so the
// distance and its powers are formed as hi + lo from the exact integer
// differences and rounded once; FP32 all the way amplified the roundings of
// r^2 about sevenfold.
__device__ __forceinline__ void geometry(const int4& a, const int4& b, const GradLaunch<float>& L, PairGeo<float>& G) {
  const Split x = split_diff(a.x, b.x, L.sx, L.sxl), y = split_diff(a.y, b.y, L.sy, L.syl),
              z = split_diff(a.z, b.z, L.sz, L.szl);
  // the leading squares added without error, everything below them in FP32
  const float xx = __fmul_rn(x.hi, x.hi), yy = __fmul_rn(y.hi, y.hi), zz = __fmul_rn(z.hi, z.hi);
  const float low = fmaf(2.f * x.hi, x.lo, fmaf(x.hi, x.hi, -xx)) + fmaf(2.f * y.hi, y.lo, fmaf(y.hi, y.hi, -yy)) +
                    fmaf(2.f * z.hi, z.lo, fmaf(z.hi, z.hi, -zz));
  const ff s1 = ff_two_sum(xx, yy), s2 = ff_two_sum(s1.hi, zz);
  const float h = s2.hi, l = low + (s1.lo + s2.lo);
  G.d[0] = __fadd_rn(x.hi, x.lo);
  G.d[1] = __fadd_rn(y.hi, y.lo);
  G.d[2] = __fadd_rn(z.hi, z.lo);
  G.r2 = h;
  const float v = rcp_approx(h);
  const float e = fmaf(-l, v, fmaf(-h, v, 1.f)), ve = v * e;
  const ff i2 = ff_quick(v, fmaf(ve, e, ve));
  const ff i6 = ff_mul(ff_mul(i2, i2), i2);
  G.r2i = ff_val(i2);
  G.v[0] = ff_val(ff_mul(i6, i6));
  G.v[1] = ff_val(i6);
  const float q = rsqrtf(h);
  G.ri = fmaf(0.5f * q, fmaf(-l * q, q, fmaf(-h * q, q, 1.f)), q);
  G.r = fmaf(h, G.ri, l * G.ri);
}
__device__ __forceinline__ void geometry(const Pos64& a, const Pos64& b, const GradLaunch<double>& L,
                                         PairGeo<double>& G) {
  G.d[0] = dfix64(a.x, b.x, L.sx);
  G.d[1] = dfix64(a.y, b.y, L.sy);
  G.d[2] = dfix64(a.z, b.z, L.sz);
  G.r2 = G.d[0] * G.d[0] + G.d[1] * G.d[1] + G.d[2] * G.d[2];
  G.ri = rsqrt_d(G.r2, float(G.r2));
  G.r = G.r2 * G.ri;
  G.r2i = G.ri * G.ri;
  G.v[1] = G.r2i * G.r2i * G.r2i;
  G.v[0] = G.v[1] * G.v[1];
}

// running sums of the per-thread accumulators
__device__ __forceinline__ void add_to(ff& sum, float v) {
  const ff t = ff_two_sum(sum.hi, v);
  sum = ff{t.hi, __fadd_rn(sum.lo, t.lo)};
}
__device__ __forceinline__ void add_lane(ff& sum, int o) {
  const ff other{__shfl_xor_sync(0xffffffffu, sum.hi, o), __shfl_xor_sync(0xffffffffu, sum.lo, o)};
  add_to(sum, other.hi);
  sum.lo = __fadd_rn(sum.lo, other.lo);
}
__device__ __forceinline__ double total_of(ff sum) { return double(sum.hi) + double(sum.lo); }
__device__ __forceinline__ void add_to(double& sum, double v) { sum += v; }
__device__ __forceinline__ void add_lane(double& sum, int o) { sum += __shfl_xor_sync(0xffffffffu, sum, o); }
__device__ __forceinline__ double total_of(double sum) { return sum; }

// The accumulators of a warp's 32 threads (own type ti, -1 without a slot),
// added per pair of types: every lane takes one of the 2 nt^2 sums (several
// lanes one where there are fewer than 32) over the threads of its type, then
// one shared-memory FP64 atomic per sum.  With an atomic per slot and sum the
// lanes of a warp waited for one another at the few addresses: 81 us at 100 000
// atoms of two types where this takes 51, 120 of eight where this takes 78.
template <typename R>
__device__ __forceinline__ void add_type_sums(int ti, int nt, const R (*s_acc)[kGradThreads], int* s_type, double* s_gc) {
  using Sum = typename std::conditional<std::is_same<R, float>::value, ff, double>::type;
  const int lane = threadIdx.x & 31, first = threadIdx.x & ~31, nsum = 2 * nt * nt;
  const int share = nt == 1 ? 16 : (nt == 2 ? 4 : 1);  // lanes per sum
  s_type[threadIdx.x] = ti;
  __syncwarp();
  for (int k0 = 0; k0 < nsum; k0 += 32 / share) {
    const int k = k0 + lane / share, part = lane % share;
    const int t = k % (2 * nt), want = k / (2 * nt);  // accumulator, own type
    Sum sum{};
    if (k < nsum)
      for (int m = 0; m < 32; m += share) {
        const int j = first + ((m + part + t * share) & 31);  // (each accumulator from another bank)
        if (s_type[j] == want) add_to(sum, s_acc[t][j]);
      }
    for (int o = share / 2; o > 0; o >>= 1) add_lane(sum, o);
    if (k < nsum && part == 0) {
      const double v = total_of(sum);
      if (v != 0.0) atomicAdd(&s_gc[k], (t & 1) ? -v : v);
    }
  }
}

// One slot's walk, its list shared by T lanes (lane q takes chunks q, q + T,
// ...): with one thread per slot a launch lasts as long as one list's chain of
// loads, 77 us at 20 000 atoms.  The partner's type selects one of the
// thread's accumulators in shared memory (s_acc[2 t + b][thread]: C12 and C6
// sums of partner type t).
template <typename R, bool CG, int T>
__device__ __forceinline__ void grad_walk(const GradWalk<R>& W, int blk, const BasisTab<R>* tab,
                                          const GradLaunch<R>& a, double* s_gc, R (*s_acc)[kGradThreads], int* s_type) {
  const int s = (blk * kGradThreads + threadIdx.x) / T, q = threadIdx.x % T;
  const bool own = s < W.nslots;
  R gi[3] = {R(0), R(0), R(0)}, gx[3] = {R(0), R(0), R(0)};
  int ti = 0;
  for (int t = 0; t < 2 * a.nt; ++t) s_acc[t][threadIdx.x] = R(0);
  if (own) {
    const auto pi = W.pos[s];
    ti = gtype(pi);
    ld3(W.g, s, gi);
    const int m = W.cnt[s], nch = (m + 3) >> 2;
    const int4* nb4 = reinterpret_cast<const int4*>(W.nbr) + s;
    int4 jj = make_int4(s, s, s, s);
    if (q < nch) jj = nb4[size_t(q) * W.nslots];
    for (int ch = q; ch < nch; ch += T) {
      int4 jn = jj;
      if (ch + T < nch) jn = nb4[size_t(ch + T) * W.nslots];
      const int rem = m - 4 * ch;  // >= 1
      const int j[4] = {jj.x, rem > 1 ? jj.y : s, rem > 2 ? jj.z : s, rem > 3 ? jj.w : s};
      GPos<R> pj[4];
      R gj[4][3];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        pj[e] = W.pos[j[e]];
        ld3(W.g, j[e], gj[e]);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int tj = gtype(pj[e]);
        const BasisTab<R>& B = tab[ti * a.nt + tj];
        PairGeo<R> G;
        geometry(pi, pj[e], a, G);
        const R rcut = CG ? B.rcp : B.rsp;
        if (!(rem > e && G.r2 < rcut * rcut)) continue;
        const R ri = G.ri;
        R p[2], p1[2], p2[2];
        basis<R, CG>(B, G, p, p1, p2);
        const R c12 = CG ? B.c12c : B.c12f, c6 = CG ? B.c6c : B.c6f;
        const R u1 = c12 * p1[0] - c6 * p1[1];
        const R u2 = c12 * p2[0] - c6 * p2[1];
        R rh[3], w[3];
        R rw = R(0), gir = R(0);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          rh[c] = G.d[c] * ri;
          w[c] = gi[c] - gj[e][c];
          rw += rh[c] * w[c];
          gir += gi[c] * rh[c];
        }
#pragma unroll
        for (int c = 0; c < 3; ++c)
          gx[c] += a.g_energy * u1 * rh[c] - (u2 * rw * rh[c] + u1 * ri * (w[c] - rw * rh[c]));
        s_acc[2 * tj][threadIdx.x] += R(0.5) * a.g_energy * p[0] - p1[0] * gir;
        s_acc[2 * tj + 1][threadIdx.x] += R(0.5) * a.g_energy * p[1] - p1[1] * gir;
      }
      jj = jn;
    }
  }
  // the slot's lanes together (T divides 32: whole slots per warp)
#pragma unroll
  for (int o = T / 2; o > 0; o >>= 1)
#pragma unroll
    for (int c = 0; c < 3; ++c) gx[c] += __shfl_xor_sync(0xffffffffu, gx[c], o);
  if (own && q == 0) st3(W.gx, W.perm[s], gx);
  add_type_sums(own ? ti : -1, a.nt, s_acc, s_type, s_gc);
}

// FP32: 80 registers a thread, six blocks per SM (us per launch at six / seven /
// eight: 16.0 / 16.5 / 18.0 at 20 000 atoms, 50.9 / 51.0 / 57.4 at 100 000);
// FP64: no bound (a bound of one block takes more registers than none)
template <typename R, int T>
__global__ void __launch_bounds__(kGradThreads, std::is_same<R, float>::value ? 6 : 0) k_pair_grad(GradLaunch<R> a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  if (*(volatile const unsigned*)a.flags & F_NOLISTS) return;
  __shared__ int s_type[kGradThreads];
  const int nrow = a.nt * a.nt;
  double* s_gc = reinterpret_cast<double*>(smem_raw);
  R(*s_acc)[kGradThreads] = reinterpret_cast<R(*)[kGradThreads]>(s_gc + 2 * nrow);
  BasisTab<R>* tab = reinterpret_cast<BasisTab<R>*>(s_acc + 2 * a.nt);
  {
    const int words = nrow * int(sizeof(BasisTab<R>) / sizeof(int));
    const int* src = reinterpret_cast<const int*>(a.tab);
    int* dst = reinterpret_cast<int*>(tab);
    for (int w = threadIdx.x; w < words; w += blockDim.x) dst[w] = src[w];
  }
  for (int q = threadIdx.x; q < 2 * nrow; q += blockDim.x) s_gc[q] = 0.0;
  __syncthreads();
  const bool cg = int(blockIdx.x) < a.nblk_cg;
  if (cg)
    grad_walk<R, true, T>(a.cg, blockIdx.x, tab, a, s_gc, s_acc, s_type);
  else
    grad_walk<R, false, T>(a.fg, blockIdx.x - a.nblk_cg, tab, a, s_gc, s_acc, s_type);
  __syncthreads();
  const int off = cg ? 2 : 0;
  for (int q = threadIdx.x; q < 2 * nrow; q += blockDim.x)
    if (s_gc[q] != 0.0) atomicAdd(&a.gc[(q >> 1) * 4 + off + (q & 1)], s_gc[q]);
}

// dL/dF (caller order, FP64) into the slot order of the FG list, then of the
// CG list (n_cg slots, 0 without one)
template <typename R>
__global__ void k_gather_g(int n_fg, int n_cg, const int* __restrict__ perm_fg, const int* __restrict__ perm_cg,
                           const double* __restrict__ g, GVec<R>* __restrict__ out_fg, GVec<R>* __restrict__ out_cg) {
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < n_fg + n_cg; k += gridDim.x * blockDim.x) {
    const int s = k < n_fg ? k : k - n_fg, i = (k < n_fg ? perm_fg : perm_cg)[s];
    const R v[3] = {R(g[3 * i]), R(g[3 * i + 1]), R(g[3 * i + 2])};
    st3(k < n_fg ? out_fg : out_cg, s, v);
  }
}

// dL/dx = FG part + CG part (hybrids), caller order, FP64 out
template <typename R>
__global__ void k_sum_gx(int n, const GVec<R>* __restrict__ gx_fg, const GVec<R>* __restrict__ gx_cg,
                         int with_cg, const DevState* st, double* __restrict__ out) {
  if (*(volatile const unsigned*)&st->flags & F_NOLISTS) return;  // the call fails: no output
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
    R a[3], b[3] = {R(0), R(0), R(0)};
    ld3(gx_fg, i, a);
    if (with_cg) ld3(gx_cg, i, b);
    out[3 * i] = double(a[0]) + double(b[0]);
    out[3 * i + 1] = double(a[1]) + double(b[1]);
    out[3 * i + 2] = double(a[2]) + double(b[2]);
  }
}

static int grid_for(int n) {
  const int b = (n + kThreads - 1) / kThreads;
  return b < 1 ? 1 : (b > 152 * 8 ? 152 * 8 : b);
}

// Threads per slot by the slots of both lists.  Measured on neopentane-like
// liquids (1.2 slots an atom), us per launch with 8 / 4 / 2 / 1 threads, of two
// types and of eight (whose sums at the end of a block take longer):
//   FP32    10 000 atoms  11.7 /  13.5 /  18.4 /  28.6    24.0 /  25.0 /  30.2 /  40.8
//           20 000        20.4 /  16.0 /  20.0 /  30.2    40.5 /  28.2 /  32.2 /  42.6
//           35 000        30.9 /  25.7 /  23.0 /  33.9    62.4 /  50.4 /  36.5 /  46.6
//           50 000        40.7 /  33.4 /  30.0 /  36.6    85.4 /  65.9 /  53.9 /  51.3
//          100 000        74.4 /  59.7 /  50.9 /  52.6     156 /   113 /  87.8 /  77.8
//          200 000         143 /   109 /  91.5 /  88.9     300 /   203 /   152 /   127
//        1 000 000         684 /   515 /   419 /   376    1457 /   958 /   674 /   527
//   FP64     5 000        93.0 /   124 /   145 /   284     114 /   141 /   157 /   296
//           10 000         195 /   176 /   220 /   267     236 /   197 /   237 /   279
//           20 000         283 /   254 /   288 /   400     350 /   287 /   309 /   416
//           40 000         493 /   466 /   431 /   510     594 /   524 /   465 /   532
//          100 000        1430 /  1250 /  1124 /  1152    1662 /  1378 /  1191 /  1273
static int grad_lanes(long long slots, int nt, bool fp64) {
  if (slots <= (fp64 ? 9000 : 14000)) return 8;
  if (slots <= (fp64 ? 35000 : 30000)) return 4;
  return fp64 || slots <= (nt <= 2 ? 180000 : 70000) ? 2 : 1;
}

template <typename R>
static cudaError_t launch_grad_t(relres_ctx* c, const double* d_grad_forces, double g_energy, double* d_grad_pos) {
  using V = GVec<R>;
  const bool do_cg = c->has_cg && c->n_h > 0;
  const double* g = d_grad_forces ? d_grad_forces : static_cast<const double*>(c->d_zero_n3);
  V* gfg = static_cast<V*>(c->d_g_fg);
  V* gcg = static_cast<V*>(c->d_g_cg);
  V* xfg = static_cast<V*>(c->d_gx_fg);
  V* xcg = static_cast<V*>(c->d_gx_cg);
  const int n_cg = do_cg ? c->n_h : 0;
  k_gather_g<R><<<grid_for(c->n + n_cg), kThreads, 0, c->stream>>>(c->n, n_cg, c->d_perm_fg, c->d_perm_cg, g, gfg, gcg);
  RELRES_LAUNCHED(c);
  const double unit = std::is_same<R, float>::value ? 4294967296.0 : 18446744073709551616.0;
  GradLaunch<R> a{};
  a.sx = R(c->box[0] / unit);
  a.sy = R(c->box[1] / unit);
  a.sz = R(c->box[2] / unit);
  a.sxl = float(c->box[0] / unit - double(a.sx));
  a.syl = float(c->box[1] / unit - double(a.sy));
  a.szl = float(c->box[2] / unit - double(a.sz));
  a.nt = c->n_types;
  a.tab = static_cast<const BasisTab<R>*>(c->d_basis);
  a.g_energy = R(g_energy);
  a.gc = c->d_gc;
  a.flags = &c->d_state->flags;
  const GPos<R>* pfg;
  const GPos<R>* pcg;
  if constexpr (std::is_same<R, float>::value) {
    pfg = c->d_pos_fg;
    pcg = c->d_pos_cg;
  } else {
    pfg = c->d_pos_fg64;
    pcg = c->d_pos_cg64;
  }
  a.fg = GradWalk<R>{c->n, pfg, walk_nbr_fg(c), walk_cnt_fg(c), c->d_perm_fg, gfg, xfg};
  a.cg = do_cg ? GradWalk<R>{c->n_h, pcg, walk_nbr_cg(c), walk_cnt_cg(c), c->d_perm_cg, gcg, xcg} : a.fg;
  const int lanes = grad_lanes(pair_slots(c), c->n_types, c->fp64), per = kGradThreads / lanes;
  const int nb_fg = (c->n + per - 1) / per;
  const int nb_cg = do_cg ? (c->n_h + per - 1) / per : 0;
  a.nblk_cg = nb_cg;
  const int nrow = c->n_types * c->n_types;
  const size_t smem = sizeof(double) * 2 * nrow + sizeof(R) * 2 * c->n_types * kGradThreads + sizeof(BasisTab<R>) * nrow;
  const cudaError_t ez = cudaMemsetAsync(c->d_gc, 0, sizeof(double) * 4 * nrow, c->stream);
  if (ez != cudaSuccess) return ez;
  if (lanes == 8)
    k_pair_grad<R, 8><<<nb_cg + nb_fg, kGradThreads, smem, c->stream>>>(a);
  else if (lanes == 4)
    k_pair_grad<R, 4><<<nb_cg + nb_fg, kGradThreads, smem, c->stream>>>(a);
  else if (lanes == 2)
    k_pair_grad<R, 2><<<nb_cg + nb_fg, kGradThreads, smem, c->stream>>>(a);
  else
    k_pair_grad<R, 1><<<nb_cg + nb_fg, kGradThreads, smem, c->stream>>>(a);
  RELRES_LAUNCHED(c);
  if (d_grad_pos) {
    k_sum_gx<R><<<grid_for(c->n), kThreads, 0, c->stream>>>(c->n, xfg, xcg, do_cg ? 1 : 0, c->d_state,
                                                                 d_grad_pos);
    RELRES_LAUNCHED(c);
  }
  return cudaGetLastError();
}

cudaError_t launch_pair_grad(relres_ctx* c, const double* d_grad_forces, double g_energy, double* d_grad_pos) {
  return c->fp64 ? launch_grad_t<double>(c, d_grad_forces, g_energy, d_grad_pos)
                 : launch_grad_t<float>(c, d_grad_forces, g_energy, d_grad_pos);
}

}  // namespace relres
