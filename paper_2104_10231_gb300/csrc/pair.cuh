// Device code shared by the FP32 pair kernels (pair.cu, pair_lanes.cu): the FG
// and CG terms of one pair, launch arguments and force accumulators.
#pragma once

#include "common.cuh"

namespace relres {

__device__ __forceinline__ int4 load_pos(const int4* p, int j) { return __ldg(p + j); }

__device__ __forceinline__ void store_force(float4* f, int i, float x, float y, float z) {
  f[i] = make_float4(x, y, z, 0.f);
}

// FP32 force coefficients of one type pair for 16-byte shared-memory loads
// (the words of PairRowF).
struct FgRow {
  float4 a;  // 4 g4, r_s+^2, 48 eps sig^12, 24 eps sig^6
  float4 b;  // r_s-, derivative of f_{s-}^{FG}: g1, 2 g2, 3 g3
};
struct CgRow {
  float4 a;  // r_s+^2, r_c+^2, r_s-, r_c-
  float4 b;  // 3 gamma_3+, 4 gamma_4+, 48 eps sig^12, 24 eps sig^6 (CG)
  float4 c;  // derivative of f_{c-}^{CG}: g1, 2 g2, 3 g3, 4 g4
};
struct PairRow {
  FgRow fg;
  CgRow cg;
};
static_assert(sizeof(PairRow) == sizeof(PairRowF), "packed by pack_pair_rows");

// Energy constants of one type pair for the FP32 path (energy steps) as
// float-float values.  Pair energies of energy steps are evaluated in
// float-float arithmetic (~48-bit): in FP32 alone, rounding that is the same
// for every pair of a type (constants, the box scale, approximate
// reciprocals) biases the total, and the FG and CG parts largely cancel in
// it, so 1e-7 of the total is out of reach; FP64 proper runs at a small
// fraction of the FP32 rate on this part.
struct FgE {
  ff c12, c6, shift, rsm, g[5];
};
struct CgE {
  ff c12, c6, gam, rsm, rcm, on0, on3, on4, close, g[5];
};
struct PairRowEnergy {
  FgE fg;
  CgE cg;
};
static_assert(sizeof(PairRowEnergy) == sizeof(PairRowE), "packed by pack_pair_rows");
__device__ __forceinline__ ff poly5_ff(const ff (&g)[5], ff d) {
  ff p = g[4];
#pragma unroll
  for (int m = 3; m >= 0; --m) p = ff_add(ff_mul(p, d), g[m]);
  return p;
}
__device__ __forceinline__ ff lj_ff(const ff& c12, const ff& c6, ff r2i) {
  const ff r6i = ff_mul(ff_mul(r2i, r2i), r2i);
  return ff_sub(ff_mul(c12, ff_mul(r6i, r6i)), ff_mul(c6, r6i));
}
// FG energy of a pair inside r_s+ (regions chosen on the leading part: the
// potential is C2 at r_s-, so a pair rounded across it changes nothing)
__device__ __forceinline__ ff fg_energy_ff(const FgE& T, float rsm2, ff r2) {
  const ff e = r2.hi < rsm2 ? lj_ff(T.c12, T.c6, ff_rcp(r2)) : poly5_ff(T.g, ff_sub(ff_sqrt(r2), T.rsm));
  return ff_sub(e, T.shift);
}
// CG energy of a pair inside r_c+
__device__ __forceinline__ ff cg_energy_ff(const CgE& T, float4 radii2, ff r2) {
  if (r2.hi < radii2.x) return T.close;
  ff e;
  if (r2.hi < radii2.y) {
    const ff d = ff_sub(ff_sqrt(r2), T.rsm);
    const ff d3 = ff_mul(ff_mul(d, d), d);
    e = ff_add(T.on0, ff_mul(d3, ff_add(ff_mul(T.on4, d), T.on3)));
  } else if (r2.hi < radii2.z) {
    e = lj_ff(T.c12, T.c6, ff_rcp(r2));
  } else {
    e = poly5_ff(T.g, ff_sub(ff_sqrt(r2), T.rcm));
  }
  return ff_sub(e, T.gam);
}

// -dU/dr / r of the FG part, every region evaluated and the right one
// selected (the LJ core by the sign of r - r_s-).  r2 >= r_s+^2 gives 0.
__device__ __forceinline__ float fg_force(const FgRow& T, float r2) {
  const float4 a = T.a, b = T.b;
  const float g4 = a.x;
  const float r2i = rcp_nr(r2);
  const float r6i = r2i * r2i * r2i;
  const float flj = r6i * (a.z * r6i - a.w) * r2i;
  const float ri = rsqrtf(r2);
  const float d = r2 * ri - b.x;
  const float fp = ((g4 * d + b.w) * d + b.z) * d + b.y;
  const float fsh = -fp * ri;
  const float fr = d < 0.f ? flj : fsh;  // r < r_s-: LJ core
  return r2 < a.y ? fr : 0.f;
}

// -dU/dr / r of the CG part, the regions below r_s- and r_c- chosen by the
// signs of r - r_s- and r - r_c-: zero below r_s- (the constant region) and
// from r_c+ on.
__device__ __forceinline__ float cg_force(const CgRow& T, float r2) {
  const float4 a = T.a, b = T.b, c = T.c;
  const float ri = rsqrtf(r2);
  const float r = r2 * ri;
  const float d = r - a.z;
  const float fon = -(d * d * (b.y * d + b.x)) * ri;
  const float r2i = ri * ri;
  const float r6i = r2i * r2i * r2i;
  const float flj = r6i * (b.z * r6i - b.w) * r2i;
  const float e = r - a.w;
  const float foff = -(((c.w * e + c.z) * e + c.y) * e + c.x) * ri;
  float fr = e < 0.f ? flj : foff;
  fr = r2 < a.x ? fon : fr;
  return (d < 0.f || !(r2 < a.y)) ? 0.f : fr;
}

// (r_s-^2, r_s+^2, r_c-^2, r_c+^2) of a CG row, for the energy regions
__device__ __forceinline__ float4 cg_radii2(const CgRow& T) {
  return make_float4(T.a.z * T.a.z, T.a.x, T.a.w * T.a.w, T.a.y);
}


struct ListWalk {
  int nslots;
  const int4* pos;
  const int* nbr;  // the list walked (pruned when pruning is on)
  const int* cnt;
  const int* perm;
  float4* f_out;
  long long* acc;  // kNQ accumulators of this list (energy, six virial components)
  // pruning launches (PRN): walk the full list and write the pruned one
  const int* nbr_full;
  const int* cnt_full;
  int* nbr_in;
  int* cnt_in;
  float rp2;  // (interaction cutoff + delta + slack)^2
  unsigned long long* tot_in;
};

struct PairLaunch {
  int nblk_cg;  // blocks [0, nblk_cg) walk the CG list, the rest the FG list
  ListWalk fg, cg;
  const PairRow* tab;          // [nt^2]
  const PairRowEnergy* tabe;   // energy steps
  int nt;
  float sx, sy, sz;
  float sxl, syl, szl;  // lo parts of L / 2^32 (float-float energies)
  const unsigned* gate;  // device flag word of the step
  int prune_on;          // prune on this launch if F_REBUILD or F_PRUNE is set
  int4* ref_p;  // PRN: positions of this pruning pass, caller order (FG walk)
  DevState* st;
};

// type-pair tables in shared memory
struct SmemTabs {
  const PairRow* row;
  const PairRowEnergy* rowe;  // energy steps
};

// Between a pair kernel's tables and its lists: waits for the kernel before it
// (the rebuild, see pair_pdl), then lets the force sum that follows start
// launching once every block of this grid is here (it waits for this grid to
// finish before reading the forces).  In this order, so that nothing behind
// this kernel runs while the lists may still change.
__device__ __forceinline__ void after_rebuild() {
  grid_dependency_wait();
  grid_dependents_launch();
}

// A launch whose lists were to be pruned by a pass of their own (or that walks
// the full lists) behind a non-finite position or an unfinished rebuild: the
// pass did not run, so the pruned lists may never have been written.  The call
// fails without reading these forces.
__device__ __forceinline__ bool lists_unpruned(const PairLaunch& a) {
  return !a.prune_on && (*(volatile const unsigned*)a.gate & F_NOLISTS) != 0u;
}

// copies n words from global to shared memory with the whole block
__device__ __forceinline__ void copy_words(void* dst, const void* src, int n) {
  for (int w = threadIdx.x; w < n; w += blockDim.x) static_cast<int*>(dst)[w] = static_cast<const int*>(src)[w];
}

// Per-thread accumulators of one walk.  The owner's force sum of the FP32
// path is kept in one of three ways (ACC, relres_set_force_accumulation):
// FP32 running sums (fx, fy, fz); compensated sums, where the (up to) four
// entries of a list chunk are summed in FP32 (kx, ...) and each chunk sum is
// added to a float-float total (fx + cx, ...) with an error-free two-sum; or
// FP64 running sums (dfx, ...), one conversion and FP64 add per entry.  The
// members a variant does not use are removed by the compiler.
struct Acc {
  float fx = 0.f, fy = 0.f, fz = 0.f;
  float kx = 0.f, ky = 0.f, kz = 0.f;
  float cx = 0.f, cy = 0.f, cz = 0.f;
  double dfx = 0.0, dfy = 0.0, dfz = 0.0;
};

// The FMAs are explicit: every kernel that sums a chunk rounds it alike.
template <int ACC>
__device__ __forceinline__ void acc_force(Acc& A, float fr, float dx, float dy, float dz) {
  if constexpr (ACC == RELRES_ACC_COMPENSATED) {
    A.kx = fmaf(fr, dx, A.kx);
    A.ky = fmaf(fr, dy, A.ky);
    A.kz = fmaf(fr, dz, A.kz);
  } else if constexpr (ACC == RELRES_ACC_FP64) {
    A.dfx += double(__fmul_rn(fr, dx));
    A.dfy += double(__fmul_rn(fr, dy));
    A.dfz += double(__fmul_rn(fr, dz));
  } else {
    A.fx = fmaf(fr, dx, A.fx);
    A.fy = fmaf(fr, dy, A.fy);
    A.fz = fmaf(fr, dz, A.fz);
  }
}

// end of a list chunk: the compensated variant moves the chunk sum into its
// float-float total
template <int ACC>
__device__ __forceinline__ void acc_chunk(Acc& A) {
  if constexpr (ACC == RELRES_ACC_COMPENSATED) {
    const ff sx = ff_two_sum(A.fx, A.kx), sy = ff_two_sum(A.fy, A.ky), sz = ff_two_sum(A.fz, A.kz);
    A.fx = sx.hi;
    A.fy = sy.hi;
    A.fz = sz.hi;
    A.cx = __fadd_rn(A.cx, sx.lo);
    A.cy = __fadd_rn(A.cy, sy.lo);
    A.cz = __fadd_rn(A.cz, sz.lo);
    A.kx = A.ky = A.kz = 0.f;
  }
}

// the owner's force sum rounded to FP32 (the width of the force buffers)
template <int ACC>
__device__ __forceinline__ void acc_final(Acc& A) {
  if constexpr (ACC == RELRES_ACC_COMPENSATED) {
    A.fx = __fadd_rn(A.fx, A.cx);
    A.fy = __fadd_rn(A.fy, A.cy);
    A.fz = __fadd_rn(A.fz, A.cz);
  } else if constexpr (ACC == RELRES_ACC_FP64) {
    A.fx = float(A.dfx);
    A.fy = float(A.dfy);
    A.fz = float(A.dfz);
  }
}

// One FP32 pair: squared distance (past every cutoff for a padding entry),
// force factor -u'(r)/r and coordinate difference.
template <bool CG>
__device__ __forceinline__ float pair_term(const int4& pi, const int4& pj, bool valid, const PairRow& T, float sx,
                                           float sy, float sz, float& fr, float& dx, float& dy, float& dz) {
  dx = dfix32(pi.x, pj.x, sx);
  dy = dfix32(pi.y, pj.y, sy);
  dz = dfix32(pi.z, pj.z, sz);
  float r2 = dx * dx + dy * dy + dz * dz;
  r2 = valid ? r2 : 3.0e38f;
  fr = CG ? cg_force(T.cg, r2) : fg_force(T.fg, r2);
  return r2;
}

// ---- pair_lanes.cu: FP32 launches of kLaneThreads-thread blocks, `lanes`
// threads per slot (1, 4 or 8; forces only: 4 or 8)
constexpr int kLaneThreads = 128;
void launch_pairs_lanes(cudaStream_t s, int acc, const PairLaunch& a, bool ev, int lanes, int grid, bool pdl);
void launch_pairs_lanes_batch(cudaStream_t s, int acc, bool ev, const BatchLaunch& b, int nrep);

// ---- pair64.cu: FP64 contexts
cudaError_t launch_pairs_f64(relres_ctx* c, bool ev, int which);
cudaError_t prepare_pairs_batch_f64(const std::vector<relres_ctx*>& cs, BatchLaunch* b, BatchLaunch* b_ev);
void launch_pairs_batch_f64(cudaStream_t s, bool ev, const BatchLaunch& b, int nrep);

}  // namespace relres
