// FP32 pair launches that spread a slot's list over several threads, and the
// FP32 energy steps.
//
// A system of a few thousand to some ten thousand atoms does not fill the part
// with one thread per slot, and its launch then lasts as long as one thread
// needs for one list: 12 us of dependent loads at 20 000 atoms, 66 us with
// energies.  Here T lanes of a warp share a slot: in each round they take T
// consecutive chunks of four entries.  The compensated force sum of the
// one-thread walk (each chunk summed in FP32, the chunk sums added in list
// order to a float-float total) is kept to the bit: the lanes leave their
// chunk sums in shared memory and three lanes add the x, y and z sums in list
// order.  A chunk past the end of the list adds exactly zero.
//
// Energy steps: every lane queues the pairs inside the cutoff that it meets
// first (the owner of the lower slot; the lists hold every pair from both
// ends) in its warp's shared-memory queue, and whole warps evaluate 32 queued
// pairs at a time, energy in float-float (see FgE) and virial from the force
// factor of the walk.  Each pair's values are converted to 64-bit fixed point
// (value * 2^32, the accumulators' own unit) and summed as integers, so energy
// and virial do not depend on the order of the lists or on T.
#include "pair.cuh"

namespace relres {

// float-float energy of one pair inside the cutoff from its exact 32-bit
// coordinate differences
template <bool CG>
__device__ __forceinline__ ff pair_energy_ff(const int4& d, const SmemTabs& S, const PairLaunch& a) {
  const ff ex = ff_fixed_diff32(d.x, 0, ff{a.sx, a.sxl});
  const ff ey = ff_fixed_diff32(d.y, 0, ff{a.sy, a.syl});
  const ff ez = ff_fixed_diff32(d.z, 0, ff{a.sz, a.szl});
  const ff r2e = ff_add(ff_add(ff_mul(ex, ex), ff_mul(ey, ey)), ff_mul(ez, ez));
  const PairRow& T = S.row[d.w];
  return CG ? cg_energy_ff(S.rowe[d.w].cg, cg_radii2(T.cg), r2e)
            : fg_energy_ff(S.rowe[d.w].fg, T.fg.b.x * T.fg.b.x, r2e);
}

// a float in units of 2^-32, rounded, as a 64-bit integer (|v| < 2^20)
__device__ __forceinline__ long long fix32(float v) { return f2ll_rn(__fmul_rn(v, 4294967296.f)); }

// Energy and virial totals of every thread of the block, in shared memory
// (touched once per queued pair; in registers they cost the walk its own).
struct PairTotals {
  long long v[kNQ][kLaneThreads];
};

// energy and virial of one queued pair added to the thread's totals
template <bool CG>
__device__ __forceinline__ void add_pair(const int4& d, float fr, const SmemTabs& S, const PairLaunch& a,
                                         PairTotals* tot) {
  const ff e = pair_energy_ff<CG>(d, S, a);
  const float x = float(d.x) * a.sx, y = float(d.y) * a.sy, z = float(d.z) * a.sz;
  const float fx = fr * x, fy = fr * y, fz = fr * z;
  const float w[6] = {fx * x, fy * y, fz * z, fx * y, fx * z, fy * z};
  // |each virial component| <= |x fx| + |y fy| + |z fz|
  if (fmaxf(fabsf(e.hi), fabsf(w[0]) + fabsf(w[1]) + fabsf(w[2])) < 1048576.f) {
    tot->v[0][threadIdx.x] += fix32(e.hi) + fix32(e.lo);
#pragma unroll
    for (int k = 0; k < 6; ++k) tot->v[k + 1][threadIdx.x] += fix32(w[k]);
  } else {  // overlapping atoms: values past the FP32 conversion's range
    tot->v[0][threadIdx.x] += to_fix_sum(double(e.hi) + double(e.lo));
#pragma unroll
    for (int k = 0; k < 6; ++k) tot->v[k + 1][threadIdx.x] += to_fix_sum(double(w[k]));
  }
}

// Queued pairs of one warp, of two classes: the plain Lennard-Jones range from
// the front, the switching ranges from the back, so that the warps that
// evaluate them run one range's arithmetic.  Fewer than 32 of a class wait
// between two rounds, and a round adds at most four per lane.
constexpr int kQueue = 2 * 31 + 4 * 32;
struct PairQueue {
  int4 d[kQueue];   // coordinate differences and type-pair row
  float fr[kQueue]; // force factor
};

// One warp's walk over the lists of its 32 / T slots.
template <bool CG, bool EV, int T, bool PRN, int ACC>
__device__ __forceinline__ void walk_lanes(const ListWalk& L, int blk, const SmemTabs& S, float4* stage,
                                           PairQueue* queue, PairTotals* tot, const PairLaunch& a,
                                           bool first_block) {
  static_assert(T == 1 || (T >= 4 && 32 % T == 0 && ACC == RELRES_ACC_COMPENSATED), "three lanes add the chunk sums");
  const int s = (blk * kLaneThreads + threadIdx.x) / T, q = threadIdx.x % T;
  const int lane = threadIdx.x & 31, base = lane - q;
  const bool own = s < L.nslots;
  const int ss = own ? s : 0;  // a valid slot for the loads of the other lanes
  const int4 pi = L.pos[ss];
  const int m = own ? (PRN ? L.cnt_full[s] : L.cnt[s]) : 0;
  const int nch = (m + 3) >> 2;
  const int4* nb4 = reinterpret_cast<const int4*>(PRN ? L.nbr_full : L.nbr) + ss;
  int4 jj = make_int4(ss, ss, ss, ss);
  if (q < nch) jj = __ldcs(nb4 + size_t(q) * L.nslots);
  const int rounds = __reduce_max_sync(0xffffffffu, (nch + T - 1) / T);
  const int row0 = pi.w * a.nt;
  __syncthreads();  // the type-pair tables
  Acc A;
  int kept = 0;
  int4 buf = make_int4(ss, ss, ss, ss);
  int waiting = 0, waiting2 = 0;  // of the Lennard-Jones range, of the others
  if constexpr (EV) {
#pragma unroll
    for (int k = 0; k < kNQ; ++k) tot->v[k][threadIdx.x] = 0;
  }
  for (int r = 0;; ++r) {
    if (r < rounds) {
      const int ch = r * T + q;
      int4 jn = jj;
      if (ch + T < nch) jn = __ldcs(nb4 + size_t(ch + T) * L.nslots);
      const int rem = m - 4 * ch;  // <= 0 past the list
      const int j[4] = {rem > 0 ? jj.x : ss, rem > 1 ? jj.y : ss, rem > 2 ? jj.z : ss, rem > 3 ? jj.w : ss};
      int4 p[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) p[e] = load_pos(L.pos, j[e]);
      float r2[4], fr[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float dx, dy, dz;
        r2[e] = pair_term<CG>(pi, p[e], rem > e, S.row[row0 + p[e].w], a.sx, a.sy, a.sz, fr[e], dx, dy, dz);
        acc_force<ACC>(A, fr[e], dx, dy, dz);
      }
      if constexpr (T == 1) {
        if (rem > 0) acc_chunk<ACC>(A);
      } else {
        float4* const st = stage + (threadIdx.x & ~31);
        st[lane] = make_float4(A.kx, A.ky, A.kz, 0.f);
        A.kx = A.ky = A.kz = 0.f;
        __syncwarp();
        const float* const sum = reinterpret_cast<const float*>(st + base) + (q & 3);
#pragma unroll
        for (int k = 0; k < T; ++k) {  // lane q < 3: component q (the others' results are not used)
          const ff v = ff_two_sum(A.fx, sum[4 * k]);
          A.fx = v.hi;
          A.cx = __fadd_rn(A.cx, v.lo);
        }
        __syncwarp();
      }
      if constexpr (PRN) {
        if constexpr (T == 1) {
          if (rem > 0) {
            int4* out4 = reinterpret_cast<int4*>(L.nbr_in) + ss;
#pragma unroll
            for (int e = 0; e < 4; ++e) keep_entry(r2[e] < L.rp2, j[e], kept, buf, out4, L.nslots);
          }
        } else {
          // in list order: the entries kept by the slot's earlier lanes, then this lane's
          const unsigned mine = ((1u << T) - 1u) << base, before = mine & ((1u << lane) - 1u);
          unsigned b[4];
          int at = kept, all = 0;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            b[e] = __ballot_sync(0xffffffffu, r2[e] < L.rp2);
            at += __popc(b[e] & before);
            all += __popc(b[e] & mine);
          }
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (r2[e] < L.rp2) {
              L.nbr_in[(size_t(at >> 2) * L.nslots + s) * 4 + (at & 3)] = j[e];
              ++at;
            }
          kept += all;
        }
      }
      if constexpr (EV) {
        PairQueue& Q = queue[threadIdx.x >> 5];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int row = row0 + p[e].w;
          const PairRow& R = S.row[row];
          const bool need = r2[e] < (CG ? R.cg.a.y : R.fg.a.y) && s < j[e];
          const bool lj = CG ? r2[e] >= R.cg.a.x && r2[e] < R.cg.a.w * R.cg.a.w : r2[e] < R.fg.b.x * R.fg.b.x;
          const unsigned b = __ballot_sync(0xffffffffu, need && lj), b2 = __ballot_sync(0xffffffffu, need && !lj);
          if (need) {
            const int k = lj ? waiting + __popc(b & ((1u << lane) - 1u))
                             : kQueue - 1 - waiting2 - __popc(b2 & ((1u << lane) - 1u));
            Q.d[k] = make_int4(int(unsigned(pi.x) - unsigned(p[e].x)), int(unsigned(pi.y) - unsigned(p[e].y)),
                               int(unsigned(pi.z) - unsigned(p[e].z)), row);
            Q.fr[k] = fr[e];
          }
          waiting += __popc(b);
          waiting2 += __popc(b2);
        }
      }
      jj = jn;
    }
    if constexpr (EV) {  // full passes of the queue; after the last round what is left
      __syncwarp();
      PairQueue& Q = queue[threadIdx.x >> 5];
      const int least = r < rounds ? 32 : 1;
      while (max(waiting, waiting2) >= least) {
        const bool lj = waiting >= least;
        const int left = lj ? waiting : waiting2, take = min(left, 32), at = left - take + lane;
        if (lj)
          waiting -= take;
        else
          waiting2 -= take;
        const int k = lj ? at : kQueue - 1 - at;
        if (lane < take) add_pair<CG>(Q.d[k], Q.fr[k], S, a, tot);
      }
      __syncwarp();
    }
    if (r >= rounds) break;
  }
  if constexpr (PRN) {
    if (own && q == 0) {
      if (T == 1) keep_tail(kept, buf, reinterpret_cast<int4*>(L.nbr_in) + ss, L.nslots);
      L.cnt_in[s] = kept;
      if (!CG) a.ref_p[L.perm[s]] = pi;
    }
    unsigned long long v[1] = {own && q == 0 ? (unsigned long long)kept : 0ull};
    __shared__ unsigned long long sh_k[kLaneThreads / 32];
    block_sum<unsigned long long, 1>(v, sh_k);
    if (threadIdx.x == 0) {
      atomicAdd(L.tot_in, v[0]);
      if (first_block) atomicAdd(&a.st->n_prunes, 1ull);
    }
  }
  if constexpr (T == 1) {
    acc_final<ACC>(A);
    if (own) store_force(L.f_out, L.perm[s], A.fx, A.fy, A.fz);
  } else if (own && q < 4) {
    reinterpret_cast<float*>(L.f_out + L.perm[s])[q] = q < 3 ? __fadd_rn(A.fx, A.cx) : 0.f;
  }
  if constexpr (EV) {
    __shared__ long long sh_e[kLaneThreads / 32][kNQ];
#pragma unroll
    for (int k = 0; k < kNQ; ++k) {
      const long long v = warp_sum(tot->v[k][threadIdx.x]);
      if (lane == 0) sh_e[threadIdx.x >> 5][k] = v;
    }
    __syncthreads();
    if (threadIdx.x < kNQ) {
      long long v = 0;
#pragma unroll
      for (int w = 0; w < kLaneThreads / 32; ++w) v += sh_e[w][threadIdx.x];
      atomicAdd(reinterpret_cast<unsigned long long*>(L.acc + threadIdx.x), (unsigned long long)v);
    }
  }
}

template <bool EV, int T>
static size_t lanes_smem(int nt) {
  const size_t nrow = size_t(nt) * nt;
  auto up = [](size_t b) { return (b + 15) / 16 * 16; };
  return up(sizeof(PairRow) * nrow) + (EV ? up(sizeof(PairRowEnergy) * nrow) + sizeof(PairQueue) * (kLaneThreads / 32) + sizeof(PairTotals) : 0) +
         (T > 1 ? sizeof(float4) * kLaneThreads : 0);
}

template <bool EV, int T, int ACC>
__device__ __forceinline__ void lanes_block(const PairLaunch& a, int bid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nrow = a.nt * a.nt;
  size_t off = 0;
  auto carve = [&](size_t bytes) {
    unsigned char* p = smem_raw + off;
    off += (bytes + 15) / 16 * 16;
    return p;
  };
  SmemTabs S{};
  PairRow* row = reinterpret_cast<PairRow*>(carve(sizeof(PairRow) * nrow));
  copy_words(row, a.tab, nrow * int(sizeof(PairRow) / sizeof(int)));
  S.row = row;
  PairQueue* queue = nullptr;
  PairTotals* tot = nullptr;
  if (EV) {
    PairRowEnergy* rowe = reinterpret_cast<PairRowEnergy*>(carve(sizeof(PairRowEnergy) * nrow));
    copy_words(rowe, a.tabe, nrow * int(sizeof(PairRowEnergy) / sizeof(int)));
    S.rowe = rowe;
    queue = reinterpret_cast<PairQueue*>(carve(sizeof(PairQueue) * (kLaneThreads / 32)));
    tot = reinterpret_cast<PairTotals*>(carve(sizeof(PairTotals)));
  }
  float4* stage = T > 1 ? reinterpret_cast<float4*>(carve(sizeof(float4) * kLaneThreads)) : nullptr;
  after_rebuild();
  // (forces only: these launches prune as they walk wherever pruning is on)
  if (EV && lists_unpruned(a)) return;
  const bool cg = bid < a.nblk_cg;
  const int blk = cg ? bid : bid - a.nblk_cg;
  const bool prn = a.prune_on && (*(volatile const unsigned*)a.gate & (F_REBUILD | F_PRUNE)) != 0u;
  if (prn) {
    if (cg)
      walk_lanes<true, EV, T, true, ACC>(a.cg, blk, S, stage, queue, tot, a, bid == 0);
    else
      walk_lanes<false, EV, T, true, ACC>(a.fg, blk, S, stage, queue, tot, a, bid == 0);
  } else {
    if (cg)
      walk_lanes<true, EV, T, false, ACC>(a.cg, blk, S, stage, queue, tot, a, bid == 0);
    else
      walk_lanes<false, EV, T, false, ACC>(a.fg, blk, S, stage, queue, tot, a, bid == 0);
  }
}

// energy steps: 96 registers a thread (five blocks per SM; at six they spill, 7 %
// slower at 20 000 atoms, at four 9 % slower), forces only: 64
template <bool EV, int T, int ACC>
__global__ void __launch_bounds__(kLaneThreads, EV ? 5 : 8) k_pair_lanes(PairLaunch a) {
  lanes_block<EV, T, ACC>(a, blockIdx.x);
}

template <bool EV, int T, int ACC>
__global__ void __launch_bounds__(kLaneThreads, EV ? 5 : 8)
    k_pair_lanes_batch(const PairLaunch* __restrict__ args, const int* __restrict__ off, int nrep) {
  const int r = batch_replica(off, nrep, blockIdx.x);
  lanes_block<EV, T, ACC>(args[r], int(blockIdx.x) - off[r]);
}

template <bool EV, int T, int ACC>
static void launch_one(cudaStream_t s, const PairLaunch& a, int grid, bool pdl) {
  launch_pdl(pdl, k_pair_lanes<EV, T, ACC>, grid, kLaneThreads, lanes_smem<EV, T>(a.nt), s, a);
}
template <bool EV, int T, int ACC>
static void launch_batch(cudaStream_t s, const BatchLaunch& b, int nrep) {
  k_pair_lanes_batch<EV, T, ACC><<<b.nblk, kLaneThreads, lanes_smem<EV, T>(b.nt), s>>>(
      static_cast<const PairLaunch*>(b.d_args), b.d_off, nrep);
}

// F<EV, T, ACC>(...) for the accumulation and the lanes of a launch
#define RELRES_LANES(F, ...)                                      \
  if (lanes == 8) {                                               \
    if (ev)                                                       \
      F<true, 8, RELRES_ACC_COMPENSATED>(__VA_ARGS__);            \
    else                                                          \
      F<false, 8, RELRES_ACC_COMPENSATED>(__VA_ARGS__);           \
  } else if (lanes == 4) {                                        \
    if (ev)                                                       \
      F<true, 4, RELRES_ACC_COMPENSATED>(__VA_ARGS__);            \
    else                                                          \
      F<false, 4, RELRES_ACC_COMPENSATED>(__VA_ARGS__);           \
  } else if (acc == RELRES_ACC_FP32) {                            \
    F<true, 1, RELRES_ACC_FP32>(__VA_ARGS__);                     \
  } else if (acc == RELRES_ACC_COMPENSATED) {                     \
    F<true, 1, RELRES_ACC_COMPENSATED>(__VA_ARGS__);              \
  } else {                                                        \
    F<true, 1, RELRES_ACC_FP64>(__VA_ARGS__);                     \
  }

void launch_pairs_lanes(cudaStream_t s, int acc, const PairLaunch& a, bool ev, int lanes, int grid, bool pdl) {
  RELRES_LANES(launch_one, s, a, grid, pdl)
}

void launch_pairs_lanes_batch(cudaStream_t s, int acc, bool ev, const BatchLaunch& b, int nrep) {
  const int lanes = b.lanes;
  RELRES_LANES(launch_batch, s, b, nrep)
}

}  // namespace relres
