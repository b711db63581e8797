// RelRes pair kernel: Eq. 20 of the paper (Section 2.5) over the two lists.
//
// The potential is evaluated split exactly into an FG part (on the FG list:
// every atom, partners within r_s+) and a CG part (on the CG list: hybrid
// sites, partners within r_c+), see PairTab in relres_internal.h.  Forces
// never depend on a shift constant, so the split changes nothing but which
// list carries which term.  One launch covers both lists: the first blocks
// walk the CG list (fewer, longer-running slots, so they start first), the
// rest walk the FG list.
//
// One thread owns one sorted slot and walks its full list four entries at a
// time.  The list is stored in chunks of four (entry k of slot s at int
// (((k >> 2) * nslots + s) << 2) + (k & 3)), so a warp reads 512 contiguous
// bytes of indices per chunk with one 16-byte streaming load per thread, and
// the next chunk's indices are requested before the current chunk is
// evaluated.  The four partner positions (16-byte packed x, y, z, type, L1/L2
// resident thanks to the Morton cell order) are gathered together, then each
// entry gets an exact wrapped integer difference converted to FP32 and its
// region selected without branches.  The owner accumulates its force in
// registers and writes it once (no atomics).  The FP64 variant (R = double)
// reads 64-bit fixed-point positions and computes every term in double; its
// energy and virial (EV template) are summed per block and added to 64-bit
// fixed-point accumulators with integer atomics.  FP32 energy steps, and the
// FP32 forces of systems too small to fill the part with one thread per slot,
// are in pair_lanes.cu.
#include "pair.cuh"

namespace relres {

// One list entry; returns its squared distance (past every cutoff for a
// padding entry), which a pruning launch compares with the pruning radius.
template <typename R, bool CG, bool EV, int ACC>
__device__ __forceinline__ R entry(const typename PosOf<R>::T& pi, const typename PosOf<R>::T& pj,
                                   bool valid, int row0, const SmemTabs& S, const PairLaunch<R>& a,
                                   Acc<R>& A) {
  const int row = row0 + ptype(pj);
  if constexpr (std::is_same<R, float>::value) {
    static_assert(!EV, "FP32 energy steps are in pair_lanes.cu");
    float fr, dx, dy, dz;
    const float r2 = pair_term<CG>(pi, pj, valid, S.row[row], a.sx, a.sy, a.sz, fr, dx, dy, dz);
    acc_force<ACC>(A, fr, dx, dy, dz);
    return r2;
  } else {
    if (!valid) return R(1e300);
    R dx, dy, dz;
    delta(pi, pj, a.sx, a.sy, a.sz, dx, dy, dz);
    const R r2 = dx * dx + dy * dy + dz * dz;
    const PairTab<R>& T = static_cast<const PairTab<R>*>(S.tab)[row];
    R fr, ep;
    const bool hit = CG ? cg_term<R, EV>(T, r2, fr, ep) : fg_term<R, EV>(T, r2, fr, ep);
    if (hit) {
      // one rounding per term (fma): the operation the ordered several-lane
      // walk repeats (walk_ordered), so both give the same bits
      A.fx = fma(fr, dx, A.fx);
      A.fy = fma(fr, dy, A.fy);
      A.fz = fma(fr, dz, A.fz);
      if (EV) {
        A.e += ep;
        A.w[0] += fr * dx * dx;
        A.w[1] += fr * dy * dy;
        A.w[2] += fr * dz * dz;
        A.w[3] += fr * dx * dy;
        A.w[4] += fr * dx * dz;
        A.w[5] += fr * dy * dz;
      }
    }
    return r2;
  }
}

// FP64 force factor of one entry and its coordinate difference (the
// arithmetic of entry()); zero for a padding entry or a pair past the cutoff.
template <bool CG>
__device__ __forceinline__ double term64(const Pos64& pi, const Pos64& pj, bool valid, int row0, const SmemTabs& S,
                                         const PairLaunch<double>& a, double d[3]) {
  double dx, dy, dz;
  delta(pi, pj, a.sx, a.sy, a.sz, dx, dy, dz);
  const double r2 = dx * dx + dy * dy + dz * dz;
  const PairTab<double>& T = static_cast<const PairTab<double>*>(S.tab)[row0 + ptype(pj)];
  double fr = 0.0, ep;
  const bool hit = valid && (CG ? cg_term<double, false>(T, r2, fr, ep) : fg_term<double, false>(T, r2, fr, ep));
  d[0] = hit ? dx : 0.0;
  d[1] = hit ? dy : 0.0;
  d[2] = hit ? dz : 0.0;
  return hit ? fr : 0.0;
}

// FP64 forces of small systems (too few slots to occupy the part with one
// thread each): TPA lanes per slot, and the same bits as one lane.  In each
// round the TPA lanes of a slot evaluate one chunk each (TPA x 4 consecutive
// entries); lanes 0, 1 and 2 of the slot then add the x, y and z terms of
// those entries in list order with the one-lane walk's operation (fma),
// taking each entry's force factor and difference from the lane that
// evaluated it.  A padding entry or a pair past the cutoff adds fma(0, 0, f)
// = f.  Every lane of the warp runs the warp's largest number of rounds (the
// shuffles take all 32 lanes).
template <bool CG, int TPA>
__device__ __forceinline__ void walk_ordered(const ListWalk<double>& L, int blk, const SmemTabs& S,
                                             const PairLaunch<double>& a) {
  static_assert(TPA >= 4 && 32 % TPA == 0, "three lanes per slot add the components");
  const int t = blk * blockDim.x + threadIdx.x;
  const int s = t / TPA, q = t % TPA;
  const int base = (threadIdx.x & 31) - q;  // the slot's first lane in the warp
  const bool own = s < L.nslots;
  const int ss = own ? s : 0;  // a valid slot for the loads of the other lanes
  const Pos64 pi = L.pos[ss];
  const int row0 = ptype(pi) * a.nt;
  const int m = own ? L.cnt[s] : 0;
  const int nch = (m + 3) >> 2;
  const int nround_w = __reduce_max_sync(0xffffffffu, (nch + TPA - 1) / TPA);
  const int4* nb4 = reinterpret_cast<const int4*>(L.nbr) + ss;
  double f = 0.0;  // lanes 0, 1, 2 of the slot: its force component q
  for (int r = 0; r < nround_w; ++r) {
    const int ch = r * TPA + q;
    const int rem = ch < nch ? m - 4 * ch : 0;
    int4 jj = make_int4(ss, ss, ss, ss);
    if (rem > 0) jj = __ldcs(nb4 + size_t(ch) * L.nslots);
    const int jv[4] = {rem > 0 ? jj.x : ss, rem > 1 ? jj.y : ss, rem > 2 ? jj.z : ss, rem > 3 ? jj.w : ss};
    double fr[4], d[4][3];
#pragma unroll
    for (int e = 0; e < 4; ++e) fr[e] = term64<CG>(pi, load_pos(L.pos, jv[e]), rem > e, row0, S, a, d[e]);
    for (int k = 0; k < TPA; ++k) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const double frk = __shfl_sync(0xffffffffu, fr[e], base + k);
        const double xk = __shfl_sync(0xffffffffu, d[e][0], base + k);
        const double yk = __shfl_sync(0xffffffffu, d[e][1], base + k);
        const double zk = __shfl_sync(0xffffffffu, d[e][2], base + k);
        f = fma(frk, q == 0 ? xk : (q == 1 ? yk : zk), f);
      }
    }
  }
  if (own && q < 3) L.f_out[3 * size_t(L.perm[s]) + q] = f;
}

// One slot's walk over its list, four entries per iteration.  TPA lanes share
// one slot (threads per atom, chosen by the autotuner): lane q of the slot
// takes chunks q, q + TPA, ... and the partial forces are summed with warp
// shuffles.  Energy steps use TPA = 1.
// PRN (pruning launches, TPA = 1): the slot walks its full list, and every
// entry within the pruning radius is appended, in list order, to its pruned
// list; the forces are the same bits as a walk of the pruned list (a dropped
// entry adds exactly zero).
template <typename R, bool CG, bool EV, int TPA, bool PRN, int ACC>
__device__ __forceinline__ void walk(const ListWalk<R>& L, int blk, const SmemTabs& S,
                                     const PairLaunch<R>& a, bool first_block) {
  static_assert(!PRN || TPA == 1, "pruning launches use one thread per slot");
  const int t = blk * blockDim.x + threadIdx.x;
  const int s = t / TPA;
  const int q = t % TPA;
  Acc<R> A;
  int kept = 0;
  if (s < L.nslots) {
    const auto pi = L.pos[s];
    const int row0 = ptype(pi) * a.nt;
    const int m = PRN ? L.cnt_full[s] : L.cnt[s];
    const int nch = (m + 3) >> 2;
    const int4* nb4 = reinterpret_cast<const int4*>(PRN ? L.nbr_full : L.nbr) + s;
    int4* out4 = reinterpret_cast<int4*>(L.nbr_in) + s;
    int4 buf = make_int4(s, s, s, s);
    int4 jj = make_int4(s, s, s, s);
    if (q < nch) jj = __ldcs(nb4 + size_t(q) * L.nslots);
    for (int ch = q; ch < nch; ch += TPA) {
      int4 jn = jj;
      if (ch + TPA < nch) jn = __ldcs(nb4 + size_t(ch + TPA) * L.nslots);
      const int rem = m - 4 * ch;  // >= 1
      const int j1 = rem > 1 ? jj.y : s, j2 = rem > 2 ? jj.z : s, j3 = rem > 3 ? jj.w : s;
      const auto p0 = load_pos(L.pos, jj.x);
      const auto p1 = load_pos(L.pos, j1);
      const auto p2 = load_pos(L.pos, j2);
      const auto p3 = load_pos(L.pos, j3);
      const R r0 = entry<R, CG, EV, ACC>(pi, p0, true, row0, S, a, A);
      const R r1 = entry<R, CG, EV, ACC>(pi, p1, rem > 1, row0, S, a, A);
      const R r2 = entry<R, CG, EV, ACC>(pi, p2, rem > 2, row0, S, a, A);
      const R r3 = entry<R, CG, EV, ACC>(pi, p3, rem > 3, row0, S, a, A);
      acc_chunk<ACC>(A);
      if (PRN) {
        keep_entry(r0 < L.rp2, jj.x, kept, buf, out4, L.nslots);
        keep_entry(r1 < L.rp2, j1, kept, buf, out4, L.nslots);
        keep_entry(r2 < L.rp2, j2, kept, buf, out4, L.nslots);
        keep_entry(r3 < L.rp2, j3, kept, buf, out4, L.nslots);
      }
      jj = jn;
    }
    if (PRN) {
      keep_tail(kept, buf, out4, L.nslots);
      L.cnt_in[s] = kept;
      if (!CG) a.ref_p[L.perm[s]] = ref_of(pi);
    }
  }
  if (PRN) {
    unsigned long long v[1] = {(unsigned long long)kept};
    __shared__ unsigned long long sh_k[1024 / 32];
    block_sum<unsigned long long, 1>(v, sh_k);
    if (threadIdx.x == 0) {
      atomicAdd(L.tot_in, v[0]);
      if (first_block) atomicAdd(&a.st->n_prunes, 1ull);
    }
  }
  acc_final<ACC>(A);
  if (TPA > 1) {  // every lane of the warp takes part (TPA divides 32)
#pragma unroll
    for (int o = TPA / 2; o > 0; o >>= 1) {
      A.fx += __shfl_xor_sync(0xffffffffu, A.fx, o);
      A.fy += __shfl_xor_sync(0xffffffffu, A.fy, o);
      A.fz += __shfl_xor_sync(0xffffffffu, A.fz, o);
    }
  }
  if (s < L.nslots && q == 0) store_force(L.f_out, L.perm[s], A.fx, A.fy, A.fz);
  if (EV) {
    double accd[kNQ];
    __shared__ double sh[(1024 / 32) * kNQ];
    accd[0] = double(A.e);
#pragma unroll
    for (int k = 0; k < 6; ++k) accd[k + 1] = double(A.w[k]);
    block_sum<double, kNQ>(accd, sh);
    if (threadIdx.x == 0) {
      // full lists: every pair was visited from both ends
#pragma unroll
      for (int k = 0; k < kNQ; ++k) acc_add(L.acc + k, 0.5 * accd[k]);
    }
  }
}

// FP32 launches are held to 64 registers a thread (the occupancy of the walk
// without pruning); the pruning walk lives in the same kernel.
template <typename R>
constexpr int pair_min_blocks(int bs) {
  return !std::is_same<R, float>::value ? 1 : 65536 / (64 * bs);
}

// One launch per step: with pruning on (one thread per slot) the kernel reads
// the device flags and, if a rebuild or the pruning trigger fired this step,
// walks the full lists and writes the pruned ones as it goes.
// The work of block `bid` of one system's pair launch.
template <typename R, bool EV, int TPA, int ACC>
__device__ __forceinline__ void pair_block(const PairLaunch<R>& a, int bid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nrow = a.nt * a.nt;
  size_t off = 0;
  auto carve = [&](size_t bytes) {
    unsigned char* p = smem_raw + off;
    off += (bytes + 15) / 16 * 16;
    return p;
  };
  SmemTabs S{};
  if constexpr (std::is_same<R, float>::value) {
    PairRow* row = reinterpret_cast<PairRow*>(carve(sizeof(PairRow) * nrow));
    copy_words(row, a.tab, nrow * int(sizeof(PairRow) / sizeof(int)));
    S.row = row;
  } else {
    PairTab<R>* tab = reinterpret_cast<PairTab<R>*>(carve(sizeof(PairTab<R>) * nrow));
    copy_words(tab, a.tab, nrow * int(sizeof(PairTab<R>) / sizeof(int)));
    S.tab = tab;
  }
  __syncthreads();
  const bool cg = bid < a.nblk_cg;
  const int blk = cg ? bid : bid - a.nblk_cg;
  if constexpr (!std::is_same<R, float>::value && TPA > 1) {
    static_assert(!EV, "FP64 energy steps use one thread per slot");
    if (cg)
      walk_ordered<true, TPA>(a.cg, blk, S, a);
    else
      walk_ordered<false, TPA>(a.fg, blk, S, a);
  } else {
    if constexpr (TPA == 1) {
      if (a.prune_on && (*(volatile const unsigned*)a.gate & (F_REBUILD | F_PRUNE)) != 0u) {
        if (cg)
          walk<R, true, EV, 1, true, ACC>(a.cg, blk, S, a, bid == 0);
        else
          walk<R, false, EV, 1, true, ACC>(a.fg, blk, S, a, bid == 0);
        return;
      }
    }
    if (cg)
      walk<R, true, EV, TPA, false, ACC>(a.cg, blk, S, a, bid == 0);
    else
      walk<R, false, EV, TPA, false, ACC>(a.fg, blk, S, a, bid == 0);
  }
}

template <typename R, bool EV, int TPA, int BS, int ACC>
__global__ void __launch_bounds__(BS, pair_min_blocks<R>(BS)) k_pair(PairLaunch<R> a) {
  // the force sum that follows may start launching once every block of this
  // grid runs (it waits for this grid to finish before reading the forces)
  grid_dependents_launch();
  pair_block<R, EV, TPA, ACC>(a, blockIdx.x);
}

// Batches (relres_batch_step): one launch over the pair work of every replica.
// Block b belongs to the replica r with off[r] <= b < off[r + 1]; its
// arguments are the replica's PairLaunch in device memory.
template <typename R, bool EV, int ACC>
__global__ void __launch_bounds__(kThreads, pair_min_blocks<R>(kThreads))
    k_pair_batch(const PairLaunch<R>* __restrict__ args, const int* __restrict__ off, int nrep) {
  const int r = batch_replica(off, nrep, blockIdx.x);
  pair_block<R, EV, 1, ACC>(args[r], int(blockIdx.x) - off[r]);
}

template <typename R>
static size_t pair_smem(int nt) {
  const size_t row = std::is_same<R, float>::value ? sizeof(PairRow) : sizeof(PairTab<double>);
  return (row * nt * nt + 15) / 16 * 16;
}

// FP32 forces with one of the launch configurations of one system, the
// owner's force sum kept as ACC (relres_accumulation)
template <int ACC>
static void launch_forces_f32(relres_ctx* c, const PairLaunch<float>& a, int grid, size_t smem) {
  switch (c->pair_cfg) {
#define RELRES_PAIR_CASE(k, T, B) \
  case k:                         \
    k_pair<float, false, T, B, ACC><<<grid, B, smem, c->stream>>>(a); \
    break;
    RELRES_PAIR_CASE(0, 1, 256)
    RELRES_PAIR_CASE(1, 1, 128)
    RELRES_PAIR_CASE(2, 1, 512)
    RELRES_PAIR_CASE(3, 2, 256)
    RELRES_PAIR_CASE(4, 4, 256)
    RELRES_PAIR_CASE(5, 8, 256)
    RELRES_PAIR_CASE(6, 2, 128)
#undef RELRES_PAIR_CASE
  }
}

// Arguments of one system's pair launch with `per` slots per block; returns
// the number of blocks (0: nothing to do).
// prune_in_kernel: the launch prunes as it walks when it is due (else the
// lists were pruned beforehand by k_prune, or pruning is off)
template <typename R>
static int make_pair_launch(const relres_ctx* c, int which, int per, bool prune_in_kernel, PairLaunch<R>* out) {
  const double unit = std::is_same<R, float>::value ? 4294967296.0 : 18446744073709551616.0;
  PairLaunch<R> a{};
  a.sx = R(c->box[0] / unit);
  a.sy = R(c->box[1] / unit);
  a.sz = R(c->box[2] / unit);
  a.sxl = float(c->box[0] / unit - double(a.sx));
  a.syl = float(c->box[1] / unit - double(a.sy));
  a.szl = float(c->box[2] / unit - double(a.sz));
  a.nt = c->n_types;
  a.tab = c->d_tab;
  a.tabe = static_cast<const PairRowEnergy*>(c->d_tabe);
  a.gate = &c->d_state->flags;
  a.ref_p = c->d_ref_p;
  a.st = c->d_state;
  const typename PosOf<R>::T* pfg;
  const typename PosOf<R>::T* pcg;
  if constexpr (std::is_same<R, float>::value) {
    pfg = c->d_pos_fg;
    pcg = c->d_pos_cg;
  } else {
    pfg = c->d_pos_fg64;
    pcg = c->d_pos_cg64;
  }
  const bool do_fg = (which & 1) != 0;
  const bool do_cg = (which & 2) && c->has_cg && c->n_h > 0;
  const R rf = R(c->rlist_fg_cut + c->prune_delta + kPruneSlack);
  a.fg = ListWalk<R>{c->n, pfg, walk_nbr_fg(c), walk_cnt_fg(c), c->d_perm_fg,
                     static_cast<ForceOut<R>*>(c->d_f_fg), c->d_acc + kAccFg,
                     c->d_nbr_fg, c->d_cnt_fg, c->d_nbr_fg_in, c->d_cnt_fg_in, rf * rf,
                     &c->d_state->tot_in_fg};
  // without a CG list the CG walk is never entered; its pointers are stand-ins
  if (do_cg) {
    const R rc = R(c->rlist_cg_cut + c->prune_delta + kPruneSlack);
    a.cg = ListWalk<R>{c->n_h, pcg, walk_nbr_cg(c), walk_cnt_cg(c), c->d_perm_cg,
                       static_cast<ForceOut<R>*>(c->d_f_cg), c->d_acc + kAccCg,
                       c->d_nbr_cg, c->d_cnt_cg, c->d_nbr_cg_in, c->d_cnt_cg_in, rc * rc,
                       &c->d_state->tot_in_cg};
  } else {
    a.cg = a.fg;
  }
  a.prune_on = prune_in_kernel ? 1 : 0;
  const int nb_fg = do_fg ? (c->n + per - 1) / per : 0;
  const int nb_cg = do_cg ? (c->n_h + per - 1) / per : 0;
  a.nblk_cg = nb_cg;
  *out = a;
  return nb_cg + nb_fg;
}

static cudaError_t launch_pairs_f64(relres_ctx* c, bool ev, int which) {
  const size_t smem = pair_smem<double>(c->n_types);
  // FP64 runs at under 2 FMA per clock per SM on this part: a system with
  // fewer 256-slot blocks than SMs spreads its slots over more SMs in 32-thread
  // blocks, and a smaller one its forces-only walks over several threads per
  // slot (walk_ordered: the same bits as one thread)
  const int bs = fp64_pair_block(c), tpa = ev ? 1 : fp64_pair_tpa(c);
  PairLaunch<double> a;
  const int grid = make_pair_launch<double>(c, which, bs / tpa, pairs_prune(c), &a);
  if (grid == 0) return cudaSuccess;
  if (bs == 32) {
    if (ev)
      k_pair<double, true, 1, 32, 0><<<grid, 32, smem, c->stream>>>(a);
    else if (tpa == kFp64SmallTpa)
      k_pair<double, false, kFp64SmallTpa, 32, 0><<<grid, 32, smem, c->stream>>>(a);
    else
      k_pair<double, false, 1, 32, 0><<<grid, 32, smem, c->stream>>>(a);
  } else if (ev) {
    k_pair<double, true, 1, kThreads, 0><<<grid, kThreads, smem, c->stream>>>(a);
  } else {
    k_pair<double, false, 1, kThreads, 0><<<grid, kThreads, smem, c->stream>>>(a);
  }
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

static cudaError_t launch_pairs_f32(relres_ctx* c, bool ev, int which) {
  const PairConfig& cfg = kPairConfigs[c->pair_cfg];
  const int lanes = ev ? fp32_lanes(c, true) : c->pair_lanes;  // 0: this file's kernels
  PairLaunch<float> a;
  const int per = lanes ? kLaneThreads / lanes : cfg.bs / cfg.tpa;
  const int grid = make_pair_launch<float>(c, which, per, pairs_prune(c), &a);
  if (grid == 0) return cudaSuccess;
  if (lanes) {
    launch_pairs_lanes(c->stream, c->force_acc, a, ev, lanes, grid);
  } else {
    const size_t smem = pair_smem<float>(c->n_types);
    if (c->force_acc == RELRES_ACC_FP32)
      launch_forces_f32<RELRES_ACC_FP32>(c, a, grid, smem);
    else if (c->force_acc == RELRES_ACC_COMPENSATED)
      launch_forces_f32<RELRES_ACC_COMPENSATED>(c, a, grid, smem);
    else
      launch_forces_f32<RELRES_ACC_FP64>(c, a, grid, smem);
  }
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

// ---- batches: the argument tables of every replica (pruning in the walk)
// uploaded once per captured graph.  Forces-only and energy launches may
// differ in slots per block, so each has its own table.
template <typename R>
static cudaError_t prepare_pairs_table(const std::vector<relres_ctx*>& cs, int per, BatchLaunch* b) {
  std::vector<PairLaunch<R>> args(cs.size());
  std::vector<int> off(cs.size() + 1, 0);
  int nt_max = 1;
  for (size_t r = 0; r < cs.size(); ++r) {
    off[r + 1] = off[r] + make_pair_launch<R>(cs[r], 3, per, cs[r]->prune_on, &args[r]);
    nt_max = std::max(nt_max, cs[r]->n_types);
  }
  b->nblk = off.back();
  b->nt = nt_max;
  return upload_batch(b, args.data(), sizeof(PairLaunch<R>) * args.size(), off);
}

cudaError_t prepare_pairs_batch(const std::vector<relres_ctx*>& cs, BatchLaunch* b, BatchLaunch* b_ev) {
  if (cs[0]->fp64) {
    const cudaError_t e = prepare_pairs_table<double>(cs, kThreads, b);
    return e != cudaSuccess ? e : prepare_pairs_table<double>(cs, kThreads, b_ev);
  }
  long long slots = 0;
  for (const relres_ctx* c : cs) slots += pair_slots(c);
  const int acc = cs[0]->force_acc, lanes = fp32_lanes_for(slots, acc, false);
  b->lanes = lanes > 1 ? lanes : 0;
  b_ev->lanes = fp32_lanes_for(slots, acc, true);
  const cudaError_t e = prepare_pairs_table<float>(cs, b->lanes ? kLaneThreads / b->lanes : kThreads, b);
  return e != cudaSuccess ? e : prepare_pairs_table<float>(cs, kLaneThreads / b_ev->lanes, b_ev);
}

template <int ACC>
static void launch_pairs_batch_f32(cudaStream_t s, const BatchLaunch& b, int nrep) {
  k_pair_batch<float, false, ACC><<<b.nblk, kThreads, pair_smem<float>(b.nt), s>>>(
      static_cast<const PairLaunch<float>*>(b.d_args), b.d_off, nrep);
}

cudaError_t launch_pairs_batch(cudaStream_t s, bool fp64, int acc, bool ev, const BatchLaunch& b, int nrep) {
  if (b.nblk == 0) return cudaSuccess;
  if (fp64) {
    const auto* args = static_cast<const PairLaunch<double>*>(b.d_args);
    const size_t smem = pair_smem<double>(b.nt);
    if (ev)
      k_pair_batch<double, true, 0><<<b.nblk, kThreads, smem, s>>>(args, b.d_off, nrep);
    else
      k_pair_batch<double, false, 0><<<b.nblk, kThreads, smem, s>>>(args, b.d_off, nrep);
  } else if (b.lanes) {
    launch_pairs_lanes_batch(s, acc, ev, b, nrep);
  } else if (acc == RELRES_ACC_FP32) {
    launch_pairs_batch_f32<RELRES_ACC_FP32>(s, b, nrep);
  } else if (acc == RELRES_ACC_COMPENSATED) {
    launch_pairs_batch_f32<RELRES_ACC_COMPENSATED>(s, b, nrep);
  } else {
    launch_pairs_batch_f32<RELRES_ACC_FP64>(s, b, nrep);
  }
  return cudaGetLastError();
}

bool pairs_prune(const relres_ctx* c) {
  if (!c->prune_on) return false;
  return c->fp64 ? fp64_pair_tpa(c) == 1 : kPairConfigs[c->pair_cfg].tpa == 1;
}

cudaError_t launch_pairs(relres_ctx* c, bool ev, int which) {
  return c->fp64 ? launch_pairs_f64(c, ev, which) : launch_pairs_f32(c, ev, which);
}

}  // namespace relres
