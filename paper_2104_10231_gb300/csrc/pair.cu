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
// registers and writes it once (no atomics).  FP32 energy steps, and the FP32
// forces of systems too small to fill the part with one thread per slot, are
// in pair_lanes.cu; FP64 contexts in pair64.cu.
#include "pair.cuh"

namespace relres {

// One list entry; returns its squared distance (past every cutoff for a
// padding entry), which a pruning launch compares with the pruning radius.
template <bool CG, int ACC>
__device__ __forceinline__ float entry(const int4& pi, const int4& pj, bool valid, int row0, const SmemTabs& S,
                                       const PairLaunch& a, Acc& A) {
  float fr, dx, dy, dz;
  const float r2 = pair_term<CG>(pi, pj, valid, S.row[row0 + pj.w], a.sx, a.sy, a.sz, fr, dx, dy, dz);
  acc_force<ACC>(A, fr, dx, dy, dz);
  return r2;
}

// One slot's walk over its list, four entries per iteration.  TPA lanes share
// one slot (threads per atom, chosen by the autotuner): lane q of the slot
// takes chunks q, q + TPA, ... and the partial forces are summed with warp
// shuffles.
// PRN (pruning launches, TPA = 1): the slot walks its full list, and every
// entry within the pruning radius is appended, in list order, to its pruned
// list; the forces are the same bits as a walk of the pruned list (a dropped
// entry adds exactly zero).
template <bool CG, int TPA, bool PRN, int ACC>
__device__ __forceinline__ void walk(const ListWalk& L, int blk, const SmemTabs& S, const PairLaunch& a,
                                     bool first_block) {
  static_assert(!PRN || TPA == 1, "pruning launches use one thread per slot");
  const int t = blk * blockDim.x + threadIdx.x;
  const int s = t / TPA;
  const int q = t % TPA;
  Acc A;
  int kept = 0;
  if (s < L.nslots) {
    const int4 pi = L.pos[s];
    const int row0 = pi.w * a.nt;
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
      const int4 p0 = load_pos(L.pos, jj.x);
      const int4 p1 = load_pos(L.pos, j1);
      const int4 p2 = load_pos(L.pos, j2);
      const int4 p3 = load_pos(L.pos, j3);
      const float r0 = entry<CG, ACC>(pi, p0, true, row0, S, a, A);
      const float r1 = entry<CG, ACC>(pi, p1, rem > 1, row0, S, a, A);
      const float r2 = entry<CG, ACC>(pi, p2, rem > 2, row0, S, a, A);
      const float r3 = entry<CG, ACC>(pi, p3, rem > 3, row0, S, a, A);
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
      if (!CG) a.ref_p[L.perm[s]] = pi;
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
}

// Launches are held to 64 registers a thread (the occupancy of the walk
// without pruning); the pruning walk lives in the same kernel.
constexpr int pair_min_blocks(int bs) { return 65536 / (64 * bs); }

// One launch per step: with pruning on (one thread per slot) the kernel reads
// the device flags and, if a rebuild or the pruning trigger fired this step,
// walks the full lists and writes the pruned ones as it goes.
// The work of block `bid` of one system's pair launch.
template <int TPA, int ACC>
__device__ __forceinline__ void pair_block(const PairLaunch& a, int bid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  PairRow* const row = reinterpret_cast<PairRow*>(smem_raw);
  copy_words(row, a.tab, a.nt * a.nt * int(sizeof(PairRow) / sizeof(int)));
  const SmemTabs S{row, nullptr};
  after_rebuild();
  if (lists_unpruned(a)) return;
  __syncthreads();
  const bool cg = bid < a.nblk_cg;
  const int blk = cg ? bid : bid - a.nblk_cg;
  if constexpr (TPA == 1) {
    if (a.prune_on && (*(volatile const unsigned*)a.gate & (F_REBUILD | F_PRUNE)) != 0u) {
      if (cg)
        walk<true, 1, true, ACC>(a.cg, blk, S, a, bid == 0);
      else
        walk<false, 1, true, ACC>(a.fg, blk, S, a, bid == 0);
      return;
    }
  }
  if (cg)
    walk<true, TPA, false, ACC>(a.cg, blk, S, a, bid == 0);
  else
    walk<false, TPA, false, ACC>(a.fg, blk, S, a, bid == 0);
}

template <int TPA, int BS, int ACC>
__global__ void __launch_bounds__(BS, pair_min_blocks(BS)) k_pair(PairLaunch a) {
  pair_block<TPA, ACC>(a, blockIdx.x);
}

// Batches (relres_batch_step): one launch over the pair work of every replica.
// Block b belongs to the replica r with off[r] <= b < off[r + 1]; its
// arguments are the replica's PairLaunch in device memory.
template <int ACC>
__global__ void __launch_bounds__(kThreads, pair_min_blocks(kThreads))
    k_pair_batch(const PairLaunch* __restrict__ args, const int* __restrict__ off, int nrep) {
  const int r = batch_replica(off, nrep, blockIdx.x);
  pair_block<1, ACC>(args[r], int(blockIdx.x) - off[r]);
}

static size_t pair_smem(int nt) { return sizeof(PairRow) * nt * nt; }

// Forces with one of the launch configurations of one system, the owner's
// force sum kept as ACC (relres_accumulation)
template <int ACC>
static void launch_forces(relres_ctx* c, const PairLaunch& a, int grid, size_t smem) {
  switch (c->pair_cfg) {
#define RELRES_PAIR_CASE(k, T, B) \
  case k:                         \
    launch_pdl(pair_pdl(c, grid, B), k_pair<T, B, ACC>, grid, B, smem, c->stream, a); \
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
static int make_pair_launch(const relres_ctx* c, int which, int per, bool prune_in_kernel, PairLaunch* out) {
  const double unit = 4294967296.0;
  PairLaunch a{};
  a.sx = float(c->box[0] / unit);
  a.sy = float(c->box[1] / unit);
  a.sz = float(c->box[2] / unit);
  a.sxl = float(c->box[0] / unit - double(a.sx));
  a.syl = float(c->box[1] / unit - double(a.sy));
  a.szl = float(c->box[2] / unit - double(a.sz));
  a.nt = c->n_types;
  a.tab = static_cast<const PairRow*>(c->d_tab);
  a.tabe = static_cast<const PairRowEnergy*>(c->d_tabe);
  a.gate = &c->d_state->flags;
  a.ref_p = c->d_ref_p;
  a.st = c->d_state;
  const bool do_fg = (which & 1) != 0;
  const bool do_cg = (which & 2) && c->has_cg && c->n_h > 0;
  const float rf = float(c->rlist_fg_cut + c->prune_delta + kPruneSlack);
  a.fg = ListWalk{c->n, c->d_pos_fg, walk_nbr_fg(c), walk_cnt_fg(c), c->d_perm_fg,
                  static_cast<float4*>(c->d_f_fg), c->d_acc + kAccFg,
                  c->d_nbr_fg, c->d_cnt_fg, c->d_nbr_fg_in, c->d_cnt_fg_in, rf * rf,
                  &c->d_state->tot_in_fg};
  // without a CG list the CG walk is never entered; its pointers are stand-ins
  if (do_cg) {
    const float rc = float(c->rlist_cg_cut + c->prune_delta + kPruneSlack);
    a.cg = ListWalk{c->n_h, c->d_pos_cg, walk_nbr_cg(c), walk_cnt_cg(c), c->d_perm_cg,
                    static_cast<float4*>(c->d_f_cg), c->d_acc + kAccCg,
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

// threads per slot of pair_lanes.cu for this launch (0: this file's kernels)
static int launch_lanes(const relres_ctx* c, bool ev) { return ev ? fp32_lanes(c, true) : c->pair_lanes; }

PairShape pair_shape(const relres_ctx* c, bool ev) {
  if (c->fp64) return PairShape{fp64_lanes(c, ev), kFp64Block};
  const int lanes = launch_lanes(c, ev);
  if (lanes) return PairShape{lanes, kLaneThreads};
  return PairShape{kPairConfigs[c->pair_cfg].tpa, kPairConfigs[c->pair_cfg].bs};
}

static cudaError_t launch_pairs_f32(relres_ctx* c, bool ev, int which) {
  const int lanes = launch_lanes(c, ev);
  const PairShape shape = pair_shape(c, ev);
  PairLaunch a;
  const int grid = make_pair_launch(c, which, shape.block / shape.threads, pairs_prune(c), &a);
  if (grid == 0) return cudaSuccess;
  if (lanes) {
    launch_pairs_lanes(c->stream, c->force_acc, a, ev, lanes, grid, pair_pdl(c, grid, kLaneThreads));
  } else {
    const size_t smem = pair_smem(c->n_types);
    if (c->force_acc == RELRES_ACC_FP32)
      launch_forces<RELRES_ACC_FP32>(c, a, grid, smem);
    else if (c->force_acc == RELRES_ACC_COMPENSATED)
      launch_forces<RELRES_ACC_COMPENSATED>(c, a, grid, smem);
    else
      launch_forces<RELRES_ACC_FP64>(c, a, grid, smem);
  }
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

// ---- batches: the argument tables of every replica (pruning in the walk)
// uploaded once per captured graph.  Forces-only and energy launches may
// differ in slots per block, so each has its own table.
static cudaError_t prepare_pairs_table(const std::vector<relres_ctx*>& cs, int per, BatchLaunch* b) {
  std::vector<PairLaunch> args(cs.size());
  std::vector<int> off(cs.size() + 1, 0);
  b->nt = 1;
  for (size_t r = 0; r < cs.size(); ++r) {
    off[r + 1] = off[r] + make_pair_launch(cs[r], 3, per, cs[r]->prune_on, &args[r]);
    b->nt = std::max(b->nt, cs[r]->n_types);
  }
  b->nblk = off.back();
  return upload_batch(b, args.data(), sizeof(PairLaunch) * args.size(), off);
}

cudaError_t prepare_pairs_batch(const std::vector<relres_ctx*>& cs, BatchLaunch* b, BatchLaunch* b_ev) {
  if (cs[0]->fp64) return prepare_pairs_batch_f64(cs, b, b_ev);
  long long slots = 0;
  for (const relres_ctx* c : cs) slots += pair_slots(c);
  const int acc = cs[0]->force_acc, lanes = fp32_lanes_for(slots, acc, false);
  b->lanes = lanes > 1 ? lanes : 0;
  b_ev->lanes = fp32_lanes_for(slots, acc, true);
  const cudaError_t e = prepare_pairs_table(cs, b->lanes ? kLaneThreads / b->lanes : kThreads, b);
  return e != cudaSuccess ? e : prepare_pairs_table(cs, kLaneThreads / b_ev->lanes, b_ev);
}

template <int ACC>
static void launch_forces_batch(cudaStream_t s, const BatchLaunch& b, int nrep) {
  k_pair_batch<ACC><<<b.nblk, kThreads, pair_smem(b.nt), s>>>(static_cast<const PairLaunch*>(b.d_args), b.d_off, nrep);
}

cudaError_t launch_pairs_batch(cudaStream_t s, bool fp64, int acc, bool ev, const BatchLaunch& b, int nrep) {
  if (b.nblk == 0) return cudaSuccess;
  if (fp64)
    launch_pairs_batch_f64(s, ev, b, nrep);
  else if (b.lanes)
    launch_pairs_lanes_batch(s, acc, ev, b, nrep);
  else if (acc == RELRES_ACC_FP32)
    launch_forces_batch<RELRES_ACC_FP32>(s, b, nrep);
  else if (acc == RELRES_ACC_COMPENSATED)
    launch_forces_batch<RELRES_ACC_COMPENSATED>(s, b, nrep);
  else
    launch_forces_batch<RELRES_ACC_FP64>(s, b, nrep);
  return cudaGetLastError();
}

bool pairs_prune(const relres_ctx* c) {
  return c->prune_on && (c->fp64 || kPairConfigs[c->pair_cfg].tpa == 1);
}

cudaError_t launch_pairs(relres_ctx* c, bool ev, int which) {
  return c->fp64 ? launch_pairs_f64(c, ev, which) : launch_pairs_f32(c, ev, which);
}

}  // namespace relres
