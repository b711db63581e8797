// RelRes pair launches of FP64 contexts: the terms of pair.cu in double, from
// 64-bit fixed-point positions.
//
// FP64 runs at 1.66 FMA per clock and SM on this part, 70 times below FP32, so
// the FP64 instructions a warp issues are what a launch costs.  One thread per
// list entry by entry issues every region's arithmetic for every entry (the
// lanes of a warp hold entries of all regions, and a quarter of the entries of
// a pruned list is past the cutoff): ~48 FP64 instructions an entry.  Here a
// warp takes 128 list entries at a time (T lanes per slot, four entries per
// lane), decides each one's region from its FP32 distance, and sorts the
// entries inside the cutoff by region in shared memory; full warps then
// evaluate 32 of them at a time, nearly always of one region, ~22 FP64
// instructions each: 116 us per step at 25 000 neopentane-like atoms, 24 us at
// 648 propane-like ones (200 and 65 entry by entry).  What is left is the FP64
// rate at 25 000 atoms, the latency of one warp's rounds at 648: fetching the
// partners of the next pass ahead gave 0 to 1 %.  A pair whose FP32 distance
// is too close to a region limit to tell the side (kNear) is kept whatever the
// side, and the FP64 distance decides when it is evaluated: the regions are
// those of an FP64 comparison (without the full shift the energy jumps at r_c+).
//
// The terms of a slot are stored by their rank in its list and added in list
// order to four sums by rank modulo four (one chain of a hundred additions by
// three lanes was a quarter of a 648-atom launch: a scheduler's FP64 unit
// takes a warp instruction every 65 cycles).  Entries past the cutoff are no
// terms (a CG pair below r_s- is none either: its constant energy is summed
// apart), so the forces are the same bits for every T, with and without
// energies and pruning.
#include "common.cuh"
#include "fbits.h"
#include "pair.cuh"

namespace relres {

struct Walk64 {
  int nslots;
  const Pos64* pos;
  const int4* pos32;  // the same positions, upper 32 bits and type
  const int* nbr;     // the list walked (pruned when pruning is on)
  const int* cnt;
  const int* perm;
  double* f_out;
  long long* acc;  // kNQ accumulators of this list (energy, six virial components)
  // pruning launches: walk the full list and write the pruned one
  const int* nbr_full;
  const int* cnt_full;
  int* nbr_in;
  int* cnt_in;
  float rp2;  // (interaction cutoff + delta + slack)^2
  unsigned long long* tot_in;
};

struct Launch64 {
  int nblk_cg;  // blocks [0, nblk_cg) walk the CG list, the rest the FG list
  Walk64 fg, cg;
  const PairTab<double>* tab;  // [nt^2]
  int nt;
  double sx, sy, sz;  // L / 2^64
  float fx, fy, fz;   // L / 2^32
  float near;         // share of r^2 within which FP32 does not decide a region
  const unsigned* gate;
  int prune_on;
  int4* ref_p;
  DevState* st;
};

// regions, in the order the entries are sorted by
enum { kCore = 0, kShell = 1, kFgRegions = 2 };                      // FG: LJ below r_s-, switching off
enum { kLj = 0, kOff = 1, kOn = 2, kCgRegions = 3 };                 // CG: below r_s- an energy only

// beside the place of an entry: the region is left to the FP64 distance
constexpr int kNear = 0x80;

// the region of a pair by its FP64 squared distance; past the cutoff (and, for
// the CG part, below r_s-) none: kOutside, kClose
enum { kOutside = 8, kClose = 9 };
template <bool CG>
__device__ __forceinline__ int region64(const PairTab<double>& T, double r2) {
  if (!CG) return !(r2 < T.rsp2) ? int(kOutside) : (r2 < T.rsm2 ? int(kCore) : int(kShell));
  if (!(r2 < T.rcp2)) return kOutside;
  if (r2 < T.rsm2) return kClose;
  return r2 < T.rsp2 ? int(kOn) : (r2 < T.rcm2 ? int(kLj) : int(kOff));
}

// values of a term: force, then (energy steps) energy and virial
constexpr int kTermF = 3, kTermEv = 3 + kNQ;

template <bool EV>
struct WarpTerms {
  double v[EV ? kTermEv : kTermF][128];  // by 4 T (slot in the warp) + rank in the slot's list
  long long px[32], py[32], pz[32];      // the slots' positions and first type-pair rows
  int row0[32];
  int j[128];  // the sorted entries: partner, FP32 squared distance, place in v
  float r2[128];
  unsigned short at[128];
};

// -u'(r)/r (and u) of one pair in the given region
template <bool CG, bool EV>
__device__ __forceinline__ void term64(int region, const PairTab<double>& T, double r2, float r2f, double& fr,
                                       double& e) {
  if (region == (CG ? int(kLj) : int(kCore))) {
    const double r2i = rcp_d(r2, r2f);
    const double r6i = r2i * r2i * r2i;
    fr = r6i * ((CG ? T.f12c : T.f12f) * r6i - (CG ? T.f6c : T.f6f)) * r2i;
    if (EV) e = r6i * ((CG ? T.c12c : T.c12f) * r6i - (CG ? T.c6c : T.c6f)) - (CG ? T.gam_cm : T.e_fg_shift);
    return;
  }
  if (region >= kOutside) {
    fr = 0.0;
    if (EV) e = CG && region == kClose ? T.e_cg_close : 0.0;
    return;
  }
  const double ri = rsqrt_d(r2, r2f);
  if (CG && region == kOn) {
    const double d = r2 * ri - T.rsm, d2 = d * d;
    fr = -(d2 * (T.ond4 * d + T.ond3)) * ri;
    if (EV) e = T.on0 + d2 * d * (T.on4 * d + T.on3) - T.gam_cm;
    return;
  }
  const double* g = CG ? T.cgo : T.fg;
  const double* gd = CG ? T.cgod : T.fgd;
  const double d = r2 * ri - (CG ? T.rcm : T.rsm);
  fr = -(((gd[3] * d + gd[2]) * d + gd[1]) * d + gd[0]) * ri;
  if (EV) e = ((((g[4] * d + g[3]) * d + g[2]) * d + g[1]) * d + g[0]) - (CG ? T.gam_cm : T.e_fg_shift);
}

// One warp's walk over the lists of its 32 / T slots.  thr: FP32 squared radii
// (r_s-, r_s+, r_c-, r_c+) per type pair.  Returns the entries this lane kept
// (pruning launches).
template <bool CG, bool EV, int T, bool PRN>
__device__ __forceinline__ unsigned long long walk64(const Walk64& L, int slot0, const PairTab<double>* tab,
                                                     const float4* thr, WarpTerms<EV>& W, const Launch64& a) {
  constexpr int NV = EV ? kTermEv : kTermF;
  constexpr int NG = T / 4;              // four lanes, one per chain, sum value g, g + NG, ...
  constexpr int NL = (NV + NG - 1) / NG;  // values of one lane
  constexpr int NR = CG ? int(kCgRegions) : int(kFgRegions);
  const int lane = threadIdx.x & 31, sl = lane / T, q = lane % T, chain = q & 3, g = q >> 2;
  const int s = slot0 + sl;
  const bool own = s < L.nslots;
  const int ss = own ? s : 0;  // a valid slot for the loads of the other lanes
  const int4 pi = L.pos32[ss];
  const int m = own ? (PRN ? L.cnt_full[s] : L.cnt[s]) : 0;
  const int nch = (m + 3) >> 2;
  const int4* nb4 = reinterpret_cast<const int4*>(PRN ? L.nbr_full : L.nbr) + ss;
  int4 jj = make_int4(ss, ss, ss, ss);
  if (q < nch) jj = __ldcs(nb4 + size_t(q) * L.nslots);
  if (q == 0) {
    const Pos64 p = L.pos[ss];
    W.px[sl] = p.x;
    W.py[sl] = p.y;
    W.pz[sl] = p.z;
    W.row0[sl] = pi.w * a.nt;
  }
  const int rounds = __reduce_max_sync(0xffffffffu, (nch + T - 1) / T);
  const int row0 = pi.w * a.nt;
  const unsigned below = (1u << lane) - 1u;
  const unsigned slot_mask = (T == 32 ? 0xffffffffu : ((1u << T) - 1u)) << (sl * T), before = slot_mask & below;
  double f[NL];
#pragma unroll
  for (int k = 0; k < NL; ++k) f[k] = 0.0;
  double close = 0.0;  // energy of the CG pairs below r_s-
  int kept = 0, done = 0;  // entries kept, terms added
  for (int r = 0; r < rounds; ++r) {
    const int ch = r * T + q;
    int4 jn = jj;
    if (ch + T < nch) jn = __ldcs(nb4 + size_t(ch + T) * L.nslots);
    const int rem = m - 4 * ch;  // <= 0 past the list
    const int j[4] = {rem > 0 ? jj.x : ss, rem > 1 ? jj.y : ss, rem > 2 ? jj.z : ss, rem > 3 ? jj.w : ss};
    float r2[4];
    int region[4], near[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int4 p = __ldg(L.pos32 + j[e]);
      const float dx = dfix32(pi.x, p.x, a.fx), dy = dfix32(pi.y, p.y, a.fy), dz = dfix32(pi.z, p.z, a.fz);
      r2[e] = rem > e ? dx * dx + dy * dy + dz * dz : 3.0e38f;
      const float4 t = thr[row0 + p.w];
      const float w = a.near * r2[e];
      float gap = fminf(fabsf(r2[e] - t.x), fabsf(r2[e] - t.y));
      if (CG) {
        gap = fminf(gap, fminf(fabsf(r2[e] - t.z), fabsf(r2[e] - t.w)));
        region[e] = !(r2[e] < t.w) || r2[e] < t.x ? -1 : (r2[e] < t.y ? int(kOn) : (r2[e] < t.z ? int(kLj) : int(kOff)));
      } else {
        region[e] = !(r2[e] < t.y) ? -1 : (r2[e] < t.x ? int(kCore) : int(kShell));
      }
      near[e] = gap <= w ? kNear : 0;
      if (near[e]) region[e] = max(region[e], 0);
      if (CG && EV && r2[e] < t.x && !near[e]) close += tab[row0 + p.w].e_cg_close;
    }
    // rank of each term in its slot's list order, and place in the sorted entries
    unsigned in[4];
    int rank = 0, terms = 0;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      in[e] = __ballot_sync(0xffffffffu, region[e] >= 0);
      rank += __popc(in[e] & before);
      terms += __popc(in[e] & slot_mask);
    }
    int total = 0, place[4] = {0, 0, 0, 0};
#pragma unroll
    for (int c = 0; c < NR; ++c)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const unsigned b = __ballot_sync(0xffffffffu, region[e] == c);
        if (region[e] == c) place[e] = total + __popc(b & below);
        total += __popc(b);
      }
    __syncwarp();  // the sums of the last round have been read
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (region[e] >= 0) {
        W.j[place[e]] = j[e];
        W.r2[place[e]] = r2[e];
        W.at[place[e]] = (unsigned short)(((region[e] | near[e]) << 8) | (4 * T * sl + rank));
        ++rank;
      }
    __syncwarp();
    for (int k = lane; k < total; k += 32) {
      const int at = W.at[k] & 0xff, from = at / (4 * T);
      const Pos64 p = L.pos[W.j[k]];
      const double dx = dfix64(W.px[from], p.x, a.sx), dy = dfix64(W.py[from], p.y, a.sy),
                   dz = dfix64(W.pz[from], p.z, a.sz);
      const PairTab<double>& T2 = tab[W.row0[from] + int(p.t)];
      const double r2d = fma(dz, dz, fma(dy, dy, dx * dx));
      int reg = W.at[k] >> 8;
      if (reg & kNear) reg = region64<CG>(T2, r2d);
      double fr, en = 0.0;
      term64<CG, EV>(reg, T2, r2d, W.r2[k], fr, en);
      const double tx = fr * dx, ty = fr * dy, tz = fr * dz;
      W.v[0][at] = tx;
      W.v[1][at] = ty;
      W.v[2][at] = tz;
      if constexpr (EV) {
        W.v[3][at] = en;
        W.v[4][at] = tx * dx;
        W.v[5][at] = ty * dy;
        W.v[6][at] = tz * dz;
        W.v[7][at] = tx * dy;
        W.v[8][at] = tx * dz;
        W.v[9][at] = ty * dz;
      }
    }
    __syncwarp();
    // four threads a slot: the sums of a round take as many additions as with
    // one chain a value, and its loads are issued together (forces only: 119.7
    // -> 116.4 us per step at 25 000 atoms) or a value of every lane at a time
    // (with energies, ten values a lane: 188 -> 174 us)
    const int k0 = (chain - done) & 3;
    if constexpr (T == 4 && !EV) {
#pragma unroll
      for (int v = 0; v < NL; ++v) {
        const double* const t = W.v[v] + 16 * sl + k0;
        double x[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) x[u] = k0 + 4 * u < terms ? t[4 * u] : 0.0;
#pragma unroll
        for (int u = 0; u < 4; ++u) f[v] += x[u];
      }
    } else if constexpr (T == 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (__any_sync(0xffffffffu, k0 + 4 * u < terms)) {
#pragma unroll
          for (int v = 0; v < NL; ++v) f[v] += k0 + 4 * u < terms ? W.v[v][16 * sl + k0 + 4 * u] : 0.0;
        }
    } else {
      for (int k = k0; k < terms; k += 4)
#pragma unroll
        for (int v = 0; v < NL; ++v)
          if (g + v * NG < NV) f[v] += W.v[g + v * NG][4 * T * sl + k];
    }
    done += terms;
    if constexpr (PRN) {
      int at = kept;
      unsigned b[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        b[e] = __ballot_sync(0xffffffffu, r2[e] < L.rp2);
        at += __popc(b[e] & before);
        kept += __popc(b[e] & slot_mask);
      }
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (r2[e] < L.rp2) {
          L.nbr_in[(size_t(at >> 2) * L.nslots + s) * 4 + (at & 3)] = j[e];
          ++at;
        }
    }
    jj = jn;
  }
#pragma unroll
  for (int v = 0; v < NL; ++v) {
    f[v] += __shfl_xor_sync(0xffffffffu, f[v], 1);
    f[v] += __shfl_xor_sync(0xffffffffu, f[v], 2);
  }
  if constexpr (CG && EV) {
#pragma unroll
    for (int o = T / 2; o > 0; o >>= 1) close += __shfl_xor_sync(0xffffffffu, close, o);
#pragma unroll
    for (int v = 0; v < NL; ++v)
      if (g + v * NG == kTermF) f[v] += close;
  }
  if (own) {
    const int i = L.perm[s];
    if (chain == 0) {
#pragma unroll
      for (int v = 0; v < NL; ++v)
        if (g + v * NG < kTermF) L.f_out[3 * size_t(i) + g + v * NG] = f[v];
    }
    if (PRN && q == 0) {
      L.cnt_in[s] = kept;
      if (!CG) a.ref_p[i] = pi;
    }
  }
  if constexpr (EV) {
    // the warp's slots added in slot order, then to the accumulators (full
    // lists: every pair was visited from both ends)
    __syncwarp();
#pragma unroll
    for (int v = 0; v < NL; ++v)
      if (chain == 0 && g + v * NG < NV) W.v[g + v * NG][sl] = own ? f[v] : 0.0;
    __syncwarp();
    if (lane < kNQ) {
      double t = 0.0;
      for (int k = 0; k < 32 / T; ++k) t += W.v[kTermF + lane][k];
      acc_add_fine(L.acc + lane, 0.5 * t);
    }
  }
  return own && q == 0 ? (unsigned long long)kept : 0ull;
}

// Whether a launch copies the type-pair rows to shared memory.  It does for up
// to two types at four threads per slot; else a term's few values come from
// global memory through the L1 cache, as the copy of every block (one warp; 22
// KB with eight types) costs more than it saves.  us per step, copied / read in
// place: 650 atoms (32 threads) of two types 26.1 / 24.2, of eight 51.0 / 24.3;
// 25 000 atoms (four) of two types 102.8 / 103.1, of four 112.2 / 103.4, of
// eight 200.9 / 104.2; 100 000 atoms 325.0 / 329.3, 328.2 / 329.6, 665 / 333.
static bool copies_rows(int lanes, int nt) { return lanes == 4 && nt <= 2; }

// shared memory of a block (one warp): FP32 radii, rows, terms
template <bool EV, bool COPY>
static size_t smem64(int nt) {
  return (sizeof(float4) + (COPY ? sizeof(PairTab<double>) : 0)) * size_t(nt) * nt + sizeof(WarpTerms<EV>);
}

template <bool EV, int T, bool COPY>
__device__ __forceinline__ void block64(const Launch64& a, int bid) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nrow = a.nt * a.nt;
  float4* const thr = reinterpret_cast<float4*>(smem_raw);
  PairTab<double>* const rows = reinterpret_cast<PairTab<double>*>(thr + nrow);
  const PairTab<double>* const tab = COPY ? rows : a.tab;
  WarpTerms<EV>& terms = *reinterpret_cast<WarpTerms<EV>*>(rows + (COPY ? nrow : 0));
  if (COPY) copy_words(rows, a.tab, nrow * int(sizeof(PairTab<double>) / sizeof(int)));
  for (int k = threadIdx.x; k < nrow; k += kFp64Block)
    thr[k] = make_float4(float(a.tab[k].rsm2), float(a.tab[k].rsp2), float(a.tab[k].rcm2), float(a.tab[k].rcp2));
  after_rebuild();
  __syncwarp();
  const bool cg = bid < a.nblk_cg;
  const int slot0 = (cg ? bid : bid - a.nblk_cg) * (32 / T);
  if (a.prune_on && (*(volatile const unsigned*)a.gate & (F_REBUILD | F_PRUNE)) != 0u) {
    const unsigned long long kept = warp_sum(cg ? walk64<true, EV, T, true>(a.cg, slot0, tab, thr, terms, a)
                                                : walk64<false, EV, T, true>(a.fg, slot0, tab, thr, terms, a));
    if (threadIdx.x == 0) {
      atomicAdd(cg ? a.cg.tot_in : a.fg.tot_in, kept);
      if (bid == 0) atomicAdd(&a.st->n_prunes, 1ull);
    }
  } else if (cg) {
    walk64<true, EV, T, false>(a.cg, slot0, tab, thr, terms, a);
  } else {
    walk64<false, EV, T, false>(a.fg, slot0, tab, thr, terms, a);
  }
}

template <bool EV, int T, bool COPY>
__global__ void __launch_bounds__(kFp64Block) k_pair64(Launch64 a) {
  block64<EV, T, COPY>(a, blockIdx.x);
}

template <bool EV, int T, bool COPY>
__global__ void __launch_bounds__(kFp64Block)
    k_pair64_batch(const Launch64* __restrict__ args, const int* __restrict__ off, int nrep) {
  const int r = batch_replica(off, nrep, blockIdx.x);
  block64<EV, T, COPY>(args[r], int(blockIdx.x) - off[r]);
}

// The FP32 squared distance of a pair and the FP64 one differ by less than this
// share of it at any region limit: each difference is rounded three times (the
// conversion, the box scale and its product) and the sum of squares three more,
// the limit once, 10 x 2^-24; the upper 32 bits of two coordinates are off by
// less than 2^-32 of the box each way, sqrt(3) of that in the distance.
static float near_share(const relres_ctx* c) {
  double rmin = c->tab_d[0].rsm;
  for (const PairTab<double>& t : c->tab_d) rmin = std::min(rmin, t.rsm);
  const double l = std::max(c->box[0], std::max(c->box[1], c->box[2]));
  return float(1e-6 + 4.0 / 4294967296.0 * l / std::max(rmin, 1e-3));
}

static int make_launch64(const relres_ctx* c, int which, int per, bool prune, Launch64* out) {
  Launch64 a{};
  a.near = near_share(c);
  a.sx = c->box[0] / 18446744073709551616.0;
  a.sy = c->box[1] / 18446744073709551616.0;
  a.sz = c->box[2] / 18446744073709551616.0;
  a.fx = float(c->box[0] / 4294967296.0);
  a.fy = float(c->box[1] / 4294967296.0);
  a.fz = float(c->box[2] / 4294967296.0);
  a.nt = c->n_types;
  a.tab = static_cast<const PairTab<double>*>(c->d_tab);
  a.gate = &c->d_state->flags;
  a.ref_p = c->d_ref_p;
  a.st = c->d_state;
  const bool do_fg = (which & 1) != 0;
  const bool do_cg = (which & 2) && c->has_cg && c->n_h > 0;
  const float rf = float(c->rlist_fg_cut + c->prune_delta + kPruneSlack);
  a.fg = Walk64{c->n, c->d_pos_fg64, c->d_pos_fg, walk_nbr_fg(c), walk_cnt_fg(c), c->d_perm_fg,
                static_cast<double*>(c->d_f_fg), c->d_acc + kAccFg, c->d_nbr_fg, c->d_cnt_fg, c->d_nbr_fg_in,
                c->d_cnt_fg_in, rf * rf, &c->d_state->tot_in_fg};
  a.cg = a.fg;  // a stand-in without a CG list
  if (do_cg) {
    const float rc = float(c->rlist_cg_cut + c->prune_delta + kPruneSlack);
    a.cg = Walk64{c->n_h, c->d_pos_cg64, c->d_pos_cg, walk_nbr_cg(c), walk_cnt_cg(c), c->d_perm_cg,
                  static_cast<double*>(c->d_f_cg), c->d_acc + kAccCg, c->d_nbr_cg, c->d_cnt_cg, c->d_nbr_cg_in,
                  c->d_cnt_cg_in, rc * rc, &c->d_state->tot_in_cg};
  }
  a.prune_on = prune ? 1 : 0;
  a.nblk_cg = do_cg ? (c->n_h + per - 1) / per : 0;
  *out = a;
  return a.nblk_cg + (do_fg ? (c->n + per - 1) / per : 0);
}

// F<EV, T, COPY>(...) for the threads per slot and types of a launch
#define RELRES_LANES64(F, NT, ...)         \
  if (ev) {                                \
    if (lanes == 32)                       \
      F<true, 32, false>(__VA_ARGS__);     \
    else if (lanes == 16)                  \
      F<true, 16, false>(__VA_ARGS__);     \
    else if (copies_rows(lanes, NT))       \
      F<true, 4, true>(__VA_ARGS__);       \
    else                                   \
      F<true, 4, false>(__VA_ARGS__);      \
  } else if (lanes == 32) {                \
    F<false, 32, false>(__VA_ARGS__);      \
  } else if (lanes == 16) {                \
    F<false, 16, false>(__VA_ARGS__);      \
  } else if (lanes == 8) {                 \
    F<false, 8, false>(__VA_ARGS__);       \
  } else if (copies_rows(lanes, NT)) {     \
    F<false, 4, true>(__VA_ARGS__);        \
  } else {                                 \
    F<false, 4, false>(__VA_ARGS__);       \
  }

template <bool EV, int T, bool COPY>
static void launch64(cudaStream_t s, const Launch64& a, int grid, bool pdl) {
  launch_pdl(pdl, k_pair64<EV, T, COPY>, grid, kFp64Block, smem64<EV, COPY>(a.nt), s, a);
}
template <bool EV, int T, bool COPY>
static void launch64_batch(cudaStream_t s, const BatchLaunch& b, int nrep) {
  k_pair64_batch<EV, T, COPY>
      <<<b.nblk, kFp64Block, smem64<EV, COPY>(b.nt), s>>>(static_cast<const Launch64*>(b.d_args), b.d_off, nrep);
}

cudaError_t launch_pairs_f64(relres_ctx* c, bool ev, int which) {
  const int lanes = pair_shape(c, ev).threads;
  Launch64 a;
  const int grid = make_launch64(c, which, kFp64Block / lanes, pairs_prune(c), &a);
  if (grid == 0) return cudaSuccess;
  RELRES_LANES64(launch64, a.nt, c->stream, a, grid, pair_pdl(c, grid, kFp64Block))
  RELRES_LAUNCHED(c);
  return cudaGetLastError();
}

// ---- batches (see pair.cu)
cudaError_t prepare_pairs_batch_f64(const std::vector<relres_ctx*>& cs, BatchLaunch* b, BatchLaunch* b_ev) {
  long long slots = 0;
  for (const relres_ctx* c : cs) slots += pair_slots(c);
  for (BatchLaunch* l : {b, b_ev}) {
    l->lanes = fp64_lanes_for(slots, l == b_ev);
    l->nt = 1;
    std::vector<Launch64> args(cs.size());
    std::vector<int> off(cs.size() + 1, 0);
    for (size_t r = 0; r < cs.size(); ++r) {
      off[r + 1] = off[r] + make_launch64(cs[r], 3, kFp64Block / l->lanes, cs[r]->prune_on, &args[r]);
      l->nt = std::max(l->nt, cs[r]->n_types);
    }
    l->nblk = off.back();
    const cudaError_t e = upload_batch(l, args.data(), sizeof(Launch64) * args.size(), off);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

void launch_pairs_batch_f64(cudaStream_t s, bool ev, const BatchLaunch& b, int nrep) {
  const int lanes = b.lanes;
  RELRES_LANES64(launch64_batch, b.nt, s, b, nrep)
}

}  // namespace relres
