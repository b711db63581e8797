// relres_pair_forces_static: a RelRes pair evaluation that allocates nothing.
//
// Some callers cannot let a library allocate device memory: a host program
// that owns the whole GPU memory budget through its own allocator and loads
// this library as a plug-in, or a latency-critical loop in which cudaMalloc /
// cudaFree (which may synchronise the device) are not allowed.  For them this
// entry point evaluates the RelRes pair forces, energy and virial of a small
// system by an all-pairs FP64 sum, with every piece of scratch memory (the
// type-pair table, packed atoms and per-block partial sums: 0.5 MB) in one
// file-scope static device array of fixed size.  The caller provides only inputs and outputs.
//
// Limits and sharing: at most RELRES_STATIC_MAX_ATOMS atoms and
// RELRES_MAX_TYPES types.  The array exists once per GPU that loads the
// library and stays allocated until the process exits.  All calls on a GPU
// share it: calls whose work overlaps on the GPU (different streams, or
// several host threads) race on it and must be serialised by the caller.
// Each call rewrites the table, atoms and partial sums it reads, and clears the
// bad-type flag before its kernels run, so stale contents from an earlier
// call are never used.
//
// Atom types live on the device, so the host cannot check them: the kernel
// skips every pair whose type index is outside [0, n_types) (no table read
// with it), writes NaN forces for such an atom and raises a flag in the static
// array, and the reduction then writes NaN energy and virial.
//
// How a call works: k_pack_static reduces every position into the box once and
// packs it as FP32 with a type code; k_allpairs_static gives each atom one
// warp, which rejects partners by their FP32 distance (32 a pass) and queues
// the others; full queues are evaluated in FP64, one pair a lane.  The FP32
// radius is widened by more than the rounding of the packed coordinates, so
// every pair inside its interaction range is evaluated, from the caller's own
// FP64 positions.  Energy and virial are summed in a fixed order from one
// partial sum per block.
//
// Set-up: the first call on each device (with that device current) looks up
// the array's device address with cudaGetSymbolAddress.
#include <atomic>
#include <cmath>
#include <cstring>

#include "common.cuh"

namespace relres {
namespace {

constexpr int kStaticThreads = 128;  // four atoms (warps) per block
constexpr int kStaticMaxBlocks = RELRES_STATIC_MAX_ATOMS / (kStaticThreads / 32);
constexpr int kMaxDevices = 64;
// Type codes of packed atoms past the valid types: an atom whose type is out
// of range (no pair with it is evaluated) and one with a non-finite coordinate
// (every pair with it is, so that the non-finite value reaches the results).
constexpr int kCodeBadType = RELRES_MAX_TYPES, kCodeNonfinite = RELRES_MAX_TYPES + 1;
constexpr int kCodes = RELRES_MAX_TYPES + 2;

struct StaticScratch {
  PairTab<double> tab[RELRES_MAX_TYPES * RELRES_MAX_TYPES];
  float4 atom[RELRES_STATIC_MAX_ATOMS];  // position in [0, L] and type code
  double partial[kNQ][kStaticMaxBlocks];
  unsigned bad_type;  // set when an atom type was outside [0, n_types)
};

static __device__ __align__(256) StaticScratch g_static_scratch;

// host-side cache of the array's device address, per device (several host
// threads may look it up at once; each finds the same address)
static std::atomic<StaticScratch*> s_scratch_ptr[kMaxDevices];

// squared FP32 distances from which a pair of types is certainly out of range
struct StaticReach {
  float r2[RELRES_MAX_TYPES * RELRES_MAX_TYPES];
};

__device__ __forceinline__ double poly5(const double* g, double d) {
  return (((g[4] * d + g[3]) * d + g[2]) * d + g[1]) * d + g[0];
}
__device__ __forceinline__ double poly4(const double* g, double d) {
  return ((g[3] * d + g[2]) * d + g[1]) * d + g[0];
}

// Eq. 20 as the sum of its FG and CG parts (see PairTab); returns -u'(r)/r
// in *fr and u(r) in *u.  Reciprocals as in the FP64 pair launches (rcp_d,
// rsqrt_d); a pair is inside at most one region of each part.
__device__ __forceinline__ void relres_pair(const PairTab<double>& T, double r2, double* fr, double* u) {
  double f = 0.0, e = 0.0;
  const float r2f = float(r2);
  const bool fg = r2 < T.rsp2, cg = r2 < T.rcp2;  // CG: zero table entries for pairs without it
  const bool core = r2 < T.rsm2, lj = cg && !fg && r2 < T.rcm2;
  if (core || lj) {  // Lennard-Jones, FG below r_s- or CG between the shells
    const double r2i = rcp_d(r2, r2f), r6i = r2i * r2i * r2i;
    f = r6i * ((core ? T.f12f : T.f12c) * r6i - (core ? T.f6f : T.f6c)) * r2i;
    e = r6i * ((core ? T.c12f : T.c12c) * r6i - (core ? T.c6f : T.c6c)) - (core ? T.e_fg_shift : T.gam_cm);
    if (core && cg) e += T.e_cg_close;
  } else if (fg || cg) {  // a smoothing shell: both parts at r_s, CG at r_c
    const double ri = rsqrt_d(r2, r2f), r = r2 * ri;
    if (fg) {
      const double d = r - T.rsm, d2 = d * d;
      f = -poly4(T.fgd, d) * ri;
      e = poly5(T.fg, d) - T.e_fg_shift;
      if (cg) {
        f -= d2 * (T.ond4 * d + T.ond3) * ri;
        e += T.on0 + d2 * d * (T.on4 * d + T.on3) - T.gam_cm;
      }
    } else {
      const double d = r - T.rcm;
      f = -poly4(T.cgod, d) * ri;
      e = poly5(T.cgo, d) - T.gam_cm;
    }
  }
  *fr = f;
  *u = e;
}

// x reduced into [0, L] (FP32; the quotient is exact for any image that FP64
// tells apart from its neighbours).
__device__ __forceinline__ float into_box(double x, double l, double il) {
  const float f = float(fma(-floor(x * il), l, x));
  return fminf(fmaxf(f, 0.f), float(l));
}

__global__ void __launch_bounds__(kThreads) k_pack_static(int n, int nt, const double* __restrict__ pos,
                                                          const int* __restrict__ type, double l0, double l1,
                                                          double l2, StaticScratch* scratch) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  bool bad = false;
  if (i < n) {
    const double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
    const int t = type[i];
    bad = t < 0 || t >= nt;
    const bool fin = isfinite(x) && isfinite(y) && isfinite(z);
    const int code = bad ? kCodeBadType : (fin ? t : kCodeNonfinite);
    scratch->atom[i] =
        make_float4(into_box(x, l0, 1.0 / l0), into_box(y, l1, 1.0 / l1), into_box(z, l2, 1.0 / l2), __int_as_float(code));
  }
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(&scratch->bad_type, 1u);
}

// distance along one axis to the nearest image, both coordinates in [0, l]
__device__ __forceinline__ float nearest(float a, float b, float l) {
  const float d = fabsf(a - b);
  return fminf(d, l - d);
}

// d - l rint(d / l).  The quotient is rounded by adding and subtracting
// 1.5 2^52; d * il may round to the other side of a half integer where d / l
// does not, which only exchanges two images at half the box, out of range.
__device__ __forceinline__ double min_image(double d, double l, double il) {
  const double t = fma(d, il, 6755399441055744.0);
  return fma(-l, t - 6755399441055744.0, d);
}

// one thread's sums: force, then energy and virial
constexpr int kSums = 3 + kNQ;
struct StaticSums {
  double v[kSums] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
};

// The sums over a warp, each left in one pair of lanes: at every level a lane
// passes on the half of its values that its partner keeps (12 FP64 additions a
// lane; ten butterflies take 50).  Returns this lane's value, its index in k
// (-1: none).
__device__ __forceinline__ double warp_sums(const StaticSums& S, int lane, int& k) {
  static_assert(kSums == 10, "split as 5 + 5, 3 + 2, 2 + 1, 1 + 1");
  const bool a = lane & 16, b = lane & 8, c = lane & 4, d = lane & 2;
  double x[6], y[4], z[2];
#pragma unroll
  for (int q = 0; q < 5; ++q)
    x[q] = (a ? S.v[q + 5] : S.v[q]) + __shfl_xor_sync(0xffffffffu, a ? S.v[q] : S.v[q + 5], 16);
  x[5] = 0.0;
#pragma unroll
  for (int q = 0; q < 3; ++q) y[q] = (b ? x[q + 3] : x[q]) + __shfl_xor_sync(0xffffffffu, b ? x[q] : x[q + 3], 8);
  y[3] = 0.0;
#pragma unroll
  for (int q = 0; q < 2; ++q) z[q] = (c ? y[q + 2] : y[q]) + __shfl_xor_sync(0xffffffffu, c ? y[q] : y[q + 2], 4);
  double t = (d ? z[1] : z[0]) + __shfl_xor_sync(0xffffffffu, d ? z[0] : z[1], 2);
  t += __shfl_xor_sync(0xffffffffu, t, 1);
  const int in = 2 * int(c) + int(d);
  k = in < (b ? 2 : 3) ? 5 * int(a) + 3 * int(b) + in : -1;
  return t;
}

// One queued pair (i, j): excluded partners are skipped here, where few
// candidates are left.
__device__ __forceinline__ void static_pair(const double* __restrict__ pos, const int* __restrict__ type, double xi,
                                            double yi, double zi, int ti, int nt, int j, double l0, double l1,
                                            double l2, double il0, double il1, double il2, const int* __restrict__ eidx,
                                            int e0, int e1, const PairTab<double>* tab, StaticSums& S) {
  for (int e = e0; e < e1; ++e)
    if (eidx[e] == j) return;
  const double dx = min_image(xi - pos[3 * j], l0, il0), dy = min_image(yi - pos[3 * j + 1], l1, il1),
               dz = min_image(zi - pos[3 * j + 2], l2, il2);
  double fr, u;
  relres_pair(tab[ti * nt + type[j]], dx * dx + dy * dy + dz * dz, &fr, &u);
  const double fx = fr * dx, fy = fr * dy, fz = fr * dz;
  S.v[0] += fx;
  S.v[1] += fy;
  S.v[2] += fz;
  S.v[3] += u;
  S.v[4] += fx * dx;
  S.v[5] += fy * dy;
  S.v[6] += fz * dz;
  S.v[7] += fx * dy;
  S.v[8] += fx * dz;
  S.v[9] += fy * dz;
}

// One warp per atom.  The FP32 test of a partner is ~20 instructions (n^2 of
// them: the floor of large n); the FP64 evaluation of the few percent that
// pass runs with full lanes from the queue, at the FP64 rate (1.66 FMA per
// clock and SM).  0.094 ms per call at 3993 propane-like atoms (18.5 with one
// thread per atom and every partner in FP64), 0.43 ms at 14 739; held to 80
// registers the loop is not unrolled: 0.20 and 1.5 ms.
__global__ void __launch_bounds__(kStaticThreads)
    k_allpairs_static(int n, int nt, const double* __restrict__ pos, const int* __restrict__ type, double l0,
                      double l1, double l2, const int* __restrict__ eoff, const int* __restrict__ eidx, int with_excl,
                      StaticReach reach, double* __restrict__ forces, StaticScratch* scratch) {
  constexpr int kWarps = kStaticThreads / 32, kUnroll = 4;
  __shared__ float s_reach[kWarps][kCodes];
  __shared__ int s_queue[kWarps][32 + 32 * kUnroll];
  __shared__ double s_sum[kWarps][kNQ];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = blockIdx.x * kWarps + w;
  StaticSums S;
  bool bad_i = false;
  if (i < n) {
    const float4 ai = scratch->atom[i];
    const int ci = __float_as_int(ai.w);
    bad_i = ci == kCodeBadType;
    if (!bad_i) {
      const int ti = type[i];
      if (lane < kCodes) {
        // partners by type code: never, always, or by the widened distance
        // (always for a non-finite atom i)
        float r2 = lane < nt ? (ci == kCodeNonfinite ? __int_as_float(0x7f800000) : reach.r2[ti * nt + lane]) : -1.f;
        if (lane == kCodeNonfinite) r2 = __int_as_float(0x7f800000);
        s_reach[w][lane] = r2;
      }
      __syncwarp();
      const double xi = pos[3 * i], yi = pos[3 * i + 1], zi = pos[3 * i + 2];
      const double il0 = 1.0 / l0, il1 = 1.0 / l1, il2 = 1.0 / l2;
      const int e0 = with_excl ? eoff[i] : 0, e1 = with_excl ? eoff[i + 1] : 0;
      const float fl0 = float(l0), fl1 = float(l1), fl2 = float(l2);
      int waiting = 0;
      float4 next[kUnroll];  // four partners a lane in flight
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) next[u] = scratch->atom[min(32 * u + lane, n - 1)];
      for (int base = 0; base < n; base += 32 * kUnroll) {
        float4 at[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
          at[u] = next[u];
          next[u] = scratch->atom[min(base + 32 * (kUnroll + u) + lane, n - 1)];
        }
        bool near[kUnroll];
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
          const int j = base + 32 * u + lane;
          const float dx = nearest(ai.x, at[u].x, fl0), dy = nearest(ai.y, at[u].y, fl1),
                      dz = nearest(ai.z, at[u].z, fl2);
          near[u] = j < n && j != i && dx * dx + dy * dy + dz * dz < s_reach[w][__float_as_int(at[u].w)];
        }
#pragma unroll
        for (int u = 0; u < kUnroll; ++u) {
          const unsigned b = __ballot_sync(0xffffffffu, near[u]);
          if (near[u]) s_queue[w][waiting + __popc(b & ((1u << lane) - 1u))] = base + 32 * u + lane;
          waiting += __popc(b);
        }
        __syncwarp();
        while (waiting >= 32) {
          waiting -= 32;
          static_pair(pos, type, xi, yi, zi, ti, nt, s_queue[w][waiting + lane], l0, l1, l2, il0, il1, il2, eidx, e0, e1,
                      scratch->tab, S);
        }
        __syncwarp();
      }
      if (lane < waiting)
        static_pair(pos, type, xi, yi, zi, ti, nt, s_queue[w][lane], l0, l1, l2, il0, il1, il2, eidx, e0, e1,
                    scratch->tab, S);
    }
  }
  int k;
  const double t = warp_sums(S, lane, k);
  if (k >= 0 && k < 3 && i < n) forces[3 * i + k] = bad_i ? __longlong_as_double(0x7ff8000000000000LL) : t;
  if (k >= 3) s_sum[w][k - 3] = t;
  __syncthreads();
  if (threadIdx.x < kNQ) {
    double v = 0.0;
#pragma unroll
    for (int q = 0; q < kWarps; ++q) v += s_sum[q][threadIdx.x];
    scratch->partial[threadIdx.x][blockIdx.x] = 0.5 * v;
  }
}

// Block q sums the q-th of the energy and virial partial sums (fixed order).
__global__ void __launch_bounds__(1024) k_allpairs_static_out(int nblocks, const StaticScratch* scratch, double* energy,
                                                              int with_energy, double* virial, int with_virial) {
  __shared__ double sh[32];
  const int q = blockIdx.x;
  double v[1] = {0.0};
  for (int b = threadIdx.x; b < nblocks; b += blockDim.x) v[0] += scratch->partial[q][b];
  block_sum<double, 1>(v, sh);
  if (threadIdx.x != 0) return;
  if (scratch->bad_type != 0u) v[0] = __longlong_as_double(0x7ff8000000000000LL);
  if (q == 0 && with_energy) energy[0] = v[0];
  if (q > 0 && with_virial) virial[q - 1] = v[0];
}

}  // namespace
}  // namespace relres

using namespace relres;

extern "C" relres_status relres_pair_forces_static(const relres_params* p, int n_atoms, const int* d_type,
                                                   const double* d_pos, const double box[3],
                                                   const int* d_excl_offsets, const int* d_excl_index,
                                                   double* d_forces, double* d_energy, double* d_virial,
                                                   void* cuda_stream) {
  if (!p || !d_type || !d_pos || !box || !d_forces) return RELRES_ERR_ARG;
  if (n_atoms < 1 || n_atoms > RELRES_STATIC_MAX_ATOMS) return RELRES_ERR_ARG;
  if ((d_excl_offsets == nullptr) != (d_excl_index == nullptr)) return RELRES_ERR_ARG;
  for (int d = 0; d < 3; ++d)
    if (!(box[d] > 0.0) || !std::isfinite(box[d])) return RELRES_ERR_ARG;
  // parameter preparation into stack buffers (no heap in this entry point's own code)
  double table[RELRES_MAX_TYPES * RELRES_MAX_TYPES * RELRES_PAIR_FIELDS];
  const relres_status ps = relres_prepare_table(p, table, int(sizeof(table) / sizeof(double)));
  if (ps != RELRES_OK) return ps;
  const int nt = p->n_types;
  double rmax = 0.0;
  StaticReach reach{};
  PairTab<double> tabs[RELRES_MAX_TYPES * RELRES_MAX_TYPES];
  std::memset(tabs, 0, sizeof(tabs));
  for (int k = 0; k < nt * nt; ++k) {
    const double* o = table + k * RELRES_PAIR_FIELDS;
    PairTab<double>& t = tabs[k];
    const double s6f = std::pow(o[1], 6.0), s6c = std::pow(o[3], 6.0);
    t.c12f = 4.0 * o[0] * s6f * s6f;
    t.c6f = 4.0 * o[0] * s6f;
    t.f12f = 12.0 * t.c12f;
    t.f6f = 6.0 * t.c6f;
    t.rsm = o[4];
    t.rsm2 = o[4] * o[4];
    t.rsp2 = o[5] * o[5];
    for (int m = 0; m < 5; ++m) t.fg[m] = o[8 + m];
    for (int m = 1; m < 5; ++m) t.fgd[m - 1] = m * o[8 + m];
    const double ws = o[5] - o[4];
    t.e_fg_shift = (((o[12] * ws + o[11]) * ws + o[10]) * ws + o[9]) * ws + o[8];
    t.c12c = 4.0 * o[2] * s6c * s6c;
    t.c6c = 4.0 * o[2] * s6c;
    t.f12c = 12.0 * t.c12c;
    t.f6c = 6.0 * t.c6c;
    t.rcm = o[6];
    t.rcm2 = o[6] * o[6];
    t.rcp2 = o[7] * o[7];
    t.on0 = o[13];
    t.on3 = o[16];
    t.on4 = o[17];
    t.ond3 = 3.0 * o[16];
    t.ond4 = 4.0 * o[17];
    for (int m = 0; m < 5; ++m) t.cgo[m] = o[18 + m];
    for (int m = 1; m < 5; ++m) t.cgod[m - 1] = m * o[18 + m];
    t.gam_cm = o[23];
    t.e_cg_close = o[13] - o[23];
    const double rk = std::fmax(o[5], o[2] > 0.0 ? o[7] : 0.0);
    rmax = std::fmax(rmax, rk);
    // beyond rk the pair's force and energy are exactly zero; widened by more
    // than the rounding of two packed coordinates and their difference
    const double wide = rk * (1.0 + 1e-5) + 1e-6 * std::fmax(box[0], std::fmax(box[1], box[2])) + 1e-3;
    reach.r2[k] = float(wide * wide * (1.0 + 1e-5));
  }
  // minimum image needs every interaction range below half the box
  if (!(rmax < 0.5 * std::fmin(box[0], std::fmin(box[1], box[2])))) return RELRES_ERR_BOX;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return RELRES_ERR_CUDA;
  StaticScratch* scratch = s_scratch_ptr[dev].load(std::memory_order_acquire);
  if (scratch == nullptr) {
    void* ptr = nullptr;
    if (cudaGetSymbolAddress(&ptr, g_static_scratch) != cudaSuccess || ptr == nullptr) return RELRES_ERR_CUDA;
    scratch = static_cast<StaticScratch*>(ptr);
    s_scratch_ptr[dev].store(scratch, std::memory_order_release);
  }
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  // the table for this call (copied from the stack; a pageable-source copy
  // returns once the source has been read) and a cleared bad-type flag
  if (cudaMemcpyAsync(scratch->tab, tabs, sizeof(PairTab<double>) * nt * nt, cudaMemcpyHostToDevice,
                      stream) != cudaSuccess)
    return RELRES_ERR_CUDA;
  if (cudaMemsetAsync(&scratch->bad_type, 0, sizeof(unsigned), stream) != cudaSuccess) return RELRES_ERR_CUDA;
  int with_excl = d_excl_offsets ? 1 : 0;
  // cudaLaunchKernel returns the status of this launch only: an earlier
  // error of unrelated work is neither reported as this call's nor cleared
  int n = n_atoms, ntt = nt;
  double l0 = box[0], l1 = box[1], l2 = box[2];
  const int* eoff = with_excl ? d_excl_offsets : d_type;
  const int* eidx = with_excl ? d_excl_index : d_type;
  void* args0[] = {&n, &ntt, const_cast<double**>(&d_pos), const_cast<int**>(&d_type), &l0, &l1, &l2, &scratch};
  if (cudaLaunchKernel(reinterpret_cast<const void*>(&k_pack_static), dim3((n_atoms + kThreads - 1) / kThreads),
                       dim3(kThreads), args0, 0, stream) != cudaSuccess)
    return RELRES_ERR_CUDA;
  void* args1[] = {&n, &ntt, const_cast<double**>(&d_pos), const_cast<int**>(&d_type), &l0, &l1, &l2,
                   const_cast<int**>(&eoff), const_cast<int**>(&eidx), &with_excl, &reach, &d_forces, &scratch};
  int nblocks = (n_atoms + kStaticThreads / 32 - 1) / (kStaticThreads / 32);
  if (cudaLaunchKernel(reinterpret_cast<const void*>(&k_allpairs_static), dim3(nblocks), dim3(kStaticThreads), args1,
                       0, stream) != cudaSuccess)
    return RELRES_ERR_CUDA;
  const StaticScratch* cscratch = scratch;
  double* e_out = d_energy ? d_energy : d_forces;
  double* w_out = d_virial ? d_virial : d_forces;
  int with_e = d_energy ? 1 : 0, with_w = d_virial ? 1 : 0;
  void* args2[] = {&nblocks, &cscratch, &e_out, &with_e, &w_out, &with_w};
  if (cudaLaunchKernel(reinterpret_cast<const void*>(&k_allpairs_static_out), dim3((with_e || with_w) ? kNQ : 1),
                       dim3(1024), args2, 0, stream) != cudaSuccess)
    return RELRES_ERR_CUDA;
  return RELRES_OK;
}
