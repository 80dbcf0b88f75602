// The FP64 form's 1D1V passes on grids of up to kMomMaxNodes nodes without the
// filter: the passes of es1d_fp64.cu with the B-spline sums written as
// polynomials of a marker's offset d from its node, so that few FP64
// instructions are left per marker (the FP64 pipe, 2 lanes per SM and clock,
// bounds this form).
//
//   gather    F_p = a_i + b_i d (+ c_i d^2): the coefficients of every node are
//             built once per block, a marker takes one FMA per order and no
//             weights.  Order 1: a = F_i, b = F_{i+1} - F_i.  Order 2:
//             c = (F_{i-1} + F_{i+1})/2 - F_i, a = F_i + c/4,
//             b = (F_{i+1} - F_{i-1})/2.
//   deposit   the moments A, A d (, A d^2) of the markers of node i, summed per
//             node; the block turns its sums into node currents when it flushes:
//             order 1 J_i += M0 - M1, J_{i+1} += M1; order 2
//             J_{i-1} += M0/8 - M1/2 + M2/2, J_i += 3/4 M0 - M2,
//             J_{i+1} += M0/8 + M1/2 + M2/2.
//             These are the B-spline weights of Sec. 2.2 term by term, so gather
//             and deposit still use one shape and Eq. exp_econs_simple holds to
//             rounding.
//             The sums are exact integers, each node's with its own unit
//             (fixed_moments.cuh).
//   factors   of a single uniformly weighted species (FOLD) are not applied
//             per marker: q w0 / h and m w0 / 2 go to the block's sums and dt q/m
//             to the tables, so that pass C's gather is v* - v^n and pass
//             E's is 2 (v^dag - v^n), with which R = |v^n|^2 + 2 v* (v^dag - v^n)
//             is one product and one FMA.
//   points    node and offset of x^{n+1/2} (pass C -> E) and of the next x*
//             (pass E -> C): 12 bytes a marker; the split of a coordinate, the
//             wrap and the tests around the root run on the integer pipe
//             (Point64, wrap_fast, root_in_range).
//   tiles     a block keeps `copies` tiles, lane l adding into copy l mod copies,
//             so that the lanes of a warp rarely meet at an address.
//   totals    each flush also adds the block's sum of M0 (the weights sum to 1),
//             so the mean current is one load instead of a reduction over the
//             grid in every block.
//   service   the last block of a launch has no markers: it writes E^{n+1} and
//             W_E, clears the currents the next pass adds into and reduces the
//             previous step's energy.
// All kernels are programmatic dependent launches: the tile is cleared before
// the wait for the previous kernel.
//
// Measured (2^23 markers, 512 nodes, order 2, ESEC2), with the general passes / with
// shared FP64 atomics in place of the fixed-point sums / with those and one unit for the
// grid / now, with a unit a node: pass C 598 / 221 / 119 / 122 us (warp instructions on
// the FP64 pipe per 32 markers 32.6 / 13.4 / 6.5 / 6.8), pass E 986 / 387 / 244 / 246 us
// (56.8 / 24.6 / 14.8 / 15.2).  20,000 markers on 64 nodes: 36.6 / 11.8 / 10.5 / 11.1 us
// a step, bound by the launches' serial parts (loads, tables, flush); 1,000 on 1792 nodes
// 43 / - / 21 / 29, the flush; 50 steps and their results 557 us with a thread's first
// marker loaded after the table is built, 540 before it.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "es1d_fp64_common.cuh"
#include "es1d_poly.cuh"
#include "fixed_moments.cuh"
#include "pdl.cuh"
#include "pic_internal.cuh"

namespace pic {
namespace {

constexpr int kMomTileBytes = 48 * 1024;  // tile copies of a block
static_assert(kFixedMaxThreads <= 512, "the kernels' launch bounds");

// k E*, E* = E^n - dt/2 (J1 - <J1>) (ESEC2) or E^n (ESEC1), into F.
template <int SCHEME>
__device__ __forceinline__ void load_estar(const Es1dConst &c, const Es1dFp64Bufs &b, int par,
                                           double k, double *F) {
  const double *E = b.E[par], *J1 = b.J1[par];
  const double mean = SCHEME == 2 && c.remove_mean ? b.Jt[par] * c.inv_nc : 0.0;
  const double kj = -k * c.hdt;
  for (int i = threadIdx.x; i < c.nc; i += blockDim.x)
    F[i] = SCHEME == 2 ? fma(kj, J1[i] - mean, k * E[i]) : k * E[i];
}

// Shared memory of a pass: the table, F (nc values, the field the coefficients
// are built from), the tile copies (16-byte aligned: F padded to two words) and the
// nodes' scale words.  On grids that those would cost the second block on an SM they
// take F's place once the table is built (c.late, one more barrier).
template <int ORDER>
struct MomShared {
  double *table, *F;
  unsigned *T, *W;
  __device__ __forceinline__ MomShared(const Es1dConst &c, double *sm) {
    table = sm;
    F = sm + (size_t)Poly<ORDER>::kWords * c.nc;
    T = (unsigned *)(F + (c.nc + 1) / 2 * 2);
    W = c.late ? (unsigned *)F : T + (size_t)2 * c.nc * (ORDER + 1) * c.copies;
  }
};

// What a pass reads of marker p (nothing past the end).
template <int SCHEME>
struct MarkerC {
  double x, v, d;
  int i;
  __device__ __forceinline__ MarkerC(const Es1dFp64Bufs &b, int64_t p, bool ok) {
    if (!ok) return;
    x = b.x[p];
    v = b.v[p];
    if (SCHEME == 2) {
      i = b.sis[p];
      d = b.sds[p];
    }
  }
};
struct MarkerE {
  double x, v, vs, d;
  int i;
  __device__ __forceinline__ MarkerE(const Es1dFp64Bufs &b, int64_t p, bool ok) {
    if (!ok) return;
    x = b.x[p];
    v = b.v[p];
    vs = b.vs[p];
    i = b.si[p];
    d = b.sd[p];
  }
};

template <int ORDER, int SCHEME, bool FOLD>
__global__ void __launch_bounds__(512, 2) mom_pass_c_kernel(Es1dConst c, Es1dFp64Bufs b, int par,
                                                            int prev_slot) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[kRedWords];
  const int nc = c.nc;
  const int nblk = (int)gridDim.x - 1;
  if ((int)blockIdx.x == nblk) {   // service block
    griddep_wait();
    griddep_launch_dependents();
    if (SCHEME == 2) {
      clear_doubles(b.J1[par ^ 1], nc);
      if (threadIdx.x == 0) b.Jt[par ^ 1] = 0.0;
    }
    if (threadIdx.x == 0) b.vmax[par ^ 1] = 0u;
    // pass E's scales, from what the pass E before recorded (all loads first)
    const ScaleMaker<> scales(b.words, b.rec, b.storm, SCHEME == 2 ? nc : 0);
    const unsigned vmax = __ldcg(b.vmax + par);
    double s = 0.0;
    if (prev_slot >= 0)
      for (int i = threadIdx.x; i < nblk; i += blockDim.x) s += b.ke_part[i];
    if (SCHEME == 2)
      scales.make((unsigned *)sm, node_reach(vmax, c.reach), c.decay, c.n_total);
    if (prev_slot >= 0) {
      const double t = block_sum_narrow(s, red);
      if (threadIdx.x == 0) {
        const double te = t + b.we[0];
        b.te[prev_slot] = te;
        if (!isfinite(te)) atomicOr(b.err, kErrNonfinite);
      }
    }
    return;
  }
  const MomShared<ORDER> m_(c, sm);
  double *table = m_.table, *F = m_.F;
  unsigned *T = m_.T, *W = m_.W;
  const int copies = c.copies;
  clear_fixed(T, 2 * nc * (ORDER + 1) * copies);
  griddep_wait();
  // (the first marker is on its way while the table is built)
  const int64_t end = chunk_end(c);
  int64_t p = blockIdx.x * c.chunk + threadIdx.x;
  MarkerC<SCHEME> m(b, p, p < end);
  const ScaleWords words(b.words + nc + 1, nc + 1);
  load_estar<SCHEME>(c, b, par, FOLD ? c.hdt_qm[0] : 1.0, F);
  if (!c.late) words.store(W);
  const double scale = FOLD ? c.qw_h[0] : 1.0;
  __syncthreads();
  build_poly<ORDER>(table, F, nc);
  __syncthreads();
  if (c.late) {
    words.store(W);
    __syncthreads();
  }
  unsigned *Tl = T + (threadIdx.x & (copies - 1));
  const double hdt = c.hdt;
  for (; p < end; p += blockDim.x, m = MarkerC<SCHEME>(b, p, p < end)) {
    const int s = FOLD ? 0 : species_of(c, p);
    const double x = m.x, v = m.v;
    Point64<ORDER> P;
    if (SCHEME == 2) {   // the point at x* that j^{n,*} was deposited at
      P.i = m.i;
      P.d = m.d;
    } else {
      P = Point64<ORDER>(__dmul_rn(wrap_fast(__fma_rn(hdt, v, x), c.L, b.err), c.inv_h), nc);
    }
    const double g = gather_poly<ORDER>(table, P.i, P.d);
    const double vs = FOLD ? __dadd_rn(v, g) : __fma_rn(c.hdt_qm[s], g, v);
    const Point64<ORDER> H(__dmul_rn(wrap_fast(__fma_rn(hdt, vs, x), c.L, b.err), c.inv_h), nc);
    b.vs[p] = vs;
    b.si[p] = H.i;
    b.sd[p] = H.d;
    double A = vs;
    if (!FOLD) A *= b.w ? c.q_h[s] * b.w[p] : c.qw_h[s];
    add_moments<ORDER>(Tl + (size_t)H.i * 2 * (ORDER + 1) * copies, copies, W + H.i, W + nc + 1, H, A, scale,
                       b.J2[par], &b.Jt[2 + par], nc);
  }
  griddep_launch_dependents();
  __syncthreads();
  flush_new(W, b.rec + nc, nc, W + nc + 1, b.storm + 2);
  flush_moments<ORDER>(T, W, copies, nc, scale, b.J2[par], &b.Jt[2 + par], ScaleRange(W[nc]));
}

template <int ORDER, int SCHEME, bool FOLD>
__global__ void __launch_bounds__(512, 2) mom_pass_e_kernel(Es1dConst c, Es1dFp64Bufs b, int par,
                                                            int slot) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[kRedWords];
  const int nc = c.nc;
  const int nblk = (int)gridDim.x - 1;
  const double *E = b.E[par], *J2 = b.J2[par];
  if ((int)blockIdx.x == nblk) {   // service block: E^{n+1}, W_E, the cleared J2
    griddep_wait();
    griddep_launch_dependents();
    const ScaleMaker<> scales(b.words + nc + 1, b.rec + nc, b.storm + 2, nc);
    const unsigned vmax = __ldcg(b.vmax + par);
    const double mean = c.remove_mean ? b.Jt[2 + par] * c.inv_nc : 0.0;
    double we = 0.0;
    for (int i = threadIdx.x; i < nc; i += blockDim.x) {
      const double en = E[i] - c.dt * (J2[i] - mean);
      b.E[par ^ 1][i] = en;
      b.J2[par ^ 1][i] = 0.0;
      we = fma(en, en, we);
    }
    const double t = block_sum_narrow(we, red);
    if (threadIdx.x == 0) {
      b.we[0] = 0.5 * c.h * t;
      b.Jt[2 + (par ^ 1)] = 0.0;
    }
    // the next pass C's scales, from what the last one recorded
    scales.make((unsigned *)sm, node_reach(vmax, c.reach), c.decay, c.n_total);
    return;
  }
  const MomShared<ORDER> m_(c, sm);
  double *table = m_.table, *F = m_.F;
  unsigned *T = m_.T, *W = m_.W;
  const int copies = c.copies;
  if (SCHEME == 2) clear_fixed(T, 2 * nc * (ORDER + 1) * copies);
  griddep_wait();
  const int64_t end = chunk_end(c);
  int64_t p = blockIdx.x * c.chunk + threadIdx.x;
  MarkerE m(b, p, p < end);
  const ScaleWords words(b.words, SCHEME == 2 ? nc + 1 : 0);
  const double scale = FOLD ? c.qw_h[0] : 1.0;
  {
    // 2 k E^{n+1/2} = 2 k E^n - k dt (j - <j>)
    const double k2 = FOLD ? 2.0 * c.dt_qm[0] : 2.0, kj = -0.5 * c.dt * k2;
    const double mean = c.remove_mean ? b.Jt[2 + par] * c.inv_nc : 0.0;
    for (int i = threadIdx.x; i < nc; i += blockDim.x) F[i] = fma(kj, J2[i] - mean, k2 * E[i]);
  }
  if (!c.late) words.store(W);
  __syncthreads();
  build_poly<ORDER>(table, F, nc);
  __syncthreads();
  if (SCHEME == 2 && c.late) {
    words.store(W);
    __syncthreads();
  }
  unsigned *Tl = T + (threadIdx.x & (copies - 1));
  const double hdt = c.hdt;
  double ke = 0.0;
  unsigned nfb = 0, vm = 0;
  for (; p < end; p += blockDim.x, m = MarkerE(b, p, p < end)) {
    const int s = FOLD ? 0 : species_of(c, p);
    const double x = m.x, v = m.v, vs = m.vs;
    double k2 = gather_poly<ORDER>(table, m.i, m.d);   // 2 (v^dag - v^n)
    if (!FOLD) k2 *= c.dt_qm[s];
    const double R = __fma_rn(vs, k2, __dmul_rn(v, v));
    double vn;
    // v^{n+1} = sqrt(R) with the sign of v^dag = v^n + k2/2, the sign of the
    // larger of the two (comparison of the bit patterns, k2's exponent one
    // less).  R has to be positive and in the root's range, the two not equal
    // and the larger above 2^-447, which makes v^dag^2 > 0; all else as Sec. 3.2
    // writes it.
    const unsigned long long av = abs_bits(v), ak2 = abs_bits(k2);
    const unsigned long long ak = ak2 >= (1ull << 52) ? ak2 - (1ull << 52) : 0ull;
    const unsigned long long big = av > ak ? av : ak;
    if (c.gamma_on && root_in_range(R) && av != ak && big >= 0x2400000000000000ull) {
      const double g = root_newton(R);
      const int sign = (av > ak ? __double2hiint(v) : __double2hiint(k2)) & 0x80000000;
      vn = __hiloint2double(sign | __double2hiint(g), __double2loint(g));
    } else {
      const double vd = __fma_rn(0.5, k2, v);
      vn = vd;
      if (c.gamma_on) {
        if (R < 0.0 || vd * vd == 0.0)
          nfb++;
        else
          vn = copysign(sqrt(R), vd);
      }
    }
    const double xn = wrap_fast(__fma_rn(c.dt, vs, x), c.L, b.err);
    b.xo[p] = xn;
    b.vo[p] = vn;
    vm = max(vm, abs_hi(vn));
    const double wp = !FOLD && b.w ? b.w[p] : 1.0;
    ke = FOLD ? __fma_rn(vn, vn, ke)
                : __fma_rn((b.w ? c.half_m[s] * wp : c.half_mw[s]) * vn, vn, ke);
    if (SCHEME == 2) {
      const Point64<ORDER> N(__dmul_rn(wrap_fast(__fma_rn(hdt, vn, xn), c.L, b.err), c.inv_h), nc);
      b.sis[p] = N.i;
      b.sds[p] = N.d;
      double A = vn;
      if (!FOLD) A *= b.w ? c.q_h[s] * wp : c.qw_h[s];
      add_moments<ORDER>(Tl + (size_t)N.i * 2 * (ORDER + 1) * copies, copies, W + N.i, W + nc + 1, N, A, scale,
                         b.J1[par ^ 1], &b.Jt[par ^ 1], nc);
    }
  }
  griddep_launch_dependents();
  flush_vmax(vm, &b.vmax[par ^ 1]);
  nfb = __reduce_add_sync(0xffffffffu, nfb);
  if ((threadIdx.x & 31) == 0 && nfb) atomicAdd(&b.fallback[slot], (unsigned long long)nfb);
  const double t = block_sum_narrow(ke, red);   // (its barriers order the tile before the flush)
  if (threadIdx.x == 0) b.ke_part[blockIdx.x] = FOLD ? c.half_mw[0] * t : t;
  if (SCHEME == 2) {
    flush_new(W, b.rec, nc, W + nc + 1, b.storm);
    flush_moments<ORDER>(T, W, copies, nc, scale, b.J1[par ^ 1], &b.Jt[par ^ 1],
                         ScaleRange(W[nc]));
  }
}

// The point of x^n + dt/2 v^n, with the rounding that every kernel of this form uses.
template <int ORDER>
__device__ __forceinline__ Point64<ORDER> mom_xstar(const Es1dConst &c, double x, double v,
                                                    unsigned *err) {
  return Point64<ORDER>(__dmul_rn(wrap_fast(__fma_rn(c.hdt, v, x), c.L, err), c.inv_h), c.nc);
}

// The nodes' largest |amounts| of the current state's deposits to the records (zero
// before) of J1 and of J2 (v* is near v), the largest |v| to vmax of parity par.
template <int ORDER>
__global__ void __launch_bounds__(512, 2) mom_absmax_kernel(Es1dConst c, Es1dFp64Bufs b,
                                                            int par) {
  __shared__ unsigned W[kMomMaxNodes];
  clear_largest(W, c.nc);
  __syncthreads();
  unsigned vm = 0;
  const int64_t end = chunk_end(c);
  for (int64_t p = blockIdx.x * c.chunk + threadIdx.x; p < end; p += blockDim.x) {
    const double v = b.v[p];
    vm = max(vm, abs_hi(v));
    const int s = species_of(c, p);
    double A = v;
    if (!c.fold) A *= b.w ? c.q_h[s] * b.w[p] : c.qw_h[s];
    raise_largest(W + mom_xstar<ORDER>(c, b.x[p], v, b.err).i, abs_hi(A) >> 20);
  }
  __syncthreads();
  flush_vmax(vm, b.vmax + par);
  flush_largest(W, b.rec, c.nc);
  flush_largest(W, b.rec + c.nc, c.nc);
}
// The first scale words (one block).
__global__ void __launch_bounds__(512) mom_scales_kernel(Es1dConst c, Es1dFp64Bufs b, int par) {
  __shared__ unsigned S[kMomMaxNodes + 2 * kMostReach];
  for (int k = 0; k < 2; k++) {
    ScaleMaker<>(b.words + k * (c.nc + 1), b.rec + k * c.nc, b.storm + 2 * k, c.nc)
        .make(S, node_reach(__ldcg(b.vmax + par), c.reach), 0, c.n_total);
    __syncthreads();
  }
}

// j^{n,*} of the current state (ESEC2 start-up and after a state change).
template <int ORDER>
__global__ void __launch_bounds__(512, 2) mom_deposit_initial_kernel(Es1dConst c, Es1dFp64Bufs b,
                                                                     int par) {
  extern __shared__ __align__(16) double sm[];
  const int nc = c.nc;
  const MomShared<ORDER> m_(c, sm);
  unsigned *T = m_.T, *W = m_.W;
  const int copies = c.copies;
  clear_fixed(T, 2 * nc * (ORDER + 1) * copies);
  ScaleWords(b.words, nc + 1).store(W);
  __syncthreads();
  unsigned *Tl = T + (threadIdx.x & (copies - 1));
  const double scale = c.fold ? c.qw_h[0] : 1.0;
  const int64_t end = chunk_end(c);
  for (int64_t p = blockIdx.x * c.chunk + threadIdx.x; p < end; p += blockDim.x) {
    const int s = species_of(c, p);
    const double v = b.v[p];
    const Point64<ORDER> N = mom_xstar<ORDER>(c, b.x[p], v, b.err);
    b.sis[p] = N.i;
    b.sds[p] = N.d;
    double A = v;
    if (!c.fold) A *= b.w ? c.q_h[s] * b.w[p] : c.qw_h[s];
    add_moments<ORDER>(Tl + (size_t)N.i * 2 * (ORDER + 1) * copies, copies, W + N.i, W + nc + 1, N, A, scale,
                       b.J1[par], &b.Jt[par], nc);
  }
  __syncthreads();
  flush_moments<ORDER>(T, W, copies, nc, scale, b.J1[par], &b.Jt[par], ScaleRange(W[nc]));
}

template <typename F>
void dispatch_mom(const Es1dConst &c, F f) {
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  auto fold = [&](auto O, auto S) {
    c.fold ? f(O, S, std::true_type()) : f(O, S, std::false_type());
  };
  if (c.order == 1) c.scheme == 1 ? fold(I1(), I1()) : fold(I1(), I2());
  else c.scheme == 1 ? fold(I2(), I1()) : fold(I2(), I2());
}

size_t mom_smem(const Es1dConst &c, int copies, bool late) {
  const size_t words = (size_t)(c.order == 1 ? 2 : 4) + (size_t)(c.order + 1) * copies;
  return sizeof(double) * (words * c.nc + (c.nc + 1) / 2 * 2) + (late ? 0 : sizeof(unsigned) * (c.nc + 2));
}
size_t mom_smem(const Es1dConst &c) { return mom_smem(c, c.copies, c.late); }

}  // namespace

// Grids whose tile and tables leave room for two blocks on an SM; the filter
// (its stencils are applied to whole tables) stays with the general passes.
bool es1d_fp64_use_moments(const Es1dConst &c) { return c.nc <= kMomMaxNodes && c.passes == 0; }

LaunchShape es1d_mom_shape(const Es1dConst &c, int nsm) {
  return fixed_shape(c.n_total, nsm, 1, c.nc / 2, mom_smem(c, 1, true) <= kTwoBlockSmem ? 2 : 1);
}

bool es1d_mom_late(const Es1dConst &c) { return mom_smem(c, 1, false) > kTwoBlockSmem; }

int es1d_mom_copies(const Es1dConst &c, LaunchShape ls) {
  return fixed_copies((int64_t)c.nc * (c.order + 1), (c.n_total + ls.grid - 1) / ls.grid,
                      kMomTileBytes);
}

int64_t es1d_mom_chunk(const Es1dConst &c, LaunchShape ls) { return fixed_chunk(c.n_total, ls); }

cudaError_t es1d_mom_prepare(const Es1dConst &c) {
  cudaError_t e = cudaSuccess;
  dispatch_mom(c, [&](auto O, auto S, auto F) {
    constexpr int ORDER = decltype(O)::value, SCHEME = decltype(S)::value;
    constexpr bool FOLD = decltype(F)::value;
    const size_t most = mom_smem(c);
    for (const void *k : {(const void *)mom_pass_c_kernel<ORDER, SCHEME, FOLD>,
                          (const void *)mom_pass_e_kernel<ORDER, SCHEME, FOLD>,
                          (const void *)mom_deposit_initial_kernel<ORDER>})
      if (e == cudaSuccess)
        e = allow_shared(k, most);
  });
  return e;
}

// (b.Jt, b.vmax, b.words and b.rec zero before) the deposits' scale and, for ESEC2, j^{n,*}
void es1d_mom_start(const Es1dConst &c, const Es1dFp64Bufs &b, int parity, LaunchShape ls,
                    cudaStream_t st) {
  (c.order == 1 ? mom_absmax_kernel<1> : mom_absmax_kernel<2>)
      <<<ls.grid, ls.block, 0, st>>>(c, b, parity);
  mom_scales_kernel<<<1, 512, 0, st>>>(c, b, parity);
  if (c.scheme == 2)
    launch_dependent(c.order == 1 ? mom_deposit_initial_kernel<1> : mom_deposit_initial_kernel<2>,
                     ls, mom_smem(c), st, false, c, b, parity);
}

void es1d_mom_pass_c(const Es1dConst &c, const Es1dFp64Bufs &b, int64_t step_index, int slot,
                     LaunchShape ls, cudaStream_t st) {
  const int par = (int)(step_index & 1);
  dispatch_mom(c, [&](auto O, auto S, auto F) {
    launch_dependent(mom_pass_c_kernel<decltype(O)::value, decltype(S)::value, decltype(F)::value>,
                     LaunchShape{ls.grid + 1, ls.block}, mom_smem(c), st, true, c, b, par, slot - 1);
  });
}

void es1d_mom_pass_e(const Es1dConst &c, const Es1dFp64Bufs &b, int64_t step_index, int slot,
                     LaunchShape ls, cudaStream_t st) {
  const int par = (int)(step_index & 1);
  dispatch_mom(c, [&](auto O, auto S, auto F) {
    launch_dependent(mom_pass_e_kernel<decltype(O)::value, decltype(S)::value, decltype(F)::value>,
                     LaunchShape{ls.grid + 1, ls.block}, mom_smem(c), st, true, c, b, par, slot);
  });
}

}  // namespace pic
