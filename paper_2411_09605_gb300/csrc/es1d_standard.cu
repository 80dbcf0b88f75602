// Standard explicit PIC, the comparison scheme of Sec. 5: Vlasov-Poisson with
// the classical leapfrog push (in 1D1V the Boris push without B) and a
// binomially filtered charge density, FP64, 1D1V.  It does not conserve
// energy; it is here to measure the energy-conserving schemes against.
//
// State: x^n, v^{n-1/2} and E^n, the field of the filtered charge of x^n.
// Two launches per step:
//   markers  every block: E^n table in shared memory; per marker E^n_p,
//     v^{n+1/2} = v^{n-1/2} + dt (q/m) E^n_p, x^{n+1} = x^n + dt v^{n+1/2},
//     the kinetic partial (1/2) m w (v^{n-1/2}^2 + v^{n+1/2}^2) / 2, and the
//     charge q w S(x_h - x^{n+1}) / h;
//   solve  Gauss's law for E^{n+1}: E_k = rho_k F_k / (i kk_k) with the filter gain
//     F_k = cos^{2p}(pi k / n) of p passes of the 1-2-1 filter (its exact
//     effect on mode k) and 0 for k = 0 (the ion background) and the Nyquist
//     mode, as a convolution of rho - <rho> with that operator's response to a
//     unit charge, one warp a node; and TE^n = KE^n + (h/2) sum (E^n)^2.
//
// The marker pass is bound by the FP64 pipe and is written like the 1D1V moment
// passes (es1d_fp64_moments.cu): polynomial gathers with dt q/m folded in (a uniform
// weight's charge is the constant 1, its moments shifts of the offset), exact
// fixed-point sums, the point of x^{n+1} kept for the next step's gather.  The
// solve was a pair of transforms by the block that finished last, one SM's FP64
// pipe while the others waited; n^2 FMAs over all SMs are faster than that at
// every n up to kStdMaxNodes (512 nodes: about 3 us against 35).
// Measured, 2^20 markers, 512 nodes, order 2: 133 -> 45 us a step.
#include <cuda_runtime.h>

#include <type_traits>

#include "es1d_fp64_common.cuh"
#include "fixed_moments.cuh"
#include "pdl.cuh"
#include "pic_internal.cuh"
#include "spectral_common.cuh"

namespace pic {
namespace {

constexpr int kStdThreads = 256;
constexpr int kStdSolveThreads = 128;            // a warp a node, one warp per SM quarter
constexpr int64_t kStdTileBytes = 48 * 1024;     // tile copies of a block

__device__ __forceinline__ int species_of_std(const StdConst &c, int64_t p) {
  int s = 0;
  while (s < c.nsp - 1 && p >= c.sp_end[s]) s++;
  return s;
}

__device__ __forceinline__ double std_qw(const StdConst &c, const StdBufs &b, int s, int64_t p) {
  return b.w ? c.q_h[s] * b.w[p] : c.qw_h[s];
}

// Words a node of the gather table: (a, b) and c of order 2, one array each.
template <int ORDER>
__device__ __forceinline__ void build_poly_std(double *table, const double *E, int n, double k) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const double f0 = k * E[i], fp = k * E[(i + 1) & (n - 1)];
    if (ORDER == 1) {
      table[i] = f0;
      table[n + i] = fp - f0;
    } else {
      const double fm = k * E[(i - 1) & (n - 1)];
      const double cc = fma(0.5, fm + fp, -f0);
      table[i] = fma(0.25, cc, f0);
      table[n + i] = 0.5 * (fp - fm);
      table[2 * n + i] = cc;
    }
  }
}

template <int ORDER>
__device__ __forceinline__ double gather_std(const double *table, int n, int i, double d) {
  if (ORDER == 1) return __fma_rn(table[n + i], d, table[i]);
  return __fma_rn(__fma_rn(table[2 * n + i], d, table[n + i]), d, table[i]);
}

__device__ __forceinline__ int64_t chunk_end(const StdConst &c) {
  const int64_t e = (blockIdx.x + 1) * c.chunk;
  return e < c.n_total ? e : c.n_total;
}

// A marker's charge at P into this lane's tile copy; the scale words W (not FOLD) lie
// after the tile.
template <int ORDER, bool FOLD>
__device__ __forceinline__ void std_deposit(unsigned *Tl, unsigned *W, const StdConst &c,
                                            const StdBufs &b, int s, int64_t p,
                                            const Point64<ORDER> &P) {
  unsigned *q = Tl + (size_t)P.i * 2 * (ORDER + 1) * c.copies;
  if (FOLD) {
    add_unit_moments<ORDER>(q, c.copies, P, c.qw_h[0], b.rho, b.rho + c.n, c.n);
  } else {
    const double A = std_qw(c, b, s, p);
    add_moments<ORDER>(q, c.copies, W + P.i, W + c.n + 1, P, A, 1.0, b.rho, b.rho + c.n, c.n);
  }
}
template <int ORDER, bool FOLD>
__device__ __forceinline__ unsigned *std_scales(unsigned *T, const StdConst &c) {
  return FOLD ? nullptr : T + (size_t)2 * (ORDER + 1) * c.n * c.copies;
}

template <int ORDER, bool FOLD>
__global__ void __launch_bounds__(kFixedMaxThreads, 2) std_step_kernel(StdConst c, StdBufs b) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[kRedWords];
  const int n = c.n, copies = c.copies;
  unsigned *T = (unsigned *)(sm + (ORDER + 1) * n), *W = std_scales<ORDER, FOLD>(T, c);
  clear_fixed(T, 2 * (ORDER + 1) * n * copies);
  griddep_wait();
  const ScaleWords words(b.words, FOLD ? 0 : n + 1);   // (W null: not stored)
  build_poly_std<ORDER>(sm, b.E, n, FOLD ? c.dt_qm[0] : 1.0);
  if (!FOLD) words.store(W);
  unsigned *Tl = T + (threadIdx.x & (copies - 1));
  __syncthreads();
  double ke = 0.0;
  unsigned vm = 0;
  const int64_t end = chunk_end(c);
  for (int64_t p = blockIdx.x * c.chunk + threadIdx.x; p < end; p += blockDim.x) {
    const int s = FOLD ? 0 : species_of_std(c, p);
    const double x = b.x[p], v = b.v[p];
    const double g = gather_std<ORDER>(sm, n, b.si[p], b.sd[p]);
    const double vn = FOLD ? __dadd_rn(v, g) : __fma_rn(c.dt_qm[s], g, v);
    if (FOLD)
      ke = __fma_rn(v, v, __fma_rn(vn, vn, ke));
    else
      ke = fma(c.half_m[s] * (b.w ? b.w[p] : c.w0[s]), 0.5 * fma(v, v, vn * vn), ke);
    const double x1 = wrap_fast(__fma_rn(c.dt, vn, x), c.L, b.err);
    b.x[p] = x1;
    b.v[p] = vn;
    if (!FOLD) vm = max(vm, abs_hi(vn));
    const Point64<ORDER> P(__dmul_rn(x1, c.inv_h), n);
    b.si[p] = P.i;   // the next step gathers there
    b.sd[p] = P.d;
    std_deposit<ORDER, FOLD>(Tl, W, c, b, s, p, P);
  }
  griddep_launch_dependents();
  if (!isfinite(ke)) atomicOr(b.err, kErrNonfinite);
  if (!FOLD) flush_vmax(vm, b.vmax);
  const double kb = block_sum_narrow(ke, red);   // (its barriers order the tile's sums)
  if (threadIdx.x == 0) b.ke_part[blockIdx.x] = FOLD ? 0.5 * c.half_m[0] * c.w0[0] * kb : kb;
  if (!FOLD) flush_new(W, b.rec, n, W + n + 1, b.storm);
  flush_moments<ORDER, 1, !FOLD>(T, W, copies, n, FOLD ? c.qw_h[0] : 1.0, b.rho, b.rho + n,
                                 FOLD ? ScaleRange(0, 0) : ScaleRange(W[n]));
}

// The nodes' largest |charges| to the records (zero before).
template <int ORDER>
__global__ void __launch_bounds__(kFixedMaxThreads, 2) std_amax_kernel(StdConst c, StdBufs b) {
  __shared__ unsigned W[kStdMaxNodes];
  clear_largest(W, c.n);
  __syncthreads();
  unsigned vm = 0;
  const int64_t end = chunk_end(c);
  for (int64_t p = blockIdx.x * c.chunk + threadIdx.x; p < end; p += blockDim.x) {
    vm = max(vm, abs_hi(b.v[p]));
    raise_largest(W + Point64<ORDER>(__dmul_rn(b.x[p], c.inv_h), c.n).i,
                  abs_hi(std_qw(c, b, species_of_std(c, p), p)) >> 20);
  }
  flush_vmax(vm, b.vmax);
  __syncthreads();
  flush_largest(W, b.rec, c.n);
}
// The first scale words (one block).
__global__ void __launch_bounds__(512) std_scales_kernel(StdConst c, StdBufs b) {
  __shared__ unsigned S[kStdMaxNodes + 2 * kMostReach];
  ScaleMaker<>(b.words, b.rec, b.storm, c.n)
      .make(S, node_reach(__ldcg(b.vmax), c.reach), 0, c.n_total);
}

// The charge and the points of x^0.
template <int ORDER, bool FOLD>
__global__ void __launch_bounds__(kFixedMaxThreads, 2) std_charge_kernel(StdConst c, StdBufs b) {
  extern __shared__ __align__(16) double sm[];
  const int n = c.n, copies = c.copies;
  unsigned *T = (unsigned *)(sm + (ORDER + 1) * n), *W = std_scales<ORDER, FOLD>(T, c);
  clear_fixed(T, 2 * (ORDER + 1) * n * copies);
  if (!FOLD) ScaleWords(b.words, n + 1).store(W);
  __syncthreads();
  unsigned *Tl = T + (threadIdx.x & (copies - 1));
  const int64_t end = chunk_end(c);
  for (int64_t p = blockIdx.x * c.chunk + threadIdx.x; p < end; p += blockDim.x) {
    const int s = FOLD ? 0 : species_of_std(c, p);
    const Point64<ORDER> P(__dmul_rn(b.x[p], c.inv_h), n);
    b.si[p] = P.i;
    b.sd[p] = P.d;
    std_deposit<ORDER, FOLD>(Tl, W, c, b, s, p, P);
  }
  __syncthreads();
  if (!FOLD) flush_new(W, b.rec, n, W + n + 1, b.storm);
  flush_moments<ORDER, 1, !FOLD>(T, W, copies, n, FOLD ? c.qw_h[0] : 1.0, b.rho, b.rho + n,
                                 FOLD ? ScaleRange(0, 0) : ScaleRange(W[n]));
}

// E^{n+1} into En from rho [n] and its total rho[n]: block 0 writes TE^n (slot >= 0)
// from the nke kinetic partials and E^n and clears the other charge buffer, each
// warp of the others forms one node's E.
__global__ void __launch_bounds__(kStdSolveThreads) std_solve_kernel(StdConst c, StdBufs b, int slot,
                                                                     int nke) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[kRedWords];
  const int n = c.n;
  double *g = sm + n;
  if (blockIdx.x > 0)   // the response does not change: loaded before the wait
    for (int i = threadIdx.x; i < n; i += blockDim.x) g[i] = __ldg(b.resp + i);
  griddep_wait();
  griddep_launch_dependents();
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i <= n; i += blockDim.x) b.rhon[i] = 0.0;
    // the next markers' scales, from what the last ones recorded
    if (!c.fold) {
      ScaleMaker<>(b.words, b.rec, b.storm, n)
          .make((unsigned *)sm, node_reach(__ldcg(b.vmax), c.reach), c.decay, c.n_total);
      __syncthreads();
      if (threadIdx.x == 0) *b.vmax = 0u;
    }
    if (slot < 0) return;
    double t = 0.0;
    for (int i = threadIdx.x; i < n; i += blockDim.x) t = fma(0.5 * c.h * b.E[i], b.E[i], t);
    for (int i = threadIdx.x; i < nke; i += blockDim.x) t += b.ke_part[i];
    const double te = block_sum_narrow(t, red);
    if (threadIdx.x == 0) b.te[slot] = te;
    return;
  }
  const double mean = b.rho[n] * c.inv_n;
  for (int i = threadIdx.x; i < n; i += blockDim.x) sm[i] = b.rho[i] - mean;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int i = ((int)blockIdx.x - 1) * (kStdSolveThreads / 32) + (int)(threadIdx.x >> 5);
  if (i >= n) return;   // (whole warps)
  double e = 0.0;
  for (int k = lane; k < n; k += 32) e = fma(g[(i - k) & (n - 1)], sm[k], e);
  for (int o = 16; o > 0; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
  if (lane == 0) b.En[i] = e;
}

// v^{-1/2} = v^0 - dt/2 (q/m) E^0_p (the start of the leapfrog).
template <int ORDER>
__global__ void __launch_bounds__(kStdThreads) std_kick_back_kernel(StdConst c, StdBufs b) {
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < c.n_total;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int s = species_of_std(c, p);
    const Shape64<ORDER> S(b.x[p] * c.inv_h, c.n);
    b.v[p] = fma(-0.5 * c.dt * c.qm[s], S.gather(b.E), b.v[p]);
  }
}

// KE^n per species with v^{n+1/2} formed but not stored (block partials
// [nsp][grid]), and from block 0 W_E^n.
template <int ORDER>
__global__ void __launch_bounds__(kStdThreads) std_energy_kernel(StdConst c, StdBufs b,
                                                                  double *ke_out, double *we) {
  __shared__ double red[33];
  for (int s = 0; s < c.nsp; s++) {
    const int64_t lo = s == 0 ? 0 : c.sp_end[s - 1], hi = c.sp_end[s];
    double acc = 0.0;
    for (int64_t p = lo + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < hi;
         p += (int64_t)gridDim.x * blockDim.x) {
      const Shape64<ORDER> S(b.x[p] * c.inv_h, c.n);
      const double v = b.v[p], vn = fma(c.dt * c.qm[s], S.gather(b.E), v);
      acc = fma(b.w ? b.w[p] : c.w0[s], 0.5 * fma(v, v, vn * vn), acc);
    }
    const double t = block_sum_d(acc, red);
    if (threadIdx.x == 0) ke_out[(size_t)s * gridDim.x + blockIdx.x] = c.half_m[s] * t;
    __syncthreads();
  }
  if (blockIdx.x == 0) {
    double a = 0.0;
    for (int i = threadIdx.x; i < c.n; i += blockDim.x) a = fma(b.E[i], b.E[i], a);
    const double t = block_sum_d(a, red);
    if (threadIdx.x == 0) *we = 0.5 * c.h * t;
  }
}

// The response of E to a unit charge at node 0, resp[d] = (2/n) sum_k g_k
// sin(2 pi k d / n) over k = 1 .. n/2 - 1, g_k = cos^{2p}(pi k / n) / kk_k; one warp
// a node, once per set-up.
__global__ void std_response_kernel(StdConst c, StdBufs b) {
  const int n = c.n, lane = threadIdx.x & 31;
  const int d = (int)blockIdx.x * ((int)blockDim.x / 32) + (int)(threadIdx.x >> 5);
  if (d >= n) return;   // (whole warps)
  double r = 0.0;
  for (int k = 1 + lane; k < n / 2; k += 32) {
    const double cs = cospi((double)k / (double)n);
    double f = 1.0;
    for (int q = 0; q < c.passes; q++) f *= cs * cs;
    const int m = (int)(((int64_t)k * d) & (n - 1));
    r += f / (2.0 * 3.141592653589793 * (double)k / c.L) * sinpi(2.0 * (double)m / (double)n);
  }
  for (int o = 16; o > 0; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  if (lane == 0) b.resp[d] = 2.0 * r / n;
}

size_t std_smem(const StdConst &c, int copies) {
  return sizeof(double) * (size_t)(c.order + 1) * (1 + (size_t)copies) * c.n +
         (c.fold ? 0 : sizeof(unsigned) * (c.n + 2));
}
size_t std_solve_smem(const StdConst &c) { return sizeof(double) * 2 * (size_t)c.n; }

template <typename F>
void dispatch_std(const StdConst &c, F f) {
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  if (c.order == 1)
    c.fold ? f(I1(), std::true_type()) : f(I1(), std::false_type());
  else
    c.fold ? f(I2(), std::true_type()) : f(I2(), std::false_type());
}

void std_solve(const StdConst &c, const StdBufs &b, int slot, LaunchShape lp, cudaStream_t st,
               bool pdl) {
  const int rows = kStdSolveThreads / 32;
  launch_dependent(std_solve_kernel, LaunchShape{1 + (c.n + rows - 1) / rows, kStdSolveThreads},
                   std_solve_smem(c), st, pdl, c, b, slot, lp.grid);
}

}  // namespace

LaunchShape std_shape(const StdConst &c, int nsm) {
  return fixed_shape(c.n_total, nsm, 0, c.n / 2, std_smem(c, 1) <= kTwoBlockSmem ? 2 : 1);
}
int std_copies(const StdConst &c, LaunchShape ls) {
  return fixed_copies((int64_t)c.n * (c.order + 1), (c.n_total + ls.grid - 1) / ls.grid,
                      kStdTileBytes);
}
int64_t std_chunk(const StdConst &c, LaunchShape ls) { return fixed_chunk(c.n_total, ls); }

cudaError_t std_prepare(const StdConst &c, const StdBufs &b, cudaStream_t st) {
  const size_t sm = std_smem(c, c.copies);
  cudaError_t e = cudaSuccess;
  dispatch_std(c, [&](auto O, auto F) {
    constexpr int ORDER = decltype(O)::value;
    constexpr bool FOLD = decltype(F)::value;
    if ((e = allow_shared(std_step_kernel<ORDER, FOLD>, sm))) return;
    if ((e = allow_shared(std_charge_kernel<ORDER, FOLD>, sm))) return;
    e = allow_shared(std_solve_kernel, std_solve_smem(c));
  });
  if (e != cudaSuccess) return e;
  std_response_kernel<<<(c.n + 3) / 4, 128, 0, st>>>(c, b);
  return cudaGetLastError();
}

// The markers of a step into b.rho, then E^{n+1} into b.En (the caller swaps E with
// En and rho with rhon).
void std_markers(const StdConst &c, const StdBufs &b, LaunchShape lp, cudaStream_t st) {
  dispatch_std(c, [&](auto O, auto F) {
    launch_dependent(std_step_kernel<decltype(O)::value, decltype(F)::value>, lp,
                     std_smem(c, c.copies), st, true, c, b);
  });
}
void std_field(const StdConst &c, const StdBufs &b, int slot, LaunchShape lp, cudaStream_t st) {
  std_solve(c, b, slot, lp, st, true);
}

// (rho, rhon, vmax, words and rec zero before) the charge of x^0 and E^0 into b.En.
void std_start_field(const StdConst &c, const StdBufs &b, LaunchShape lp, cudaStream_t st) {
  if (!c.fold) {
    (c.order == 1 ? std_amax_kernel<1> : std_amax_kernel<2>)<<<lp.grid, lp.block, 0, st>>>(c, b);
    std_scales_kernel<<<1, 512, 0, st>>>(c, b);
  }
  dispatch_std(c, [&](auto O, auto F) {
    std_charge_kernel<decltype(O)::value, decltype(F)::value>
        <<<lp.grid, lp.block, std_smem(c, c.copies), st>>>(c, b);
  });
  std_solve(c, b, -1, lp, st, false);
}

void std_kick_back(const StdConst &c, const StdBufs &b, LaunchShape lp, cudaStream_t st) {
  if (c.order == 1)
    std_kick_back_kernel<1><<<lp.grid, kStdThreads, 0, st>>>(c, b);
  else
    std_kick_back_kernel<2><<<lp.grid, kStdThreads, 0, st>>>(c, b);
}

void std_energy(const StdConst &c, const StdBufs &b, double *ke_out, double *we, LaunchShape lp,
                cudaStream_t st) {
  if (c.order == 1)
    std_energy_kernel<1><<<lp.grid, kStdThreads, 0, st>>>(c, b, ke_out, we);
  else
    std_energy_kernel<2><<<lp.grid, kStdThreads, 0, st>>>(c, b, ke_out, we);
}

}  // namespace pic
