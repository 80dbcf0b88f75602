// The FP64 form's 2D3V Yee step with point shapes where a cell has markers enough
// (em2d_use_moments; em2d_fp64.cu states the scheme and keeps the other runs), written to spare the FP64 pipe, which
// bounds the marker passes (2 lanes per SM and clock):
//
//   gather    a component's B-spline interpolant in a cell is a polynomial of the
//             marker's offsets, sum_pq C_pq dx^p dy^q (order 1: 4 coefficients,
//             order 2: 9).  The grid kernels write the coefficients of every cell
//             once, times dt/2 (q/m) of a single species; a marker takes 3 (8) FMAs
//             a component and no weights.  Components on the same nodes lie side by
//             side: (Ex, By), (Ey, Bx), Ez, Bz.
//   deposit   the moments A dx^p dy^q of a marker's amount to its cell, with global
//             FP64 atomics; the grid kernels turn them into node currents with the
//             same polynomials, so gather and deposit use one shape (Eq.
//             exp_econs_simple to rounding).  q w0 / |h| of a single uniform species
//             is applied there.  Order 1: the four moments of a cell are one 32-byte
//             sector; four lanes exchange their moments so that each atomic
//             instruction covers whole sectors.
//   points    integer-node offsets of both axes and the half-node offsets derived
//             from them (pass C -> E at x^{n+1/2}, pass E -> C at the next x*).
//   scale     with h = dt/2 (q/m): pass C's gathers give u - v^n and t; pass E's
//             d' = h (E + v* x B) = (v^dag - v^n) / 2 (gamma_series in
//             es1d_fp64_common.cuh takes the correction from there).
//
// Measured (128 x 128, 2^20 markers, order 1; FP64 pipe 85% busy in both passes,
// 62 and 78 warp instructions on it per 32 markers): pass C 268 -> 128 us, pass E
// 340 -> 160 us, a step 665 -> 340 us; the grid kernels went 4 -> 10 us each.
//
// Grid kernels: one block a 32 x 8 tile of one component, the field (and its rim)
// in shared memory, then the coefficients.
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>

#include "em2d_common.cuh"
#include "fixed_moments.cuh"
#include "pdl.cuh"
#include "pic_internal.cuh"

namespace pic {
namespace {

constexpr int kTX = 32, kTY = 8;           // tile of a grid block
constexpr int kPassThreads = 256;

// Coefficient tables: place of component f (Ex, Ey, Ez, Bx, By, Bz) of cell 0 and
// the stride between cells, in units of K2 = (order + 1)^2 words.
__device__ __forceinline__ void table_place(int f, int nc, int &base, int &stride) {
  // (Ex, By) | (Ey, Bx) | Ez | Bz
  stride = f == 2 || f == 5 ? 1 : 2;
  base = f == 0 ? 0 : f == 4 ? 1 : f == 1 ? 2 * nc : f == 3 ? 2 * nc + 1 : f == 2 ? 4 * nc : 5 * nc;
}

// The current of component d at node (i, j) from the cells' moments M [nc][K2].
template <int ORDER>
__device__ double node_current(const double *M, int i, int j, int nx, int ny) {
  constexpr int K2 = (ORDER + 1) * (ORDER + 1);
  const int im = i == 0 ? nx - 1 : i - 1, jm = j == 0 ? ny - 1 : j - 1;
  if (ORDER == 1) {
    const double *c00 = M + (size_t)K2 * (j * nx + i), *c10 = M + (size_t)K2 * (j * nx + im);
    const double *c01 = M + (size_t)K2 * (jm * nx + i), *c11 = M + (size_t)K2 * (jm * nx + im);
    // weights (1 - dx)(1 - dy), dx (1 - dy) from the cell to the left, ...
    return ((c00[0] - c00[1]) - (c00[2] - c00[3])) + (c10[1] - c10[3]) + (c01[2] - c01[3]) + c11[3];
  }
  const int ip = i + 1 == nx ? 0 : i + 1, jp = j + 1 == ny ? 0 : j + 1;
  const int ci[3] = {im, i, ip}, cj[3] = {jm, j, jp};
  double s = 0.0;
#pragma unroll
  for (int b = 0; b < 3; b++) {
    double r[3] = {0.0, 0.0, 0.0};   // the row's sums over x, by power of dy
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const double *m = M + (size_t)K2 * (cj[b] * nx + ci[a]);
#pragma unroll
      for (int q = 0; q < 3; q++) {
        // the cell's nearest node is ci[a]: this node is its right (a = 0), own or
        // left (a = 2) neighbour
        const double m0 = m[3 * q], m1 = m[3 * q + 1], m2 = m[3 * q + (ORDER == 2 ? 2 : 0)];
        r[q] += a == 1 ? fma(0.75, m0, -m2)
                       : fma(0.125, m0, 0.5 * (a == 0 ? m2 + m1 : m2 - m1));
      }
    }
    s += b == 1 ? fma(0.75, r[0], -r[2]) : fma(0.125, r[0], 0.5 * (b == 0 ? r[2] + r[1] : r[2] - r[1]));
  }
  return s;
}

// The coefficients of cell (tx, ty) of the tile from the field F, whose rows are
// kTX + 2 wide with the rim's first node at (-1, -1).
template <int ORDER>
__device__ __forceinline__ void store_coefs(const double (*F)[kTX + 2], int tx, int ty,
                                            double *out) {
  if (ORDER == 1) {
    const double a = F[ty + 1][tx + 1], b = F[ty + 1][tx + 2] - a, c = F[ty + 2][tx + 1] - a;
    const double e = (F[ty + 2][tx + 2] - F[ty + 2][tx + 1]) - b;
    *(double2 *)out = make_double2(a, b);
    *(double2 *)(out + 2) = make_double2(c, e);
  } else {
    double r[3][3];   // [row][power of dx]
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const double fm = F[ty + b][tx], f0 = F[ty + b][tx + 1], fp = F[ty + b][tx + 2];
      const double cc = fma(0.5, fm + fp, -f0);
      r[b][0] = fma(0.25, cc, f0);
      r[b][1] = 0.5 * (fp - fm);
      r[b][2] = cc;
    }
#pragma unroll
    for (int p = 0; p < 3; p++) {
      const double cc = fma(0.5, r[0][p] + r[2][p], -r[1][p]);
      out[p] = fma(0.25, cc, r[1][p]);
      out[3 + p] = 0.5 * (r[2][p] - r[0][p]);
      out[6 + p] = cc;
    }
  }
}

// FULL false, K1: tables of E* = E^n + dt/2 (c^2 curl Bp - j^{n,*}) (ESEC1: E^n) and
// of Bp; clears J2.  FULL true, K3: E^{n+1} = E^n + dt (c^2 curl Bp - j^{*,n+1/2})
// and the table of E^{n+1/2} in E*'s place; clears J1.  blockIdx.y: the component.
template <int ORDER, bool FULL>
__global__ void __launch_bounds__(kTX * kTY) em_grid_kernel(Em2dConst c, Em2dBufs b) {
  constexpr int K2 = (ORDER + 1) * (ORDER + 1);
  __shared__ double F[kTY + 2][kTX + 2];
  const int nx = c.nx, ny = c.ny, nc = nx * ny, f = blockIdx.y;
  const int tiles_x = (nx + kTX - 1) / kTX;
  const int i0 = ((int)blockIdx.x % tiles_x) * kTX, j0 = ((int)blockIdx.x / tiles_x) * kTY;
  const int tx = threadIdx.x % kTX, ty = threadIdx.x / kTX;
  const double k = c.fold ? c.hdt_qm[0] : 1.0, qa = c.fold ? c.qw_a[0] : 1.0;
  griddep_wait();
  griddep_launch_dependents();
  for (int t = threadIdx.x; t < (kTY + 2) * (kTX + 2); t += kTX * kTY) {
    const int lx = t % (kTX + 2), ly = t / (kTX + 2);
    const int i = wrapi(i0 + lx - 1, nx), j = wrapi(j0 + ly - 1, ny), a = j * nx + i;
    double v;
    if (f >= 3) {
      v = b.Bp[(f - 3) * nc + a];
    } else {
      const double e = b.E[f * nc + a];
      if (!FULL) {
        v = e;
        if (c.scheme == 2)
          v = fma(0.5 * c.dt, fma(c.c2, curl_b(c, b.Bp, i, j, f),
                                  -qa * node_current<ORDER>(b.M1 + (size_t)K2 * f * nc, i, j, nx, ny)),
                  e);
      } else {
        const double en =
            fma(c.dt, fma(c.c2, curl_b(c, b.Bp, i, j, f),
                          -qa * node_current<ORDER>(b.M2 + (size_t)K2 * f * nc, i, j, nx, ny)), e);
        // a tile writes its own nodes
        if (lx >= 1 && lx <= kTX && ly >= 1 && ly <= kTY && i0 + lx - 1 < nx && j0 + ly - 1 < ny)
          b.En[f * nc + a] = en;
        v = 0.5 * (e + en);
      }
    }
    F[ly][lx] = k * v;
  }
  __syncthreads();
  const int i = i0 + tx, j = j0 + ty;
  if (i >= nx || j >= ny) return;
  int base, stride;
  table_place(f, nc, base, stride);
  store_coefs<ORDER>(F, tx, ty, b.T + (size_t)K2 * (base + (size_t)stride * (j * nx + i)));
  if (f < 3) {
    double *m = (FULL ? b.M1 : b.M2) + (size_t)K2 * (f * nc + j * nx + i);
#pragma unroll
    for (int q = 0; q < K2; q++) m[q] = 0.0;
  }
}

// A point: the integer-node cells and offsets of both axes, and the half-node ones
// (xi - 1/2: the same node where the offset reaches the cell's middle, else the
// one before).
template <int ORDER>
struct Point2 {
  int xI, yI;
  double dxI, dyI, dxH, dyH;
  __device__ __forceinline__ static bool upper(double d) {
    return ORDER == 1 ? __double2hiint(d) >= 0x3fe00000 : __double2hiint(d) >= 0;
  }
  __device__ __forceinline__ int xH(int nx) const {
    return upper(dxI) ? xI : (xI == 0 ? nx - 1 : xI - 1);
  }
  __device__ __forceinline__ int yH(int ny) const {
    return upper(dyI) ? yI : (yI == 0 ? ny - 1 : yI - 1);
  }
  __device__ __forceinline__ void load(const double *sd, const int *si, int64_t p, int64_t n) {
    xI = si[p];
    yI = si[n + p];
    dxI = sd[p];
    dyI = sd[n + p];
    dxH = sd[2 * n + p];
    dyH = sd[3 * n + p];
  }
  __device__ __forceinline__ void store(double *sd, int *si, int64_t p, int64_t n) const {
    si[p] = xI;
    si[n + p] = yI;
    sd[p] = dxI;
    sd[n + p] = dyI;
    sd[2 * n + p] = dxH;
    sd[3 * n + p] = dyH;
  }
  // the point of (x + s vx, y + s vy), wrapped, with the one rounding all kernels use
  __device__ __forceinline__ void set(const Em2dConst &c, double x, double y, double s, double vx,
                                      double vy, unsigned *err) {
    const Point64<ORDER> X(__dmul_rn(wrap_fast(__fma_rn(s, vx, x), c.Lx, err), c.inv_hx), c.nx);
    const Point64<ORDER> Y(__dmul_rn(wrap_fast(__fma_rn(s, vy, y), c.Ly, err), c.inv_hy), c.ny);
    xI = X.i;
    yI = Y.i;
    dxI = X.d;
    dyI = Y.d;
    dxH = __dadd_rn(dxI, upper(dxI) ? -0.5 : 0.5);
    dyH = __dadd_rn(dyI, upper(dyI) ? -0.5 : 0.5);
  }
};

// sum_pq C[q][p] dx^p dy^q
template <int ORDER>
__device__ __forceinline__ double eval2(const double *C, double dx, double dy) {
  if constexpr (ORDER == 1) {
    const double2 ab = *(const double2 *)C, ce = *((const double2 *)C + 1);
    return __fma_rn(__fma_rn(ce.y, dx, ce.x), dy, __fma_rn(ab.y, dx, ab.x));
  } else {
    double r[3];
#pragma unroll
    for (int q = 0; q < 3; q++)
      r[q] = __fma_rn(__fma_rn(C[3 * q + 2], dx, C[3 * q + 1]), dx, C[3 * q]);
    return __fma_rn(__fma_rn(r[2], dy, r[1]), dy, r[0]);
  }
}

// E and B at P from the table.
template <int ORDER>
__device__ __forceinline__ void gather2(const double *T, const Point2<ORDER> &P, int nx, int ny,
                                        double (&e)[3], double (&bb)[3]) {
  constexpr int K2 = (ORDER + 1) * (ORDER + 1);
  const size_t nc = (size_t)nx * ny;
  const int xH = P.xH(nx), yH = P.yH(ny);
  const double *a = T + K2 * 2 * (size_t)(P.yI * nx + xH);              // (Ex, By)
  const double *b = T + K2 * 2 * (nc + (size_t)(yH * nx + P.xI));       // (Ey, Bx)
  const double *z = T + K2 * (4 * nc + (size_t)(P.yI * nx + P.xI));     // Ez
  const double *w = T + K2 * (5 * nc + (size_t)(yH * nx + xH));         // Bz
  e[0] = eval2<ORDER>(a, P.dxH, P.dyI);
  bb[1] = eval2<ORDER>(a + K2, P.dxH, P.dyI);
  e[1] = eval2<ORDER>(b, P.dxI, P.dyH);
  bb[0] = eval2<ORDER>(b + K2, P.dxI, P.dyH);
  e[2] = eval2<ORDER>(z, P.dxI, P.dyI);
  bb[2] = eval2<ORDER>(w, P.dxH, P.dyH);
}

// The moments of an amount A at offsets (dx, dy) of a cell, added to M [nc][K2].
// Every lane of the warp calls it (on: this lane has a marker).
template <int ORDER>
__device__ __forceinline__ void deposit2(double *M, int cell, double dx, double dy, double A,
                                         bool on) {
  if (ORDER == 1) {
    double m[4];
    m[0] = A;
    m[1] = __dmul_rn(A, dx);
    m[2] = __dmul_rn(A, dy);
    m[3] = __dmul_rn(m[1], dy);
    // 4 x 4 transposition among the lanes 4 g .. 4 g + 3: afterwards m[r] is moment
    // `lane & 3` of the group's marker r
    const int j = threadIdx.x & 3;
    {
      const bool up = j & 1;
#pragma unroll
      for (int r = 0; r < 4; r += 2) {
        const double x = __shfl_xor_sync(0xffffffffu, up ? m[r] : m[r + 1], 1);
        if (up) m[r] = x;
        else m[r + 1] = x;
      }
    }
    {
      const bool up = j & 2;
#pragma unroll
      for (int r = 0; r < 2; r++) {
        const double x = __shfl_xor_sync(0xffffffffu, up ? m[r] : m[r + 2], 2);
        if (up) m[r] = x;
        else m[r + 2] = x;
      }
    }
    const int mine = on ? cell : -1;
#pragma unroll
    for (int r = 0; r < 4; r++) {
      const int cr = __shfl_sync(0xffffffffu, mine, r, 4);
      if (cr >= 0) atomicAdd(&M[4 * (size_t)cr + j], m[r]);
    }
  } else if (on) {
    double *q = M + 9 * (size_t)cell;
    double r = A;
#pragma unroll
    for (int b = 0; b < 3; b++) {
      const double m1 = __dmul_rn(r, dx);
      atomicAdd(q + 3 * b, r);
      atomicAdd(q + 3 * b + 1, m1);
      atomicAdd(q + 3 * b + 2, __dmul_rn(m1, dx));
      if (b < 2) r = __dmul_rn(r, dy);
    }
  }
}

template <int ORDER>
__device__ __forceinline__ void deposit_j2(const Em2dConst &c, double *M, const Point2<ORDER> &P,
                                           const double (&A)[3], bool on) {
  constexpr int K2 = (ORDER + 1) * (ORDER + 1);
  const int nx = c.nx;
  const size_t nc = (size_t)nx * c.ny;
  const int xH = P.xH(nx), yH = P.yH(c.ny);
  deposit2<ORDER>(M, P.yI * nx + xH, P.dxH, P.dyI, A[0], on);
  deposit2<ORDER>(M + K2 * nc, yH * nx + P.xI, P.dxI, P.dyH, A[1], on);
  deposit2<ORDER>(M + 2 * K2 * nc, P.yI * nx + P.xI, P.dxI, P.dyI, A[2], on);
}

__device__ __forceinline__ int species_of2m(const Em2dConst &c, int64_t p) {
  int s = 0;
  while (s < c.nsp - 1 && p >= c.sp_end[s]) s++;
  return s;
}

template <int ORDER, bool FOLD>
__global__ void __launch_bounds__(kPassThreads, 2) em_mom_c_kernel(Em2dConst c, Em2dBufs b) {
  griddep_wait();
  const int64_t n = c.n_total, beg = blockIdx.x * c.chunk;
  const int64_t end = beg + c.chunk < n ? beg + c.chunk : n;
  for (int64_t p0 = beg; p0 < end; p0 += blockDim.x) {   // whole warps: the deposits shuffle
    const bool on = p0 + threadIdx.x < end;
    const int64_t p = p0 + threadIdx.x;   // lanes past the end work on zeros
    const int s = FOLD ? 0 : species_of2m(c, p);
    const double x = on ? b.x[p] : 0.0, y = on ? b.y[p] : 0.0;
    const double v[3] = {on ? b.vx[p] : 0.0, on ? b.vy[p] : 0.0, on ? b.vz[p] : 0.0};
    Point2<ORDER> P{};
    if (!b.sds)
      P.set(c, x, y, c.hdt, v[0], v[1], b.err);
    else if (on)   // the point x* that j^{n,*} was deposited at
      P.load(b.sds, b.sis, p, n);
    double u[3], t[3];
    gather2<ORDER>(b.T, P, c.nx, c.ny, u, t);
#pragma unroll
    for (int d = 0; d < 3; d++) {
      if (FOLD) {
        u[d] = __dadd_rn(v[d], u[d]);
      } else {
        u[d] = __fma_rn(c.hdt_qm[s], u[d], v[d]);
        t[d] = __dmul_rn(c.hdt_qm[s], t[d]);
      }
    }
    // v* - v* x t = u  ->  v* = (u + u x t + (u.t) t) / (1 + |t|^2)
    const double ut = __fma_rn(u[2], t[2], __fma_rn(u[1], t[1], __dmul_rn(u[0], t[0])));
    const double inv = recip_newton(
        __fma_rn(t[2], t[2], __fma_rn(t[1], t[1], __fma_rn(t[0], t[0], 1.0))));
    double vs[3];
#pragma unroll
    for (int d = 0; d < 3; d++) {
      const int d1 = (d + 1) % 3, d2 = (d + 2) % 3;
      const double w = __fma_rn(-u[d2], t[d1], __fma_rn(u[d1], t[d2], u[d]));
      vs[d] = __dmul_rn(__fma_rn(ut, t[d], w), inv);
    }
    P.set(c, x, y, c.hdt, vs[0], vs[1], b.err);   // x^{n+1/2}
    double A[3] = {vs[0], vs[1], vs[2]};
    if (!FOLD) {
      const double q = b.w && on ? c.q_a[s] * b.w[p] : c.qw_a[s];
#pragma unroll
      for (int d = 0; d < 3; d++) A[d] *= q;
    }
    if (on) {
      b.vsx[p] = vs[0];
      b.vsy[p] = vs[1];
      b.vsz[p] = vs[2];
      P.store(b.sd, b.si, p, n);
    }
    deposit_j2<ORDER>(c, b.M2, P, A, on);
  }
  griddep_launch_dependents();
}

template <int ORDER, bool FOLD>
__global__ void __launch_bounds__(kPassThreads, 2) em_mom_e_kernel(Em2dConst c, Em2dBufs b,
                                                                   int slot) {
  __shared__ double red[kRedWords];
  griddep_wait();
  const int64_t n = c.n_total, beg = blockIdx.x * c.chunk;
  const int64_t end = beg + c.chunk < n ? beg + c.chunk : n;
  double ke = 0.0;
  unsigned nfb = 0, bad = 0;
  for (int64_t p0 = beg; p0 < end; p0 += blockDim.x) {
    const bool on = p0 + threadIdx.x < end;
    const int64_t p = p0 + threadIdx.x;   // lanes past the end work on zeros
    const int s = FOLD ? 0 : species_of2m(c, p);
    Point2<ORDER> P{};
    if (on) P.load(b.sd, b.si, p, n);
    double d[3], bb[3];
    gather2<ORDER>(b.T, P, c.nx, c.ny, d, bb);
    const double vs[3] = {on ? b.vsx[p] : 0.0, on ? b.vsy[p] : 0.0, on ? b.vsz[p] : 0.0};
    const double v[3] = {on ? b.vx[p] : 0.0, on ? b.vy[p] : 0.0, on ? b.vz[p] : 0.0};
    double vn[3], A0 = 0.0, vd2 = 0.0;   // vn: v^dag first
#pragma unroll
    for (int a = 0; a < 3; a++) {
      const int a1 = (a + 1) % 3, a2 = (a + 2) % 3;
      d[a] = __fma_rn(-vs[a2], bb[a1], __fma_rn(vs[a1], bb[a2], d[a]));
      if (!FOLD) d[a] *= c.hdt_qm[s];
      vn[a] = __fma_rn(2.0, d[a], v[a]);
      const double br = __dadd_rn(__dadd_rn(vs[a], -v[a]), -d[a]);   // v* - v^n - Delta/2
      A0 = a == 0 ? __dmul_rn(br, d[0]) : __fma_rn(br, d[a], A0);
      vd2 = a == 0 ? __dmul_rn(vn[0], vn[0]) : __fma_rn(vn[a], vn[a], vd2);
    }
    if (c.gamma_on) {
      double gm;
      if (gamma_series(__dmul_rn(4.0, A0), vd2, gm)) {
#pragma unroll
        for (int a = 0; a < 3; a++) vn[a] = __fma_rn(gm, vn[a], vn[a]);
      } else if (on) {
        double R = 0.0, v2 = 0.0;
#pragma unroll
        for (int a = 0; a < 3; a++) {
          R = fma(vs[a], d[a], R);
          v2 = fma(v[a], v[a], v2);
        }
        gm = gamma_root(fma(4.0, R, v2), vd2, nfb);   // Gamma = sqrt(R) / |v^dag|
#pragma unroll
        for (int a = 0; a < 3; a++) vn[a] *= gm;
      }
    }
    const double xn = wrap_fast(__fma_rn(c.dt, vs[0], on ? b.x[p] : 0.0), c.Lx, b.err);
    const double yn = wrap_fast(__fma_rn(c.dt, vs[1], on ? b.y[p] : 0.0), c.Ly, b.err);
    const double q2 = __fma_rn(vn[2], vn[2], __fma_rn(vn[1], vn[1], __dmul_rn(vn[0], vn[0])));
    if (on) {
      ke = FOLD ? __dadd_rn(ke, q2)
                : __fma_rn(b.w ? c.half_m[s] * b.w[p] : c.half_mw[s], q2, ke);
      if (((unsigned)__double2hiint(q2) & 0x7ff00000u) == 0x7ff00000u &&
          !isfinite(vn[0] + vn[1] + vn[2]))
        bad = kErrNonfinite;
      b.vx[p] = vn[0];
      b.vy[p] = vn[1];
      b.vz[p] = vn[2];
      b.x[p] = xn;
      b.y[p] = yn;
    }
    if (c.scheme == 2) {
      Point2<ORDER> N;
      N.set(c, xn, yn, c.hdt, vn[0], vn[1], b.err);
      double A[3] = {vn[0], vn[1], vn[2]};
      if (!FOLD) {
        const double q = b.w && on ? c.q_a[s] * b.w[p] : c.qw_a[s];
#pragma unroll
        for (int a = 0; a < 3; a++) A[a] *= q;
      }
      if (on) N.store(b.sds, b.sis, p, n);   // the next pass C gathers there
      deposit_j2<ORDER>(c, b.M1, N, A, on);
    }
  }
  griddep_launch_dependents();
  if (bad) atomicOr(b.err, bad);
  nfb = __reduce_add_sync(0xffffffffu, nfb);
  if ((threadIdx.x & 31) == 0 && nfb) atomicAdd(&b.fallback[slot], (unsigned long long)nfb);
  const double t = block_sum_narrow(ke, red);
  if (threadIdx.x == 0) b.ke_part[blockIdx.x] = FOLD ? c.half_mw[0] * t : t;
}

// j^{n,*} of the current state (start-up and after a state change)
template <int ORDER, bool FOLD>
__global__ void __launch_bounds__(kPassThreads, 2) em_mom_start_kernel(Em2dConst c, Em2dBufs b) {
  const int64_t n = c.n_total, beg = blockIdx.x * c.chunk;
  const int64_t end = beg + c.chunk < n ? beg + c.chunk : n;
  for (int64_t p0 = beg; p0 < end; p0 += blockDim.x) {
    const bool on = p0 + threadIdx.x < end;
    const int64_t p = p0 + threadIdx.x;   // lanes past the end work on zeros
    const int s = FOLD ? 0 : species_of2m(c, p);
    double A[3] = {on ? b.vx[p] : 0.0, on ? b.vy[p] : 0.0, on ? b.vz[p] : 0.0};
    Point2<ORDER> N;
    N.set(c, on ? b.x[p] : 0.0, on ? b.y[p] : 0.0, c.hdt, A[0], A[1], b.err);
    if (!FOLD) {
      const double q = b.w && on ? c.q_a[s] * b.w[p] : c.qw_a[s];
#pragma unroll
      for (int a = 0; a < 3; a++) A[a] *= q;
    }
    if (on) N.store(b.sds, b.sis, p, n);
    deposit_j2<ORDER>(c, b.M1, N, A, on);
  }
}

template <typename F>
void dispatch_em2(const Em2dConst &c, F f) {
  using I1 = std::integral_constant<int, 1>;
  using I2 = std::integral_constant<int, 2>;
  if (c.order == 1)
    c.fold ? f(I1(), std::true_type()) : f(I1(), std::false_type());
  else
    c.fold ? f(I2(), std::true_type()) : f(I2(), std::false_type());
}

template <bool FULL>
void grid_launch(const Em2dConst &c, const Em2dBufs &b, int comps, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(((c.nx + kTX - 1) / kTX) * ((c.ny + kTY - 1) / kTY), comps);
  cfg.blockDim = dim3(kTX * kTY);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (c.order == 1)
    cudaLaunchKernelEx(&cfg, em_grid_kernel<1, FULL>, c, b);
  else
    cudaLaunchKernelEx(&cfg, em_grid_kernel<2, FULL>, c, b);
}

}  // namespace

// A marker costs less here (order 1: 0.31 ns of a step against 0.62, order 2: 0.56
// against 0.98), a node more, 0.3 and 1.5 to 2 ns a step: its coefficients and
// moments are 576 (order 2: 1296) bytes, written twice.  Order 1: a marker a node
// pays for it, less some that the six launches' overlap pays for.  Order 2: five
// markers a node, eleven where the coefficients (432 bytes a node) leave the L2, and
// some more for launches that take longer; all runs on grids of up to 64 x 64.  us a
// step (ESEC2), general passes / these: order 1, 1024 x 1024, 10^5 markers 248 / 542,
// 2^21 markers 1406 / 1153; order 2, 256 x 256, 10^5 markers 162 / 267, 2^19 markers
// 581 / 450; 1024 x 1024, 2^23 markers 8112 / 8691.
bool em2d_use_moments(const Em2dConst &c) {
  const int64_t nodes = (int64_t)c.nx * c.ny;
  if (c.order == 1) return c.n_total + (1 << 14) >= nodes + nodes / 8;
  return nodes <= 64 * 64 || c.n_total >= (nodes <= 1 << 18 ? 5 : 11) * nodes + 45'000;
}

// Two blocks of up to 256 per SM, each with an equal run of markers.  No warp is
// without: one that is lets the next launch's blocks take the SMs before the others
// are done (64 x 64, order 2, 57,344 markers: 135 us a step, with these 81).
LaunchShape em2d_mom_shape(const Em2dConst &c, int nsm) {
  const int64_t most = 2 * (int64_t)nsm;
  const int64_t chunk = ((c.n_total + most - 1) / most + 31) / 32 * 32;
  return LaunchShape{c.n_total ? (int)((c.n_total + chunk - 1) / chunk) : 1,
                     (int)std::min<int64_t>(kPassThreads, std::max<int64_t>(chunk, 32))};
}
int64_t em2d_mom_chunk(const Em2dConst &c, LaunchShape ls) { return fixed_chunk(c.n_total, ls); }

void em2d_mom_k1(const Em2dConst &c, const Em2dBufs &b, cudaStream_t st) {
  grid_launch<false>(c, b, 6, st);
}
void em2d_mom_k3(const Em2dConst &c, const Em2dBufs &b, cudaStream_t st) {
  grid_launch<true>(c, b, 3, st);
}
void em2d_mom_pass_c(const Em2dConst &c, const Em2dBufs &b, LaunchShape lp, cudaStream_t st) {
  dispatch_em2(c, [&](auto O, auto F) {
    launch_dependent(em_mom_c_kernel<decltype(O)::value, decltype(F)::value>, lp, 0, st, true, c, b);
  });
}
void em2d_mom_pass_e(const Em2dConst &c, const Em2dBufs &b, int slot, LaunchShape lp,
                     cudaStream_t st) {
  dispatch_em2(c, [&](auto O, auto F) {
    launch_dependent(em_mom_e_kernel<decltype(O)::value, decltype(F)::value>, lp, 0, st, true, c, b,
                     slot);
  });
}
void em2d_mom_start(const Em2dConst &c, const Em2dBufs &b, LaunchShape lp, cudaStream_t st) {
  dispatch_em2(c, [&](auto O, auto F) {
    em_mom_start_kernel<decltype(O)::value, decltype(F)::value>
        <<<lp.grid, lp.block, 0, st>>>(c, b);
  });
}

}  // namespace pic
