// Advection-diffusion (Helmholtz-type) velocity solve of the fractional step, with no-slip
// ghost rows, by scheduled relaxed Jacobi (SRJ): Sec. "Governing Equations and Numerical
// Methods" (the momentum equation split into an advection-diffusion step solved with SRJ and
// the pressure Poisson equation), Sec. "Results and Discussions" (the diagonally dominant
// advection-diffusion system), Sec. "GPU Porting" item 2 (no-slip on the immersed surface).
//
// System (the paper gives no discretisation; reading): one velocity component u solves
//   fluid row i:  D_i u_i - alpha sum_d c_{i,d} v_nb = f_i,  D_i = 1 + alpha sum_d c_{i,d}
//                 (c: the pressure system's 7-point coefficients, zero across the walls;
//                 v_nb the neighbour, the ghost cell or, across a cut membrane link, the
//                 neighbour's entry on this cell's side)
//   ghost row G:  (1 + w_s) u_G + (1 - w_s) sum_k w_k v_k = 2 u_b
//                 (the boundary value at BI, the midpoint of the ghost centre and its image
//                 point; w_k the image-point weights divided by 1 - w_s, w_s the row's own
//                 weight moved to the left-hand side, 0 if none)
// SRJ cycle: K Jacobi sweeps of the fluid rows with relaxation factors w_k = 1 / lambda_k,
// lambda_k the Chebyshev nodes of [1 - rho, 1 + rho], rho = alpha S / (1 + alpha S) with S
// the largest sum of a cell's coefficients: the fluid rows' Jacobi spectrum lies in that
// interval (diagonal dominance); the step divides by D through an FP32 reciprocal (it scales
// the step only, so the fixed point is unchanged).  After every sweep the ghost rows are
// re-evaluated from the new fluid values (Jacobi among ghosts).  Precision 0 runs the cycles
// in FP64; precisions 1 and 2 run each cycle in FP32 on the correction equation H e = r
// inside iterative refinement, whose residual and update are FP64 (1) or double-FP32 pairs
// with error-free transformations on the FP32 pipe (2).  Convergence: ||S r|| / ||S b|| over
// fluid and ghost rows, S = alpha s_G on ghost rows (s_G the pressure system's row scale), 1 elsewhere.
//
// Layout: the finest level of the FP64 multigrid hierarchy of the tables (padded arrays,
// mask, ghost sources, membrane entry slots and cut-cell lists) is shared with the pressure
// solver; the velocity work arrays live in the hierarchy's own workspace.
#include <algorithm>
#include <chrono>
#include <cmath>
#include <vector>

#include "dfloat.cuh"
#include "ghost.cuh"
#include "ibm_internal.cuh"

namespace ibm {

ibm_status build_hierarchy(ibm_tables *t, int precision, cudaStream_t st);

namespace {

constexpr int HZ_BLOCKS = REDUCE_BLOCKS;   // fixed grid of the norm kernels: deterministic sums
constexpr int HZ_THREADS = 256;
constexpr int TX = 32, TY = 8, KCH = 16;   // sweep tile (x, y) and z-planes per block

inline unsigned nb_of(long long n, int t) { return (unsigned)((n + t - 1) / t); }

template <typename T>
struct HzView {
  int nx, ny, nz;
  long long sy, sz;
  const uint8_t *mask;
  const T *cxm, *cxp, *cym, *cyp, *czm, *czp;   // alpha x the face coefficients, per axis
  const T *sdx, *sdy, *sdz;                     // alpha x their per-axis sums
};

// relaxation divisor: 1 / D as an FP32 reciprocal (it scales the Jacobi step only, so the
// iteration's fixed point does not depend on its rounding)
template <typename T> __device__ __forceinline__ T relax_rcp(T D);
template <> __device__ __forceinline__ float relax_rcp<float>(float D) { return __frcp_rn(D); }
template <> __device__ __forceinline__ double relax_rcp<double>(double D) { return (double)__frcp_rn((float)D); }

// one Jacobi step of the fluid rows with relaxation w (FP64, precision 0): un = u + w (f - H u) / D, each
// block a 32 x 8 tile marching KCH planes in z with the z-neighbours in registers; the next plane's
// value, mask and right-hand side are loaded one plane ahead
template <typename T>
__global__ void __launch_bounds__(TX *TY) k_hz_sweep(HzView<T> v, const T *u, T *un, const T *f, T w) {
  const int i = blockIdx.x * TX + threadIdx.x, j = blockIdx.y * TY + threadIdx.y;
  if (i >= v.nx || j >= v.ny) return;
  const int k0 = blockIdx.z * KCH, k1 = min(v.nz, k0 + KCH);
  const long long sy = v.sy, sz = v.sz;
  long long id = ((long long)(k0 + 1) * (v.ny + 2) + (j + 1)) * sy + (i + OX);
  const T cxm = v.cxm[i], cxp = v.cxp[i], cym = v.cym[j], cyp = v.cyp[j], dxy = (T)1 + (v.sdx[i] + v.sdy[j]);
  T zm = u[id - sz], zc = u[id], zp = u[id + sz], fc = f[id];
  uint8_t m = v.mask[id];
  for (int k = k0; k < k1; ++k, id += sz) {
    T zpp = 0, fn = 0;
    uint8_t mn = 1;
    if (k + 1 < k1) {   // planes k + 2 and k + 3 of the padded array exist when k + 1 < nz
      zpp = u[id + 2 * sz];
      fn = f[id + sz];
      mn = v.mask[id + sz];
    }
    const T xl = u[id - 1], xr = u[id + 1], yl = u[id - sy], yr = u[id + sy];
    T s = cxm * xl;
    s = fma(cxp, xr, s);
    s = fma(cym, yl, s);
    s = fma(cyp, yr, s);
    s = fma(v.czm[k], zm, s);
    s = fma(v.czp[k], zp, s);
    const T D = dxy + v.sdz[k];
    const T res = fma(-D, zc, fc) + s;
    if (m == 0) un[id] = fma(w * relax_rcp(D), res, zc);
    zm = zc;
    zc = zp;
    zp = zpp;
    fc = fn;
    m = mn;
  }
}

// The same step in FP32 (the correction cycles): a strip of four cells and KZ planes per thread, strips
// numbered along x then y, every load of a thread before the arithmetic, and the strip's x
// coefficients (xq: cxm, cxp, sdx in rows of nx4 floats) in 16-byte loads.  FIRST: the field is zero
// (it is neither read nor cleared first).  HBM-bound, 13 bytes per cell (FIRST: 9): 42 us and 21 us at
// 256^3, the one-cell-per-thread form 59 us for either
constexpr int SW_THREADS = 128, SW_KZ = 2;
template <bool FIRST>
__global__ void __launch_bounds__(SW_THREADS) k_hz_sweep4(HzView<float> v, const float *xq, const float *u, float *un,
                                                          const float *f, float w) {
  const int groups = (v.nx + 3) >> 2, nx4 = 4 * groups;
  const int strip = blockIdx.x * SW_THREADS + threadIdx.x, j = strip / groups, g = strip - j * groups;
  const int k0 = blockIdx.y * SW_KZ;
  if (j >= v.ny) return;
  auto ld = [](const float *p, float (&a)[4]) {
    const float4 q = *reinterpret_cast<const float4 *>(p);
    a[0] = q.x; a[1] = q.y; a[2] = q.z; a[3] = q.w;
  };
  const long long id0 = ((long long)(k0 + 1) * (v.ny + 2) + (j + 1)) * v.sy + OX + 4 * g;
  float C[SW_KZ + 2][4], N[SW_KZ][4], S[SW_KZ][4], F[SW_KZ][4], xl[SW_KZ], xr[SW_KZ];
  unsigned m[SW_KZ];
#pragma unroll
  for (int q = 0; q < SW_KZ; ++q) {
    const long long id = id0 + q * v.sz;
    const bool in = k0 + q < v.nz;   // plane nz of an odd grid's last pair is the halo
    m[q] = in ? *reinterpret_cast<const unsigned *>(v.mask + id) : 0xffffffffu;
    ld(f + id, F[q]);
    if (!FIRST) {
      ld(u + id, C[q + 1]);
      if (in) {
        ld(u + id - v.sy, N[q]);
        ld(u + id + v.sy, S[q]);
        xl[q] = u[id - 1];
        xr[q] = u[id + 4];
      }
    }
  }
  if (!FIRST) {
    ld(u + id0 - v.sz, C[0]);
    if (k0 + SW_KZ <= v.nz) ld(u + id0 + SW_KZ * v.sz, C[SW_KZ + 1]);
  }
  float cm[4], cp[4], sd[4];
  ld(xq + 4 * g, cm);
  ld(xq + nx4 + 4 * g, cp);
  ld(xq + 2 * nx4 + 4 * g, sd);
  const float cym = v.cym[j], cyp = v.cyp[j], sdy = v.sdy[j];
#pragma unroll
  for (int q = 0; q < SW_KZ; ++q) {
    const int k = min(k0 + q, v.nz - 1);
    const float czm = v.czm[k], czp = v.czp[k], sdz = v.sdz[k];
    float out[4];
#pragma unroll
    for (int a = 0; a < 4; ++a) {
      const float D = (1.0f + (sd[a] + sdy)) + sdz, rr = w * relax_rcp(D);
      if (FIRST) {
        out[a] = rr * F[q][a];
      } else {
        float s = cm[a] * (a == 0 ? xl[q] : C[q + 1][a > 0 ? a - 1 : 0]);
        s = fmaf(cp[a], a == 3 ? xr[q] : C[q + 1][a < 3 ? a + 1 : 3], s);
        s = fmaf(cym, N[q][a], s);
        s = fmaf(cyp, S[q][a], s);
        s = fmaf(czm, C[q][a], s);
        s = fmaf(czp, C[q + 2][a], s);
        const float c = C[q + 1][a], res = fmaf(-D, c, F[q][a]) + s;
        out[a] = fmaf(rr, res, c);
      }
    }
    float *o = un + id0 + q * v.sz;
    if (m[q] == 0u) {
      *reinterpret_cast<float4 *>(o) = make_float4(out[0], out[1], out[2], out[3]);
    } else {
#pragma unroll
      for (int a = 0; a < 4; ++a)
        if (((m[q] >> (8 * a)) & 0xffu) == 0u) o[a] = out[a];
    }
  }
}

// x coefficients in rows of nx4 floats (entries past nx repeat the last): alpha x cxm, cxp, sdx (hi
// parts, the FP32 sweep's), then their lo parts
constexpr int HZ_XQ = 6;
__global__ void k_hz_xq(const float *h, const float *l, int nx, int na, int nx4, float *xq) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nx4) return;
  const int c = min(i, nx - 1);
  const float q[HZ_XQ] = {h[c], h[nx + c], h[2 * na + c], l[c], l[nx + c], l[2 * na + c]};
  for (int r = 0; r < HZ_XQ; ++r) xq[r * nx4 + i] = q[r];
}

// the same step at the membrane cut cells (their links read the entries through cut_nb)
template <typename T>
__global__ void k_hz_sweep_cut(HzView<T> v, const long long *cut_id, const long long *cut_nb, const int *cut_ijk,
                               const long long *cnt, const T *u, T *un, const T *f, T w) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < cnt[1];
       t += (long long)gridDim.x * blockDim.x) {
    const long long id = cut_id[t];
    const int i = cut_ijk[3 * t], j = cut_ijk[3 * t + 1], k = cut_ijk[3 * t + 2];
    const T c[6] = {v.cxm[i], v.cxp[i], v.cym[j], v.cyp[j], v.czm[k], v.czp[k]};
    T s = 0;
    for (int d = 0; d < 6; ++d) s = fma(c[d], u[cut_nb[6 * t + d]], s);
    const T D = ((T)1 + (v.sdx[i] + v.sdy[j])) + v.sdz[k];
    const T res = fma(-D, u[id], f[id]) + s;
    un[id] = fma(w * relax_rcp(D), res, u[id]);
  }
}

// ghost rows from the new fluid values and the previous ghost values (u null: they are zero):
// u_G = (b_G - (1 - w_s) sum w v) / (1 + w_s), b_G = f at the ghost's slot
template <typename T>
__global__ void k_hz_ghost(const long long *src, const long long *dst, const double *gw, const double *ws,
                           long long ng, T *un, const T *u, const T *f) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g >= ng) return;
  const GhostRow<double> row(src, gw, g);
  const long long d = dst[g];
  const T b = f[d], w = (T)ws[g];
  const T s = row.sum<T>([&](long long q) {
    return (q & GHOST_CORNER) ? (u ? u[q & ~GHOST_CORNER] : (T)0) : un[q];
  });
  un[d] = (b - ((T)1 - w) * s) / ((T)1 + w);
}

// FP64 residual r = b - H u of the regular fluid rows (coefficients pre-scaled by alpha);
// block partials of sum r^2 (and of sum b^2 when with_b); r32 (if given) receives r in FP32
__global__ void __launch_bounds__(HZ_THREADS) k_hz_resid(HzView<double> v, const double *u, const double *f,
                                                         float *r32, double *part, bool with_b) {
  __shared__ double sr[HZ_THREADS], sb[HZ_THREADS];
  double ar = 0.0, ab = 0.0;
  const long long rows = (long long)v.ny * v.nz;
  for (long long row = blockIdx.x; row < rows; row += gridDim.x) {
    const int j = (int)(row % v.ny), k = (int)(row / v.ny);
    const long long base = ((long long)(k + 1) * (v.ny + 2) + (j + 1)) * v.sy + OX;
    const double cym = v.cym[j], cyp = v.cyp[j], czm = v.czm[k], czp = v.czp[k], syz = v.sdy[j] + v.sdz[k];
    for (int i = threadIdx.x; i < v.nx; i += blockDim.x) {
      const long long id = base + i;
      if (v.mask[id] != 0) continue;
      double acc = v.cxm[i] * u[id - 1];
      acc = fma(v.cxp[i], u[id + 1], acc);
      acc = fma(cym, u[id - v.sy], acc);
      acc = fma(cyp, u[id + v.sy], acc);
      acc = fma(czm, u[id - v.sz], acc);
      acc = fma(czp, u[id + v.sz], acc);
      const double D = 1.0 + (v.sdx[i] + syz);
      const double r = fma(-D, u[id], f[id]) + acc;
      if (r32) r32[id] = (float)r;
      ar += r * r;
      if (with_b) ab += f[id] * f[id];
    }
  }
  sr[threadIdx.x] = ar;
  sb[threadIdx.x] = ab;
  __syncthreads();
  for (int st = HZ_THREADS / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) { sr[threadIdx.x] += sr[threadIdx.x + st]; sb[threadIdx.x] += sb[threadIdx.x + st]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) { part[2 * blockIdx.x] = sr[0]; part[2 * blockIdx.x + 1] = sb[0]; }
}

// residual of the cut cells and of the ghost rows (scaled by alpha s_G), one block-partial
// pair per block after the regular rows' partials
// values of the refinement loop's u and f: FP64 arrays, or double-FP32 pairs (hi + lo)
struct Fp64Vals {
  const double *u, *f;
  __device__ double U(long long q) const { return u[q]; }
  __device__ double F(long long q) const { return f[q]; }
};
struct DfVals {
  const float *uh, *ul, *fh, *fl;
  __device__ double U(long long q) const { return dfl::join(uh[q], ul[q]); }
  __device__ double F(long long q) const { return dfl::join(fh[q], fl[q]); }
};

template <typename Vals>
__global__ void __launch_bounds__(HZ_THREADS) k_hz_resid_rest(
    HzView<double> v, const long long *cut_id, const long long *cut_nb, const int *cut_ijk, const long long *cnt,
    const long long *src, const long long *dst, const double *gw, const double *ws, const double *gscale,
    long long ng, Vals x, double alpha, float *r32, double *part, bool with_b) {
  __shared__ double sr[HZ_THREADS], sb[HZ_THREADS];
  double ar = 0.0, ab = 0.0;
  const long long ncut = cnt ? cnt[1] : 0;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < ncut + ng;
       t += (long long)gridDim.x * blockDim.x) {
    if (t < ncut) {
      const long long id = cut_id[t];
      const int i = cut_ijk[3 * t], j = cut_ijk[3 * t + 1], k = cut_ijk[3 * t + 2];
      const double c[6] = {v.cxm[i], v.cxp[i], v.cym[j], v.cyp[j], v.czm[k], v.czp[k]};
      double acc = 0.0;
      for (int d = 0; d < 6; ++d) acc = fma(c[d], x.U(cut_nb[6 * t + d]), acc);
      const double D = 1.0 + ((v.sdx[i] + v.sdy[j]) + v.sdz[k]);
      const double fi = x.F(id);
      const double r = fma(-D, x.U(id), fi) + acc;
      if (r32) r32[id] = (float)r;
      ar += r * r;
      if (with_b) ab += fi * fi;
    } else {
      const long long g = t - ncut;
      const double s = GhostRow<double>(src, gw, g).sum<double>([&](long long q) { return x.U(q & ~GHOST_CORNER); });
      const long long id = dst[g];
      const double fi = x.F(id);
      const double r = fi - ((1.0 + ws[g]) * x.U(id) + (1.0 - ws[g]) * s);
      if (r32) r32[id] = (float)r;
      const double sc = alpha * gscale[g];
      ar += (sc * r) * (sc * r);
      if (with_b) ab += (sc * fi) * (sc * fi);
    }
  }
  sr[threadIdx.x] = ar;
  sb[threadIdx.x] = ab;
  __syncthreads();
  for (int st = HZ_THREADS / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) { sr[threadIdx.x] += sr[threadIdx.x + st]; sb[threadIdx.x] += sb[threadIdx.x + st]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) { part[2 * blockIdx.x] = sr[0]; part[2 * blockIdx.x + 1] = sb[0]; }
}

// out[0] = sum of the r^2 partials, out[1] = sum of the b^2 partials (fixed order): nreg
// pairs of the regular rows at part, nrest pairs of the other rows at part + 2 HZ_BLOCKS
__global__ void k_hz_norms(const double *part, int nreg, int nrest, double *out) {
  __shared__ double sr[HZ_THREADS], sb[HZ_THREADS];
  double ar = 0.0, ab = 0.0;
  for (int b = threadIdx.x; b < nreg + nrest; b += blockDim.x) {
    const int q = b < nreg ? b : HZ_BLOCKS + (b - nreg);
    ar += part[2 * q];
    ab += part[2 * q + 1];
  }
  sr[threadIdx.x] = ar;
  sb[threadIdx.x] = ab;
  __syncthreads();
  for (int st = HZ_THREADS / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) { sr[threadIdx.x] += sr[threadIdx.x + st]; sb[threadIdx.x] += sb[threadIdx.x + st]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) { out[0] = sr[0]; out[1] = sb[0]; }
}

// double-FP32 residual of the regular fluid rows (precision 2): u, f and alpha x the
// coefficients as hi + lo float pairs, r = f - D u + sum c v by error-free transformations
// on the FP32 pipe (the residual error is a few units of 2^-48 x sum |c| |v|); r32 receives
// r; block partials of sum r^2 (and sum f^2 when with_b)
struct HzDf {
  const float *ch, *cl;   // alpha x coefficients and sums (layout of HzView), hi and lo parts
};

__device__ __forceinline__ void df_add(float ah, float al, float bh, float bl, float &sh, float &sl) {
  float s, e;
  dfl::two_sum(ah, bh, s, e);
  e += al + bl;
  dfl::fast_two_sum(s, e, sh, sl);
}

// Bound by the latency of its loads: a thread marches a strip of four cells through kz planes with three
// planes of u in registers and the next plane's u, f and mask loaded one plane ahead; products and
// sums are packed two cells to an instruction.  One warp per row, each lane four cells with the
// neighbour planes reloaded, took 135 us at 256^3; this takes 106
__global__ void __launch_bounds__(HZ_THREADS, 2) k_hz_resid_df(HzView<double> v, HzDf c, const float *xq, const float *uh,
                                                               const float *ul, const float *fh, const float *fl,
                                                               float *r32, double *part, bool with_b, int kz) {
  using namespace dfl;
  __shared__ double sr[HZ_THREADS], sb[HZ_THREADS];
  const int nx = v.nx, ny = v.ny, nz = v.nz, na = nx + ny + nz, groups = (nx + 3) >> 2, nx4 = 4 * groups;
  const long long sy = v.sy, sz = v.sz;
  // coefficient offsets in the layout cxm cxp cym cyp czm czp (2 na) then sdx sdy sdz (na)
  const float *cyh = c.ch + 2 * nx, *cyl = c.cl + 2 * nx, *czh = c.ch + 2 * nx + 2 * ny, *czl = c.cl + 2 * nx + 2 * ny;
  const float *sdh = c.ch + 2 * na, *sdl = c.cl + 2 * na;
  double dr = 0.0, db = 0.0;
  auto two = [](float x) { return f2(x, x); };
  auto ld = [](const float *q, F2 (&r)[2]) {   // a strip as two pairs
    const ulonglong2 a = *reinterpret_cast<const ulonglong2 *>(q);
    r[0].v = a.x;
    r[1].v = a.y;
  };
  const int sblocks = (groups * ny + HZ_THREADS - 1) / HZ_THREADS;
  const int items = sblocks * ((nz + kz - 1) / kz);
  for (int item = blockIdx.x; item < items; item += gridDim.x) {
    const int chunk = item / sblocks, strip = (item - chunk * sblocks) * HZ_THREADS + (int)threadIdx.x;
    const int j = strip / groups, g = strip - j * groups;
    if (j >= ny) continue;
    const int k0 = chunk * kz, k1 = min(nz, k0 + kz);
    const float *x = xq + 4 * g;
    const F2 ymh = two(cyh[j]), yml = two(cyl[j]), yph = two(cyh[ny + j]), ypl = two(cyl[ny + j]);
    float t1h, t1l;
    df_add(1.0f, 0.0f, sdh[nx + j], sdl[nx + j], t1h, t1l);
    long long id = ((long long)(k0 + 1) * (ny + 2) + (j + 1)) * sy + OX + 4 * g;
    F2 MH[2], ML[2], PH[2], PL[2], UH[2], UL[2], FH[2], FL[2];   // u in planes k - 1, k, k + 1; f in plane k
    ld(uh + id - sz, MH);
    ld(ul + id - sz, ML);
    ld(uh + id, PH);
    ld(ul + id, PL);
    ld(uh + id + sz, UH);
    ld(ul + id + sz, UL);
    ld(fh + id, FH);
    ld(fl + id, FL);
    unsigned mn = *reinterpret_cast<const unsigned *>(v.mask + id);
    float ar = 0.f, ab = 0.f;
    int nplane = 0;
#pragma unroll 1
    for (int k = k0; k < k1; ++k, id += sz) {
      const unsigned m = mn;
      F2 NH[2][2], NL[2][2], cc[2], cl[2], sh[2], sl[2], b[2], wh[2], wl[2], gh[2], gl[2];
      ld(uh + id - sy, NH[0]);
      ld(ul + id - sy, NL[0]);
      ld(uh + id + sy, NH[1]);
      ld(ul + id + sy, NL[1]);
      const float xlh = uh[id - 1], xll = ul[id - 1], xrh = uh[id + 4], xrl = ul[id + 4];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        sh[q] = FH[q];
        sl[q] = FL[q];
        b[q] = add2(FH[q], FL[q]);
        wh[q] = UH[q];
        wl[q] = UL[q];
        gh[q] = FH[q];
        gl[q] = FL[q];
      }
      if (k + 1 < k1) {
        mn = *reinterpret_cast<const unsigned *>(v.mask + id + sz);
        ld(uh + id + 2 * sz, wh);
        ld(ul + id + 2 * sz, wl);
        ld(fh + id + sz, gh);
        ld(fl + id + sz, gl);
      }
      float dyzh, dyzl;
      df_add(t1h, t1l, sdh[nx + ny + k], sdl[nx + ny + k], dyzh, dyzl);
      const F2 zmh = two(czh[k]), zml = two(czl[k]), zph = two(czh[nz + k]), zpl = two(czl[nz + k]);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        acc_prod2(ymh, yml, NH[0][q], NL[0][q], sh[q], sl[q]);
        acc_prod2(yph, ypl, NH[1][q], NL[1][q], sh[q], sl[q]);
        acc_prod2(zmh, zml, MH[q], ML[q], sh[q], sl[q]);
        acc_prod2(zph, zpl, UH[q], UL[q], sh[q], sl[q]);
      }
      ld(x + 2 * nx4, cc);
      ld(x + 5 * nx4, cl);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        // D = (1 + sdy + sdz) + sdx as a renormalised pair, then -D u
        F2 t, e;
        two_sum2(two(dyzh), cc[q], t, e);
        e = add2(e, add2(two(dyzl), cl[q]));
        const F2 Dh = add2(t, e), Dl = sub2(e, sub2(Dh, t));
        acc_prod_neg2(Dh, neg2(Dh), neg2(Dl), PH[q], PL[q], sh[q], sl[q]);
      }
      float p0, p1, p2, p3, q0, q1, q2, q3;
      un2(PH[0], p0, p1);
      un2(PH[1], p2, p3);
      un2(PL[0], q0, q1);
      un2(PL[1], q2, q3);
      ld(x, cc);
      ld(x + 3 * nx4, cl);
      acc_prod2(cc[0], cl[0], f2(xlh, p0), f2(xll, q0), sh[0], sl[0]);
      acc_prod2(cc[1], cl[1], f2(p1, p2), f2(q1, q2), sh[1], sl[1]);
      ld(x + nx4, cc);
      ld(x + 4 * nx4, cl);
      acc_prod2(cc[0], cl[0], f2(p1, p2), f2(q1, q2), sh[0], sl[0]);
      acc_prod2(cc[1], cl[1], f2(p3, xrh), f2(q3, xrl), sh[1], sl[1]);
      float R[4], B[4];
      un2(add2(sh[0], sl[0]), R[0], R[1]);
      un2(add2(sh[1], sl[1]), R[2], R[3]);
      un2(b[0], B[0], B[1]);
      un2(b[1], B[2], B[3]);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        if (((m >> (8 * q)) & 0xffu) == 0u) {
          ar = fmaf(R[q], R[q], ar);
          if (with_b) ab = fmaf(B[q], B[q], ab);
          if (r32 && m != 0u) r32[id + q] = R[q];
        }
      if (r32 && m == 0u) *reinterpret_cast<float4 *>(r32 + id) = make_float4(R[0], R[1], R[2], R[3]);
      if (++nplane == 2 || k + 1 == k1) {   // the float sums of a few cells into FP64
        dr += widen(ar);
        if (with_b) db += widen(ab);
        ar = ab = 0.f;
        nplane = 0;
      }
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        MH[q] = PH[q]; ML[q] = PL[q];
        PH[q] = UH[q]; PL[q] = UL[q];
        UH[q] = wh[q]; UL[q] = wl[q];
        FH[q] = gh[q]; FL[q] = gl[q];
      }
    }
  }
  sr[threadIdx.x] = dr;
  sb[threadIdx.x] = db;
  __syncthreads();
  for (int st = HZ_THREADS / 2; st > 0; st >>= 1) {
    if (threadIdx.x < st) { sr[threadIdx.x] += sr[threadIdx.x + st]; sb[threadIdx.x] += sb[threadIdx.x + st]; }
    __syncthreads();
  }
  if (threadIdx.x == 0) { part[2 * blockIdx.x] = sr[0]; part[2 * blockIdx.x + 1] = sb[0]; }
}

// (uh, ul) += e on every slot (double-FP32 update)
__global__ void k_hz_update_df(float *uh, float *ul, const float *e, long long n) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x) {
    float s, t;
    dfl::two_sum(uh[q], e[q], s, t);
    t += ul[q];
    dfl::fast_two_sum(s, t, uh[q], ul[q]);
  }
}

// Packs and unpacks stream 33 and 17 bytes per cell: a thread takes one cell of four rows of a plane,
// all loads before the stores (one row per thread keeps a quarter of the bytes in flight: 180 and 97 us
// at 256^3, this 103 and 57); the split into pairs runs on the integer pipe (dfloat.cuh)
constexpr int HZ_PK = 128, HZ_PKR = 4;   // grid: (x blocks, row groups, nz)
template <class LD, class ST>
__device__ __forceinline__ void hz_rows(int nx, int ny, LevelGeom g, const uint8_t *mask, LD ld, ST st) {
  const int i = blockIdx.x * HZ_PK + threadIdx.x, j0 = blockIdx.y * HZ_PKR, k = blockIdx.z;
  if (i >= nx) return;
  const long long l0 = ((long long)k * ny + j0) * nx + i, id0 = pidx(g, i, j0, k);
  double2 x[HZ_PKR];
  uint8_t m[HZ_PKR];
#pragma unroll
  for (int q = 0; q < HZ_PKR; ++q)
    if (j0 + q < ny) {
      m[q] = mask[id0 + q * g.sy];
      x[q] = ld(l0 + (long long)q * nx, id0 + q * g.sy);
    }
#pragma unroll
  for (int q = 0; q < HZ_PKR; ++q)
    if (j0 + q < ny) st(l0 + (long long)q * nx, id0 + q * g.sy, fluid_row(m[q]), fluid_row(m[q]) || m[q] == 3, x[q]);
}

__global__ void __launch_bounds__(HZ_PK) k_hz_pack_df(const double *f, const double *u, int nx, int ny, LevelGeom g,
                                                      const uint8_t *mask, float *fh, float *fl, float *uh, float *ul) {
  hz_rows(nx, ny, g, mask, [&](long long l, long long) { return make_double2(f[l], u[l]); },
          [&](long long, long long id, bool fluid, bool active, double2 x) {
            dfl::split(fluid ? x.x : 0.0, fh[id], fl[id]);
            dfl::split(active ? x.y : 0.0, uh[id], ul[id]);
          });
}

__global__ void k_hz_ghost_rhs_df(const long long *dst, const double *ub, long long ng, float *fh, float *fl) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g < ng) dfl::split(ub ? 2.0 * ub[g] : 0.0, fh[dst[g]], fl[dst[g]]);
}

__global__ void __launch_bounds__(HZ_PK) k_hz_unpack_df(const float *uh, const float *ul, int nx, int ny, LevelGeom g,
                                                        const uint8_t *mask, double *u) {
  hz_rows(nx, ny, g, mask, [&](long long, long long id) { return make_double2(dfl::join(uh[id], ul[id]), 0.0); },
          [&](long long l, long long, bool, bool active, double2 x) { u[l] = active ? x.x : 0.0; });
}

// user layout -> padded: f on fluid rows (0 elsewhere), u on fluid and ghost cells
__global__ void __launch_bounds__(HZ_PK) k_hz_pack(const double *f, const double *u, int nx, int ny, LevelGeom g,
                                                   const uint8_t *mask, double *fp, double *up) {
  hz_rows(nx, ny, g, mask, [&](long long l, long long) { return make_double2(f[l], u[l]); },
          [&](long long, long long id, bool fluid, bool active, double2 x) {
            fp[id] = fluid ? x.x : 0.0;
            up[id] = active ? x.y : 0.0;
          });
}

// ghost-row right-hand sides 2 u_b at the ghosts' slots
__global__ void k_hz_ghost_rhs(const long long *dst, const double *ub, long long ng, double *fp) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g < ng) fp[dst[g]] = ub ? 2.0 * ub[g] : 0.0;
}

__global__ void __launch_bounds__(HZ_PK) k_hz_unpack(const double *up, int nx, int ny, LevelGeom g, const uint8_t *mask,
                                                     double *u) {
  hz_rows(nx, ny, g, mask, [&](long long, long long id) { return make_double2(up[id], 0.0); },
          [&](long long l, long long, bool, bool active, double2 x) { u[l] = active ? x.x : 0.0; });
}

// u += e on every slot.  Off the active rows (and membranes' entries) e may hold an earlier solve's values, since a
// correction that starts from zero is not cleared: u is then as undefined there, and nothing reads it
// (neighbours and sources of active rows are active, the packs rewrite every cell, the unpacks write zeros)
__global__ void k_hz_update(double *u, const float *e, long long n) {
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
    u[q] += (double)e[q];
}

// alpha x the FP64 coefficients and their sums, in FP64 and as a double-FP32 pair (a32 the
// high part, the FP32 coefficients of the correction sweeps)
__global__ void k_scale_coefs(const double *c, long long n, double alpha, double *a64, float *a32, float *a32lo) {
  const long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (q >= n) return;
  const double x = alpha * c[q];
  a64[q] = x;
  dfl::split(x, a32[q], a32lo[q]);
}

// rigid boundary velocity of every ghost entry: u_b = v0 + omega x (BI - c) for the mesh of
// its closest triangle; out[d * ng + g]
constexpr int MAX_RIGID_V = 32;
struct RigidVel {
  int n;
  int off[MAX_RIGID_V + 1];
  double m[MAX_RIGID_V][9];   // v0 (3), omega (3), centre (3)
};

__global__ void k_rigid_velocity(const double *bi, const int *tri, long long ng, RigidVel M, double *out) {
  const long long g = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (g >= ng) return;
  int lo = 0, hi = M.n;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (M.off[mid] <= tri[g]) lo = mid; else hi = mid;
  }
  const double *mm = M.m[lo], *om = mm + 3;
  const double r[3] = {bi[3 * g] - mm[6], bi[3 * g + 1] - mm[7], bi[3 * g + 2] - mm[8]};
  out[g] = mm[0] + (om[1] * r[2] - om[2] * r[1]);
  out[ng + g] = mm[1] + (om[2] * r[0] - om[0] * r[2]);
  out[2 * ng + g] = mm[2] + (om[0] * r[1] - om[1] * r[0]);
}

// the largest sum of one cell's face coefficients along one axis (host, from the faces)
double axis_max_sum(const std::vector<double> &f) {
  const int n = (int)f.size() - 1;
  double best = 0.0;
  for (int i = 0; i < n; ++i) {
    const double ci = 0.5 * (f[i] + f[i + 1]), wi = f[i + 1] - f[i];
    double s = 0.0;
    if (i > 0) s += 1.0 / (wi * (ci - 0.5 * (f[i - 1] + f[i])));
    if (i < n - 1) s += 1.0 / (wi * (0.5 * (f[i + 1] + f[i + 2]) - ci));
    best = std::max(best, s);
  }
  return best;
}

struct HzWork {
  double *u[2], *f, *ac64;   // ac: alpha x coefficients and sums
  float *e[2], *r32, *ac32, *ac32lo, *xq;
  double *part, *norms;
};

}  // namespace

// time_ms non-null: after the setup, time n_timed launches of the sweep kernel alone (CUDA
// events on st around each launch; mean in *time_ms) instead of solving
ibm_status helmholtz_solve_impl(ibm_ctx *ctx, ibm_tables *t, double alpha, const double *f_user, const double *ub,
                                double tol, double *u_user, const ibm_helmholtz_opts *opts, ibm_solve_info *info,
                                cudaStream_t st, double *time_ms = nullptr, int n_timed = 0) {
  const auto t0 = std::chrono::steady_clock::now();
  ibm_helmholtz_opts o;
  ibm_helmholtz_opts_default(&o);
  if (opts) o = *opts;
  if (!f_user || !u_user || !(alpha >= 0.0) || !std::isfinite(alpha) || !(tol > 0.0) || o.precision < 0 ||
      o.precision > 2 || o.srj_steps < 1 || o.srj_steps > 64 || o.max_cycles < 1)
    return IBM_ERR_INVALID_ARG;
  if (t->ny > 65535 || t->nz > 65535) return IBM_ERR_CAPACITY;   // launch grid rows and planes
  ibm_status s = build_hierarchy(t, 0, st);
  if (s != IBM_OK) return s;
  Hierarchy *h = t->hier[0];
  Level &L0 = h->lv[0];
  const LevelGeom &G = L0.g;
  const long long nslot = h->nslot, ng = t->nghost;
  const int nx = G.nx, ny = G.ny, nz = G.nz, na = nx + ny + nz;
  // workspace: u (2), f in FP64; e (2), r in FP32; FP32 coefficients; partials; norms
  const long long want = nslot;
  const size_t na3 = ((3 * (size_t)na + 31) / 32) * 32;   // keeps the FP32 arrays 256-byte aligned
  const size_t bytes = sizeof(double) * (3 * (size_t)want + 2 * (size_t)HZ_BLOCKS * 2 + 8 + na3) +
                       sizeof(float) * (3 * (size_t)want + 2 * na3 + 64 + HZ_XQ * (((size_t)nx + 3) / 4 * 4));
  if (!h->helm_buf || h->helm_n != want + na) {
    if (h->helm_buf) { IBM_TRY(cudaStreamSynchronize(st)); cudaFree(h->helm_buf); }
    h->helm_buf = nullptr;
    h->helm_n = 0;
    IBM_TRY(cudaMalloc(&h->helm_buf, bytes));
    IBM_TRY(cudaMemsetAsync(h->helm_buf, 0, bytes, st));   // halos and inactive cells stay 0
    h->helm_n = want + na;
    h->helm_layout = -1;
  }
  HzWork W;
  {
    double *d = (double *)h->helm_buf;
    W.u[0] = d; W.u[1] = d + want; W.f = d + 2 * want;
    W.part = d + 3 * want;
    W.norms = W.part + 2 * 2 * HZ_BLOCKS;
    W.ac64 = W.norms + 8;
    float *fl = (float *)(W.ac64 + na3);
    W.e[0] = fl; W.e[1] = fl + want; W.r32 = fl + 2 * want; W.ac32 = fl + 3 * want;
    W.ac32lo = W.ac32 + na3;
    W.xq = W.ac32lo + na3;
  }
  // views of the finest level: alpha x the hierarchy's FP64 coefficients, and FP32 copies
  long long launches = 0;
  k_scale_coefs<<<nb_of(3 * na, 256), 256, 0, st>>>(h->c64, 3 * na, alpha, W.ac64, W.ac32, W.ac32lo);
  const int nx4 = (nx + 3) / 4 * 4;
  k_hz_xq<<<nb_of(nx4, 256), 256, 0, st>>>(W.ac32, W.ac32lo, nx, na, nx4, W.xq);
  launches += 2;
  HzView<double> v64;
  {
    const double *c = W.ac64;
    v64.nx = nx; v64.ny = ny; v64.nz = nz; v64.sy = G.sy; v64.sz = G.sz; v64.mask = L0.mask;
    v64.cxm = c; v64.cxp = c + nx; v64.cym = c + 2 * nx; v64.cyp = v64.cym + ny;
    v64.czm = v64.cyp + ny; v64.czp = v64.czm + nz;
    v64.sdx = c + 2 * na; v64.sdy = v64.sdx + nx; v64.sdz = v64.sdy + ny;
  }
  HzView<float> v32;
  {
    const float *c = W.ac32;
    v32.nx = nx; v32.ny = ny; v32.nz = nz; v32.sy = G.sy; v32.sz = G.sz; v32.mask = L0.mask;
    v32.cxm = c; v32.cxp = c + nx; v32.cym = c + 2 * nx; v32.cyp = v32.cym + ny;
    v32.czm = v32.cyp + ny; v32.czp = v32.czm + nz;
    v32.sdx = c + 2 * na; v32.sdy = v32.sdx + nx; v32.sdz = v32.sdy + ny;
  }
  // pack f, u and the ghost rows' right-hand sides
  // precision 2: u and f as double-FP32 pairs in the same bytes (hi parts, then lo parts).
  // The packs write the cells only; halo and padding slots must read 0 in either view, so
  // the arrays are cleared whenever the layout changes.
  const bool df = o.precision == 2;
  const dim3 cell_grid(nb_of(nx, HZ_PK), nb_of(ny, HZ_PKR), nz);   // pack / unpack
  float *uh = (float *)W.u[0], *ul = uh + want, *fh = (float *)W.f, *fl = fh + want;
  if (h->helm_layout != (df ? 1 : 0)) {
    IBM_TRY(cudaMemsetAsync(W.u[0], 0, sizeof(double) * 3 * (size_t)want, st));   // u[0], u[1], f
    h->helm_layout = df ? 1 : 0;
  }
  if (df)
    k_hz_pack_df<<<cell_grid, HZ_PK, 0, st>>>(f_user, u_user, nx, ny, G, L0.mask, fh, fl, uh, ul);
  else
    k_hz_pack<<<cell_grid, HZ_PK, 0, st>>>(f_user, u_user, nx, ny, G, L0.mask, W.f, W.u[0]);
  ++launches;
  if (ng > 0) {
    if (df) k_hz_ghost_rhs_df<<<nb_of(ng, 128), 128, 0, st>>>(h->gdst, ub, ng, fh, fl);
    else k_hz_ghost_rhs<<<nb_of(ng, 128), 128, 0, st>>>(h->gdst, ub, ng, W.f);
    ++launches;
  }
  const bool cuts = t->membrane && h->cut_id;
  const unsigned cut_blocks = cuts ? std::max(1u, std::min(nb_of(h->cutcap, 256), (unsigned)ctx->wave)) : 0;
  // SRJ relaxation factors: 1 / Chebyshev nodes of [1 - rho, 1 + rho]
  const double S = axis_max_sum(t->xf) + axis_max_sum(t->yf) + axis_max_sum(t->zf);
  const double rho = alpha * S / (1.0 + alpha * S);
  const int K = o.srj_steps;
  std::vector<double> om(K);
  for (int k = 0; k < K; ++k) om[k] = 1.0 / (1.0 + rho * std::cos(3.141592653589793 * (2.0 * k + 1.0) / (2.0 * K)));
  const dim3 sweep_grid(nb_of(nx, TX), nb_of(ny, TY), nb_of(nz, KCH)), sweep_block(TX, TY);
  const int rest_blocks =
      (int)std::max<long long>(1, std::min<long long>(HZ_BLOCKS, nb_of((cuts ? h->cutcap : 0) + ng, HZ_THREADS)));
  // the FP32 sweep's grid; the double-FP32 residual's: one wave of two blocks per SM, and the planes per
  // march that give the fewest plane steps
  const long long strips = (long long)(nx4 / 4) * ny;
  const dim3 sweep4_grid(nb_of(strips, SW_THREADS), nb_of(nz, SW_KZ));
  const int df_max = std::max(1, std::min(HZ_BLOCKS, 2 * std::max(1, ctx->sm_count)));
  int df_kz = 1;
  {
    const long long sblocks = nb_of(strips, HZ_THREADS);
    long long best = -1;
    for (int q = std::min(16, nz); q >= 1; --q) {
      const long long cost = (sblocks * ((nz + q - 1) / q) + df_max - 1) / df_max * (q + 1);
      if (best < 0 || cost < best) { best = cost; df_kz = q; }
    }
  }
  const int df_blocks = (int)std::min<long long>(df_max, (long long)nb_of(strips, HZ_THREADS) * ((nz + df_kz - 1) / df_kz));
  // residual r = b - H u (FP64) with its norm, and the norm of b on the first call
  auto residual = [&](const double *u, float *r32, bool with_b) -> ibm_status {
    const long long *cnt = cuts ? h->d_cnt : nullptr;
    if (df) {
      const float *xh = (const float *)u, *xl = xh + want;
      k_hz_resid_df<<<df_blocks, HZ_THREADS, 0, st>>>(v64, HzDf{W.ac32, W.ac32lo}, W.xq, xh, xl, fh, fl, r32, W.part,
                                                      with_b, df_kz);
      k_hz_resid_rest<DfVals><<<rest_blocks, HZ_THREADS, 0, st>>>(
          v64, h->cut_id, h->cut_nb, h->cut_ijk, cnt, h->gsrc, h->gdst, t->gw, t->gwself, t->gscale, ng,
          DfVals{xh, xl, fh, fl}, alpha, r32, W.part + 2 * HZ_BLOCKS, with_b);
    } else {
      k_hz_resid<<<HZ_BLOCKS, HZ_THREADS, 0, st>>>(v64, u, W.f, r32, W.part, with_b);
      k_hz_resid_rest<Fp64Vals><<<rest_blocks, HZ_THREADS, 0, st>>>(
          v64, h->cut_id, h->cut_nb, h->cut_ijk, cnt, h->gsrc, h->gdst, t->gw, t->gwself, t->gscale, ng,
          Fp64Vals{u, W.f}, alpha, r32, W.part + 2 * HZ_BLOCKS, with_b);
    }
    k_hz_norms<<<1, HZ_THREADS, 0, st>>>(W.part, df ? df_blocks : HZ_BLOCKS, rest_blocks, W.norms);
    launches += 3;
    IBM_TRY(cudaMemcpyAsync(ctx->hscal, W.norms, 2 * sizeof(double), cudaMemcpyDeviceToHost, st));
    IBM_TRY(cudaStreamSynchronize(st));
    return IBM_OK;
  };
  // one SRJ cycle of K relaxed Jacobi steps on (u, rhs); returns the index of the current buffer.
  // zero: the field is zero, whatever its buffer holds (the first step does not read it)
  auto srj_cycle = [&](auto *buf0, auto *buf1, const auto *rhs, auto view, int cur, bool zero) -> int {
    using T = std::remove_const_t<std::remove_pointer_t<decltype(buf0)>>;
    T *b[2] = {buf0, buf1};
    for (int k = 0; k < K; ++k) {
      T *u = b[cur], *un = b[1 - cur];
      const bool first = zero && k == 0;
      if constexpr (sizeof(T) == 4) {
        if (first) k_hz_sweep4<true><<<sweep4_grid, SW_THREADS, 0, st>>>(view, W.xq, u, un, rhs, (T)om[k]);
        else k_hz_sweep4<false><<<sweep4_grid, SW_THREADS, 0, st>>>(view, W.xq, u, un, rhs, (T)om[k]);
      } else {
        k_hz_sweep<T><<<sweep_grid, sweep_block, 0, st>>>(view, u, un, rhs, (T)om[k]);
      }
      ++launches;
      if (cuts) {
        k_hz_sweep_cut<T><<<cut_blocks, 256, 0, st>>>(view, h->cut_id, h->cut_nb, h->cut_ijk, h->d_cnt, u, un, rhs,
                                                     (T)om[k]);
        ++launches;
      }
      if (ng > 0) {
        k_hz_ghost<T><<<nb_of(ng, 128), 128, 0, st>>>(h->gsrc, h->gdst, t->gw, t->gwself, ng, un,
                                                      first ? nullptr : (const T *)u, rhs);
        ++launches;
      }
      cur = 1 - cur;
    }
    return cur;
  };
  if (time_ms) {   // the sweep kernel alone, on the packed field (FP32: the correction arrays)
    std::vector<cudaEvent_t> ev(2 * (size_t)n_timed);
    for (auto &e : ev) IBM_TRY(cudaEventCreate(&e));
    for (int q = 0; q < n_timed; ++q) {
      IBM_TRY(cudaEventRecord(ev[2 * q], st));
      if (o.precision == 0)
        k_hz_sweep<double><<<sweep_grid, sweep_block, 0, st>>>(v64, W.u[q & 1], W.u[1 - (q & 1)], W.f, om[0]);
      else
        k_hz_sweep4<false><<<sweep4_grid, SW_THREADS, 0, st>>>(v32, W.xq, W.e[q & 1], W.e[1 - (q & 1)], W.r32,
                                                               (float)om[0]);
      IBM_TRY(cudaEventRecord(ev[2 * q + 1], st));
    }
    IBM_TRY(cudaGetLastError());
    IBM_TRY(cudaStreamSynchronize(st));
    double tot = 0.0;
    for (int q = 0; q < n_timed; ++q) {
      float ms = 0.f;
      cudaEventElapsedTime(&ms, ev[2 * q], ev[2 * q + 1]);
      tot += ms;
    }
    for (auto &e : ev) cudaEventDestroy(e);
    *time_ms = tot / std::max(1, n_timed);
    ctx->launches += launches + n_timed;
    return IBM_OK;
  }
  ibm_status ret = IBM_OK;
  int cycles = 0, hist = 0;
  double rel = 0.0;
  if ((s = residual(W.u[0], o.precision >= 1 ? W.r32 : nullptr, true)) != IBM_OK) return s;
  const double bnorm = std::sqrt(ctx->hscal[1]);
  double r0 = std::sqrt(ctx->hscal[0]);
  int cur = 0;
  if (!std::isfinite(bnorm) || !std::isfinite(r0)) {
    ret = IBM_ERR_DIVERGED;
    rel = r0 / bnorm;
  } else if (bnorm == 0.0) {
    IBM_TRY(cudaMemsetAsync(W.u[0], 0, sizeof(double) * want, st));
    rel = 0.0;
  } else {
    rel = r0 / bnorm;
    while (rel > tol) {
      if (cycles >= o.max_cycles) { ret = IBM_ERR_NOT_CONVERGED; break; }
      if (o.precision == 0) {
        cur = srj_cycle(W.u[0], W.u[1], (const double *)W.f, v64, cur, false);
        if ((s = residual(W.u[cur], nullptr, false)) != IBM_OK) return s;
      } else {
        // the correction starts from zero; the membranes' cut cells read it, so there it is cleared
        if (cuts) IBM_TRY(cudaMemsetAsync(W.e[0], 0, sizeof(float) * want, st));
        const int ec = srj_cycle(W.e[0], W.e[1], (const float *)W.r32, v32, 0, !cuts);
        if (df) k_hz_update_df<<<ctx->wave, 256, 0, st>>>(uh, ul, W.e[ec], want);
        else k_hz_update<<<ctx->wave, 256, 0, st>>>(W.u[cur], W.e[ec], want);
        ++launches;
        if ((s = residual(W.u[cur], W.r32, false)) != IBM_OK) return s;
      }
      ++cycles;
      const double rn = std::sqrt(ctx->hscal[0]);
      rel = rn / bnorm;
      if (info && info->resid_history && hist < info->history_cap) info->resid_history[hist++] = rel;
      if (!std::isfinite(rel) || rn > 1e6 * std::max(r0, bnorm)) { ret = IBM_ERR_DIVERGED; break; }
    }
  }
  if (df) k_hz_unpack_df<<<cell_grid, HZ_PK, 0, st>>>(uh, ul, nx, ny, G, L0.mask, u_user);
  else k_hz_unpack<<<cell_grid, HZ_PK, 0, st>>>(W.u[cur], nx, ny, G, L0.mask, u_user);
  ++launches;
  IBM_TRY(cudaGetLastError());
  IBM_TRY(cudaStreamSynchronize(st));
  ctx->launches += launches;
  if (info) {
    info->cycles = cycles;
    info->history_len = hist;
    info->rel_resid = rel;
    info->lambda = 0.0;
    info->ms_total = std::chrono::duration<double, std::milli>(std::chrono::steady_clock::now() - t0).count();
  }
  return ret;
}

ibm_status helmholtz_sweeps_timed_impl(ibm_ctx *ctx, ibm_tables *t, double alpha, int precision, int nsweeps,
                                       const double *f_user, double *u_user, cudaStream_t st, double *ms) {
  if (!ms || nsweeps < 1 || nsweeps > 4096) return IBM_ERR_INVALID_ARG;
  ibm_helmholtz_opts o;
  ibm_helmholtz_opts_default(&o);
  o.precision = precision;
  return helmholtz_solve_impl(ctx, t, alpha, f_user, nullptr, 1.0, u_user, &o, nullptr, st, ms, nsweeps);
}

ibm_status boundary_velocity_rigid_impl(ibm_tables *T, const double *motions, int nmesh, double *ub,
                                        cudaStream_t st) {
  if (nmesh < 1 || nmesh + 1 != (int)T->mesh_tri_off.size() || !motions || !ub) return IBM_ERR_INVALID_ARG;
  if (nmesh > MAX_RIGID_V) return IBM_ERR_CAPACITY;
  RigidVel M;
  M.n = nmesh;
  for (int m = 0; m <= nmesh; ++m) M.off[m] = T->mesh_tri_off[m];
  for (int m = 0; m < nmesh; ++m)
    for (int q = 0; q < 9; ++q) M.m[m][q] = motions[9 * m + q];
  const long long ng = T->nghost;
  if (ng > 0) {
    k_rigid_velocity<<<nb_of(ng, 256), 256, 0, st>>>(T->gbi, T->gtri, ng, M, ub);
    T->ctx->launches += 1;
  }
  IBM_TRY(cudaGetLastError());
  return IBM_OK;
}

}  // namespace ibm
