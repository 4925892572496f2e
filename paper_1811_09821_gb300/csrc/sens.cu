// Step (c): compliance C = f^T u (Eq. 1 with z = f) and the design sensitivities
// dC/drho_s = -E'(rho_s) w_s,  w_s = u_e^T K0_s u_e = integral over subcell s of eps^T D0 eps,
// E'(rho) = q rho^(q-1) (E0 - Emin).  The compliance problem is self-adjoint (adjoint = -u), so u
// is the only field needed; it is re-gathered per element from the stored global vector.
//
// Two kernels.  Both gather the element's displacement in FP64 and remove its best-fit rigid motion
// (translation and rotation, which K0_s annihilates) in FP64.
//
// FP64 (sens_poly_kernel): the energy density eps^T D0 eps is a polynomial of degree <= 2p per axis,
// so its values on one (2p+1) x (2p+1) Gauss grid of the element determine it, and its integrals
// over the d x d subcells are two small products with the integrals W of the grid's Lagrange
// polynomials over the subcells: w = W en W^T.  For Q3 and 8 x 8 subcells that is 49 strain
// evaluations in place of 1024.  Its weights have both signs, so its error is relative to the element's
// largest w: subcells below 1/64 of that (Q1: 1/16) are integrated by the subcell's own (p+1) x (p+1) Gauss points, a
// sum of squares with positive weights (w >= 0 for u = v, error relative to sqrt(w w_max)).  The
// 1D tables are formed in double-double and rounded once: rounded products of Lagrange factors were
// the larger part of either form's error.  Against extended precision (orders 1..6, d = 3 and 8; rough,
// smooth and bending fields; 2-norm): point sums over every subcell with rounded tables 2e-16 to 1.5e-15, this
// form 1.7e-16 to 3.9e-16, nowhere the larger but for 2.4e-16 against 2.2e-16 at p = 4, d = 8.  Bound by the
// FP64 pipes (2 FMA per clock and SM): a block takes several elements and spreads each stage over all
// its threads.  480 x 240 Q3/d8 elements: 12.25 ms with point sums over every subcell, 0.76 ms with the
// polynomial for every one, 0.87 ms with the small ones directly.
//
// FP32 (sens_kernel, MTO_MIXED): one warp per element; strains at the (p+1) x (p+1) Gauss points of
// every subcell from a sum-factorised tensor evaluation on the element's d(p+1) x d(p+1) point grid;
// each point adds eps^T D0 eps (a sum of non-negative terms) to its subcell.
#include <cmath>

#include "mto_internal.cuh"

namespace mto {

constexpr int kSensQMax = 2 * MTO_P_MAX + 1;

// points per axis of the FP64 kernel's grid: enough for degree 2p, or the subcell's own Gauss rule for d = 1
__host__ __device__ constexpr int sens_q(int p, int d) { return d == 1 ? p + 1 : 2 * p + 1; }

namespace {

// Double-double arithmetic (Dekker 1971: a value is the unevaluated sum of two doubles, about 106 bits)
// for the tables below.
struct DD {
  double h, l;
};

__device__ __forceinline__ DD dd_norm(double h, double l) {   // |h| >= |l|
  const double s = __dadd_rn(h, l);
  return {s, __dsub_rn(l, __dsub_rn(s, h))};
}
__device__ __forceinline__ DD operator+(DD a, DD b) {
  const double s = __dadd_rn(a.h, b.h), t = __dsub_rn(s, a.h);
  const double e = __dadd_rn(__dsub_rn(a.h, __dsub_rn(s, t)), __dsub_rn(b.h, t));
  return dd_norm(s, __dadd_rn(e, __dadd_rn(a.l, b.l)));
}
__device__ __forceinline__ DD operator-(DD a, DD b) { return a + DD{-b.h, -b.l}; }
__device__ __forceinline__ DD operator*(DD a, DD b) {
  const double p = __dmul_rn(a.h, b.h);
  return dd_norm(p, fma(a.h, b.h, -p) + fma(a.h, b.l, a.l * b.h));
}
__device__ __forceinline__ DD operator/(DD a, DD b) {
  const double q = a.h / b.h;
  const DD r = a - b * DD{q, 0.0};
  return dd_norm(q, r.h / b.h);
}
__device__ __forceinline__ DD dd(double x) { return {x, 0.0}; }

// (P_n, P_{n-1}) at x by the three-term recurrence
__device__ __forceinline__ void dd_legendre(int n, DD x, DD* pn, DD* pn1) {
  DD a = dd(1.0), b = x;
  for (int k = 2; k <= n; ++k) {
    const DD c = (dd(2 * k - 1) * x * b - dd(k - 1) * a) / dd(k);
    a = b;
    b = c;
  }
  *pn = n == 0 ? dd(1.0) : b;
  *pn1 = a;
}

// 1 / prod_{j != a} (z_a - z_j)
__device__ __forceinline__ DD dd_bary(const double* z, int n, int a) {
  DD v = dd(1.0);
  for (int j = 0; j < n; ++j)
    if (j != a) v = v * (dd(z[a]) - dd(z[j]));
  return dd(1.0) / v;
}

// Lagrange polynomial l_a on the nodes z and its derivative, c = dd_bary(z, n, a)
__device__ __forceinline__ DD dd_lagrange(const double* z, int n, int a, DD c, DD x) {
  for (int j = 0; j < n; ++j)
    if (j != a) c = c * (x - dd(z[j]));
  return c;
}
__device__ __forceinline__ DD dd_lagrange_der(const double* z, int n, int a, DD c, DD x) {
  DD s = dd(0.0);
  for (int i = 0; i < n; ++i) {
    if (i == a) continue;
    DD t = c;
    for (int j = 0; j < n; ++j)
      if (j != a && j != i) t = t * (x - dd(z[j]));
    s = s + t;
  }
  return s;
}

}  // namespace

// Tables of a (p, d) class.  FP64 (Q = sens_q Gauss points x_g): [L: N1 x Q][Dx: N1 x Q][Dy: N1 x Q]
// [W: d x Q][Z: N1] with L = l_a(x_g), Dx = 2/hx l_a'(x_g), Dy = 2/hy l_a'(x_g),
// W = integral over subcell i of the Lagrange polynomial of point g, Z the GLL nodes; then for d > 1 the
// subcells' own points xi_g = -1 + (2 i + 1 + x_k)/d, G = d (p+1): [L: G x N1][Dx: G x N1][Dy: G x N1]
// [w: N1] with the weights w_k / d.
// FP32: [L: N1 x G][D: N1 x G][W: G] at the same points, W = w_k / d (the 1D subcell Jacobian).
__host__ __device__ constexpr int sens_tab_len(int p, int d) {
  return (3 * sens_q(p, d) + 1) * (p + 1) + d * sens_q(p, d) + (d > 1 ? (3 * d * (p + 1) + 1) * (p + 1) : 0);
}

__global__ void __launch_bounds__(256) sens_table_kernel(int p, int d, double hx, double hy, double* __restrict__ tab,
                                                         float* __restrict__ tabf) {
  const int n1 = p + 1, G = d * n1, Q = sens_q(p, d), t = threadIdx.x;
  __shared__ double z[kPMaxTab + 1], gx[kPMaxTab + 1], gw[kPMaxTab + 1], qx[kSensQMax], qw[kSensQMax];
  __shared__ DD xk[kPMaxTab + 1], wk[kPMaxTab + 1], cz[kPMaxTab + 1], cq[kSensQMax];
  if (t == 0) gll_nodes(p, z);
  if (t == 32) gauss_rule(n1, gx, gw);
  if (t == 64) gauss_rule(Q, qx, qw);
  __syncthreads();
  for (int k = t; k < 2 * n1 * G + G; k += blockDim.x) {
    double v;
    if (k < 2 * n1 * G) {
      int which = k / (n1 * G), r = k % (n1 * G), a = r / G, g = r % G;
      int i = g / n1, kk = g % n1;
      double xi = -1.0 + (2.0 * i + 1.0 + gx[kk]) / d;
      v = which == 0 ? lagrange_val(z, n1, a, xi) : lagrange_der(z, n1, a, xi);
    } else {
      v = gw[(k - 2 * n1 * G) % n1] / d;
    }
    tabf[k] = (float)v;
  }
  if (t < n1) {   // the (p+1)-point rule: one Newton step from the rounded node, w = 2 (1 - x^2) / (n P_{n-1})^2
    DD pn, pn1, x = dd(gx[t]);
    dd_legendre(n1, x, &pn, &pn1);
    x = x - pn * (dd(1.0) - x * x) / (dd(n1) * (pn1 - x * pn));
    dd_legendre(n1, x, &pn, &pn1);
    xk[t] = x;
    wk[t] = dd(2.0) * (dd(1.0) - x * x) / (dd(n1) * pn1 * dd(n1) * pn1);
  }
  if (t >= 32 && t < 32 + n1) cz[t - 32] = dd_bary(z, n1, t - 32);
  if (t >= 64 && t < 64 + Q) cq[t - 64] = dd_bary(qx, Q, t - 64);
  __syncthreads();
  auto point = [&](int g) { return (dd(2 * (g / n1) + 1) + xk[g % n1]) / dd(d) - dd(1.0); };
  auto value = [&](int which, int a, DD x) {   // 0: l_a, 1: 2/hx l_a', 2: 2/hy l_a'
    return which == 0 ? dd_lagrange(z, n1, a, cz[a], x).h
                      : (dd(2.0) / dd(which == 1 ? hx : hy) * dd_lagrange_der(z, n1, a, cz[a], x)).h;
  };
  const int nt = n1 * Q, nz = 3 * nt + d * Q, np = G * n1, len = sens_tab_len(p, d);
  for (int k = t; k < len; k += blockDim.x) {
    double v;
    if (k < 3 * nt) {
      v = value(k / nt, k % nt / Q, dd(qx[k % Q]));
    } else if (k < nz) {
      const int i = (k - 3 * nt) / Q, g = (k - 3 * nt) % Q;
      DD s = dd(0.0);
      if (d == 1) s = wk[g];   // Q = p + 1
      else
        for (int kk = 0; kk < n1; ++kk) s = s + wk[kk] / dd(d) * dd_lagrange(qx, Q, g, cq[g], point(i * n1 + kk));
      v = s.h;
    } else if (k < nz + n1) {
      v = z[k - nz];
    } else if (k < nz + n1 + 3 * np) {
      const int r = k - nz - n1;
      v = value(r / np, r % n1, point(r % np / n1));
    } else {
      v = (wk[k - nz - n1 - 3 * np] / dd(d)).h;
    }
    tab[k] = v;
  }
}

namespace {

__device__ __forceinline__ double wsum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The FP32 quadrature: w_s = u_e^T K0_s u_e (compliance, self-adjoint).
template <int PO>
__global__ void __launch_bounds__(128) sens_kernel(
    int n, int d, const int* __restrict__ elem, const int* __restrict__ slot, const int* __restrict__ gmap,
    const Constraint* __restrict__ cons, const double* __restrict__ u, const double* __restrict__ rho,
    const int64_t* __restrict__ design_off, double E0, double Emin, double q, double nu, double hx, double hy,
    const float* __restrict__ tab, const double* __restrict__ Z, double* __restrict__ dc) {
  constexpr int N1 = PO + 1, NN = N1 * N1;
  static_assert(NN <= 64, "two nodes per lane at most");
  const int G = d * N1;
  extern __shared__ unsigned char smem_raw[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // per-warp shared layout: A[4][N1][G], part[G], U[2][NN]
  const size_t per_warp = (size_t)(4 * N1 * G + G + 2 * NN) * sizeof(float);
  float* A = reinterpret_cast<float*>(smem_raw + warp * per_warp);
  float* part = A + 4 * N1 * G;
  float* U = part + G;
  const int k = blockIdx.x * (blockDim.x >> 5) + warp;
  if (k >= n) return;
  const int e = elem[k], sl = slot[k];
  const float* L = tab;
  const float* Dd = tab + N1 * G;
  const float* W = tab + 2 * N1 * G;

  // gather (FP64) and remove the best-fit rigid motion in FP64 (lanes stride over nodes)
  {
    double sux = 0.0, suy = 0.0, snum = 0.0, sden = 0.0;
    double ux[2], uy[2], xl[2], yl[2];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int ln = lane + 32 * r;
      ux[r] = uy[r] = xl[r] = yl[r] = 0.0;
      if (ln < NN) {
        int g = gmap[(size_t)sl * NN + ln];
        if (g >= 0) {
          ux[r] = u[2 * (size_t)g];
          uy[r] = u[2 * (size_t)g + 1];
        } else {
          const Constraint& c = cons[-g - 1];
          for (int j = 0; j < c.cnt; ++j) {
            ux[r] += c.w[j] * u[2 * (size_t)c.node[j]];
            uy[r] += c.w[j] * u[2 * (size_t)c.node[j] + 1];
          }
        }
        xl[r] = 0.5 * Z[ln % N1] * hx;   // node coordinates about the element centre (FP64 GLL nodes)
        yl[r] = 0.5 * Z[ln / N1] * hy;
        sux += ux[r];
        suy += uy[r];
        snum += xl[r] * uy[r] - yl[r] * ux[r];
        sden += xl[r] * xl[r] + yl[r] * yl[r];
      }
    }
    const double tx = wsum(sux) / NN, ty = wsum(suy) / NN;
    const double om = wsum(snum) / wsum(sden);
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int ln = lane + 32 * r;
      if (ln < NN) {
        U[ln] = (float)(ux[r] - tx + om * yl[r]);
        U[NN + ln] = (float)(uy[r] - ty - om * xl[r]);
      }
    }
  }
  __syncwarp();

  // stage 1 (x direction): A_c[b][g] = sum_a U_c[b][a] L[a][g],  Ad_c[b][g] = sum_a U_c[b][a] D[a][g]
  for (int g = lane; g < G; g += 32) {
#pragma unroll
    for (int b = 0; b < N1; ++b) {
      float a0 = 0, a1 = 0, d0 = 0, d1 = 0;
#pragma unroll
      for (int a = 0; a < N1; ++a) {
        const float l = L[a * G + g], dl = Dd[a * G + g];
        const float v0 = U[b * N1 + a], v1 = U[NN + b * N1 + a];
        a0 = fma(v0, l, a0);
        d0 = fma(v0, dl, d0);
        a1 = fma(v1, l, a1);
        d1 = fma(v1, dl, d1);
      }
      A[(0 * N1 + b) * G + g] = a0;
      A[(1 * N1 + b) * G + g] = d0;
      A[(2 * N1 + b) * G + g] = a1;
      A[(3 * N1 + b) * G + g] = d1;
    }
  }
  __syncwarp();

  // stage 2 (y direction) and the energy density at every point
  const float sx = (float)(2.0 / hx), sy = (float)(2.0 / hy), jac = (float)(0.25 * hx * hy);
  const double f = 1.0 / (1.0 - nu * nu);
  const float D11 = (float)f, D12 = (float)(f * nu), D33 = (float)(f * 0.5 * (1.0 - nu));
  const double dE = E0 - Emin;
  const int64_t off = design_off[e];
  for (int j = 0; j < d; ++j) {
    for (int g = lane; g < G; g += 32) {
      float acc = 0;
      for (int kk = 0; kk < N1; ++kk) {
        const int gy = j * N1 + kk;
        float ex = 0, ey = 0, g0 = 0, g1 = 0;
#pragma unroll
        for (int b = 0; b < N1; ++b) {
          const float lb = L[b * G + gy], db = Dd[b * G + gy];
          ex = fma(A[(1 * N1 + b) * G + g], lb, ex);   // d ux / d xi
          g0 = fma(A[(0 * N1 + b) * G + g], db, g0);   // d ux / d eta
          g1 = fma(A[(3 * N1 + b) * G + g], lb, g1);   // d uy / d xi
          ey = fma(A[(2 * N1 + b) * G + g], db, ey);   // d uy / d eta
        }
        const float exx = ex * sx, eyy = ey * sy, gam = g0 * sy + g1 * sx;
        const float en = D11 * (exx * exx + eyy * eyy) + D12 * (exx * eyy + eyy * exx) + D33 * gam * gam;
        acc = fma(W[gy], en, acc);
      }
      part[g] = acc * W[g] * jac;
    }
    __syncwarp();
    for (int i = lane; i < d; i += 32) {
      float w = 0;
      for (int kk = 0; kk < N1; ++kk) w += part[i * N1 + kk];
      const int s = j * d + i;
      const double r = rho[off + s];
      dc[off + s] = -q * pow(r, q - 1.0) * dE * (double)w;
    }
    __syncwarp();
  }
}

// The FP64 kernel (see the head of this file).  A block of 128 threads takes EB elements (a power of
// two, 4..32); each stage is a flat loop over the items of all of them.
constexpr int kSensThreads = 128;
// Subcells below this share of the element's largest |w| are integrated directly.  Down to it the polynomial's
// error, relative to the subcell's own w, was 0.3 to 1.1 times that of point sums with rounded tables in most
// classes of the study (1.7 times in the worst, bending Q4 elements with 8 x 8 subcells); it grows with the
// inverse of the share.
__host__ __device__ constexpr double sens_direct_share(int p) { return p == 1 ? 1.0 / 16.0 : 1.0 / 64.0; }

// doubles of shared memory per element of the x-contracted fields (later the subcells' w), and in all
__host__ __device__ constexpr int sens_work_doubles(int p, int d, int nf) {
  return nf * 4 * (p + 1) * sens_q(p, d) > d * d ? nf * 4 * (p + 1) * sens_q(p, d) : d * d;
}
__host__ __device__ constexpr int sens_elem_doubles(int p, int d, int nf) {
  const int nn = (p + 1) * (p + 1), Q = sens_q(p, d);
  return nf * (2 * nn + 3) + sens_work_doubles(p, d, nf) + Q * Q + d * Q + (d * d + 3) / 4;
}

// (exx + nu eyy)(exx' + nu eyy') + (1 - nu^2) eyy eyy' + (1 - nu)/2 gam gam': the energy density over 1 / (1 - nu^2)
template <int NF>
__device__ __forceinline__ double sens_density(const double (&ax)[NF], const double (&ey)[NF], const double (&gm)[NF],
                                               double c1, double c2) {
  constexpr int o = NF - 1;
  return fma(ax[0], ax[o], fma(c1 * ey[0], ey[o], c2 * gm[0] * gm[o]));
}

// Column kx of the (p+1) x (p+1) Gauss points of subcell (i, j): the energy density integrated along y, of the
// fields at Uf[NF][2][NN]; tab: the tables of the subcells' points.
template <int PO, int NF>
__device__ __forceinline__ double sens_direct(const double* __restrict__ Uf, const double* __restrict__ tab, int d, int i,
                                              int j, int kx, double nu, double c1, double c2) {
  constexpr int N1 = PO + 1, NN = N1 * N1;
  const int np = d * N1 * N1;
  const double *L = tab, *Dx = L + np, *Dy = Dx + np, *w1 = Dy + np;
  const double *lx = L + (i * N1 + kx) * N1, *dx = Dx + (i * N1 + kx) * N1;
  double A[NF][4][N1];
#pragma unroll
  for (int fld = 0; fld < NF; ++fld)
#pragma unroll
    for (int b = 0; b < N1; ++b) {
      double a0 = 0.0, d0 = 0.0, a1 = 0.0, d1 = 0.0;
#pragma unroll
      for (int a = 0; a < N1; ++a) {
        const double l = __ldg(lx + a), dl = __ldg(dx + a);
        const double v0 = Uf[fld * 2 * NN + b * N1 + a], v1 = Uf[fld * 2 * NN + NN + b * N1 + a];
        a0 = fma(v0, l, a0);
        d0 = fma(v0, dl, d0);
        a1 = fma(v1, l, a1);
        d1 = fma(v1, dl, d1);
      }
      A[fld][0][b] = a0;
      A[fld][1][b] = d0;
      A[fld][2][b] = a1;
      A[fld][3][b] = d1;
    }
  double t = 0.0;
#pragma unroll 1
  for (int ky = 0; ky < N1; ++ky) {
    const double *ly = L + (j * N1 + ky) * N1, *dy = Dy + (j * N1 + ky) * N1;
    double ax[NF], ey[NF], gm[NF];
#pragma unroll
    for (int fld = 0; fld < NF; ++fld) {
      double ex = 0.0, e2 = 0.0, ga = 0.0;
#pragma unroll
      for (int b = 0; b < N1; ++b) {
        const double lb = __ldg(ly + b), db = __ldg(dy + b);
        ex = fma(A[fld][1][b], lb, ex);
        ga = fma(A[fld][0][b], db, ga);
        ga = fma(A[fld][3][b], lb, ga);
        e2 = fma(A[fld][2][b], db, e2);
      }
      ax[fld] = fma(nu, e2, ex);
      ey[fld] = e2;
      gm[fld] = ga;
    }
    t = fma(__ldg(w1 + ky), sens_density<NF>(ax, ey, gm, c1, c2), t);
  }
  return t;
}

template <int PO, int NF>
__global__ void __launch_bounds__(kSensThreads, NF == 1 ? (PO <= 3 ? 6 : 4) : (PO <= 3 ? 4 : 2)) sens_poly_kernel(
    int n, int d, int Q, int EB, const int* __restrict__ elem, const int* __restrict__ slot,
    const int* __restrict__ gmap, const Constraint* __restrict__ cons, const double* __restrict__ u,
    const double* __restrict__ v, const double* __restrict__ rho, const int64_t* __restrict__ design_off, double E0,
    double Emin, double q, double nu, double hx, double hy, const double* __restrict__ tab, double* __restrict__ dc,
    double* __restrict__ eout) {
  constexpr int N1 = PO + 1, NN = N1 * N1;
  extern __shared__ double sd[];
  const int t = threadIdx.x;
  const int NQ = N1 * Q, ntab = 3 * NQ + d * Q + N1;
  const double *L = sd, *Dx = sd + NQ, *Dy = Dx + NQ, *W = Dy + NQ, *Z = W + d * Q;
  double* U = sd + ntab;                       // [EB][NF][2][NN]
  double* rig = U + EB * NF * 2 * NN;          // [EB][NF][3] translation and rotation
  double* A = rig + EB * NF * 3;               // [EB][NF][4][N1][Q]
  double* ws = A;                              // [EB][d][d] w of the subcells, once A is used up
  double* en = A + EB * sens_work_doubles(PO, d, NF);   // [EB][Q][Q] energy density (y, x)
  double* T = en + EB * Q * Q;                 // [EB][d][Q] integrated along x (subcell, y point)
  unsigned short* list = reinterpret_cast<unsigned short*>(T + EB * d * Q);   // [EB][d][d] small subcells
  __shared__ int n_list;
  __shared__ double part[kSensThreads];
  if (t == 0) n_list = 0;
  for (int k = t; k < ntab; k += kSensThreads) sd[k] = tab[k];
  const int base = blockIdx.x * EB;
  const int ne = min(EB, n - base);
  // gather (FP64)
  for (int it = t; it < ne * NF * NN; it += kSensThreads) {
    const int el = it / (NF * NN), fld = it / NN % NF, ln = it % NN;
    const double* x = fld == 0 ? u : v;
    const int g = gmap[(size_t)slot[base + el] * NN + ln];
    double ux = 0.0, uy = 0.0;
    if (g >= 0) {
      ux = x[2 * (size_t)g];
      uy = x[2 * (size_t)g + 1];
    } else {
      const Constraint& c = cons[-g - 1];
      for (int j = 0; j < c.cnt; ++j) {
        ux += c.w[j] * x[2 * (size_t)c.node[j]];
        uy += c.w[j] * x[2 * (size_t)c.node[j] + 1];
      }
    }
    U[(el * NF + fld) * 2 * NN + ln] = ux;
    U[(el * NF + fld) * 2 * NN + NN + ln] = uy;
  }
  __syncthreads();
  // least-squares rigid motion about the element centre
  for (int it = t; it < ne * NF * 3; it += kSensThreads) {
    const int k = it % 3;
    const double* Uf = U + (it / 3) * 2 * NN;
    double s = 0.0;
    if (k < 2) {
      for (int ln = 0; ln < NN; ++ln) s += Uf[k * NN + ln];
      s /= NN;
    } else {
      double den = 0.0;
      for (int ln = 0; ln < NN; ++ln) {
        const double x = 0.5 * hx * Z[ln % N1], y = 0.5 * hy * Z[ln / N1];
        s += x * Uf[NN + ln] - y * Uf[ln];
        den += x * x + y * y;
      }
      s /= den;
    }
    rig[it] = s;
  }
  __syncthreads();
  for (int it = t; it < ne * NF * NN; it += kSensThreads) {
    const int ef = it / NN, ln = it % NN;
    double* Uf = U + ef * 2 * NN;
    Uf[ln] = Uf[ln] - rig[3 * ef] + rig[3 * ef + 2] * (0.5 * hy * Z[ln / N1]);
    Uf[NN + ln] = Uf[NN + ln] - rig[3 * ef + 1] - rig[3 * ef + 2] * (0.5 * hx * Z[ln % N1]);
  }
  __syncthreads();
  // stage 1 (along x), per row b of nodes and grid column g: ux and uy by L and by Dx
  for (int it = t; it < ne * NF * NQ; it += kSensThreads) {
    const int ef = it / NQ, b = it % NQ / Q, g = it % Q;
    const double* Uf = U + ef * 2 * NN + b * N1;
    double a0 = 0.0, d0 = 0.0, a1 = 0.0, d1 = 0.0;
#pragma unroll
    for (int a = 0; a < N1; ++a) {
      const double l = L[a * Q + g], dl = Dx[a * Q + g], v0 = Uf[a], v1 = Uf[NN + a];
      a0 = fma(v0, l, a0);
      d0 = fma(v0, dl, d0);
      a1 = fma(v1, l, a1);
      d1 = fma(v1, dl, d1);
    }
    double* Af = A + (ef * 4 * N1 + b) * Q + g;
    Af[0] = a0;
    Af[NQ] = d0;
    Af[2 * NQ] = a1;
    Af[3 * NQ] = d1;
  }
  __syncthreads();
  // stage 2 (along y): strains and the energy density over 1 / (1 - nu^2) at every grid point
  const double c1 = 1.0 - nu * nu, c2 = 0.5 * (1.0 - nu);
  for (int it = t; it < ne * Q * Q; it += kSensThreads) {
    const int el = it / (Q * Q), h = it % (Q * Q) / Q, g = it % Q;
    double ax[NF], ey[NF], gm[NF];
#pragma unroll
    for (int fld = 0; fld < NF; ++fld) {
      const double* Af = A + (el * NF + fld) * 4 * NQ + g;
      double ex = 0.0, e2 = 0.0, ga = 0.0;
#pragma unroll
      for (int b = 0; b < N1; ++b) {
        const double lb = L[b * Q + h], db = Dy[b * Q + h];
        ex = fma(Af[NQ + b * Q], lb, ex);       // d ux / d x
        ga = fma(Af[b * Q], db, ga);            // d ux / d y
        ga = fma(Af[3 * NQ + b * Q], lb, ga);   // + d uy / d x
        e2 = fma(Af[2 * NQ + b * Q], db, e2);   // d uy / d y
      }
      ax[fld] = fma(nu, e2, ex);
      ey[fld] = e2;
      gm[fld] = ga;
    }
    en[it] = sens_density<NF>(ax, ey, gm, c1, c2);
  }
  __syncthreads();
  // integrals over the subcells: along x, then along y
  for (int it = t; it < ne * d * Q; it += kSensThreads) {
    const int el = it / (d * Q), i = it % (d * Q) / Q, h = it % Q;
    const double* e = en + (el * Q + h) * Q;
    double s = 0.0;
    for (int g = 0; g < Q; ++g) s = fma(W[i * Q + g], e[g], s);
    T[it] = s;
  }
  __syncthreads();
  const double jac = 0.25 * hx * hy / (1.0 - nu * nu), dE = E0 - Emin;
  const bool cube = q == 3.0;
  const int tpe = kSensThreads / EB;   // threads per element, at most 32
  const int el = t / tpe, S = d * d;
  double top = 0.0;
  if (el < ne)
    for (int s = t % tpe; s < S; s += tpe) {
      const double* Wj = W + (s / d) * Q;
      const double* Ti = T + (el * d + s % d) * Q;
      double w = 0.0;
      for (int h = 0; h < Q; ++h) w = fma(Wj[h], Ti[h], w);
      ws[el * S + s] = w;
      top = fmax(top, fabs(w));
    }
  if (d > 1) {   // (one subcell: its Gauss points are the grid's)
    for (int o = tpe >> 1; o > 0; o >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, o));
    if (el < ne)
      for (int s = t % tpe; s < S; s += tpe)
        if (!(fabs(ws[el * S + s]) >= sens_direct_share(PO) * top))   // also where w is not a number
          list[atomicAdd(&n_list, 1)] = (unsigned short)(el << 8 | s);
    __syncthreads();
    // a thread per column of points (one per subcell left small meshes waiting for its chain)
    constexpr int kItems = kSensThreads / N1;
    const int small = n_list;
    const double* w1 = tab + ntab + 3 * d * N1 * N1;
    for (int first = 0; first < small; first += kItems) {
      const int it = first + t / N1;
      if (t < kItems * N1 && it < small) {
        const int le = list[it] >> 8, s = list[it] & 255;
        part[t] = sens_direct<PO, NF>(U + le * NF * 2 * NN, tab + ntab, d, s % d, s / d, t % N1, nu, c1, c2);
      }
      __syncthreads();
      if (t < min(kItems, small - first)) {
        const int e = list[first + t];
        double w = 0.0;
#pragma unroll
        for (int kx = 0; kx < N1; ++kx) w = fma(__ldg(w1 + kx), part[t * N1 + kx], w);
        ws[(e >> 8) * S + (e & 255)] = w;
      }
      __syncthreads();
    }
  }
  double energy = 0.0;   // sum_s E(rho_s) w_s (eout)
  if (el < ne) {
    const int64_t off = design_off[elem[base + el]];
    for (int s = t % tpe; s < S; s += tpe) {
      const double w = ws[el * S + s] * jac, r = rho[off + s];
      if (dc) dc[off + s] = -q * (cube ? r * r : pow(r, q - 1.0)) * dE * w;
      if (eout) energy += (Emin + (cube ? r * r * r : pow(r, q)) * dE) * w;
    }
  }
  if (eout) {
    for (int o = tpe >> 1; o > 0; o >>= 1) energy += __shfl_xor_sync(0xffffffffu, energy, o);
    if (el < ne && t % tpe == 0) eout[elem[base + el]] = energy;
  }
}

template <int PO, int NF>
mto_status launch_poly(mto_handle h, const BClass& b, const double* u, const double* v, const double* rho,
                       const mto_material* m, double* dc, double* eout) {
  const int Q = sens_q(PO, b.d), ntab = (3 * Q + 1) * (PO + 1) + b.d * Q;
  const int per = sens_elem_doubles(PO, b.d, NF);
  // elements per block: as many as fit about 36 KB (six blocks per SM), fewer while the launch has less
  // than two blocks per SM
  int EB = 32;
  while (EB > 4 && (EB * per * 8 > 36 * 1024 || b.n < EB * 304)) EB /= 2;
  const size_t smem = sizeof(double) * ((size_t)EB * per + ntab);
  static_assert(8 * (4 * sens_elem_doubles(PO, MTO_D_MAX, NF) + (3 * sens_q(PO, MTO_D_MAX) + 1) * (PO + 1) +
                     MTO_D_MAX * sens_q(PO, MTO_D_MAX)) + 8 * kSensThreads + 16 <= 48 * 1024, "four elements of the largest count fit 48 KB");
  sens_poly_kernel<PO, NF><<<(b.n + EB - 1) / EB, kSensThreads, smem, h->stream>>>(
      b.n, b.d, Q, EB, b.elem, b.slot, h->pc[b.p].gmap, h->cons_d, u, v, rho, h->design_off_d, m->E0, m->Emin, m->q,
      m->nu, h->hx, h->hy, b.stab, dc, eout);
  return mto_after_launch(h, "sens_poly_kernel");
}

// the FP32 quadrature (MTO_MIXED sensitivities)
template <int PO>
mto_status launch_sens(mto_handle h, const BClass& b, const double* u, const double* rho, const mto_material* m,
                       double* dc) {
  constexpr int N1 = PO + 1, warps = 4;
  auto smem_bytes = [](int d) { return sizeof(float) * warps * (size_t)(4 * N1 * d * N1 + d * N1 + 2 * N1 * N1); };
  const size_t smem = smem_bytes(b.d);
  MTO_TRY(allow_smem(h, sens_kernel<PO>, smem_bytes(MTO_D_MAX)));
  const PClass& c = h->pc[b.p];
  const int Q = sens_q(PO, b.d);
  sens_kernel<PO><<<(b.n + warps - 1) / warps, 32 * warps, smem, h->stream>>>(
      b.n, b.d, b.elem, b.slot, c.gmap, h->cons_d, u, rho, h->design_off_d, m->E0, m->Emin, m->q, m->nu,
      h->hx, h->hy, b.stabf, b.stab + 3 * N1 * Q + b.d * Q, dc);
  return mto_after_launch(h, "sens_kernel");
}

template <int NF>
mto_status sens_all(mto_handle h, const double* u, const double* v, const double* rho, const mto_material* m,
                    double* dc, double* eout = nullptr) {
  for (auto& b : h->bc) {
    switch (b.p) {
      case 1: MTO_TRY((launch_poly<1, NF>(h, b, u, v, rho, m, dc, eout))); break;
      case 2: MTO_TRY((launch_poly<2, NF>(h, b, u, v, rho, m, dc, eout))); break;
      case 3: MTO_TRY((launch_poly<3, NF>(h, b, u, v, rho, m, dc, eout))); break;
      case 4: MTO_TRY((launch_poly<4, NF>(h, b, u, v, rho, m, dc, eout))); break;
      case 5: MTO_TRY((launch_poly<5, NF>(h, b, u, v, rho, m, dc, eout))); break;
      case 6: MTO_TRY((launch_poly<6, NF>(h, b, u, v, rho, m, dc, eout))); break;
    }
  }
  return MTO_OK;
}

mto_status sens_all32(mto_handle h, const double* u, const double* rho, const mto_material* m, double* dc) {
  for (auto& b : h->bc) {
    switch (b.p) {
      case 1: MTO_TRY(launch_sens<1>(h, b, u, rho, m, dc)); break;
      case 2: MTO_TRY(launch_sens<2>(h, b, u, rho, m, dc)); break;
      case 3: MTO_TRY(launch_sens<3>(h, b, u, rho, m, dc)); break;
      case 4: MTO_TRY(launch_sens<4>(h, b, u, rho, m, dc)); break;
      case 5: MTO_TRY(launch_sens<5>(h, b, u, rho, m, dc)); break;
      case 6: MTO_TRY(launch_sens<6>(h, b, u, rho, m, dc)); break;
    }
  }
  return MTO_OK;
}

}  // namespace

mto_status build_sens_tables(mto_handle h) {
  for (auto& b : h->bc) {
    const int n1 = b.p + 1, G = b.d * n1;
    MTO_TRY(mto_alloc(h, &b.stab, (size_t)sens_tab_len(b.p, b.d)));
    MTO_TRY(mto_alloc(h, &b.stabf, (size_t)2 * n1 * G + G));
    sens_table_kernel<<<1, 256, 0, h->stream>>>(b.p, b.d, h->hx, h->hy, b.stab, b.stabf);
    MTO_TRY(mto_after_launch(h, "sens_table_kernel"));
  }
  return MTO_OK;
}

mto_status sensitivity(mto_handle h, const double* u, const double* f, const double* rho, const mto_material* m,
                       int precision, double* dc, double* C) {
  {
  TimedScope ts(h, F_SENS);
  if (precision == MTO_FP64) MTO_TRY((sens_all<1>(h, u, nullptr, rho, m, dc)));
  else MTO_TRY(sens_all32(h, u, rho, m, dc));
  MTO_TRY(dot64(h, f, u, h->ndof, h->red + 8));
  }
  if (C) {
    MTO_TRY(mto_cuda_check(h, cudaMemcpyAsync(h->host_pinned + 8, h->red + 8, sizeof(double), cudaMemcpyDeviceToHost, h->stream), "copy"));
    MTO_TRY(mto_cuda_check(h, cudaStreamSynchronize(h->stream), "sync"));
    *C = h->host_pinned[8];
  }
  return MTO_OK;
}

// dJ/drho_s = -E'(rho_s) v_e^T K0_s u_e for an objective J = z^T u with the adjoint field v
// solving K v = z (Eq. 1; v = u for compliance).  FP64 quadrature.
mto_status sensitivity_adjoint(mto_handle h, const double* u, const double* v, const double* rho,
                               const mto_material* m, double* dc) {
  TimedScope ts(h, F_SENS);
  return sens_all<2>(h, u, v, rho, m, dc);
}

// Compliance of an approximate displacement in its energy form, C(u) = 2 f^T u - u^T K u
// (= C* - ||u* - u||_K^2 for the exact u*, so its error is second order in the displacement's):
// u^T K u as the sum of the element energies sum_s E(rho_s) u_e^T K0_s u_e, each after the FP64
// removal of the element's rigid motion (free of the cancellation of a global u^T (K u)), summed
// over the elements in a fixed order.
mto_status compliance_energy(mto_handle h, const double* u, const double* f, const double* rho,
                             const mto_material* m, double* C) {
  {
    TimedScope ts(h, F_SENS);
    MTO_TRY((sens_all<1>(h, u, nullptr, rho, m, nullptr, h->dbuf)));
    MTO_TRY(sum64(h, h->dbuf, h->nel, h->red + 10));
    MTO_TRY(dot64(h, f, u, h->ndof, h->red + 11));
  }
  MTO_TRY(mto_cuda_check(h, cudaMemcpyAsync(h->host_pinned + 10, h->red + 10, 2 * sizeof(double),
                                            cudaMemcpyDeviceToHost, h->stream), "copy"));
  MTO_TRY(mto_cuda_check(h, cudaStreamSynchronize(h->stream), "sync"));
  *C = 2.0 * h->host_pinned[11] - h->host_pinned[10];
  return MTO_OK;
}

}  // namespace mto
