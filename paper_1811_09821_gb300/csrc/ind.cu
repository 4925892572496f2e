// Step (d): the composite refinement indicator and the dp map update (Sec. 3.2, 3.3), and the
// optimality-criteria design update.  All FP64 or its equal (the QR error's matrices from the sliced
// tensor-core sums where those are no further off, see qr_kernel): the integer maps must match the oracle
// exactly, so every floating-point decision is taken in double with a fixed reduction order.
#include <algorithm>
#include <cmath>
#include <vector>

#include <math_constants.h>

#include "mto_internal.cuh"

namespace mto {
namespace {

// Basis constants shared by the indicator kernels: GLL nodes of orders 1..kPMaxTab, Gauss rules of
// 1..kPMaxTab+2 points, and for the Kelly edges the Lagrange derivatives at both ends of an element
// (dn[p][0]: -1, dn[p][1]: +1) and the Lagrange values at the points of an n-point rule (lv[p][n]).
// Filled once per handle by basis_table_kernel.
struct BasisTab {
  double gll[kPMaxTab + 1][kPMaxTab + 1];
  double gx[kPMaxTab + 3][kPMaxTab + 3];
  double gw[kPMaxTab + 3][kPMaxTab + 3];
  double dn[kPMaxTab + 1][2][kPMaxTab + 1];
  double lv[kPMaxTab + 1][kPMaxTab + 3][kPMaxTab + 3][kPMaxTab + 1];
};

__global__ void __launch_bounds__(256) basis_table_kernel(BasisTab* t) {
  const int i = threadIdx.x;
  if (i >= 1 && i <= kPMaxTab) gll_nodes(i, t->gll[i]);
  if (i >= 33 && i <= 32 + kPMaxTab + 2) gauss_rule(i - 32, t->gx[i - 32], t->gw[i - 32]);
  __syncthreads();
  for (int k = i; k < (kPMaxTab + 1) * 2 * (kPMaxTab + 1); k += blockDim.x) {
    const int a = k % (kPMaxTab + 1), end = k / (kPMaxTab + 1) % 2, p = k / (2 * (kPMaxTab + 1));
    if (p >= 1 && a <= p) t->dn[p][end][a] = lagrange_der(t->gll[p], p + 1, a, end ? 1.0 : -1.0);
  }
  constexpr int NG = kPMaxTab + 3;
  for (int k = i; k < (kPMaxTab + 1) * NG * NG * (kPMaxTab + 1); k += blockDim.x) {
    const int a = k % (kPMaxTab + 1), g = k / (kPMaxTab + 1) % NG, n = k / ((kPMaxTab + 1) * NG) % NG;
    const int p = k / ((kPMaxTab + 1) * NG * NG);
    if (p >= 1 && a <= p && n >= 1 && g < n) t->lv[p][n][g][a] = lagrange_val(t->gll[p], p + 1, a, t->gx[n][g]);
  }
}

// Both components of local node ln of the element in slot `slot` (through its constraint if hanging)
__device__ __forceinline__ void gather_node(int nn, int slot, int ln, const int* __restrict__ gmap,
                                            const Constraint* __restrict__ cons, const double* __restrict__ u,
                                            double* ue) {
  int g = gmap[(size_t)slot * nn + ln];
  double a = 0.0, b = 0.0;
  if (g >= 0) {
    a = u[2 * (size_t)g];
    b = u[2 * (size_t)g + 1];
  } else {
    const Constraint& c = cons[-g - 1];
    for (int k = 0; k < c.cnt; ++k) {
      a += c.w[k] * u[2 * (size_t)c.node[k]];
      b += c.w[k] * u[2 * (size_t)c.node[k] + 1];
    }
  }
  ue[2 * ln] = a;
  ue[2 * ln + 1] = b;
}

__device__ __forceinline__ double warp_sum_all(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

struct ClassPtrs {
  const int* gmap[kPMaxTab + 1];
};

// ------------------------------------------------------------------------------------ Kelly
// Adds sign x the normal derivative (along +x or +y) of one element's field at the Gauss points of
// one of its edges to (jx, jy).  The trace of the normal derivative is contracted first: along the
// normal by the derivatives at the element's end (end: 0 the low, 1 the high side), then along the
// edge by the values at the Gauss points: 2 (p + 1) (p + 1 + nq) FMAs, where products of Lagrange
// polynomials formed per point took thousands of FP64 instructions and divisions.
constexpr int kEdgeQ = MTO_P_MAX + 1;   // Gauss points of an edge of the largest order

__device__ __forceinline__ void add_edge_trace(const BasisTab* __restrict__ B, int p, int slot,
                                               const int* __restrict__ gmap, const Constraint* __restrict__ cons,
                                               const double* __restrict__ u, bool vertical, int end, int nq,
                                               double scale, double (&jx)[kEdgeQ], double (&jy)[kEdgeQ]) {
  const int n1 = p + 1;
  const int* gm = gmap + (size_t)slot * n1 * n1;
  const double* dn = B->dn[p][end];
  const int sn = vertical ? 1 : n1, st = vertical ? n1 : 1;   // node strides along the normal and the edge
  for (int b = 0; b < n1; ++b) {
    double tx = 0.0, ty = 0.0;
#pragma unroll 4
    for (int a = 0; a < n1; ++a) {
      const int g = gm[b * st + a * sn];
      double ux, uy;
      if (g >= 0) {
        ux = u[2 * (size_t)g];   // u is the caller's: 8-byte aligned at the least
        uy = u[2 * (size_t)g + 1];
      } else {
        const Constraint& c = cons[-g - 1];
        ux = uy = 0.0;
        for (int k = 0; k < c.cnt; ++k) {
          ux += c.w[k] * u[2 * (size_t)c.node[k]];
          uy += c.w[k] * u[2 * (size_t)c.node[k] + 1];
        }
      }
      tx = fma(dn[a], ux, tx);
      ty = fma(dn[a], uy, ty);
    }
    tx *= scale;
    ty *= scale;
#pragma unroll
    for (int g = 0; g < kEdgeQ; ++g)
      if (g < nq) {
        const double w = B->lv[p][nq][g][b];
        jx[g] = fma(w, tx, jx[g]);
        jy[g] = fma(w, ty, jy[g]);
      }
  }
}

// Edge term c_F * integral_F [du/dn]^2 ds (Eq. 9) for every interior edge: horizontal edges
// first (id iy*nelx + ix, between elements below and above), then vertical edges.  One thread per
// edge, bound by the FP64 pipes (about 150 FMAs per edge between Q3 elements).  Measured with the
// selection kernels below: the indicators of a 320 x 160 adaptive mesh 22.1 -> 10.9 ms (10.5 ms of
// them were this kernel, forming Lagrange products and their divisions per point); on the
// 1024 x 512 beam this kernel took 34 ms.
__global__ void __launch_bounds__(128) kelly_edge_kernel(
    int nelx, int nely, const int* __restrict__ p_of, const int* __restrict__ slot_of, ClassPtrs cp,
    const Constraint* __restrict__ cons, const double* __restrict__ u, const BasisTab* __restrict__ B, double hx,
    double hy, double* __restrict__ edge_val) {
  const int64_t nH = (int64_t)(nely + 1) * nelx, nV = (int64_t)nely * (nelx + 1);
  const double hF = sqrt(hx * hx + hy * hy);
  for (int64_t id = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; id < nH + nV; id += (int64_t)gridDim.x * blockDim.x) {
    const bool vertical = id >= nH;
    int eA, eB;
    if (!vertical) {
      int iy = (int)(id / nelx), ix = (int)(id % nelx);
      if (iy == 0 || iy == nely) { edge_val[id] = 0.0; continue; }
      eA = (iy - 1) * nelx + ix; eB = iy * nelx + ix;
    } else {
      int64_t v = id - nH;
      int iy = (int)(v / (nelx + 1)), ix = (int)(v % (nelx + 1));
      if (ix == 0 || ix == nelx) { edge_val[id] = 0.0; continue; }
      eA = iy * nelx + ix - 1; eB = iy * nelx + ix;
    }
    const double len = vertical ? hy : hx, sc = 2.0 / (vertical ? hx : hy);
    const int pA = p_of[eA], pB = p_of[eB];
    const int pF = pA > pB ? pA : pB;
    const int nq = pF + 1;
    double jx[kEdgeQ], jy[kEdgeQ];
#pragma unroll
    for (int g = 0; g < kEdgeQ; ++g) jx[g] = jy[g] = 0.0;
    add_edge_trace(B, pA, slot_of[eA], cp.gmap[pA], cons, u, vertical, 1, nq, sc, jx, jy);
    add_edge_trace(B, pB, slot_of[eB], cp.gmap[pB], cons, u, vertical, 0, nq, -sc, jx, jy);
    double val = 0.0;
#pragma unroll
    for (int g = 0; g < kEdgeQ; ++g)
      if (g < nq) val += B->gw[nq][g] * (jx[g] * jx[g] + jy[g] * jy[g]) * 0.5 * len;
    edge_val[id] = hF / (2.0 * pF) * val;
  }
}

// Gamma^a_e = sum of its four edge terms in the fixed order left, right, bottom, top.
__global__ void kelly_sum_kernel(int nelx, int nely, const double* __restrict__ edge_val, double* __restrict__ ga) {
  const int64_t nH = (int64_t)(nely + 1) * nelx, nel = (int64_t)nelx * nely;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nel; e += (int64_t)gridDim.x * blockDim.x) {
    int ix = (int)(e % nelx), iy = (int)(e / nelx);
    double s = edge_val[nH + (int64_t)iy * (nelx + 1) + ix];
    s += edge_val[nH + (int64_t)iy * (nelx + 1) + ix + 1];
    s += edge_val[(int64_t)iy * nelx + ix];
    s += edge_val[(int64_t)(iy + 1) * nelx + ix];
    ga[e] = s;
  }
}

// ------------------------------------------------------------------------------------ Gamma^d
// smallest and largest order key; one pair of atomics per block
__global__ void __launch_bounds__(256) minmax_kernel(int64_t n, const double* __restrict__ rho,
                                                     unsigned long long* __restrict__ mm) {
  unsigned long long lo = ~0ULL, hi = 0ULL;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    unsigned long long k = order_key(rho[i]);
    lo = k < lo ? k : lo;
    hi = k > hi ? k : hi;
  }
  __shared__ unsigned long long sl[8], sh[8];
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long a = __shfl_xor_sync(0xffffffffu, lo, o), b = __shfl_xor_sync(0xffffffffu, hi, o);
    lo = a < lo ? a : lo;
    hi = b > hi ? b : hi;
  }
  if ((threadIdx.x & 31) == 0) {
    sl[threadIdx.x >> 5] = lo;
    sh[threadIdx.x >> 5] = hi;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
    lo = sl[w] < lo ? sl[w] : lo;
    hi = sh[w] > hi ? sh[w] : hi;
  }
  atomicMin(&mm[0], lo);
  atomicMax(&mm[1], hi);
}

__device__ double key_to_double(unsigned long long k) {
  unsigned long long u = (k >> 63) ? (k & 0x7fffffffffffffffULL) : ~k;
  double v;
  memcpy(&v, &u, 8);
  return v;
}

// Density indicator (Sec. 3.2.2): per element, the cells' band contributions in cell order.  A warp
// takes 32 consecutive elements: its lanes form the contributions of 32 cells of one element at a
// time (coalesced; the bands are compared on the order keys, off the FP64 pipes), and then each lane
// adds its own element's in cell order, so the sums are those of a serial loop.  The division by
// the cell count is a product where the count is a power of two (exact either way).
constexpr int kGdWarps = 4;
__global__ void __launch_bounds__(32 * kGdWarps) gamma_d_kernel(
    int64_t nel, const int64_t* __restrict__ off, const double* __restrict__ rho,
    const unsigned long long* __restrict__ mm, int cycle, double alpha, double beta, double* __restrict__ gd) {
  __shared__ double tile[kGdWarps][32][33];
  const double rmin = key_to_double(mm[0]), rmax = key_to_double(mm[1]);
  const double ravg = 0.5 * (rmax + rmin);
  const double fac = ravg * exp(-beta * (cycle - 1));
  const double rl = rmin + (1.0 - alpha) * fac, ru = rmax - (1.0 - alpha) * fac;
  const double cl = rmin + alpha * fac, cu = rmax - alpha * fac;
  // -0 and +0 compare equal: zero is added to every key's value first
  auto key = [](double v) { return order_key(__longlong_as_double(__double_as_longlong(v) == (1ll << 63) ? 0ll : __double_as_longlong(v))); };
  // a NaN bound fails its comparison: the largest key as a lower bound, the smallest as an upper one
  auto lower = [&](double v) { return v == v ? key(v) : ~0ULL; };
  auto upper = [&](double v) { return v == v ? key(v) : 0ULL; };
  const unsigned long long krl = lower(rl), kru = upper(ru), kcl = upper(cl), kcu = lower(cu);
  const unsigned long long kav_hi = upper(ravg), kav_lo = lower(ravg);
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  double(*T)[33] = tile[wib];
  const int64_t nw = (int64_t)gridDim.x * kGdWarps;
  for (int64_t base = 32 * (blockIdx.x * (int64_t)kGdWarps + wib); base < nel; base += 32 * nw) {
    const int64_t e = base + lane;
    const int64_t a = e < nel ? off[e] : 0;
    const int n = e < nel ? (int)(off[e + 1] - a) : 0;
    const double nd = (double)n, inv = 1.0 / nd;
    const int nmax = __reduce_max_sync(0xffffffffu, n);
    double g = 0.0;
    for (int c0 = 0; c0 < nmax; c0 += 32) {
#pragma unroll 4
      for (int k = 0; k < 32; ++k) {
        const int nk = __shfl_sync(0xffffffffu, n, k);
        const int64_t ak = __shfl_sync(0xffffffffu, a, k);
        const double ndk = __shfl_sync(0xffffffffu, nd, k), ik = __shfl_sync(0xffffffffu, inv, k);
        const bool p2 = (nk & (nk - 1)) == 0;
        if (c0 >= nk) continue;
        double t = 0.0;
        if (c0 + lane < nk) {
          const double r = rho[ak + c0 + lane];
          const unsigned long long kr = key(r);
          double x = 0.0;
          if ((unsigned long long)(__double_as_longlong(r) & 0x7fffffffffffffffll) <= 0x7ff0000000000000ull) {   // no NaN
            if (krl <= kr && kr <= kav_hi) x = r - rl;
            else if (kav_lo < kr && kr <= kru) x = ru - r;
            else if (kr <= kcl) x = r - cl;     // subtracting cl - r
            else if (kr >= kcu) x = cu - r;
          }
          t = p2 ? x * ik : x / ndk;
        }
        T[k][lane] = t;
      }
      __syncwarp();
      const int m = min(32, n - c0);
      for (int j = 0; j < m; ++j) g += T[lane][j];
      __syncwarp();
    }
    if (e < nel) gd[e] = g;
  }
}

// ------------------------------------------------------------------------------------ QR error
// One warp per element of a (p, d) class (Eq. 14).  Shared layout (doubles): A[L1] (the order p+1
// matrix, lower triangle packed by rows, A_ij at i (i + 1) / 2 + j, factorised in place as
// L D L^T), f[n0], f1[n1], u1[n1], ue[n0], rd[n1] (reciprocal pivots), cl[n1] (the pivot
// column before scaling), pr[3 n1] (the pinned rows of the unmodified matrix); E[S], the moduli, in the
// place of the last three until they are needed; with n0 = 2 (p+1)^2, n1 = 2 (p+2)^2,
// L1 = n1 (n1 + 1) / 2 rounded up.
// K^(p+1) = sum_s E_s K0_s comes as rows formed on the tensor cores (tc_rows, d <= 8), or is summed
// here from the table (rows null, and the elements that `sliced_rows_hold` turns away: 81.6 k of 115 k FMAs
// of a Q3/d8 element).  With rows the FP64 pipes (2 FMA per clock and SM) are 75 % busy, the rest is the
// L D L^T's shared-memory round trips: 12,800 Q3/d8 elements 1.2 ms.  A graded design, most of whose
// elements sum, takes 3.2 ms and is bound by L1 (a lane's table row lies S doubles from the next lane's).
// Indicators of a 320 x 160 adaptive mesh, graded: 10.9 ms with sums, 6.9 with rows, 9.7 with both by this rule.
// eps is invariant to rigid motions of u^(p), which are removed first (FP64) so that the element
// energies carry no cancellation.
//
// The sliced rows are exact to about 2^-54 of the element's largest modulus times the column's largest
// table entry, the FP64 sums to a few 2^-53 of the sum of each entry's own terms.  Those are alike while the
// moduli are; beside void, entries that only soft subcells carry are far below the row's scale.
// In extended precision (orders 1..5, d = 2..8, fields of solved shape) the error of eps with rows was, as
// a geometric mean over the elements of a class, 0.8 to 1.1 times that with sums for fronts of a factor of
// 16, up to 1.7 times for 125 and up to 4.5 times for 1e9: rows serve the elements within kQRContrast.
constexpr double kQRContrast = 16.0;

// dynamic shared memory of qr_kernel (its layout above)
size_t qr_smem_bytes(int p, int S) {
  const int n0 = 2 * (p + 1) * (p + 1), n1 = 2 * (p + 2) * (p + 2);
  return sizeof(double) * ((size_t)qr_row_len(p + 1) + 2 * n0 + 2 * n1 + std::max(5 * n1, S));
}

// whether the moduli's extremes over the element (lo, hi; ok: every one is a number of at least 0) let the rows be used
__device__ __forceinline__ bool sliced_rows_hold(bool ok, double lo, double hi) {
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  return __all_sync(0xffffffffu, ok) && hi <= kQRContrast * lo;
}

__global__ void __launch_bounds__(32) qr_kernel(int p, int d, int n, int first, const int* __restrict__ elem,
                                                const int* __restrict__ slot, int L, const int* __restrict__ gmap,
                                                const Constraint* __restrict__ cons, const double* __restrict__ K64,
                                                const double* __restrict__ rows, const double* __restrict__ K0T1,
                                                const double* __restrict__ R, const double* __restrict__ u,
                                                const double* __restrict__ rho, const int64_t* __restrict__ off,
                                                double E0, double Emin, double q, const BasisTab* __restrict__ B,
                                                double hx, double hy, double* __restrict__ eps) {
  extern __shared__ __align__(16) double sh[];
  const int lane = threadIdx.x;
  const int k = first + blockIdx.x;
  if (k >= n) return;
  const int e = elem[k], sl = slot[k];
  const int n1d = p + 1;
  const int na = (p + 1) * (p + 1), nb = (p + 2) * (p + 2);
  const int n0 = 2 * na, n1 = 2 * nb, S = d * d;
  const int P1 = packed_size(n1), L1 = qr_row_len(p + 1);
  double* A = sh;
  double* f = A + L1;
  double* f1 = f + n0;
  double* u1 = f1 + n1;
  double* ue = u1 + n1;
  double* rd = ue + n0;
  double* cl = rd + n1;
  double* pr = cl + n1;
  double* E = rd;   // S doubles (the launch's shared memory covers S > 5 n1)
  bool ok = true;
  double lo = CUDART_INF, hi = 0.0;
  for (int s = lane; s < S; s += 32) {
    const double r = rho[off[e] + s];
    const double m = Emin + (q == 3.0 ? r * r * r : pow(r, q)) * (E0 - Emin);
    E[s] = m;
    ok = ok && m >= 0.0;
    lo = fmin(lo, m);
    hi = fmax(hi, m);
  }
  const bool sliced = rows && sliced_rows_hold(ok, lo, hi);
  if (sliced) {
    const double2* src = reinterpret_cast<const double2*>(rows + (size_t)blockIdx.x * L1);
    for (int c = lane; c < L1 / 2; c += 32) reinterpret_cast<double2*>(A)[c] = src[c];
  }
  // gather u_e (lanes over nodes), then remove its least-squares rigid motion about the element
  // centre (translations and rotation; node sums over the warp)
  for (int ln = lane; ln < na; ln += 32) gather_node(na, sl, ln, gmap, cons, u, ue);
  __syncwarp();
  {
    const double* z = B->gll[p];
    double tx = 0.0, ty = 0.0, num = 0.0, den = 0.0;
    for (int ln = lane; ln < na; ln += 32) {
      const double x = 0.5 * hx * z[ln % n1d], y = 0.5 * hy * z[ln / n1d];
      tx += ue[2 * ln];
      ty += ue[2 * ln + 1];
      num += x * ue[2 * ln + 1] - y * ue[2 * ln];
      den += x * x + y * y;
    }
    tx = warp_sum_all(tx) / na;
    ty = warp_sum_all(ty) / na;
    const double om = warp_sum_all(num) / warp_sum_all(den);
    for (int ln = lane; ln < na; ln += 32) {
      const double x = 0.5 * hx * z[ln % n1d], y = 0.5 * hy * z[ln / n1d];
      ue[2 * ln] = ue[2 * ln] - tx + om * y;
      ue[2 * ln + 1] = ue[2 * ln + 1] - ty - om * x;
    }
  }
  __syncwarp();
  // f = K_e u_e (order p, FP64 element matrix of the build: row i of the circulant-diagonal layout from
  // D_k[i] and D_k[i - k]) and J^(p) = u^T f / 2
  double jp = 0.0;
  const double* Ke = K64 + (size_t)sl * L;
  for (int i = lane; i < n0; i += 32) {
    double s = 0.0;
    for (int kk = 0; 2 * kk <= n0; ++kk) {
      const int j = i + kk < n0 ? i + kk : i + kk - n0, jm = i >= kk ? i - kk : i - kk + n0;
      s += Ke[kk * n0 + i] * ue[j];
      if (kk > 0 && 2 * kk < n0) s += Ke[kk * n0 + jm] * ue[jm];
    }
    f[i] = s;
    jp += ue[i] * s;
  }
  for (int o = 16; o > 0; o >>= 1) jp += __shfl_xor_sync(0xffffffffu, jp, o);
  jp *= 0.5;
  __syncwarp();
  // f1 = R f per component
  for (int i = lane; i < n1; i += 32) {
    const int jn = i >> 1, c = i & 1;
    double s = 0.0;
    for (int kk = 0; kk < na; ++kk) s += R[jn * na + kk] * f[2 * kk + c];
    f1[i] = s;
  }
  if (!sliced) {
    // K^(p+1) (table rows by upper packed index (i <= j)) into the lower triangle
    for (int c = lane; c < P1; c += 32) {
      double s = 0.0;
      const double* kc = K0T1 + (size_t)c * S;
      for (int t = 0; t < S; ++t) s = fma(E[t], kc[t], s);
      int i = 0, rem = c;
      while (rem >= n1 - i) { rem -= n1 - i; ++i; }
      const int j = i + rem;
      A[j * (j + 1) / 2 + i] = s;
    }
  }
  __syncwarp();
  // pinned DOFs of the (p+1) element: u_x, u_y at the bottom-left vertex, u_y at the bottom-right
  // vertex; their values are those of u^(p) at the same vertices
  const int fx[3] = {0, 1, 2 * (p + 1) + 1};
  const double v[3] = {ue[0], ue[1], ue[2 * p + 1]};
  auto at = [&](int a, int b) -> double { return a >= b ? A[a * (a + 1) / 2 + b] : A[b * (b + 1) / 2 + a]; };
  // the pinned rows before the modification (for J^(p+1)), and the right-hand side on free DOFs
  for (int i = lane; i < n1; i += 32) {
    const double k0 = at(i, fx[0]), k1 = at(i, fx[1]), k2 = at(i, fx[2]);
    pr[i] = k0;
    pr[n1 + i] = k1;
    pr[2 * n1 + i] = k2;
    double r = f1[i] - k0 * v[0] - k1 * v[1] - k2 * v[2];
    for (int k = 0; k < 3; ++k)
      if (i == fx[k]) r = v[k];
    u1[i] = r;
  }
  __syncwarp();
  // identity rows and columns on the pinned DOFs
  for (int k = 0; k < 3; ++k)
    for (int i = lane; i < n1; i += 32) {
      const int a = i > fx[k] ? i : fx[k], b = i > fx[k] ? fx[k] : i;
      A[a * (a + 1) / 2 + b] = i == fx[k] ? 1.0 : 0.0;
    }
  __syncwarp();
  // A = L D L^T (right-looking).  Column c: the pivot's reciprocal into rd[c], the column kept
  // unscaled in cl and scaled into L; the trailing update A_ij -= L_ic cl_j (c < j <= i) runs over
  // the m (m + 1) / 2 pairs of the trailing block spread evenly over the lanes: pair
  // t = s (s + 1) / 2 + r (0 <= r <= s < m) is row n1 - 1 - r, column n1 - 1 - s.  A pinned column is
  // the identity's: nothing to update.
  for (int c = 0; c < n1; ++c) {
    if (c == fx[0] || c == fx[1] || c == fx[2]) {
      if (lane == 0) rd[c] = 1.0;
      continue;
    }
    const double inv = newton_rcp(A[c * (c + 1) / 2 + c]);
    for (int i = c + 1 + lane; i < n1; i += 32) {
      const double a = A[i * (i + 1) / 2 + c];
      cl[i] = a;
      A[i * (i + 1) / 2 + c] = a * inv;
    }
    if (lane == 0) rd[c] = inv;
    __syncwarp();
    const int m = n1 - 1 - c;
    const int T = m * (m + 1) / 2;
    for (int t = lane; t < T; t += 32) {
      int s = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
      while (s * (s + 1) / 2 > t) --s;
      while ((s + 1) * (s + 2) / 2 <= t) ++s;
      const int r = t - s * (s + 1) / 2;
      const int i = n1 - 1 - r, j = n1 - 1 - s;
      A[i * (i + 1) / 2 + j] -= A[i * (i + 1) / 2 + c] * cl[j];
    }
    __syncwarp();
  }
  // L y = b, y <- D^-1 y, L^T x = y, column by column (each solved entry updates the rest over the
  // lanes; a pinned column has nothing to give)
  for (int j = 0; j < n1; ++j) {
    if (j == fx[0] || j == fx[1] || j == fx[2]) continue;
    const double yj = u1[j];
    for (int i = j + 1 + lane; i < n1; i += 32) u1[i] -= A[i * (i + 1) / 2 + j] * yj;
    __syncwarp();
  }
  for (int i = lane; i < n1; i += 32) u1[i] *= rd[i];
  __syncwarp();
  for (int j = n1 - 1; j >= 0; --j) {
    if (j == fx[0] || j == fx[1] || j == fx[2]) continue;
    const double xj = u1[j];
    for (int i = lane; i < j; i += 32) u1[i] -= A[j * (j + 1) / 2 + i] * xj;
    __syncwarp();
  }
  // J^(p+1) = u1^T K u1 / 2 = (u1_f^T f1_f + v^T (K u1)_pinned) / 2: on the free rows K u1 is the
  // right-hand side f1, on the pinned rows the saved rows of the unmodified matrix give it
  double j1 = 0.0;
  for (int i = lane; i < n1; i += 32) {
    const bool pin = i == fx[0] || i == fx[1] || i == fx[2];
    if (!pin) j1 += u1[i] * f1[i];
    j1 += u1[i] * (v[0] * pr[i] + v[1] * pr[n1 + i] + v[2] * pr[2 * n1 + i]);
  }
  for (int o = 16; o > 0; o >>= 1) j1 += __shfl_xor_sync(0xffffffffu, j1, o);
  j1 *= 0.5;
  if (lane == 0) eps[e] = j1 == 0.0 ? 0.0 : 1.0 - jp / j1;
}

// ------------------------------------------------------------------------------------ selection
// k-th smallest (0-based) composite key (order_key(v_i), i) among the items that take part, found by
// radix selection over the 64-bit key (8 passes of 8 bits) and then the index among equal keys.
// Up to two ranks of the same values are selected together; the last block of a pass to finish
// picks the digits (a scan over the 256 counters), so a selection is 9 launches with nothing between
// them.  State of target t: st[2 t] the prefix, st[2 t + 1] the rank remaining.
__device__ __forceinline__ bool participates(int mode, double v) {
  return mode == 0 ? true : mode == 1 ? (v < 0.0) : (v > 0.0);
}

// inclusive scan over the 256 threads of a block
__device__ __forceinline__ unsigned scan256(unsigned v, unsigned* ws) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  if (lane == 31) ws[w] = v;
  __syncthreads();
  unsigned add = 0;
  for (int k = 0; k < w; ++k) add += ws[k];
  __syncthreads();
  return v + add;
}

struct SelRanks {
  unsigned long long k[2];
};

// the counters hist [2][256] and cnt are zero between launches
__global__ void __launch_bounds__(256) sel_pass_kernel(int64_t n, const double* __restrict__ v, int mode, int nt,
                                                       SelRanks ranks, int shift, unsigned long long* __restrict__ st,
                                                       unsigned* __restrict__ hist, unsigned* __restrict__ cnt) {
  __shared__ unsigned hs[2][256], ws[8];
  __shared__ int last;
  const int t = threadIdx.x;
  hs[0][t] = hs[1][t] = 0;
  __syncthreads();
  const unsigned long long himask = shift >= 56 ? 0ULL : (~0ULL << (shift + 8));
  const unsigned long long p0 = shift >= 56 ? 0ULL : st[0], p1 = shift >= 56 ? 0ULL : st[2];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + t; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const double x = v[i];
    if (!participates(mode, x)) continue;
    const unsigned long long key = order_key(x);
    const unsigned d = (unsigned)(key >> shift) & 255u;
    if ((key & himask) == p0) atomicAdd(&hs[0][d], 1u);
    if (nt > 1 && (key & himask) == p1) atomicAdd(&hs[1][d], 1u);
  }
  __syncthreads();
  for (int q = 0; q < nt; ++q)
    if (hs[q][t]) atomicAdd(&hist[256 * q + t], hs[q][t]);
  __threadfence();
  __syncthreads();
  if (t == 0) last = atomicAdd(cnt, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int q = 0; q < nt; ++q) {
    const unsigned c = __ldcg(hist + 256 * q + t);
    hist[256 * q + t] = 0;
    const unsigned inc = scan256(c, ws);
    const unsigned long long r = shift >= 56 ? ranks.k[q] : st[2 * q + 1];
    const unsigned long long pre = shift >= 56 ? 0ULL : st[2 * q];
    __syncthreads();
    // the first digit whose inclusive count exceeds the rank (the last one for a rank beyond the count)
    if ((inc - c <= r && r < inc) || (t == 255 && r >= inc)) {
      st[2 * q] = pre | ((unsigned long long)t << shift);
      st[2 * q + 1] = r - (inc - c);
    }
  }
  if (t == 0) *cnt = 0u;
}

// the index of the item of remaining rank among those equal to the selected key, and the result
// (key, index) to out[2 q], out[2 q + 1].  part: [2][gridDim.x] counts per block (a block takes
// consecutive items).
__global__ void __launch_bounds__(256) sel_index_kernel(int64_t n, const double* __restrict__ v, int mode, int nt,
                                                        const unsigned long long* __restrict__ st,
                                                        unsigned* __restrict__ part, unsigned* __restrict__ cnt,
                                                        unsigned long long* __restrict__ out0,
                                                        unsigned long long* __restrict__ out1) {
  __shared__ unsigned ws[8];
  __shared__ int last, s_block;
  __shared__ unsigned long long s_rank, s_idx;
  const int t = threadIdx.x;
  const int64_t per = (n + gridDim.x - 1) / gridDim.x;
  auto match = [&](int64_t i, unsigned long long key) {
    const double x = v[i];
    return participates(mode, x) && order_key(x) == key;
  };
  for (int q = 0; q < nt; ++q) {
    const unsigned long long key = st[2 * q];
    unsigned c = 0;
    for (int64_t i = blockIdx.x * per + t; i < n && i < (blockIdx.x + 1) * per; i += 256) c += match(i, key);
    const unsigned tot = scan256(c, ws);
    if (t == 255) part[q * gridDim.x + blockIdx.x] = tot;
  }
  __threadfence();
  __syncthreads();
  if (t == 0) last = atomicAdd(cnt, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int q = 0; q < nt; ++q) {
    const unsigned long long key = st[2 * q];
    if (t == 0) {
      s_block = -1;
      s_idx = ~0ULL;
    }
    __syncthreads();
    // gridDim.x <= 256: one block's count per thread
    const unsigned c = t < (int)gridDim.x ? __ldcg(part + q * gridDim.x + t) : 0u;
    const unsigned inc = scan256(c, ws);
    const unsigned long long r = st[2 * q + 1];
    if (inc - c <= r && r < inc) {
      s_block = t;
      s_rank = r - (inc - c);
    }
    __syncthreads();
    if (s_block >= 0) {
      unsigned long long rank = s_rank;
      const int64_t end = min(n, (s_block + 1) * per);
      for (int64_t i0 = s_block * per; i0 < end; i0 += 256) {
        const int64_t i = i0 + t;
        const unsigned m = i < end && match(i, key);
        const unsigned im = scan256(m, ws);
        if (m && im - 1 == rank) s_idx = (unsigned long long)i;
        __syncthreads();
        if (s_idx != ~0ULL) break;
        if (t == 255) s_rank = rank - im;   // not among these: the total of this piece comes off
        __syncthreads();
        rank = s_rank;
      }
    }
    __syncthreads();
    if (t == 0) {
      unsigned long long* out = q ? out1 : out0;
      out[0] = key;
      out[1] = s_idx;
    }
    __syncthreads();
  }
  if (t == 0) *cnt = 0u;
}

__device__ __forceinline__ bool comp_less(double v, int64_t i, unsigned long long key, unsigned long long idx) {
  unsigned long long k = order_key(v);
  return k < key || (k == key && (unsigned long long)i < idx);
}

__global__ void count_sign_kernel(int64_t n, const double* __restrict__ v, unsigned long long* __restrict__ out) {
  unsigned long long neg = 0, pos = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    neg += v[i] < 0.0;
    pos += v[i] > 0.0;
  }
  atomicAdd(&out[0], neg);
  atomicAdd(&out[1], pos);
}

// Analysis (step 2), density (step 3c) and the flags.  thr: [0..3] analysis coarsen threshold
// (key, idx) and whether it applies, analysis refine threshold; [..] density thresholds.
struct Thresholds {
  unsigned long long ac_key, ac_idx, ar_key, ar_idx, dc_key, dc_idx, dr_key, dr_idx;
  int ac_mode, ar_mode, dc_mode, dr_mode;   // 0 none, 1 all, 2 threshold
};

__device__ __forceinline__ bool in_low(int mode, double v, int64_t i, unsigned long long k, unsigned long long x) {
  return mode == 1 || (mode == 2 && comp_less(v, i, k, x));
}
__device__ __forceinline__ bool in_high(int mode, double v, int64_t i, unsigned long long k, unsigned long long x) {
  return mode == 1 || (mode == 2 && !comp_less(v, i, k, x));
}

__global__ void flags_kernel(int64_t nel, const int* __restrict__ p_in, const double* __restrict__ ga,
                             const double* __restrict__ gd, const unsigned long long* __restrict__ selbuf,
                             Thresholds th, int p_max, int* __restrict__ p_out, int* __restrict__ theta_out) {
  // thresholds computed on the device live in selbuf: [0..1] analysis coarsen, [2..3] analysis
  // refine, [4..5] density coarsen, [6..7] density refine (key, index)
  if (th.ac_mode == 2) { th.ac_key = selbuf[0]; th.ac_idx = selbuf[1]; }
  if (th.ar_mode == 2) { th.ar_key = selbuf[2]; th.ar_idx = selbuf[3]; }
  if (th.dc_mode == 2) { th.dc_key = selbuf[4]; th.dc_idx = selbuf[5]; }
  if (th.dr_mode == 2) { th.dr_key = selbuf[6]; th.dr_idx = selbuf[7]; }
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nel; e += (int64_t)gridDim.x * blockDim.x) {
    int p = p_in[e], t = 0;
    if (in_low(th.ac_mode, ga[e], e, th.ac_key, th.ac_idx)) { t = -1; p = p > 1 ? p - 1 : 1; }
    if (in_high(th.ar_mode, ga[e], e, th.ar_key, th.ar_idx)) { t = 1; p = p + 1 < p_max ? p + 1 : p_max; }
    const double g = gd[e];
    if (g < 0.0 && in_low(th.dc_mode, g, e, th.dc_key, th.dc_idx)) {
      if (p == 1) t = -2;
      else if (t == 0) p -= 1;
    }
    if (g > 0.0 && in_high(th.dr_mode, g, e, th.dr_key, th.dr_idx) && (t == 0 || t == -1))
      p = p + 1 < p_max ? p + 1 : p_max;
    p_out[e] = p;
    theta_out[e] = t;
  }
}

// one Jacobi sweep of p_k <- max(p_k, max_{edge neighbours} p_j - 2)
__global__ void smooth_kernel(int nelx, int nely, const int* __restrict__ a, int* __restrict__ b) {
  const int64_t nel = (int64_t)nelx * nely;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nel; e += (int64_t)gridDim.x * blockDim.x) {
    int ix = (int)(e % nelx), iy = (int)(e / nelx);
    int m = a[e];
    int nb = -1000;
    if (ix > 0) nb = max(nb, a[e - 1]);
    if (ix + 1 < nelx) nb = max(nb, a[e + 1]);
    if (iy > 0) nb = max(nb, a[e - nelx]);
    if (iy + 1 < nely) nb = max(nb, a[e + nelx]);
    b[e] = max(m, nb - 2);
  }
}

__device__ int isqrt_dev(int v) {
  int r = 0;
  while ((r + 1) * (r + 1) <= v) ++r;
  return r;
}

__global__ void final_kernel(int64_t nel, const int* __restrict__ p_s, const int* __restrict__ theta,
                             const double* __restrict__ eqr, double alpha_qr, int p_max, int d_max,
                             int32_t* __restrict__ p_new, int32_t* __restrict__ d_new, int8_t* __restrict__ th_out) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nel; e += (int64_t)gridDim.x * blockDim.x) {
    int p = p_s[e], t = theta[e];
    int nd = 2 * (p + 1) * (p + 1) - 3;
    if (nd > d_max) nd = d_max;
    int d = t == -2 ? 1 : isqrt_dev(nd);
    if (eqr[e] > alpha_qr) p = p + 1 < p_max ? p + 1 : p_max;
    p_new[e] = p;
    d_new[e] = d;
    th_out[e] = (int8_t)t;
  }
}

// ------------------------------------------------------------------------------------ OC
// rho_new_j = clip(rho_j (B_j / lambda)^eta, max(0, rho_j - m), min(1, rho_j + m)), B_j = -dc_j / dv_j,
// written as t_j c with t_j = rho_j B_j^eta formed once and c = lambda^-eta.  The volume of a trial
// lambda is sum_j dv_j clip(t_j c, lo_j, hi_j) = sum_j clip(T_j c, L_j, H_j) with T, L, H the values
// scaled by their subcell's area (dv > 0 commutes with the clip).  The clip is taken on the integer
// pipes (non-negative doubles order like their bit patterns).
//
// The bisection on [0, 1e9] visits the same midpoints and ends in the same interval as a loop that sums
// every value at every midpoint (about 64 passes over all values; 7.8 ms for 8.4 million values, now
// 1.5 ms), but does not look at every value each time:
//  - while the lower end is 0 the midpoints are 1e9 2^-k, and the volume falls as lambda grows, so the
//    first k whose volume exceeds the target is searched for, from a guess on a sample of the values: a
//    pass at the guess and one at its neighbour where the guess holds (at most ten);
//  - from then on the interval is [l, 2 l], and a value whose clip is settled over the whole interval
//    (at L, at H, or T c throughout) only adds to a constant or to the slope.  Each block keeps the
//    values of its own segment that are not settled yet, compacted in order, so a pass reads about half
//    of the one before.
// All sums are taken in a fixed order, and the last block of a launch takes the step, so the whole update
// is a chain of launches with no host round trips.  Small designs run in one block.
constexpr int kOCBlock = 256;
constexpr int kOCSmall = 4096;      // values of the one-block path (above, its 42 rounds on one SM's FP64 pipes cost
                                    // more than the launches)
constexpr int kOCSample = 8192;
constexpr int kOCMaxIt = 128;       // bisection steps in all, as in a plain loop
constexpr int kOCLocate = 10;       // passes that find k: the guess, its neighbour, 7 halvings of 1..129
constexpr int kOCSteps = 34;        // halvings from [l, 2 l] to a relative width of 1e-10

struct OCState {
  int lo, hi;         // largest k known not to exceed the target (0: none), smallest known to (129: none)
  int cand, tries;
  int its, done;
  double l1, l2;
  double c1, c2, cm;  // lambda^-eta at l1, l2 and the midpoint
};

__device__ __forceinline__ double oc_pow(double x, double eta) { return eta == 0.5 ? sqrt(x) : pow(x, eta); }
__device__ __forceinline__ double oc_c(double lam, double eta) { return eta == 0.5 ? 1.0 / sqrt(lam) : pow(lam, -eta); }
__device__ __forceinline__ double oc_mid(int k) { return ldexp(1e9, -k); }   // exact halvings

// clip(x, lo, hi) for non-negative lo <= hi (x >= 0 or -0) by signed 64-bit compares of the bits
__device__ __forceinline__ double clip_nonneg(double x, double lo, double hi) {
  long long xi = __double_as_longlong(x);
  const long long li = __double_as_longlong(lo), hi_ = __double_as_longlong(hi);
  xi = xi > li ? xi : li;
  xi = xi < hi_ ? xi : hi_;
  return __longlong_as_double(xi);
}

// block-wide sum (fixed order), valid in thread 0
template <int BLOCK>
__device__ __forceinline__ double oc_block_sum(double v, double* ws) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = v;
  __syncthreads();
  double b = 0.0;
  if (threadIdx.x < 32) {
    b = threadIdx.x < BLOCK / 32 ? ws[threadIdx.x] : 0.0;
    for (int o = BLOCK / 64; o > 0; o >>= 1) b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  return b;
}

// the next k to look at, or the interval once k is known
__device__ void oc_located(OCState* st, int k, bool over, double eta) {
  if (over) st->hi = k;
  else st->lo = k;
  st->tries++;
  if (st->hi == st->lo + 1) {
    st->its = min(st->hi, kOCMaxIt);
    st->l1 = st->hi <= kOCMaxIt ? oc_mid(st->hi) : 0.0;
    st->l2 = oc_mid(st->lo);
    st->done = st->its >= kOCMaxIt;
    st->c1 = oc_c(st->l1, eta);
    st->c2 = oc_c(st->l2, eta);
    st->cm = oc_c(0.5 * (st->l1 + st->l2), eta);
  } else if (st->tries == 1) {
    st->cand = over ? k - 1 : k + 1;
  } else {
    st->cand = (st->lo + st->hi) / 2;
  }
}

// one bisection step with the volume at the midpoint
__device__ void oc_step(OCState* st, bool over, double eta, double tol) {
  const double mid = 0.5 * (st->l1 + st->l2);
  if (over) {
    st->l1 = mid;
    st->c1 = st->cm;
  } else {
    st->l2 = mid;
    st->c2 = st->cm;
  }
  st->its++;
  if ((st->l2 - st->l1) / (st->l1 + st->l2) <= tol || st->its >= kOCMaxIt) st->done = 1;
  st->cm = oc_c(0.5 * (st->l1 + st->l2), eta);
}

// t_j, and the area-scaled T_j = dv t_j, L_j = dv max(0, rho_j - m), H_j = dv min(1, rho_j + m)
__global__ void __launch_bounds__(kOCBlock) oc_prep_kernel(int64_t nel, const int64_t* __restrict__ off,
                                                           const int* __restrict__ dmap, double hx, double hy,
                                                           const double* __restrict__ rho,
                                                           const double* __restrict__ dc, double move, double eta,
                                                           double* __restrict__ t, double* __restrict__ T,
                                                           double* __restrict__ Lo, double* __restrict__ Hi) {
  const int lane = threadIdx.x & 31;
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  double dv = 0.0, inv = 0.0;
  int dlast = 0;
  bool exact = false;
  for (int64_t e = w0; e < nel; e += nw) {
    const int d = dmap[e];
    if (d != dlast) {
      dlast = d;
      dv = hx * hy / ((double)d * d);
      inv = 1.0 / dv;
      // a power of two divides exactly as a product
      exact = (__double_as_longlong(dv) & 0xfffffffffffffll) == 0;
    }
    for (int64_t j = off[e] + lane; j < off[e + 1]; j += 32) {
      const double r = rho[j];
      const double g = fmax(-dc[j], 0.0);
      const double tj = r * oc_pow(exact ? g * inv : g / dv, eta);
      t[j] = tj;
      T[j] = dv * tj;
      Lo[j] = dv * fmax(0.0, r - move);
      Hi[j] = dv * fmin(1.0, r + move);
    }
  }
}

// a guess of k from every (n / kOCSample)-th value, taken for as many of the others (one block)
__global__ void __launch_bounds__(1024) oc_guess_kernel(int64_t n, const double* __restrict__ T,
                                                        const double* __restrict__ Lo, const double* __restrict__ Hi,
                                                        double eta, double target, OCState* __restrict__ st) {
  __shared__ double ws[32], ck[kOCMaxIt + 1];
  __shared__ int over;
  if (threadIdx.x <= kOCMaxIt) ck[threadIdx.x] = oc_c(oc_mid(threadIdx.x), eta);
  const int64_t stride = (n + kOCSample - 1) / kOCSample, ns = (n + stride - 1) / stride;
  constexpr int PER = kOCSample / 1024;
  double tv[PER], lv[PER], hv[PER];
#pragma unroll
  for (int k = 0; k < PER; ++k) {
    const int64_t i = threadIdx.x + 1024 * k;
    tv[k] = lv[k] = hv[k] = 0.0;
    if (i < ns) {
      tv[k] = T[i * stride];
      lv[k] = Lo[i * stride];
      hv[k] = Hi[i * stride];
    }
  }
  int lo = 0, hi = kOCMaxIt + 1;
  while (hi > lo + 1) {
    __syncthreads();
    const int k = (lo + hi) / 2;
    const double c = ck[k];
    double s = 0.0;
#pragma unroll
    for (int j = 0; j < PER; ++j) s += clip_nonneg(tv[j] * c, lv[j], hv[j]);
    s = oc_block_sum<1024>(s, ws);
    if (threadIdx.x == 0) over = s * ((double)n / (double)ns) > target;
    __syncthreads();
    if (over) hi = k;
    else lo = k;
  }
  if (threadIdx.x == 0) {
    st->lo = 0;
    st->hi = kOCMaxIt + 1;
    st->cand = min(max(hi, 1), kOCMaxIt);
    st->tries = st->its = st->done = 0;
  }
}

// the volume at 1e9 2^-cand over all values
__global__ void __launch_bounds__(kOCBlock) oc_locate_kernel(int64_t n, const double* __restrict__ T,
                                                             const double* __restrict__ Lo,
                                                             const double* __restrict__ Hi, double eta, double target,
                                                             OCState* __restrict__ st, double* __restrict__ part,
                                                             unsigned* __restrict__ cnt) {
  if (st->hi == st->lo + 1) return;
  __shared__ double ws[kOCBlock / 32];
  __shared__ int last;
  __shared__ double s_c;
  const int k = st->cand;
  if (threadIdx.x == 0) s_c = oc_c(oc_mid(k), eta);
  __syncthreads();
  const double c = s_c;
  double s = 0.0;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x)
    s += clip_nonneg(T[j] * c, Lo[j], Hi[j]);
  s = oc_block_sum<kOCBlock>(s, ws);
  if (threadIdx.x == 0) {
    part[blockIdx.x] = s;
    __threadfence();
    last = atomicAdd(cnt, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double tot = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += kOCBlock) tot += __ldcg(part + i);
  tot = oc_block_sum<kOCBlock>(tot, ws);
  if (threadIdx.x == 0) {
    oc_located(st, k, tot > target, eta);
    *cnt = 0u;
  }
}

// One bisection step from [l1, l2], l1 > 0.  Block b holds seg consecutive places of T, Lo, Hi; the first
// cnt_b of them are its unsettled values (first: all of them), with acc[b], acc[G + b] the constant and the
// slope of the settled ones.  part: [2][gridDim.x].
__global__ void __launch_bounds__(kOCBlock) oc_pass_kernel(int64_t n, int seg, int first, double* __restrict__ T,
                                                           double* __restrict__ Lo, double* __restrict__ Hi,
                                                           double eta, double target, double tol,
                                                           OCState* __restrict__ st, int* __restrict__ left,
                                                           double* __restrict__ acc, double* __restrict__ part,
                                                           unsigned* __restrict__ cnt) {
  if (st->done) return;
  __shared__ double ws[kOCBlock / 32];
  __shared__ int wc[kOCBlock / 32];
  __shared__ int last;
  const int G = gridDim.x, b = blockIdx.x, t = threadIdx.x, lane = t & 31, w = t >> 5;
  const double c1 = st->c1, c2 = st->c2, cm = st->cm;
  const int64_t base = (int64_t)b * seg;
  const int cntb = first ? (int)max((int64_t)0, min((int64_t)seg, n - base)) : left[b];
  double sc = 0.0, sl = 0.0, su = 0.0;
  int out = 0;
  for (int i0 = 0; i0 < cntb; i0 += kOCBlock) {
    const int i = i0 + t;
    bool keep = false;
    double tv = 0.0, lv = 0.0, hv = 0.0;
    if (i < cntb) {
      tv = T[base + i];
      lv = Lo[base + i];
      hv = Hi[base + i];
      const long long lb = __double_as_longlong(lv), hb = __double_as_longlong(hv);
      const long long a = __double_as_longlong(tv * c2), z = __double_as_longlong(tv * c1);   // least and largest T c
      if (a >= hb || lb >= hb) sc += hv;   // lb > hb (a density outside [0, 1]): the clip gives H
      else if (z <= lb) sc += lv;
      else if (a >= lb && z <= hb) sl += tv;
      else {
        keep = true;
        su += clip_nonneg(tv * cm, lv, hv);
      }
    }
    // compact in order: the places written lie at or before those read so far
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) wc[w] = __popc(m);
    __syncthreads();   // also: every value of this piece has been read
    int at = out + __popc(m & ((1u << lane) - 1u)), tot = 0;
    for (int k = 0; k < kOCBlock / 32; ++k) {
      if (k < w) at += wc[k];
      tot += wc[k];
    }
    if (keep && at != i) {
      T[base + at] = tv;
      Lo[base + at] = lv;
      Hi[base + at] = hv;
    }
    out += tot;
    __syncthreads();
  }
  sc = oc_block_sum<kOCBlock>(sc, ws);
  sl = oc_block_sum<kOCBlock>(sl, ws);
  su = oc_block_sum<kOCBlock>(su, ws);
  if (t == 0) {
    const double C = (first ? 0.0 : acc[b]) + sc, S = (first ? 0.0 : acc[G + b]) + sl;
    acc[b] = C;
    acc[G + b] = S;
    left[b] = out;
    part[b] = C + su;
    part[G + b] = S;
    __threadfence();
    last = atomicAdd(cnt, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double tc = 0.0, ts = 0.0;
  for (int i = t; i < G; i += kOCBlock) {
    tc += __ldcg(part + i);
    ts += __ldcg(part + G + i);
  }
  tc = oc_block_sum<kOCBlock>(tc, ws);
  ts = oc_block_sum<kOCBlock>(ts, ws);
  if (t == 0) {
    oc_step(st, fma(ts, cm, tc) > target, eta, tol);
    *cnt = 0u;
  }
}

// the whole bisection of at most kOCSmall values in one block
__global__ void __launch_bounds__(1024) oc_small_kernel(int n, const double* __restrict__ T,
                                                        const double* __restrict__ Lo, const double* __restrict__ Hi,
                                                        double eta, double target, double tol,
                                                        OCState* __restrict__ st_out) {
  extern __shared__ double osm[];
  __shared__ double ws[32], s_c;
  __shared__ OCState st;
  double *Ts = osm, *Ls = osm + n, *Hs = osm + 2 * n;
  for (int j = threadIdx.x; j < n; j += 1024) {
    Ts[j] = T[j];
    Ls[j] = Lo[j];
    Hs[j] = Hi[j];
  }
  if (threadIdx.x == 0) {
    st.lo = 0;
    st.hi = kOCMaxIt + 1;
    st.cand = (kOCMaxIt + 1) / 2;
    st.tries = 1;
    st.its = st.done = 0;
  }
  __syncthreads();
  while (!st.done) {   // at most 8 + 34 rounds
    const bool locate = st.hi != st.lo + 1;
    const int k = st.cand;
    if (threadIdx.x == 0) s_c = locate ? oc_c(oc_mid(k), eta) : st.cm;
    __syncthreads();
    const double c = s_c;
    double s = 0.0;
    for (int j = threadIdx.x; j < n; j += 1024) s += clip_nonneg(Ts[j] * c, Ls[j], Hs[j]);
    s = oc_block_sum<1024>(s, ws);
    if (threadIdx.x == 0) {
      if (locate) oc_located(&st, k, s > target, eta);
      else oc_step(&st, s > target, eta, tol);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) *st_out = st;
}

__global__ void __launch_bounds__(kOCBlock) oc_write_kernel(int64_t n, const double* __restrict__ rho,
                                                            const double* __restrict__ t, double move, double eta,
                                                            const OCState* __restrict__ st, double* __restrict__ out) {
  __shared__ double s_c;
  if (threadIdx.x == 0) s_c = oc_c(0.5 * (st->l1 + st->l2), eta);
  __syncthreads();
  const double c = s_c;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n; j += (int64_t)gridDim.x * blockDim.x) {
    const double r = rho[j];
    out[j] = fmin(fmax(t[j] * c, fmax(0.0, r - move)), fmin(1.0, r + move));
  }
}

// ------------------------------------------------------------------------------------ host side
mto_status ensure_basis(mto_handle h, BasisTab** out) {
  if (!h->basis_tab) {
    MTO_TRY(mto_alloc(h, reinterpret_cast<unsigned char**>(&h->basis_tab), sizeof(BasisTab)));
    basis_table_kernel<<<1, 256, 0, h->stream>>>(reinterpret_cast<BasisTab*>(h->basis_tab));
    MTO_TRY(mto_after_launch(h, "basis_table_kernel"));
  }
  *out = reinterpret_cast<BasisTab*>(h->basis_tab);
  return MTO_OK;
}

// Selection of the items of ranks k[0 .. nt) among the participating values; each (key, index) pair
// to out[q][0..1] (device).
mto_status select_kth(mto_handle h, const double* v, int64_t n, int mode, int nt, const SelRanks& k,
                      unsigned long long* out0, unsigned long long* out1) {
  unsigned long long* st = h->sel + 32;
  unsigned* cnt = reinterpret_cast<unsigned*>(h->sel + 48);
  unsigned* hist = reinterpret_cast<unsigned*>(h->sel + 64);   // [2][256]
  const int grd = grid_for(n, 1024, 152 * 2);
  for (int shift = 56; shift >= 0; shift -= 8) {
    sel_pass_kernel<<<grd, 256, 0, h->stream>>>(n, v, mode, nt, k, shift, st, hist, cnt);
    MTO_TRY(mto_after_launch(h, "sel_pass_kernel"));
  }
  sel_index_kernel<<<grid_for(n, 1024, 256), 256, 0, h->stream>>>(n, v, mode, nt, st, hist + 512, cnt, out0, out1);
  return mto_after_launch(h, "sel_index_kernel");
}

}  // namespace

mto_status map_update(mto_handle h, const double* ga, const double* gd, const double* eqr,
                      const mto_indicator_opts* o, int32_t* pn, int32_t* dn, int8_t* th) {
  const int64_t nel = h->nel;
  const int grd = grid_for(nel, 256, 152 * 4);
  unsigned long long* selbuf = h->sel + 8;         // 8 values: the four (key, index) thresholds
  Thresholds T;
  memset(&T, 0, sizeof(T));
  // analysis step: floor(frac * nel) lowest / highest Gamma^a
  const int64_t nc = (int64_t)std::floor(o->frac_a_coarsen * (double)nel);
  const int64_t nr = (int64_t)std::floor(o->frac_a_refine * (double)nel);
  T.ac_mode = nc >= nel ? 1 : nc > 0 ? 2 : 0;
  T.ar_mode = nr >= nel ? 1 : nr > 0 ? 2 : 0;
  if (T.ac_mode == 2 && T.ar_mode == 2)
    MTO_TRY(select_kth(h, ga, nel, 0, 2, SelRanks{{(unsigned long long)nc, (unsigned long long)(nel - nr)}}, selbuf + 0,
                       selbuf + 2));
  else if (T.ac_mode == 2)
    MTO_TRY(select_kth(h, ga, nel, 0, 1, SelRanks{{(unsigned long long)nc, 0}}, selbuf + 0, nullptr));
  else if (T.ar_mode == 2)
    MTO_TRY(select_kth(h, ga, nel, 0, 1, SelRanks{{(unsigned long long)(nel - nr), 0}}, selbuf + 2, nullptr));
  // density step: fractions of the negative / positive Gamma^d elements
  if (o->alpha_d_coarsen >= 1.0) T.dc_mode = 1;
  if (o->alpha_d_refine >= 1.0) T.dr_mode = 1;
  if (T.dc_mode == 0 || T.dr_mode == 0) {
    unsigned long long* cnt = h->sel + 18;
    MTO_TRY(mto_cuda_check(h, cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), h->stream), "memset"));
    count_sign_kernel<<<grd, 256, 0, h->stream>>>(nel, gd, cnt);
    MTO_TRY(mto_after_launch(h, "count_sign_kernel"));
    unsigned long long hc[2];
    MTO_TRY(mto_cuda_check(h, cudaMemcpyAsync(hc, cnt, sizeof(hc), cudaMemcpyDeviceToHost, h->stream), "copy"));
    MTO_TRY(mto_cuda_check(h, cudaStreamSynchronize(h->stream), "sync"));
    MTO_TRY(tc_check(h, TC_INDICATOR));
    const int64_t nneg = (int64_t)hc[0], npos = (int64_t)hc[1];
    if (T.dc_mode == 0) {
      const int64_t kc = (int64_t)std::floor(o->alpha_d_coarsen * (double)nneg);
      if (kc >= nneg) T.dc_mode = 1;
      else if (kc > 0) {
        T.dc_mode = 2;
        MTO_TRY(select_kth(h, gd, nel, 1, 1, SelRanks{{(unsigned long long)kc, 0}}, selbuf + 4, nullptr));
      }
    }
    if (T.dr_mode == 0) {
      const int64_t kr = (int64_t)std::floor(o->alpha_d_refine * (double)npos);
      if (kr >= npos) T.dr_mode = 1;
      else if (kr > 0) {
        T.dr_mode = 2;
        MTO_TRY(select_kth(h, gd, nel, 2, 1, SelRanks{{(unsigned long long)(npos - kr), 0}}, selbuf + 6, nullptr));
      }
    }
  }
  int* pa = h->ibuf;
  int* pb = h->ibuf + nel;
  int* tt = h->ibuf + 2 * nel;
  flags_kernel<<<grd, 256, 0, h->stream>>>(nel, h->p_d, ga, gd, selbuf, T, o->p_max, pa, tt);
  MTO_TRY(mto_after_launch(h, "flags_kernel"));
  for (int s = 0; s < MTO_P_MAX; ++s) {
    smooth_kernel<<<grd, 256, 0, h->stream>>>(h->nelx, h->nely, pa, pb);
    MTO_TRY(mto_after_launch(h, "smooth_kernel"));
    int* tmp = pa; pa = pb; pb = tmp;
  }
  final_kernel<<<grd, 256, 0, h->stream>>>(nel, pa, tt, eqr, o->alpha_qr, o->p_max, o->d_max, pn, dn, th);
  return mto_after_launch(h, "final_kernel");
}

mto_status indicators(mto_handle h, const double* u, const double* rho, const mto_material* m,
                      const mto_indicator_opts* o, double* ga, double* gd, double* eqr, int32_t* pn, int32_t* dn,
                      int8_t* th) {
  TimedScope ts(h, F_INDICATOR);
  const int64_t nel = h->nel;
  BasisTab* B;
  MTO_TRY(ensure_basis(h, &B));
  // outputs the caller did not ask for go to scratch
  double* ga_ = ga ? ga : h->dbuf;
  double* gd_ = gd ? gd : h->dbuf + nel;
  double* eq_ = eqr ? eqr : h->edge_buf + (h->n_edges);     // after the edge values
  ClassPtrs cp;
  for (int p = 0; p <= kPMaxTab; ++p) {
    cp.gmap[p] = p <= MTO_P_MAX ? h->pc[p].gmap : nullptr;
  }
  // Kelly
  kelly_edge_kernel<<<grid_for(h->n_edges, 128, 152 * 64), 128, 0, h->stream>>>(
      h->nelx, h->nely, h->p_d, h->slot_d, cp, h->cons_d, u, B, h->hx, h->hy, h->edge_buf);
  MTO_TRY(mto_after_launch(h, "kelly_edge_kernel"));
  kelly_sum_kernel<<<grid_for(nel, 256), 256, 0, h->stream>>>(h->nelx, h->nely, h->edge_buf, ga_);
  MTO_TRY(mto_after_launch(h, "kelly_sum_kernel"));
  // density indicator
  unsigned long long* mm = h->sel + 16;
  MTO_TRY(mto_cuda_check(h, cudaMemsetAsync(mm, 0xff, sizeof(*mm), h->stream), "memset"));
  MTO_TRY(mto_cuda_check(h, cudaMemsetAsync(mm + 1, 0, sizeof(*mm), h->stream), "memset"));
  minmax_kernel<<<grid_for(h->design_len, 1024, 152 * 4), 256, 0, h->stream>>>(h->design_len, rho, mm);
  MTO_TRY(mto_after_launch(h, "minmax_kernel"));
  gamma_d_kernel<<<grid_for(nel, 32 * kGdWarps, 152 * 6), 32 * kGdWarps, 0, h->stream>>>(
      nel, h->design_off_d, rho, mm, o->cycle, o->alpha, o->beta, gd_);
  MTO_TRY(mto_after_launch(h, "gamma_d_kernel"));
  ++h->tc_tag[TC_INDICATOR];
  // QR error per (p, d) class, in chunks of elements whose rows fit 448 MB, full waves of the row
  // kernel (128 elements per SM) where a chunk is that large (38,912 elements of Q3)
  for (size_t ci = 0; ci < h->bc.size(); ++ci) {
    const BClass& b = h->bc[ci];
    const BClass& b1 = h->bc_qr[ci];
    const PClass& c = h->pc[b.p];
    const int L1 = qr_row_len(b.p + 1);
    bool tc = h->build_path == MTO_BUILD_TENSOR && b1.tcB;
    const size_t smem = qr_smem_bytes(b.p, b.S);
    MTO_TRY(allow_smem(h, qr_kernel, qr_smem_bytes(MTO_P_MAX, MTO_D_MAX * MTO_D_MAX)));
    int chunk = b.n;
    if (tc) {
      const int wave = 152 * 128;
      const int most = (int)(((size_t)448 << 20) / (sizeof(double) * L1));
      chunk = std::min(b.n, most >= wave ? most / wave * wave : most / 128 * 128);
      if ((size_t)chunk * L1 > h->qr_cap) {
        if (h->qr_rows) {
          MTO_TRY(mto_cuda_check(h, cudaStreamSynchronize(h->stream), "sync"));
          cudaFree(h->qr_rows);
          h->qr_rows = nullptr;
          h->bytes -= (int64_t)(h->qr_cap * sizeof(double));
          h->qr_cap = 0;
        }
        // where the device has not that much left: smaller chunks, or the sums in the kernel
        while (mto_alloc(h, &h->qr_rows, (size_t)chunk * L1) != MTO_OK && chunk > 128)
          chunk = (chunk / 2 + 127) / 128 * 128;
        if (h->qr_rows) h->qr_cap = (size_t)chunk * L1;
        else {
          tc = false;
          chunk = b.n;
        }
        cudaGetLastError();
        h->err.clear();
      }
    }
    for (int first = 0; first < b.n; first += chunk) {
      const int cn = std::min(chunk, b.n - first);
      if (tc) MTO_TRY(tc_rows(h, b, b1, L1, first, cn, nullptr, rho, m, h->qr_rows, nullptr, nullptr,
                              TC_INDICATOR));
      qr_kernel<<<cn, 32, smem, h->stream>>>(b.p, b.d, b.n, first, b.elem, b.slot, c.L, c.gmap, h->cons_d, c.K64,
                                             tc ? h->qr_rows : nullptr, b1.K0T, h->qr[b.p].R, u, rho,
                                             h->design_off_d, m->E0, m->Emin, m->q, B, h->hx, h->hy, eq_);
      MTO_TRY(mto_after_launch(h, "qr_kernel"));
    }
  }
  if (!pn && !dn && !th) return MTO_OK;
  if (!pn || !dn || !th) return mto_fail(h, MTO_EINVAL, "mto_indicator: p_new, d_new and theta go together");
  return map_update(h, ga_, gd_, eq_, o, pn, dn, th);
}

mto_status oc_update(mto_handle h, const double* rho, const double* dc, double volfrac, double move, double eta,
                     double* rho_new, double* lambda) {
  TimedScope ts(h, F_OC);
  const int64_t nel = h->nel;
  const int64_t n = h->design_len;
  if (!h->oc_t) MTO_TRY(mto_alloc(h, &h->oc_t, (size_t)4 * n));   // t, T, L, H
  double* T = h->oc_t + n;
  double* Lo = T + n;
  double* Hi = Lo + n;
  // segments of at least 1024 values, at most one full wave of blocks
  const int seg = (int)std::max<int64_t>(1024, (n + 152 * 8 - 1) / (152 * 8));
  const int grd = (int)((n + seg - 1) / seg);
  if (!h->oc_work) MTO_TRY(mto_alloc(h, &h->oc_work, sizeof(OCState) + (size_t)152 * 8 * (4 * sizeof(double) + sizeof(int)) + 64));
  OCState* st = reinterpret_cast<OCState*>(h->oc_work);
  double* part = reinterpret_cast<double*>(h->oc_work + round_up((int)sizeof(OCState), 16));   // [2][grd]
  double* acc = part + 2 * 152 * 8;                                                            // [2][grd]
  int* left = reinterpret_cast<int*>(acc + 2 * 152 * 8);
  unsigned* cnt = reinterpret_cast<unsigned*>(h->flags + 9);
  MTO_TRY(mto_cuda_check(h, cudaMemsetAsync(cnt, 0, sizeof(int), h->stream), "memset"));
  const double target = volfrac * (double)h->nelx * h->nely * h->hx * h->hy, tol = 1e-10;
  oc_prep_kernel<<<grid_for(nel * 32, kOCBlock, 152 * 8), kOCBlock, 0, h->stream>>>(
      nel, h->design_off_d, h->d_d, h->hx, h->hy, rho, dc, move, eta, h->oc_t, T, Lo, Hi);
  MTO_TRY(mto_after_launch(h, "oc_prep_kernel"));
  if (n <= kOCSmall) {
    const size_t smem = 3 * sizeof(double) * (size_t)n;
    MTO_TRY(allow_smem(h, oc_small_kernel, 3 * sizeof(double) * kOCSmall));
    oc_small_kernel<<<1, 1024, smem, h->stream>>>((int)n, T, Lo, Hi, eta, target, tol, st);
    MTO_TRY(mto_after_launch(h, "oc_small_kernel"));
  } else {
    oc_guess_kernel<<<1, 1024, 0, h->stream>>>(n, T, Lo, Hi, eta, target, st);
    MTO_TRY(mto_after_launch(h, "oc_guess_kernel"));
    for (int it = 0; it < kOCLocate; ++it) {
      oc_locate_kernel<<<grd, kOCBlock, 0, h->stream>>>(n, T, Lo, Hi, eta, target, st, part, cnt);
      MTO_TRY(mto_after_launch(h, "oc_locate_kernel"));
    }
    for (int it = 0; it < kOCSteps; ++it) {
      oc_pass_kernel<<<grd, kOCBlock, 0, h->stream>>>(n, seg, it == 0, T, Lo, Hi, eta, target, tol, st, left, acc, part,
                                                      cnt);
      MTO_TRY(mto_after_launch(h, "oc_pass_kernel"));
    }
  }
  oc_write_kernel<<<grid_for(n, kOCBlock, 152 * 8), kOCBlock, 0, h->stream>>>(n, rho, h->oc_t, move, eta, st, rho_new);
  MTO_TRY(mto_after_launch(h, "oc_write_kernel"));
  if (lambda) {
    MTO_TRY(mto_cuda_check(h, cudaMemcpyAsync(h->host_pinned + 16, &st->l1, 2 * sizeof(double), cudaMemcpyDeviceToHost, h->stream), "copy"));
    MTO_TRY(mto_cuda_check(h, cudaStreamSynchronize(h->stream), "sync"));
    *lambda = 0.5 * (h->host_pinned[16] + h->host_pinned[17]);
  }
  return MTO_OK;
}

}  // namespace mto
