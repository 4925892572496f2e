// The P2 density filter of Sec. 2.1 (Eqs. 4-5) at the subcell centres and its adjoint:
//   rho~_s = sum_t H_st rho_t / W_s,   H_st = R - dist(c_s, c_t) for |c_s - c_t| < R,   W_s = sum_t H_st
//   g_t    = sum_s H_st g~_s / W_s     (the chain rule of the sensitivities)
// over all subcells of the mesh (across element edges), summed in a fixed order.
//
// Between elements of the same design count d the distance of two subcells depends only on their
// offset on the fine grid, so the weights come from one small table per d (one square root per
// offset and call).  A mesh of one d is a plain stencil on its fine grid: one FMA per neighbour, and
// W_s, the same for every subcell whose stencil lies inside the mesh, is summed only near its
// boundary.  On mixed meshes the offsets to neighbours of another count take their square root as
// they are met.  Bound by the FP64 pipes (2 FMA per clock and SM): the divisions and square roots
// per pair, tens of FP64 instructions each, were nearly all of the former time.  320 x 160 elements
// of 4 x 4 subcells, radius 0.6: filter and adjoint 37.5 ms before, 0.17 ms with the tables.
#include <algorithm>
#include <cmath>
#include <vector>

#include "mto_internal.cuh"

namespace mto {
namespace {

// Table of one design count d: the weights H[dj][di] = max(R - dist, 0) of the offsets
// 0 <= di <= kx, 0 <= dj <= ky on the fine grid (row stride kx + 1), per dj the largest di of positive
// weight (-1: none), and the sum over the whole stencil.
struct FilterTab {
  int kx[MTO_D_MAX + 1], ky[MTO_D_MAX + 1];   // largest offsets within R
  int h0[MTO_D_MAX + 1], e0[MTO_D_MAX + 1];   // first entry of d's weights and of its row extents
};

// one block per design count in `mask`
__global__ void __launch_bounds__(256) filter_table_kernel(FilterTab ft, unsigned mask, double hx, double hy, double R,
                                                           double* __restrict__ H, int* __restrict__ ext,
                                                           double* __restrict__ Wfull) {
  const int d = blockIdx.x + 1;
  if (!(mask >> d & 1u)) return;
  const int kx = ft.kx[d], ky = ft.ky[d], n1 = kx + 1;
  double* Hd = H + ft.h0[d];
  __shared__ double ws[8];
  double sum = 0.0;
  for (int k = threadIdx.x; k < n1 * (ky + 1); k += blockDim.x) {
    const int di = k % n1, dj = k / n1;
    const double tx = di * hx / d, ty = dj * hy / d;
    const double dist = sqrt(tx * tx + ty * ty);
    const double w = dist < R ? R - dist : 0.0;
    Hd[k] = w;
    sum += w * ((di ? 2 : 1) * (dj ? 2 : 1));
  }
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if ((threadIdx.x & 31) == 0) ws[threadIdx.x >> 5] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 8; ++w) sum += ws[w];
    // the usual small stencils: in the order of the cells' own sums, whose rounding it then shares
    if ((2 * kx + 1) * (2 * ky + 1) <= 512) {
      sum = 0.0;
      for (int dj = -ky; dj <= ky; ++dj)
        for (int di = -kx; di <= kx; ++di) sum += Hd[abs(dj) * n1 + abs(di)];
    }
    Wfull[d] = sum;
  }
  for (int dj = threadIdx.x; dj <= ky; dj += blockDim.x) {
    int e = -1;
    while (e < kx && Hd[dj * n1 + e + 1] > 0.0) ++e;
    ext[ft.e0[d] + dj] = e;
  }
}

// kScale: y_s = x_s / W_s (the adjoint's first pass); kForward: sum_t H_st x_t / W_s; kSum: sum_s H_st y_s
enum FilterMode { kScale = 0, kForward = 1, kSum = 2 };
constexpr int kFTX = 32, kFTY = 32;   // fine cells per block (256 threads, 4 rows each)

// a mesh of one design count d: a stencil on the (nely d) x (nelx d) grid
template <int MODE>
__global__ void __launch_bounds__(256) filter_uniform_kernel(int nelx, int nely, int d, int kx, int ky,
                                                             const double* __restrict__ H,
                                                             const int* __restrict__ ext,
                                                             const double* __restrict__ Wfull,
                                                             const double* __restrict__ x, double* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char fsm[];
  const int n1 = kx + 1, nh = n1 * (ky + 1);
  double* Hs = reinterpret_cast<double*>(fsm);
  long long* row = reinterpret_cast<long long*>(Hs + nh);       // [kFTY + 2 ky] packed offset of a grid row
  int* col = reinterpret_cast<int*>(row + kFTY + 2 * ky);       // [kFTX + 2 kx] and of a grid column
  int* es = col + kFTX + 2 * kx;                                // [ky + 1]
  const int NX = nelx * d, NY = nely * d;
  const int c0 = blockIdx.x * kFTX, r0 = blockIdx.y * kFTY;
  const int t = threadIdx.x;
  for (int k = t; k < nh; k += 256) Hs[k] = H[k];
  for (int k = t; k <= ky; k += 256) es[k] = ext[k];
  for (int k = t; k < kFTX + 2 * kx; k += 256) {
    const int c = c0 - kx + k;
    col[k] = (c >= 0 && c < NX) ? c / d * d * d + c % d : 0;
  }
  for (int k = t; k < kFTY + 2 * ky; k += 256) {
    const int r = r0 - ky + k;
    row[k] = (r >= 0 && r < NY) ? (long long)(r / d) * nelx * d * d + r % d * d : 0;
  }
  __syncthreads();
  const int c = c0 + (t & 31);
  if (c >= NX) return;
  const int cl = kx + (t & 31);
  for (int rr = t >> 5; rr < kFTY; rr += 8) {
    const int r = r0 + rr;
    if (r >= NY) return;
    const int rl = ky + rr;
    const int j0 = max(-ky, -r), j1 = min(ky, NY - 1 - r);
    double acc = 0.0;
    if (MODE == kScale) {
      acc = x[row[rl] + col[cl]];
    } else {
      for (int dj = j0; dj <= j1; ++dj) {
        const int aj = abs(dj), e = es[aj];
        const double* xr = x + row[rl + dj];
        const double* Hr = Hs + aj * n1;
        const int i0 = max(-e, -c), i1 = min(e, NX - 1 - c);
        for (int di = i0; di <= i1; ++di) acc = fma(Hr[abs(di)], xr[col[cl + di]], acc);
      }
    }
    if (MODE != kSum) {
      double W = *Wfull;
      if (c < kx || c + kx >= NX || r < ky || r + ky >= NY) {
        W = 0.0;
        for (int dj = j0; dj <= j1; ++dj) {
          const int aj = abs(dj), e = es[aj];
          const int i0 = max(-e, -c), i1 = min(e, NX - 1 - c);
          for (int di = i0; di <= i1; ++di) W += Hs[aj * n1 + abs(di)];
        }
      }
      acc /= W;
    }
    out[row[rl] + col[cl]] = acc;
  }
}

// any design counts: a block takes kFEl consecutive elements and spreads their subcells over its threads
constexpr int kFEl = 32;

template <int MODE>
__global__ void __launch_bounds__(128) filter_mixed_kernel(int nelx, int nely, double hx, double hy, double R,
                                                           int reach, FilterTab ft, const double* __restrict__ H,
                                                           const int* __restrict__ ext,
                                                           const int* __restrict__ dmap,
                                                           const int64_t* __restrict__ off,
                                                           const double* __restrict__ x, double* __restrict__ out) {
  __shared__ int first[kFEl + 1];
  __shared__ double cen[MTO_D_MAX + 1][MTO_D_MAX];   // subcell centres (i + 1/2) / d
  const int nel = nelx * nely, e0 = blockIdx.x * kFEl, ne = min(kFEl, nel - e0);
  for (int k = threadIdx.x; k < (MTO_D_MAX + 1) * MTO_D_MAX; k += blockDim.x)
    if (k / MTO_D_MAX > k % MTO_D_MAX) cen[k / MTO_D_MAX][k % MTO_D_MAX] = (k % MTO_D_MAX + 0.5) / (k / MTO_D_MAX);
  for (int k = threadIdx.x; k <= ne; k += blockDim.x) first[k] = (int)(off[e0 + k] - off[e0]);
  __syncthreads();
  for (int it = threadIdx.x; it < first[ne]; it += blockDim.x) {
    int lo = 0, hi = ne;   // the element holding subcell `it`
    while (hi - lo > 1) {
      const int m = (lo + hi) >> 1;
      if (first[m] <= it) lo = m; else hi = m;
    }
    const int e = e0 + lo, ex = e % nelx, ey = e / nelx, d = dmap[e];
    const int s = it - first[lo], i = s % d, j = s / d;
    const int64_t self = off[e] + s;
    const double cx = (ex + cen[d][i]) * hx, cy = (ey + cen[d][j]) * hy;
    const int kx = ft.kx[d], ky = ft.ky[d];
    const double* Hd = H + ft.h0[d];
    const int* ed = ext + ft.e0[d];
    double wsum = 0.0, acc = 0.0;
    for (int ny = max(ey - reach, 0); ny <= min(ey + reach, nely - 1); ++ny) {
      // distance from the centre to the neighbour row's y-range
      const double dy0 = fmax(fmax(ny * hy - cy, cy - (ny + 1) * hy), 0.0);
      if (dy0 >= R) continue;
      for (int nx = max(ex - reach, 0); nx <= min(ex + reach, nelx - 1); ++nx) {
        const double dx0 = fmax(fmax(nx * hx - cx, cx - (nx + 1) * hx), 0.0);
        if (dx0 * dx0 + dy0 * dy0 >= R * R) continue;
        const int n = ny * nelx + nx, dn = dmap[n];
        const double* xn = x + off[n];
        if (dn == d) {   // offsets on the common fine grid; a value out of reach is not touched (it may be no number)
          const int bi = (nx - ex) * d - i, bj = (ny - ey) * d - j;
          const int j0 = max(0, -ky - bj), j1 = min(d - 1, ky - bj);
          for (int jj = j0; jj <= j1; ++jj) {
            const int aj = abs(bj + jj), i0 = max(0, -ed[aj] - bi), i1 = min(d - 1, ed[aj] - bi);
            const double* Hr = Hd + aj * (kx + 1);
            for (int ii = i0; ii <= i1; ++ii) {
              const double w = Hr[abs(bi + ii)];
              if (MODE != kSum) wsum += w;
              if (MODE != kScale) acc = fma(w, xn[jj * d + ii], acc);
            }
          }
        } else {
          for (int jj = 0; jj < dn; ++jj) {
            const double ty = (ny + cen[dn][jj]) * hy - cy, ty2 = ty * ty;
            if (ty2 >= R * R) continue;
            for (int ii = 0; ii < dn; ++ii) {
              const double tx = (nx + cen[dn][ii]) * hx - cx;
              const double d2 = fma(tx, tx, ty2);
              if (d2 >= R * R) continue;
              const double w = R - sqrt(d2);
              if (!(w > 0.0)) continue;
              if (MODE != kSum) wsum += w;
              if (MODE != kScale) acc = fma(w, xn[jj * dn + ii], acc);
            }
          }
        }
      }
    }
    out[self] = MODE == kScale ? x[self] / wsum : MODE == kForward ? acc / wsum : acc;
  }
}

// Design transfer between per-element design counts: new subcell (i, j) of element e takes the
// area-weighted mean of the old subcells it overlaps (overlap lengths per axis, both layouts
// uniform over the element); an unchanged count copies the values.  One warp per element, lanes
// over its new subcells.
__global__ void __launch_bounds__(128) transfer_kernel(int nel, const int* __restrict__ d_old,
                                                       const int64_t* __restrict__ off_old,
                                                       const int* __restrict__ d_new,
                                                       const int64_t* __restrict__ off_new,
                                                       const double* __restrict__ rho_old,
                                                       double* __restrict__ rho_new) {
  const int e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5, lane = threadIdx.x & 31;
  if (e >= nel) return;
  const int dn = d_new[e], dO = d_old[e];
  const double* src = rho_old + off_old[e];
  double* dst = rho_new + off_new[e];
  for (int s = lane; s < dn * dn; s += 32) {
    if (dn == dO) {
      dst[s] = src[s];
      continue;
    }
    const int i = s % dn, j = s / dn;
    const double ax0 = (double)i / dn, ax1 = (double)(i + 1) / dn;
    const double ay0 = (double)j / dn, ay1 = (double)(j + 1) / dn;
    double acc = 0.0;
    for (int l = 0; l < dO; ++l) {
      const double oy = fmax(0.0, fmin(ay1, (double)(l + 1) / dO) - fmax(ay0, (double)l / dO));
      if (oy == 0.0) continue;
      for (int k = 0; k < dO; ++k) {
        const double ox = fmax(0.0, fmin(ax1, (double)(k + 1) / dO) - fmax(ax0, (double)k / dO));
        acc += ox * oy * src[l * dO + k];
      }
    }
    dst[s] = acc * dn * dn;
  }
}

}  // namespace

mto_status transfer_design(mto_handle h, const int* d_old_host, const double* rho_old, double* rho_new) {
  const int64_t nel = h->nel;
  std::vector<int64_t> off(nel + 1, 0);
  for (int64_t e = 0; e < nel; ++e) {
    if (d_old_host[e] < 1 || d_old_host[e] > MTO_D_MAX)
      return mto_fail(h, MTO_EINVAL, "mto_transfer_design: old design count outside 1..MTO_D_MAX");
    off[e + 1] = off[e] + (int64_t)d_old_host[e] * d_old_host[e];
  }
  int* dd = nullptr;
  int64_t* od = nullptr;
  MTO_TRY(mto_cuda_check(h, cudaMalloc(&dd, nel * sizeof(int)), "cudaMalloc"));
  mto_status st = mto_cuda_check(h, cudaMalloc(&od, (nel + 1) * sizeof(int64_t)), "cudaMalloc");
  if (st == MTO_OK)
    st = mto_cuda_check(h, cudaMemcpyAsync(dd, d_old_host, nel * sizeof(int), cudaMemcpyHostToDevice, h->stream), "copy");
  if (st == MTO_OK)
    st = mto_cuda_check(h, cudaMemcpyAsync(od, off.data(), (nel + 1) * sizeof(int64_t), cudaMemcpyHostToDevice, h->stream),
                        "copy");
  if (st == MTO_OK) {
    transfer_kernel<<<(int)((nel * 32 + 127) / 128), 128, 0, h->stream>>>((int)nel, dd, od, h->d_d, h->design_off_d,
                                                                        rho_old, rho_new);
    st = mto_after_launch(h, "transfer_kernel");
  }
  if (st == MTO_OK) st = mto_cuda_check(h, cudaStreamSynchronize(h->stream), "sync");
  cudaFree(dd);
  cudaFree(od);
  return st;
}

mto_status density_filter(mto_handle h, double R, const double* x, double* out, bool adjoint) {
  TimedScope ts(h, F_BUILD);
  const int nel = (int)h->nel;
  const double hmin = h->hx < h->hy ? h->hx : h->hy;
  const int reach = (int)std::ceil(R / hmin);
  // tables of the design counts present (radius at most 4 elements: offsets up to 4 d)
  FilterTab ft;
  unsigned mask = 0;
  int nh = 0, next = 0;
  for (auto& b : h->bc) mask |= 1u << b.d;
  for (int d = 0; d <= MTO_D_MAX; ++d) {
    ft.kx[d] = std::min(4 * d, (int)std::floor(R * d / h->hx));
    ft.ky[d] = std::min(4 * d, (int)std::floor(R * d / h->hy));
    ft.h0[d] = nh;
    ft.e0[d] = next;
    if (!(mask >> d & 1u)) continue;
    nh += (ft.kx[d] + 1) * (ft.ky[d] + 1);
    next += ft.ky[d] + 1;
  }
  constexpr int kHMax = 25040, kEMax = 8 * 72;   // sums of (4 d + 1)^2 and of 4 d + 1 over d = 1..16
  if (!h->filt_H) {
    MTO_TRY(mto_alloc(h, &h->filt_H, (size_t)kHMax + MTO_D_MAX + 1));
    MTO_TRY(mto_alloc(h, &h->filt_ext, (size_t)kEMax));
  }
  double* Wfull = h->filt_H + kHMax;
  filter_table_kernel<<<MTO_D_MAX, 256, 0, h->stream>>>(ft, mask, h->hx, h->hy, R, h->filt_H, h->filt_ext, Wfull);
  MTO_TRY(mto_after_launch(h, "filter_table_kernel"));
  if (adjoint && !h->filt_W) MTO_TRY(mto_alloc(h, &h->filt_W, (size_t)h->design_len));
  if ((mask & (mask - 1)) == 0) {
    const int d = h->bc[0].d, kx = ft.kx[d], ky = ft.ky[d];
    const size_t smem = sizeof(double) * (kx + 1) * (ky + 1) + 8 * (kFTY + 2 * ky) + 4 * (kFTX + 2 * kx + ky + 1) + 16;
    const dim3 grid((h->nelx * d + kFTX - 1) / kFTX, (h->nely * d + kFTY - 1) / kFTY);
    auto go = [&](auto kernel, const double* in, double* o) -> mto_status {
      kernel<<<grid, 256, smem, h->stream>>>(h->nelx, h->nely, d, kx, ky, h->filt_H + ft.h0[d], h->filt_ext + ft.e0[d],
                                             Wfull + d, in, o);
      return mto_after_launch(h, "filter_uniform_kernel");
    };
    if (!adjoint) return go(filter_uniform_kernel<kForward>, x, out);
    MTO_TRY(go(filter_uniform_kernel<kScale>, x, h->filt_W));
    return go(filter_uniform_kernel<kSum>, h->filt_W, out);
  }
  auto go = [&](auto kernel, const double* in, double* o) -> mto_status {
    kernel<<<(nel + kFEl - 1) / kFEl, 128, 0, h->stream>>>(h->nelx, h->nely, h->hx, h->hy, R, reach, ft, h->filt_H,
                                                           h->filt_ext, h->d_d, h->design_off_d, in, o);
    return mto_after_launch(h, "filter_mixed_kernel");
  };
  if (!adjoint) return go(filter_mixed_kernel<kForward>, x, out);
  MTO_TRY(go(filter_mixed_kernel<kScale>, x, h->filt_W));
  return go(filter_mixed_kernel<kSum>, h->filt_W, out);
}

}  // namespace mto
