// Step (a) on the 5th-generation tensor cores: K_e = sum_s E(rho_s) K0_s (Eqs. 2-3, App. B
// composite rule) for every element of a (p, d) class as one GEMM per class,
//   C[e][pos] = sum_s E[e][s] * K0[c(pos)][s],
// M = elements, N = positions of the circulant-diagonal element row, K = subcells.
//
// The element matrices need FP64 accuracy (on the binary designs a relative error of 1e-13 in K_e
// moves the compliance by ~1e-6), so the products cannot be plain BF16 products.  The GEMM is made
// exact by slicing (an Ozaki-type error-free splitting): each element's moduli row is scaled by a
// power of two sigma_e (max |E| <= sigma_e) and each K0 column by a power of two tau_pos, and both
// are cut into 8 slices of 7 bits (56 bits), E/sigma = sum_i a_i 2^-7i and K0/tau = sum_j b_j 2^-7j
// with integer a_i, b_j in [-127, 127] (exact in BF16).  Every slice product a_i . b_j
// over K <= 64 subcells is an integer below 2^20, and all pairs of one level g = i + j share the
// weight 2^-7g: each level accumulates its (at most 8) slice GEMMs in one FP32 TMEM accumulator
// exactly (sums below 2^23).  Levels g = 2..10 are kept (the dropped levels weigh below 2^-51 of
// the row/column scale, the operands' truncation 2^-56).
//
// The epilogue stays off the FP64 pipes (2 FMA per clock and SM on GB300: one FP64 instruction per
// stored entry of the 1024 x 512 beam costs 0.47 ms): the nine level sums are integers, so an entry
// is one 80-bit integer times a power of two, which integer instructions round to FP64 (once, to
// nearest even) and split into the FP32 pair.
//
// One CTA per 128 elements and range of N tiles (16 positions each; the tiles of small classes are
// spread over several CTAs so that the chip fills).  The A slices (8 x 128 x K) are formed in
// shared memory from rho once.  Warp 8 feeds the tensor cores: B slices of a tile by one bulk copy
// into a ring of three, then per K step one tcgen05.mma (kind::f16, BF16 x BF16 -> FP32, M = 128)
// per A slice i against the stacked B slices 1 .. min(8, 10 - i): B slice j times A slice i belongs
// to level i + j, and the level accumulators lie side by side in TMEM, so the products of one A
// slice with all its B slices are one MMA of up to N = 128 (the A slice is read once for all of
// them).  Two TMEM stages of 9 x 16 columns let the MMAs of a tile run under the epilogue of the
// tile before.  Warps 0-7 read their row's 8 positions with tcgen05.ld and write whole sectors of
// their rows through a small shared staging.
// Operands use the no-swizzle K-major core-matrix layout (8 rows x 16 bytes per core matrix).
// Every wait is bounded: on expiry the CTA records an error word that the host reads (tc_check), waits for
// its own copies and MMAs in flight, and its rows are NaN from there on.
//
// Measured (build and one operator product together): 480 x 240 Q3/d8, mixed: 5.32 ms with an FP64
// epilogue of 24 FP64 instructions per entry and 43 single-slice MMAs per K step, 1.10 ms now;
// 320 x 160 adaptive maps (16 classes), FP64: 11.8 ms, 1.62 ms with this epilogue, 1.02 ms with the diagonal
// spread over the local nodes as well.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include <math_constants.h>

#include "mto_internal.cuh"

namespace mto {
namespace {

constexpr int kTM = 128;        // elements per CTA (MMA M)
constexpr int kTN = 16;         // positions per N tile
constexpr int kBRing = 3;       // B tiles in flight
constexpr int kEpiWarps = 8;    // epilogue warps (one more feeds the tensor cores)
constexpr int kSlices = 8;      // slices per operand (8 x 7 = 56 bits)
constexpr int kSliceBits = 7;
constexpr int kOpBits = kSlices * kSliceBits;
constexpr int kLevels = 9;      // levels g = i + j = 2..10
constexpr int kTmemCols = 512;  // two stages of 9 x 16 = 144 columns, 256 apart
constexpr int kTmemStage = 256;
// staging rows of an epilogue warp: 8 doubles or 8 floats and 16 bytes of padding (conflict-free
// 16-byte stores by 32 lanes)
constexpr int kStRow64 = 80, kStRow32 = 48;
constexpr int kStWarp = 32 * (kStRow64 + 2 * kStRow32);

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
}

__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// 8 consecutive 32-bit TMEM columns of this thread's lane
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
      : "r"(taddr)
      : "memory");
}

__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major, no swizzle.  lbo = byte stride between core matrices
// along K, sbo = byte stride between 8-row groups.
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version
  return d;                // base offset 0, relative LBO, layout type 0 (no swizzle)
}

// Instruction descriptor, kind::f16: BF16 A and B, FP32 accumulator, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// byte offset of element (row, k) in the no-swizzle K-major core-matrix layout of a rows x kpad
// BF16 tile
__host__ __device__ __forceinline__ uint32_t core_off(int row, int k, int kpad) {
  return (uint32_t)(((row >> 3) * (kpad >> 3) + (k >> 3)) * 128 + (row & 7) * 16 + (k & 7) * 2);
}

__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// bounded wait for the phase of parity `parity`; false when the limit expires
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, unsigned limit) {
  for (unsigned n = 0; n < limit; ++n)
    if (mbar_try_wait(bar, parity)) return true;
  return false;
}

__device__ __forceinline__ void tc_bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// B operand tables of a class: per N tile, 8 slices of kTN x kpad BF16 in the core layout (so the
// slices of a tile stack along N), and per position the exponent of its power-of-two scale tau.  One
// thread per (position, subcell).
__global__ void tc_btable_kernel(int S, int kpad, int L, int ntile, const double* __restrict__ K0T,
                                 const int* __restrict__ posc, unsigned short* __restrict__ Bt,
                                 int* __restrict__ tau) {
  const int pos = blockIdx.x;
  if (pos >= ntile * kTN) return;
  __shared__ double colmax;
  const int c = pos < L ? posc[pos] : -1;
  if (threadIdx.x < 32) {
    double m = 0.0;
    if (c >= 0)
      for (int s = threadIdx.x; s < S; s += 32) m = fmax(m, fabs(K0T[(size_t)c * S + s]));
    for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (threadIdx.x == 0) colmax = m;
  }
  __syncthreads();
  int ex = 0;
  if (colmax > 0.0) frexp(colmax, &ex);   // colmax < 2^ex
  const double sc = ldexp(1.0, -ex);
  if (threadIdx.x == 0) tau[pos] = ex;
  const int tile = pos / kTN, row = pos % kTN;
  for (int s = threadIdx.x; s < kpad; s += blockDim.x) {
    const double w = (c >= 0 && s < S) ? K0T[(size_t)c * S + s] * sc : 0.0;   // |w| < 1
    const double aw = fabs(w);
    const unsigned long long W = (unsigned long long)ldexp(aw, kOpBits);   // floor(|w| 2^56)
    for (int j = 0; j < kSlices; ++j) {
      const int bits = (int)((W >> (kOpBits - kSliceBits * (j + 1))) & 127ull);
      const float v = (w < 0.0 ? -1.0f : 1.0f) * (float)bits;
      const unsigned short b = (unsigned short)(__float_as_uint(v) >> 16);   // exact: |v| <= 127
      unsigned char* base = reinterpret_cast<unsigned char*>(Bt) +
                            ((size_t)tile * kSlices + j) * (size_t)kTN * kpad * 2;
      *reinterpret_cast<unsigned short*>(base + core_off(row, s, kpad)) = b;
    }
  }
}

// sig[] of a row with a modulus that is not finite: all its entries are NaN, as the FP64 sums give them
constexpr int kRowNaN = 1 << 20;

// rows: element k of the class (first <= k < n) is output row slot[k], or row k - first without slots.
// Kh null: FP64 rows only.  err: the host's error word (pinned), which receives `tag` when a wait expires.
__global__ void __launch_bounds__(32 * (kEpiWarps + 1), 1) tc_build_kernel(
    int n, int first, int S, int kpad, int L, int ntile, int tiles_per_cta, const int* __restrict__ elem,
    const int* __restrict__ slot, const int64_t* __restrict__ design_off, const double* __restrict__ rho, double E0,
    double Emin, double q, const unsigned short* __restrict__ Bt, const int* __restrict__ tau,
    double* __restrict__ K64, float* __restrict__ Kh, float* __restrict__ Kl, unsigned limit, volatile int* err, int tag) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t a_slice = (uint32_t)kTM * kpad * 2, b_slice = (uint32_t)kTN * kpad * 2;
  const uint32_t b_tile = kSlices * b_slice;
  unsigned char* As = smem;
  unsigned char* Bs = As + kSlices * a_slice;
  unsigned char* stage = Bs + kBRing * b_tile;
  uint64_t* bfull = reinterpret_cast<uint64_t*>(stage + kEpiWarps * kStWarp);   // [kBRing] B tile landed
  uint64_t* full = bfull + kBRing;    // [2] MMAs of a TMEM stage done
  uint64_t* empty = full + 2;         // [2] TMEM stage read by all epilogue warps
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(empty + 2);
  int* sig = reinterpret_cast<int*>(tmem_slot + 2);   // [kTM] exponents of sigma_e
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int base = first + blockIdx.x * kTM;
  const int tile0 = blockIdx.y * tiles_per_cta;
  const int nt = min(tiles_per_cta, ntile - tile0);

  if (warp == 0) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  if (warp == kEpiWarps && lane == 0) {
    for (int b = 0; b < kBRing; ++b) mbar_init(bfull + b, 1);
    for (int b = 0; b < 2; ++b) {
      mbar_init(full + b, 1);
      mbar_init(empty + b, kEpiWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    for (int i = 0; i < kBRing && i < nt; ++i) {
      mbar_expect(bfull + i, b_tile);
      tc_bulk_g2s(Bs + i * b_tile, reinterpret_cast<const unsigned char*>(Bt) + (size_t)(tile0 + i) * b_tile, b_tile,
                  bfull + i);
    }
  }

  // A slices: one element row per warp at a time, two subcells per lane (coalesced rho, packed
  // 32-bit stores).  Moduli E_s scaled by sigma_e and cut into 8 x 7 bits and their sign by integer shifts;
  // q = 3 takes products instead of pow (both run on the FP64 pipes).
  if (warp < kEpiWarps) {
    const bool cube = q == 3.0;
    const double dE = E0 - Emin;
    auto modulus = [&](double r) { return Emin + (cube ? r * r * r : pow(r, q)) * dE; };
    const int s0 = 2 * lane;
#pragma unroll 4
    for (int r = warp; r < kTM; r += kEpiWarps) {
      const int k = base + r;
      double r0 = 0.0, r1 = 0.0;
      const bool v0 = k < n && s0 < S, v1 = k < n && s0 + 1 < S;
      if (v0) {
        const int64_t off = design_off[elem[k]];
        r0 = rho[off + s0];
        if (v1) r1 = rho[off + s0 + 1];
      }
      const unsigned long long e0 = v0 ? (unsigned long long)__double_as_longlong(modulus(r0)) : 0ull;
      const unsigned long long e1 = v1 ? (unsigned long long)__double_as_longlong(modulus(r1)) : 0ull;
      // sigma_e = 2^ex > max |E|: from the largest exponent
      const int xm = __reduce_max_sync(0xffffffffu, max((int)(e0 >> 52) & 0x7ff, (int)(e1 >> 52) & 0x7ff));
      const int ex = max(xm, 1) - 1022;
      if (lane == 0) sig[r] = xm < 0x7ff ? ex : kRowNaN;
      if (s0 < kpad) {
        const unsigned sgn = (unsigned)(e0 >> 63) << 15 | (unsigned)(e1 >> 63) << 31;
        const unsigned long long V0 = fixed56(e0, ex), V1 = fixed56(e1, ex);
        unsigned char* dst = As + core_off(r, s0, kpad);
#pragma unroll
        for (int i = 0; i < kSlices; ++i) {
          const int sh = kOpBits - kSliceBits * (i + 1);
          const unsigned a0 = __float_as_uint((float)(int)((V0 >> sh) & 127ull)) >> 16;
          const unsigned a1 = __float_as_uint((float)(int)((V1 >> sh) & 127ull)) & 0xffff0000u;
          *reinterpret_cast<unsigned*>(dst + i * a_slice) = sgn | a0 | a1;   // BF16 of integers <= 127: exact
        }
      }
    }
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool ok = true;

  if (warp == kEpiWarps) {
    if (lane == 0) {
      const uint32_t sbo = (uint32_t)(kpad >> 3) * 128u;
      const int kst = kpad / 16;
      const uint32_t a0 = smem_u32(As);
      int issued = min(kBRing, nt), committed = 0;
      for (int it = 0; it < nt && ok; ++it) {
        const int st = it & 1;
        ok = mbar_wait(bfull + it % kBRing, (uint32_t)((it / kBRing) & 1), limit);
        if (ok && it >= 2) ok = mbar_wait(empty + st, (uint32_t)(((it >> 1) - 1) & 1), limit);
        if (!ok) break;
        tc_fence_after();
        const uint32_t b0 = smem_u32(Bs + (it % kBRing) * b_tile);
        const uint32_t d0 = tmem + (uint32_t)(st * kTmemStage);
        auto mma = [&](int i, int j, int nj, int ks, uint32_t acc) {   // A slice i times B slices j .. j + nj - 1
          umma_bf16(d0 + (uint32_t)((i + j - 2) * kTN), smem_desc(a0 + (uint32_t)(i - 1) * a_slice + ks * 256u, 128u, sbo),
                    smem_desc(b0 + (uint32_t)(j - 1) * b_slice + ks * 256u, 128u, sbo), idesc_bf16(kTM, kTN * nj), acc);
        };
        // slice 2 first: it starts levels 3..10; slice 1 then starts level 2 and adds to the others
        for (int ks = 0; ks < kst; ++ks) mma(2, 1, kSlices, ks, ks > 0);
        mma(1, 1, 1, 0, 0);
        mma(1, 2, kSlices - 1, 0, 1);
        for (int ks = 1; ks < kst; ++ks) mma(1, 1, kSlices, ks, 1);
        for (int i = 3; i <= kSlices; ++i)
          for (int ks = 0; ks < kst; ++ks) mma(i, 1, kLevels + 1 - i, ks, 1);
        umma_commit(full + st);
        committed = it + 1;
        // refill the ring slot of the tile before, whose MMAs are done once its stage is committed
        if (it >= 1 && it - 1 + kBRing < nt) {
          const int nx = it - 1 + kBRing;
          ok = mbar_wait(full + (st ^ 1), (uint32_t)(((it - 1) >> 1) & 1), limit);
          if (!ok) break;
          mbar_expect(bfull + nx % kBRing, b_tile);
          tc_bulk_g2s(Bs + (nx % kBRing) * b_tile, reinterpret_cast<const unsigned char*>(Bt) + (size_t)(tile0 + nx) * b_tile,
                      b_tile, bfull + nx % kBRing);
          issued = nx + 1;
        }
      }
      if (!ok) {
        // a wait expired: every copy that was issued lands, and every MMA ends, before the CTA gives up its memory
        for (int i = max(0, issued - kBRing); i < issued; ++i)
          mbar_wait(bfull + i % kBRing, (uint32_t)((i / kBRing) & 1), kTcPolls);
        if (committed > 0)
          mbar_wait(full + ((committed - 1) & 1), (uint32_t)(((committed - 1) >> 1) & 1), kTcPolls);
      }
    }
    __syncwarp();
  } else {
    const int row = (warp & 3) * 32 + lane, c0 = (warp >> 2) * 8;
    const int k = base + row;
    const int sl = k < n ? (slot ? slot[k] : k - first) : -1;
    const int sexp = sig[row];
    unsigned char* st64 = stage + warp * kStWarp;
    unsigned char* sth = st64 + 32 * kStRow64;
    unsigned char* stl = sth + 32 * kStRow32;
    int it = 0;
    for (; it < nt; ++it) {
      const int st = it & 1;
      ok = mbar_wait(full + st, (uint32_t)((it >> 1) & 1), limit);
      if (!__all_sync(0xffffffffu, ok)) {
        ok = false;
        break;
      }
      tc_fence_after();
      uint32_t v[kLevels][8];
      const uint32_t src = tmem + (uint32_t)(st * kTmemStage + c0) + ((uint32_t)((warp & 3) * 32) << 16);
#pragma unroll
      for (int g = 0; g < kLevels; ++g) tmem_ld8(src + (uint32_t)(g * kTN), v[g]);
      tmem_wait_ld();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(empty + st);
      const int pos0 = (tile0 + it) * kTN + c0;
      if (pos0 < L) {
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          int I[kLevels];
#pragma unroll
          for (int g = 0; g < kLevels; ++g) I[g] = __float2int_rn(__uint_as_float(v[g][c]));
          // pairs of levels fit 32 bits (2^30 + 2^23); units: level 6 for H, level 10 for Lw
          const int p0 = I[0] * 128 + I[1], p1 = I[2] * 128 + I[3], p2 = I[5] * 128 + I[6], p3 = I[7] * 128 + I[8];
          const long long H = (long long)p0 * (1 << 21) + (long long)p1 * 128 + I[4];
          const long long Lw = (long long)p2 * (1 << 14) + p3;
          unsigned long long bits = levels_to_double(H, Lw, sexp + __ldg(tau + pos0 + c));
          if (sexp == kRowNaN) bits = 0x7ff8000000000000ull;
          *reinterpret_cast<unsigned long long*>(st64 + lane * kStRow64 + c * 8) = bits;
          if (Kh) {
            float hi, lo;
            split_pair(bits, hi, lo);
            *reinterpret_cast<float*>(sth + lane * kStRow32 + c * 4) = hi;
            *reinterpret_cast<float*>(stl + lane * kStRow32 + c * 4) = lo;
          }
        }
        __syncwarp();
        // whole sectors: 4 lanes per 64-byte row piece of the FP64 rows, 2 lanes per FP32 piece
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = 8 * i + (lane >> 2), o = 2 * (lane & 3);
          const int rs = __shfl_sync(0xffffffffu, sl, r);
          if (rs >= 0 && pos0 + o < L)
            *reinterpret_cast<double2*>(K64 + (size_t)rs * L + pos0 + o) =
                *reinterpret_cast<const double2*>(st64 + r * kStRow64 + o * 8);
        }
        if (Kh) {
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const int r = 16 * i + (lane >> 1), o = 4 * (lane & 1);
            const int rs = __shfl_sync(0xffffffffu, sl, r);
            if (rs >= 0 && pos0 + o < L) {
              const size_t at = (size_t)rs * L + pos0 + o;
              *reinterpret_cast<float4*>(Kh + at) = *reinterpret_cast<const float4*>(sth + r * kStRow32 + o * 4);
              *reinterpret_cast<float4*>(Kl + at) = *reinterpret_cast<const float4*>(stl + r * kStRow32 + o * 4);
            }
          }
        }
        __syncwarp();
      }
    }
    for (; it < nt && sl >= 0; ++it)   // after an expired wait
      for (int pos = (tile0 + it) * kTN + c0; pos < min((tile0 + it) * kTN + c0 + 8, L); ++pos) {
        const size_t at = (size_t)sl * L + pos;
        K64[at] = CUDART_NAN;
        if (Kh) Kh[at] = Kl[at] = CUDART_NAN_F;
      }
  }
  tc_fence_before();
  if (__syncthreads_or(!ok) && t == 0) *err = tag;
  tc_fence_after();
  if (warp == 0) tmem_dealloc(tmem, kTmemCols);
}

}  // namespace

// Per (p, d) class with d <= 8: B slice tables (once per nu) for the tensor-core build, and for the
// QR indicator's order p + 1 matrices (in its packed row order).
mto_status tc_tables(mto_handle h) {
  for (int qr = 0; qr < 2; ++qr) {
    for (auto& b : qr ? h->bc_qr : h->bc) {
      if (b.S > 64) continue;
      const int L = qr ? qr_row_len(b.p) : h->pc[b.p].L;
      const int* pos = qr ? h->qr[b.p - 1].pos : h->pc[b.p].posc;
      const int kpad = (b.S + 15) / 16 * 16;
      const int ntile = (L + kTN - 1) / kTN;
      if (!b.tcB) {
        MTO_TRY(mto_alloc(h, &b.tcB, (size_t)ntile * kSlices * kTN * kpad));
        MTO_TRY(mto_alloc(h, &b.tcTau, (size_t)ntile * kTN));
      }
      tc_btable_kernel<<<ntile * kTN, 64, 0, h->stream>>>(b.S, kpad, L, ntile, b.K0T, pos, b.tcB, b.tcTau);
      MTO_TRY(mto_after_launch(h, "tc_btable_kernel"));
    }
  }
  return MTO_OK;
}

namespace {
// Dynamic shared memory of the build kernel, at least 120 KB so that one CTA (and one 512-column
// TMEM allocation) is resident per SM.
size_t tc_smem_bytes(int kpad) {
  const size_t need = (size_t)kSlices * (kTM + kBRing * kTN) * kpad * 2 + kEpiWarps * kStWarp + 8 * (kBRing + 4) + 8 +
                      4 * kTM + 64;
  return need < 120 * 1024 ? 120 * 1024 : need;
}
}  // namespace

// Rows sum_s E(rho_s) K0_s of elements first .. first + n - 1 of a class (its elements and counts from
// `b`, the tables from `tab`): to row slot[k] of K64 (and the pair), or to row k - first without slots.
// The N tiles of few elements are split over CTAs (each forms its elements' A slices again, about the
// cost of three tiles) until the launch has about one CTA per SM.
mto_status tc_rows(mto_handle h, const BClass& b, const BClass& tab, int L, int first, int n, const int* slot,
                   const double* rho, const mto_material* m, double* K64, float* Kh, float* Kl, TcUse use) {
  const int kpad = (b.S + 15) / 16 * 16;
  const int ntile = (L + kTN - 1) / kTN;
  const size_t smem = tc_smem_bytes(kpad);
  MTO_TRY(allow_smem(h, tc_build_kernel, tc_smem_bytes(64)));
  const int gx = (n + kTM - 1) / kTM;
  const int gy = std::max(1, std::min(ntile, 152 / gx));
  const int per = (ntile + gy - 1) / gy;
  tc_build_kernel<<<dim3(gx, (ntile + per - 1) / per), 32 * (kEpiWarps + 1), smem, h->stream>>>(
      first + n, first, b.S, kpad, L, ntile, per, b.elem, slot, h->design_off_d, rho, m->E0, m->Emin, m->q, tab.tcB,
      tab.tcTau, K64, Kh, Kl, h->tc_polls, h->host_flags + 9 + use, h->tc_tag[use]);
  return mto_after_launch(h, "tc_build_kernel");
}

// The tensor-core build of one (p, d) class (d <= 8).
mto_status tc_build_class(mto_handle h, const BClass& b, const double* rho, const mto_material* m, int precision) {
  const PClass& c = h->pc[b.p];
  const bool mixed = precision == MTO_MIXED;
  return tc_rows(h, b, b, c.L, 0, b.n, b.slot, rho, m, c.K64, mixed ? c.K32 : nullptr, mixed ? c.K32lo : nullptr,
                 TC_BUILD);
}

// After a synchronisation of the stream: whether a wait of the current build (or the last indicator's
// rows) expired.
mto_status tc_check(mto_handle h, TcUse use) {
  if (h->host_flags[9 + use] != h->tc_tag[use] || h->tc_tag[use] == 0) return MTO_OK;
  return mto_fail(h, MTO_ETIMEOUT, use == TC_BUILD ? "element build: a bounded device wait expired"
                                                   : "QR indicator: a bounded device wait expired");
}

}  // namespace mto
