// Stand-alone batched transforms (in place) for the kernel sweep.   grid = batch * L
#include "d2mhe_kernels_common.cuh"

namespace {

template <int LOGN, int G, int WIDE>
__global__ void __launch_bounds__(ntt_threads_ct(LOGN, G), ntt_minb_ct(LOGN, G))
    k_ntt_fwd(DevView v, const __grid_constant__ LimbParams lp, u64* __restrict__ polys) {
  const u32 l = blockIdx.x % v.L;
  const LimbTab& lt = lp.limbs[l];
  u64* row = polys + (size_t)blockIdx.x * v.n;
  ntt_forward<LOGN, G, WIDE>(
      poly_smem(), lt, v.logn, [&](u32 j) { return row[j]; },
      [&](int, u32 q, u64(&x)[8]) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = shoup_full(x[k], 1, lt.one_sh, lt.p);
        store_octet(row + 8 * (size_t)q, x);
      });
}

template <int LOGN, int G, int WIDE>
__global__ void __launch_bounds__(ntt_threads_ct(LOGN, G), ntt_minb_ct(LOGN, G))
    k_ntt_inv(DevView v, const __grid_constant__ LimbParams lp, u64* __restrict__ polys) {
  const u32 l = blockIdx.x % v.L;
  const LimbTab& lt = lp.limbs[l];
  u64* row = polys + (size_t)blockIdx.x * v.n;
  ntt_inverse<LOGN, G, WIDE>(
      poly_smem(), lt, v.logn,
      [&](int, u32 q, u64(&x)[8]) {
        const ulonglong2* s = reinterpret_cast<const ulonglong2*>(row + 8 * (size_t)q);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          ulonglong2 t = s[k];
          x[2 * k] = t.x;
          x[2 * k + 1] = t.y;
        }
      },
      [&](u32 j, u64 val) { row[j] = shoup_full(val, lt.ninv, lt.ninv_sh, lt.p); });
}


// ---- two-pass transforms for N = 2^15, 2^16 (one polynomial does not fit one CTA) ----------
// Pass A applies the first SA = log2 N - 12 stages in registers: thread o owns the 2^SA
// coefficients o + k * 4096 (coalesced across threads; every thread uses the same 2^SA - 1
// twiddles).  After it the array is 2^SA independent blocks of 4096, each finished by the
// shared-memory engine with the twiddles of its sub-tree (pass B).  The inverse runs B then A.
// Between the passes values are lazily reduced: below 8p with one conditional subtraction per butterfly (MODE_STRICT);
// WIDE primes take 16 stages without any; below 2^60 (LAZY60) three stages fit and the fourth's operands are reduced.
// Forward at N = 32768 (three stages) the conditional subtractions cost nothing and the kernel without them is the slower
// one (444 rows mod 54-bit primes, both passes: 150.7 us with them, 153.8 without; inverse 153.2 / 142.4; N = 65536
// forward 327 / 317): there WIDE primes take MODE_STRICT.
template <int SA, bool INV, int MODE>
__global__ void __launch_bounds__(256)
    k_ntt_strided(DevView v, const __grid_constant__ LimbParams lp, u64* __restrict__ polys) {
  constexpr int R = 1 << SA;
  const u32 r = blockIdx.x >> 4;  // polynomial-limb; 16 CTAs of 256 columns each
  const LimbTab& lt = lp.limbs[r % v.L];
  const Mod md(lt);
  const u32 o = (blockIdx.x & 15u) * blockDim.x + threadIdx.x;  // < 4096
  u64* row = polys + (size_t)r * v.n + o;
  if (!D2MHE_CHK(v.chk, (size_t)o + ((size_t)(R - 1) << 12), v.n, SITE_LOAD)) return;
  u64 x[R];
#pragma unroll
  for (int k = 0; k < R; ++k) x[k] = row[(size_t)k << 12];
  if (!INV) {
#pragma unroll
    for (int s = 0; s < SA; ++s) {
      const int m = 1 << s, half = R >> (s + 1);
#pragma unroll
      for (int i = 0; i < m; ++i) {
        const ulonglong2 w = __ldg(lt.W + m + i);
#pragma unroll
        for (int j = 0; j < half; ++j) {
          u64& X = x[i * 2 * half + j];
          if (MODE == MODE_LAZY60 && s == 3) X = reduce_small(X, md);  // p, 5p, 9p, 13p before the stages
          ct_bfly<MODE>(X, x[i * 2 * half + j + half], w, md);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < R; ++k) row[(size_t)k << 12] = x[k];
  } else {
#pragma unroll
    for (int s = SA - 1; s >= 0; --s) {
      const int m = 1 << s, half = R >> (s + 1);
#pragma unroll
      for (int i = 0; i < m; ++i) {
        const ulonglong2 w = __ldg(lt.IW + m + i);
#pragma unroll
        for (int j = 0; j < half; ++j) {
          u64 &X = x[i * 2 * half + j], &Y = x[i * 2 * half + j + half];
          // sums double from 4p: WIDE adds what they have reached; LAZY60 (8p) brings both below 3p from the second on
          if (MODE == MODE_LAZY60 && s < SA - 1) X = reduce_small(X, md), Y = reduce_small(Y, md);
          gs_bfly<MODE>(X, Y, w, md, md.fourp << (SA - 1 - s));
        }
      }
    }
#pragma unroll
    for (int k = 0; k < R; ++k) row[(size_t)k << 12] = shoup_full(x[k], lt.ninv, lt.ninv_sh, lt.p);
  }
}

// Pass B: block b of polynomial-limb r; grid = batch * L * 2^soff.
template <int LOGN, int G, int WIDE>
__global__ void __launch_bounds__(ntt_threads_ct(LOGN, G), ntt_minb_ct(LOGN, G))
    k_ntt_fwd_blk(DevView v, const __grid_constant__ LimbParams lp, u64* __restrict__ polys, u32 soff) {
  const u32 b = blockIdx.x & ((1u << soff) - 1), r = blockIdx.x >> soff;
  const LimbTab& lt = lp.limbs[r % v.L];
  u64* row = polys + (size_t)r * v.n + ((size_t)b << LOGN);
  ntt_forward<LOGN, G, WIDE>(
      poly_smem(), lt, LOGN, [&](u32 j) { return row[j]; },
      [&](int, u32 q, u64(&x)[8]) {
#pragma unroll
        for (int k = 0; k < 8; ++k) x[k] = shoup_full(x[k], 1, lt.one_sh, lt.p);
        store_octet(row + 8 * (size_t)q, x);
      },
      soff, b);
}
template <int LOGN, int G, int WIDE>
__global__ void __launch_bounds__(ntt_threads_ct(LOGN, G), ntt_minb_ct(LOGN, G))
    k_ntt_inv_blk(DevView v, const __grid_constant__ LimbParams lp, u64* __restrict__ polys, u32 soff) {
  const u32 b = blockIdx.x & ((1u << soff) - 1), r = blockIdx.x >> soff;
  const LimbTab& lt = lp.limbs[r % v.L];
  u64* row = polys + (size_t)r * v.n + ((size_t)b << LOGN);
  ntt_inverse<LOGN, G, WIDE>(
      poly_smem(), lt, LOGN,
      [&](int, u32 q, u64(&x)[8]) {
        const ulonglong2* s = reinterpret_cast<const ulonglong2*>(row + 8 * (size_t)q);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          ulonglong2 t = s[k];
          x[2 * k] = t.x;
          x[2 * k + 1] = t.y;
        }
      },
      [&](u32 j, u64 val) { row[j] = val; },  // below 4p; pass A scales and reduces
      soff, b);
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

static int ntt_mode(const DevView& v) { return v.wide ? MODE_WIDE : v.below60 ? MODE_LAZY60 : MODE_STRICT; }

static cudaError_t ntt_two_pass(const DevView& v, const LimbParams& lp, cudaStream_t s, u64* polys,
                                u32 batch, bool inverse) {
  const u32 soff = v.logn - 12, rows = batch * v.L;
  const size_t smem = poly_bytes(4096);
  const u32 grid_a = rows * 16;
  const u32 grid_b = rows << soff, threads = ntt_threads(4096, D2MHE_G12);
  const int mode = ntt_mode(v);
  cudaError_t e = cudaSuccess;
#define D2MHE_STRIDED(INV_, MODE_)                                              \
  do {                                                                          \
    if (soff == 3)                                                              \
      k_ntt_strided<3, INV_, !INV_ && MODE_ == MODE_WIDE ? MODE_STRICT : MODE_>  \
          <<<grid_a, 256, 0, s>>>(v, lp, polys);                                \
    else                                                                        \
      k_ntt_strided<4, INV_, MODE_><<<grid_a, 256, 0, s>>>(v, lp, polys);       \
    e = cudaGetLastError();                                                     \
  } while (0)
#define D2MHE_BLOCKS(KERNEL, MODE_) \
  e = launch_clustered(KERNEL<12, D2MHE_G12, MODE_>, grid_b, threads, smem, s, 1, v, lp, polys, soff)
#define D2MHE_TWO_PASS(MODE_)                 \
  do {                                        \
    if (!inverse) {                           \
      D2MHE_STRIDED(false, MODE_);            \
      if (e != cudaSuccess) return e;         \
      D2MHE_BLOCKS(k_ntt_fwd_blk, MODE_);     \
    } else {                                  \
      D2MHE_BLOCKS(k_ntt_inv_blk, MODE_);     \
      if (e != cudaSuccess) return e;         \
      D2MHE_STRIDED(true, MODE_);             \
    }                                         \
  } while (0)
  if (mode == MODE_WIDE)
    D2MHE_TWO_PASS(MODE_WIDE);
  else if (mode == MODE_LAZY60)
    D2MHE_TWO_PASS(MODE_LAZY60);
  else
    D2MHE_TWO_PASS(MODE_STRICT);
#undef D2MHE_STRIDED
#undef D2MHE_BLOCKS
#undef D2MHE_TWO_PASS
  return e;
}

// one-pass sizes: the instantiation for the ring degree and the arithmetic mode
#define D2MHE_NTT_MODE(KERNEL, LOGN_, G_)                                                                      \
  do {                                                                                                         \
    const u32 grid = batch * v.L, threads = ntt_threads(v.n, G_);                                              \
    const size_t smem = poly_bytes(v.n);                                                                       \
    if (mode == MODE_WIDE) return launch_clustered(KERNEL<LOGN_, G_, MODE_WIDE>, grid, threads, smem, s, 1, v, lp, polys);   \
    if (mode == MODE_LAZY60)                                                                                   \
      return launch_clustered(KERNEL<LOGN_, G_, MODE_LAZY60>, grid, threads, smem, s, 1, v, lp, polys);        \
    return launch_clustered(KERNEL<LOGN_, G_, MODE_STRICT>, grid, threads, smem, s, 1, v, lp, polys);          \
  } while (0)
#define D2MHE_NTT_SIZE(KERNEL)                                 \
  switch (v.logn) {                                            \
    case 11: D2MHE_NTT_MODE(KERNEL, 11, 1);                    \
    case 12: D2MHE_NTT_MODE(KERNEL, 12, D2MHE_G12);            \
    case 13: D2MHE_NTT_MODE(KERNEL, 13, D2MHE_G13);            \
    case 14: D2MHE_NTT_MODE(KERNEL, 14, D2MHE_G14);            \
    default: D2MHE_NTT_MODE(KERNEL, 0, 1);                     \
  }

cudaError_t ntt(const DevView& v, const LimbParams& lp, cudaStream_t s, u64* polys, u32 batch, bool inverse) {
  if (v.logn > 14) return ntt_two_pass(v, lp, s, polys, batch, inverse);
  const int mode = ntt_mode(v);
  if (inverse) {
    D2MHE_NTT_SIZE(k_ntt_inv)
  } else {
    D2MHE_NTT_SIZE(k_ntt_fwd)
  }
}

}  // namespace D2MHE_LAUNCH_NS
