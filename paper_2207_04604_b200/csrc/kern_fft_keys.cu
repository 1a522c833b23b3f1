// Transforms for the double-precision ring products that serve many products: key shares and public keys, point by point as
// exact as a double can be, and the polynomials u and mu_k, which do not depend on the limb.
#include "d2mhe_fft_block.cuh"

namespace {

// A key's transform in double-double arithmetic, rounded to double once at the end: the error bound of the products needs
// every point of it to about one unit (see d2mhe_fft.cuh).  One thread block transforms the m = 256 R points of a group
// in shared memory, a radix-2 stage at a time from the top, which leaves Z_k at the bit-reversed place; roots of unity are
// products of two table entries.  in(j): coefficient j, a whole number.  row: the group's n points, as fft_store leaves
// them, times 1/n (a power of two: exact).
// Bound by the double-precision pipe: 240 operations a butterfly, 12 stages of 2048.  Once per key.
constexpr u32 KEY_THREADS = 512;
template <int LOGN>
constexpr size_t key_smem() {
  return (size_t)FftGeo<LOGN>::NG * sizeof(ddc);
}
template <int LOGN, class In>
__device__ __forceinline__ void fft_key(const DevView& v, u32 group, double2* __restrict__ row, In in) {
  using G = FftGeo<LOGN>;
  constexpr u32 m = G::NG, order = 8 * m, LM = LOGN - (G::GR == 2 ? 2 : 1);
  dd* re = reinterpret_cast<dd*>(smem_raw);
  dd* im = re + m;
  const ddc *coarse = v.fft.roots, *fine = coarse + order / FFT_ROOT_FINE;
  auto root = [&](u32 k) { return dd_root(coarse, fine, order, k); };
  for (u32 j = threadIdx.x; j < m; j += KEY_THREADS) {
    ddc z{dd{in(j), 0.0}, dd{in(j + G::n), 0.0}};
    if (G::GR == 2)  // z_j +- q z_(j + m), q = e^(i pi / 4)
      z = dd_cadd(z, dd_cmul(ddc{dd{in(j + m), 0.0}, dd{in(j + m + G::n), 0.0}}, root(m + 4 * m * group)));
    z = dd_cmul(z, root(G::GR == 1 ? 2 * j : group ? 0u - 3 * j : j));
    re[j] = z.r, im[j] = z.i;
  }
#pragma unroll 1
  for (int lg = (int)LM - 1; lg >= 0; --lg) {
    __syncthreads();
    const u32 len = 1u << lg;
    for (u32 b = threadIdx.x; b < m / 2; b += KEY_THREADS) {
      const u32 j = b & (len - 1), lo = ((b >> lg) << (lg + 1)) + j, hi = lo + len;
      if (!D2MHE_CHK(v.chk, hi, m, SITE_STAGED)) continue;
      const ddc x{re[lo], im[lo]}, y{re[hi], im[hi]};
      const ddc s = dd_cadd(x, y), d = dd_cmul(dd_csub(x, y), root(j * (4 * m >> lg)));
      re[lo] = s.r, im[lo] = s.i;
      re[hi] = d.r, im[hi] = d.i;
    }
  }
  __syncthreads();
  constexpr double scale = 1.0 / (double)G::n;
  for (u32 i = threadIdx.x; i < m; i += KEY_THREADS) {  // point kA of thread (kC, kB)
    const u32 kA = i / G::TG, t = i % G::TG, k = (t >> 4) + (u32)G::R * ((t & 15u) + 16u * kA);
    const u32 at = __brev(k) >> (32 - LM);
    const u32 slot = kA * G::T + group * G::TG + t;
    if (!D2MHE_CHK(v.chk, at, m, SITE_STAGED) || !D2MHE_CHK(v.chk, slot, G::n, SITE_STORE)) continue;
    row[slot] = make_double2(re[at].h * scale, im[at].h * scale);
  }
}

// s_k of the listed parties, sampled again from its stream (one transform serves every limb).   grid = n_parties * GR
template <int LOGN>
__global__ void __launch_bounds__(KEY_THREADS)
    k_fft_secret(DevView v, const u32* __restrict__ parties, u32 tag, double2* __restrict__ dst) {
  using G = FftGeo<LOGN>;
  const u32 party = parties[blockIdx.x / G::GR];
  if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY)) return;
  const Stream st(v.seed, tag, 0, party, 0);
  fft_key<LOGN>(v, blockIdx.x % G::GR, dst + (size_t)party * G::n, [&](u32 j) { return (double)st.ternary(j); });
}

// Sampled polynomials (bytes as sample_streams leaves them in the order of the double-precision kernels), transformed.
// Every stride-th polynomial of src.   grid = polynomials; dst: [grid][n]
template <int LOGN>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_fft_samples(DevView v, const uint4* __restrict__ src, u32 stride, double2* __restrict__ dst) {
  using G = FftGeo<LOGN>;
  const FftSmem<LOGN> sm(v);
  double xr[16], xi[16];
  fft_samples_forward(sm, v.fft, src + (size_t)blockIdx.x * stride * (v.n / 16), xr, xi);
  fft_store(sm, dst + (size_t)blockIdx.x * G::n, xr, xi);
}

// Residue rows, limb r mod L of row r: both parts (PARTS = 2), or whole rows below 2^30 (PARTS = 1).
// grid = rows * PARTS * GR; src: [..][N], dst: [..][PARTS][n].
// users != null: row r is row r mod 2L of user users[r / 2L], in the parts of Conversion.
template <int LOGN, int PARTS>
__global__ void __launch_bounds__(KEY_THREADS)
    k_fft_rows(DevView v, const __grid_constant__ LimbParams lp, const u64* __restrict__ src, const u32* __restrict__ users,
               double2* __restrict__ dst) {
  using G = FftGeo<LOGN>;
  const u32 half = (blockIdx.x / G::GR) % PARTS;
  size_t r = blockIdx.x / G::GR / PARTS;
  if (users) {
    const u32 user = users[r / (2 * v.L)];
    if (!D2MHE_CHK(v.chk, user, v.K, SITE_PARTY)) return;
    r = (size_t)user * 2 * v.L + r % (2 * v.L);
  }
  const LimbTab& lt = lp.limbs[r % v.L];
  const u64* row = src + r * v.n;
  const u64 p = lt.p;
  const u32 h = users ? lt.fftc.h : lt.fft.h;
  fft_key<LOGN>(v, blockIdx.x % G::GR, dst + (PARTS * r + half) * G::n, [&](u32 j) {
    if (!D2MHE_CHK(v.chk, j, v.n, SITE_LOAD)) return 0.0;
    const u64 c = __ldg(row + j);
    if (PARTS == 1) return (double)((long long)c - (c > (p >> 1) ? (long long)p : 0ll));
    int lo, hi;
    fft_split(c, p, h, lo, hi);
    return (double)(half ? hi : lo);
  });
}

// Test hook: warp 0 does not announce that it has read the exchange area, so the second wait runs into the limit, and those
// after it give up at once.  No copies in flight, no tensor memory.
__global__ void __launch_bounds__(FftGeo<12>::T) k_wait_selftest(DevView v, int tries) {
  FftSmem<12, 0> sm(v);
  sm.tries = tries;
  if (threadIdx.x == 0) sm.init();
  __syncthreads();
  sm.acquire();
  if (threadIdx.x >= 32) sm.release();
  for (int i = 0; i < 8; ++i) sm.acquire();
  __syncthreads();
  if (threadIdx.x == 0) sm.finish(v);
}

template <int LOGN>
cudaError_t launch_secret(const DevView& v, cudaStream_t s, const u32* parties_dev, u32 n_parties, u32 tag, double2* dst) {
  cudaError_t e = set_smem(k_fft_secret<LOGN>, key_smem<LOGN>());
  if (e != cudaSuccess) return e;
  k_fft_secret<LOGN><<<n_parties * FftGeo<LOGN>::GR, KEY_THREADS, key_smem<LOGN>(), s>>>(v, parties_dev, tag, dst);
  return cudaGetLastError();
}
template <int LOGN>
cudaError_t launch_samples(const DevView& v, cudaStream_t s, const void* src, u32 stride, u32 polys, double2* dst) {
  using G = FftGeo<LOGN>;
  cudaError_t e = set_smem(k_fft_samples<LOGN>, G::ex_bytes);
  if (e != cudaSuccess) return e;
  k_fft_samples<LOGN><<<polys, G::T, G::ex_bytes, s>>>(v, reinterpret_cast<const uint4*>(src), stride, dst);
  return cudaGetLastError();
}
template <int LOGN, int PARTS>
cudaError_t launch_rows(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* src, const u32* users_dev, u32 rows,
                        double2* dst) {
  cudaError_t e = set_smem(k_fft_rows<LOGN, PARTS>, key_smem<LOGN>());
  if (e != cudaSuccess) return e;
  k_fft_rows<LOGN, PARTS><<<rows * PARTS * FftGeo<LOGN>::GR, KEY_THREADS, key_smem<LOGN>(), s>>>(v, lp, src, users_dev, dst);
  return cudaGetLastError();
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

// dst: [K][n], rows of the listed parties only
cudaError_t fft_secret(const DevView& v, cudaStream_t s, const u32* parties_dev, u32 n_parties, u32 tag, double2* dst) {
  switch (v.logn) {
    case 12: return launch_secret<12>(v, s, parties_dev, n_parties, tag, dst);
    case 13: return launch_secret<13>(v, s, parties_dev, n_parties, tag, dst);
    case 14: return launch_secret<14>(v, s, parties_dev, n_parties, tag, dst);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t wait_selftest(const DevView& v, cudaStream_t s, u32 tries) {
  const size_t smem = FftGeo<12>::smem_bytes(0);
  const cudaError_t e = set_smem(k_wait_selftest, smem);
  if (e != cudaSuccess) return e;
  k_wait_selftest<<<1, FftGeo<12>::T, smem, s>>>(v, (int)tries);
  return cudaGetLastError();
}

// every stride-th of the polynomials in src; dst: [polys][n]
cudaError_t fft_samples(const DevView& v, cudaStream_t s, const void* src, u32 stride, u32 polys, double2* dst) {
  switch (v.logn) {
    case 12: return launch_samples<12>(v, s, src, stride, polys, dst);
    case 13: return launch_samples<13>(v, s, src, stride, polys, dst);
    case 14: return launch_samples<14>(v, s, src, stride, polys, dst);
    default: return cudaErrorInvalidValue;
  }
}

// src: rows of N residues (of the listed users: 2L rows each); dst: [rows][2][n], or [rows][n] whole (32-bit words)
cudaError_t fft_rows(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* src, const u32* users_dev, u32 rows,
                     bool whole, double2* dst) {
  switch (whole ? v.logn + 100 : v.logn) {
    case 12: return launch_rows<12, 2>(v, lp, s, src, users_dev, rows, dst);
    case 13: return launch_rows<13, 2>(v, lp, s, src, users_dev, rows, dst);
    case 14: return launch_rows<14, 2>(v, lp, s, src, users_dev, rows, dst);
    case 112: return launch_rows<12, 1>(v, lp, s, src, users_dev, rows, dst);
    case 113: return launch_rows<13, 1>(v, lp, s, src, users_dev, rows, dst);
    case 114: return launch_rows<14, 1>(v, lp, s, src, users_dev, rows, dst);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace D2MHE_LAUNCH_NS
