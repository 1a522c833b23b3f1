// Transforms for the double-precision ring products that serve many products: key shares, public keys, and the
// polynomials u and mu_k, which do not depend on the limb.
#include "d2mhe_fft_block.cuh"

namespace {

// s_k of the listed parties, sampled again from its stream (one transform serves every limb), times 1/n (a power of
// two: exact).   grid = n_parties
template <int LOGN>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_fft_secret(DevView v, const u32* __restrict__ parties, u32 tag, double2* __restrict__ dst) {
  using G = FftGeo<LOGN>;
  const u32 party = parties[blockIdx.x];
  if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY)) return;
  double xr[16], xi[16];
  const Stream st(v.seed, tag, 0, party, 0);
  fft_forward<LOGN>(FftSmem<LOGN>(), v.fft, xr, xi, [&](u32 j) {
    return cpx{small_to_double(st.ternary(j)), small_to_double(st.ternary(j + G::n))};
  });
  fft_store<LOGN>(dst + (size_t)party * G::n, xr, xi, 1.0 / (double)G::n);
}

// Sampled polynomials (bytes as sample_streams leaves them in the order of the double-precision kernels), transformed.
// Every stride-th polynomial of src.   grid = polynomials; dst: [grid][n]
template <int LOGN>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_fft_samples(DevView v, const uint4* __restrict__ src, u32 stride, double2* __restrict__ dst) {
  using G = FftGeo<LOGN>;
  const FftSmem<LOGN> sm;
  const uint4* poly = src + (size_t)blockIdx.x * stride * (v.n / 16);
  // number i of thread t is coefficient fft_coef(i): a column's coefficients are this thread's, or (two groups) this
  // thread's and the one's at the same place of the other group
  u32 w[G::GR * 8];
#pragma unroll
  for (int g = 0; g < G::GR; ++g)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint4 a = __ldg(poly + sm.tg + g * G::TG + h * G::T);
      w[8 * g + 4 * h] = a.x, w[8 * g + 4 * h + 1] = a.y, w[8 * g + 4 * h + 2] = a.z, w[8 * g + 4 * h + 3] = a.w;
    }
  auto value = [&](int word, int byte) {
    return small_to_double((int)__byte_perm(w[word], 0, 0x4440 | byte) - D2MHE_GAUSS_B);
  };
  double xr[16], xi[16];
  fft_forward_at<LOGN>(sm, v.fft, xr, xi, [&](auto c_, auto j_, auto h_) {
    // digit j of column c; h: the upper half of the coefficients below n (two groups)
    constexpr int j = decltype(j_)::value;
    if constexpr (G::GR == 2) {  // i = (j & 7) + 8 (h + 2 imaginary) of group j / 8
      constexpr int base = 8 * (j / 8) + 2 * decltype(h_)::value + (j & 7) / 4;
      return cpx{value(base, j & 3), value(base + 4, j & 3)};
    } else {  // i = 2R c + j + R imaginary
      constexpr int i = 2 * G::R * decltype(c_)::value + j;
      return cpx{value(i / 4, i & 3), value((i + G::R) / 4, i & 3)};
    }
  });
  fft_store<LOGN>(dst + (size_t)blockIdx.x * G::n, xr, xi, 1.0);
}

// Both parts of residue rows, times 1/n.   grid = rows * 2; limb of row r = r mod L; src: [..][N], dst: [..][2][n].
// users != null: row r is row r mod 2L of user users[r / 2L].
template <int LOGN>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_fft_rows(DevView v, const __grid_constant__ LimbParams lp, const u64* __restrict__ src, const u32* __restrict__ users,
               double2* __restrict__ dst) {
  using G = FftGeo<LOGN>;
  const u32 half = blockIdx.x & 1u;
  size_t r = blockIdx.x >> 1;
  if (users) {
    const u32 user = users[r / (2 * v.L)];
    if (!D2MHE_CHK(v.chk, user, v.K, SITE_PARTY)) return;
    r = (size_t)user * 2 * v.L + r % (2 * v.L);
  }
  const LimbTab& lt = lp.limbs[r % v.L];
  const u64* row = src + r * v.n;
  double xr[16], xi[16];
  fft_forward<LOGN>(FftSmem<LOGN>(), v.fft, xr, xi, [&](u32 j) {
    if (!D2MHE_CHK(v.chk, j + G::n, v.n, SITE_LOAD)) return cpx{0.0, 0.0};
    return fft_split_pair(row, j, G::n, half, lt);
  });
  fft_store<LOGN>(dst + (2 * r + half) * G::n, xr, xi, 1.0 / (double)G::n);
}

// KERNEL<LOGN> with the exchange area as its shared memory
#define D2MHE_FFT_LAUNCH(KERNEL, LOGN_, grid, ...)                                                      \
  case LOGN_: {                                                                                         \
    cudaError_t e_ = set_smem(KERNEL<LOGN_>, FftGeo<LOGN_>::ex_bytes);                                  \
    if (e_ != cudaSuccess) return e_;                                                                   \
    KERNEL<LOGN_><<<grid, FftGeo<LOGN_>::T, FftGeo<LOGN_>::ex_bytes, s>>>(__VA_ARGS__);                 \
    return cudaGetLastError();                                                                          \
  }
#define D2MHE_FFT_DISPATCH(KERNEL, grid, ...)         \
  switch (v.logn) {                                   \
    D2MHE_FFT_LAUNCH(KERNEL, 12, grid, __VA_ARGS__)   \
    D2MHE_FFT_LAUNCH(KERNEL, 13, grid, __VA_ARGS__)   \
    D2MHE_FFT_LAUNCH(KERNEL, 14, grid, __VA_ARGS__)   \
    default: return cudaErrorInvalidValue;            \
  }

}  // namespace

namespace D2MHE_LAUNCH_NS {

// dst: [K][n], rows of the listed parties only
cudaError_t fft_secret(const DevView& v, cudaStream_t s, const u32* parties_dev, u32 n_parties, u32 tag, double2* dst) {
  D2MHE_FFT_DISPATCH(k_fft_secret, n_parties, v, parties_dev, tag, dst)
}

// every stride-th of the polynomials in src; dst: [polys][n]
cudaError_t fft_samples(const DevView& v, cudaStream_t s, const void* src, u32 stride, u32 polys, double2* dst) {
  D2MHE_FFT_DISPATCH(k_fft_samples, polys, v, reinterpret_cast<const uint4*>(src), stride, dst)
}

// src: rows of N residues (of the listed users: 2L rows each); dst: [rows][2][n]
cudaError_t fft_rows(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* src, const u32* users_dev, u32 rows,
                     double2* dst) {
  D2MHE_FFT_DISPATCH(k_fft_rows, rows * 2, v, lp, src, users_dev, dst)
}

}  // namespace D2MHE_LAUNCH_NS
