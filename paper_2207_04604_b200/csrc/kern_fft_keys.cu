// Transforms of key material for the double-precision ring products.
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

template <int LOGN>
cudaError_t launch_secret(const DevView& v, cudaStream_t s, const u32* parties_dev, u32 n_parties, u32 tag, double2* dst) {
  using G = FftGeo<LOGN>;
  cudaError_t e = set_smem(k_fft_secret<LOGN>, G::ex_bytes);
  if (e != cudaSuccess) return e;
  k_fft_secret<LOGN><<<n_parties, G::T, G::ex_bytes, s>>>(v, parties_dev, tag, dst);
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

}  // namespace D2MHE_LAUNCH_NS
