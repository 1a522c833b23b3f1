// MBFV.Convert shares by double-precision FFT: (s_k c_1 + mu_k p_{0,i} + e_{0,k}, mu_k p_{1,i} + e_{1,k}), and the
// products c_1 sk_i of BFV.Decrypt under a user's own key.
#include <algorithm>

#include "d2mhe_fft_block.cuh"

namespace {

// One thread block = one (recipient, ciphertext, limb); it walks over its part of the parties.  The transforms of both
// parts of c_1 stay in tensor memory; those of s_k, mu_k (made once per share by k_fft_samples) and the recipient's
// public key come from L2: h_0 is one inverse transform per part, of the sum of two products.
// noise: the bytes of mu, e_0, e_1, N each per share.   grid: fft_deal, rows = n_units * L
template <int LOGN, bool MIXED>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_convert_fft(DevView v, const __grid_constant__ LimbParams lp, const u64* __restrict__ agg,
                  const u32* __restrict__ recipients, const u32* __restrict__ parties, u32 n_parties, u32 n_cts,
                  u32 unit_first, const double2* __restrict__ mu_fft, const uint4* __restrict__ noise,
                  u64* __restrict__ shares, FftDeal deal) {
  using G = FftGeo<LOGN>;
  constexpr int n = G::n;
  u32 block_part, split;
  const u32 rest = fft_dealt<MIXED>(deal, blockIdx.x, block_part, split);
  const u32 l = rest % v.L, ulocal = rest / v.L, unit = unit_first + ulocal;
  if (block_part >= n_parties) return;
  const u32 irec = unit / n_cts, cl = unit % n_cts, tid = threadIdx.x;
  u32 recipient = recipients[irec];
  if (!D2MHE_CHK(v.chk, recipient, v.K, SITE_PARTY)) recipient = 0;
  const LimbTab& lt = lp.limbs[l];
  FftSmem<LOGN, 2> sm(v);
  if (tid == 0) sm.init();
  if (tid < 32) tmem_alloc(sm.slot, G::tmem_cols(2));
  __syncthreads();
  const u32 tbase = *sm.slot, tm = tmem_thread_base(tbase, 2 * G::WORDS);
  const size_t row = (size_t)l * v.n, poly = (size_t)v.L * v.n;
  const u64* c1 = agg + ((size_t)unit * 2 + 1) * poly + row;
  double xr[16], xi[16];
#pragma unroll 1
  for (u32 half = 0; half < 2; ++half) {
    fft_forward<LOGN>(sm, v.fft, xr, xi, [&](u32 j) {
      if (!D2MHE_CHK(v.chk, j + n, v.n, SITE_LOAD)) return cpx{0.0, 0.0};
      return fft_split_pair(c1, j, n, half, lt.p, lt.fftc.h);
    });
    fft_to_tmem(tm + half * G::WORDS, xr, xi);
  }
  tmem_store_done();
  const double2* pk = v.upk_fft + ((size_t)recipient * 2 * v.L + l) * 2 * n;  // [component][part], components 2 L n apart
  u32 a = block_part, i = 0;  // i = 2 component + part
#pragma unroll 1
  while (a < n_parties) {
    u32 party = parties[a];
    if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY)) party = 0;
    const size_t share = (size_t)ulocal * n_parties + a;
    const u32 comp = i >> 1;
    const bool high = (i & 1u) != 0;
    u64* out = shares + ((((size_t)irec * n_parties + a) * n_cts + cl) * 2 + comp) * poly + row;
    const double2* key = pk + ((size_t)comp * v.L * 2 + (high ? 1 : 0)) * n;
    FftNoise<LOGN> nz;
    cpx tw[G::COLS];
    if (comp == 0) {
      fft_load(sm, v.s_fft + (size_t)party * n, xr, xi);
      fft_product_sum(sm, tm + (high ? G::WORDS : 0), mu_fft + share * n, key, xr, xi);
    } else {
      fft_load(sm, mu_fft + share * n, xr, xi);
      fft_product_row(sm, key, xr, xi);
    }
    fft_inverse<LOGN>(sm, v.fft, xr, xi, tw, [&] {
      if (high) nz.load(noise + ((share * 3 + 1 + comp) * v.n) / 16, v.chk);
    });
    fft_finish<LOGN>(sm, lt, lt.fftc, tw, xr, xi, high, nz, [&](u32 j, u64 s) {
      if (D2MHE_CHK(v.chk, j, v.n, SITE_STORE)) __stcs(out + j, fft_canon(s, lt));
    });
    i = (i + 1) & 3u;
    if (i == 0) a += split;
  }
  __syncthreads();
  if (tid == 0) sm.finish(v);
  if (tid < 32) tmem_free(tbase, G::tmem_cols(2));
}

template <int LOGN>
cudaError_t launch_convert(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg,
                           const u32* recipients_dev, const u32* parties_dev, u32 n_parties, u32 n_cts, u32 unit_first,
                           u32 n_units, const double2* mu_fft, const void* noise, u64* shares) {
  using G = FftGeo<LOGN>;
  const FftDeal deal = fft_deal(v.sms * G::CTAS, n_units * v.L, n_parties, FFT_WORK_CONVERT);
  const auto kernel = deal.whole ? k_convert_fft<LOGN, true> : k_convert_fft<LOGN, false>;
  const cudaError_t e = set_smem(kernel, G::smem_bytes(2));
  if (e != cudaSuccess) return e;
  kernel<<<deal.blocks, G::T, G::smem_bytes(2), s>>>(
      v, lp, agg, recipients_dev, parties_dev, n_parties, n_cts, unit_first, mu_fft,
      reinterpret_cast<const uint4*>(noise), shares, deal);
  return cudaGetLastError();
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

// scratch: at least n_parties * 11 N bytes per unit (transforms of mu_k, bytes of mu, e_0, e_1)
cudaError_t convert_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg,
                        const u32* recipients_dev, u32 n_rec, const u32* parties_dev, u32 n_parties, u32 ct_first,
                        u32 n_cts, u64* shares, void* scratch, size_t scratch_bytes, u32* launches) {
  const size_t per_unit = (size_t)n_parties * 11 * v.n;
  const u32 n_units = n_rec * n_cts;
  u32 per_batch = (u32)std::min<size_t>(scratch_bytes / per_unit, n_units);
  if (per_batch == 0) return cudaErrorInvalidValue;
  per_batch = whole_wave_batch(v, per_batch, n_units, v.L);
  for (u32 first = 0; first < n_units; first += per_batch) {
    const u32 nu = std::min(per_batch, n_units - first);
    double2* mu_fft = reinterpret_cast<double2*>(scratch);
    unsigned char* noise = reinterpret_cast<unsigned char*>(scratch) + (size_t)nu * n_parties * 8 * v.n;
    cudaError_t e = sample_streams(v, s, recipients_dev, parties_dev, n_parties, ct_first, n_cts, first, nu,
                                   kSampleConvert, true, noise);
    if (e != cudaSuccess) return e;
    e = fft_samples(v, s, noise, 3, nu * n_parties, mu_fft);
    if (e != cudaSuccess) return e;
    switch (v.logn) {
#define D2MHE_CONVERT(LOGN_)                                                                                          \
  case LOGN_:                                                                                                         \
    e = launch_convert<LOGN_>(v, lp, s, agg, recipients_dev, parties_dev, n_parties, n_cts, first, nu, mu_fft, noise, \
                              shares);                                                                                \
    break
      D2MHE_CONVERT(12);
      D2MHE_CONVERT(13);
      D2MHE_CONVERT(14);
#undef D2MHE_CONVERT
      default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    *launches += 3;
  }
  return cudaSuccess;
}

}  // namespace D2MHE_LAUNCH_NS
