// MBFV.Bootstrap shares by double-precision FFT: (s_k c_1 - Lambda M_k + e_{0,k}, -s_k alpha + Lambda M_k + e_{1,k}).
#include <algorithm>

#include "d2mhe_fft_block.cuh"

namespace {

// One thread block = one (recipient, ciphertext, limb) and component; it walks over its part of the parties.  The
// component's fixed factor (c_1, or -alpha) stays in tensor memory, as in the share kernel.
// alpha: [units][L][N] residues; noise: the bytes of e_0, e_1, N each per share; masks: M_k, N words per share.
// grid: fft_deal, rows = n_units * L * 2
template <int LOGN, bool MIXED>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_boot_fft(DevView v, const __grid_constant__ LimbParams lp, const u64* __restrict__ agg,
               const u32* __restrict__ parties, u32 n_parties, u32 n_cts, u32 unit_first, const u64* __restrict__ alpha,
               const uint4* __restrict__ noise, const u32* __restrict__ masks, u64* __restrict__ shares, FftDeal deal) {
  using G = FftGeo<LOGN>;
  constexpr int n = G::n;
  u32 part, split;
  const u32 row_comp = fft_dealt<MIXED>(deal, blockIdx.x, part, split), comp = row_comp & 1u, rest = row_comp / 2;
  const u32 l = rest % v.L, ulocal = rest / v.L, unit = unit_first + ulocal;
  if (part >= n_parties) return;
  const u32 irec = unit / n_cts, cl = unit % n_cts, tid = threadIdx.x;
  const LimbTab& lt = lp.limbs[l];
  FftSmem<LOGN> sm(v);
  if (tid == 0) sm.init();
  if (tid < 32) tmem_alloc(sm.slot, G::tmem_cols(2));
  __syncthreads();
  const u32 tbase = *sm.slot, tm = tmem_thread_base(tbase, 2 * G::WORDS);
  const size_t row = (size_t)l * v.n, poly = (size_t)v.L * v.n;
  const u64* fixed = comp ? alpha + (size_t)ulocal * poly + row : agg + ((size_t)unit * 2 + 1) * poly + row;
  const double sign = comp ? -1.0 : 1.0;
  double xr[16], xi[16];
#pragma unroll 1
  for (u32 half = 0; half < 2; ++half) {
    fft_forward<LOGN>(sm, v.fft, xr, xi, [&](u32 j) {
      if (!D2MHE_CHK(v.chk, j + n, v.n, SITE_LOAD)) return cpx{0.0, 0.0};
      const cpx z = fft_split_pair(fixed, j, n, half, lt.p, lt.fft.h);
      return cpx{z.r * sign, z.i * sign};
    });
    fft_to_tmem(tm + half * G::WORDS, xr, xi);
  }
  tmem_store_done();
  auto key_of = [&](u32 a) {
    u32 party = parties[a];
    if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY)) party = 0;
    return v.s_fft + (size_t)party * n;
  };
  const double2* key = key_of(part);
  u32 a = part;
  bool high = false;
#pragma unroll 1
  while (a < n_parties) {
    const double2* next = high && a + split < n_parties ? key_of(a + split) : key;
    const size_t share = (size_t)ulocal * n_parties + a;
    u64* out = shares + ((((size_t)irec * n_parties + a) * n_cts + cl) * 2 + comp) * poly + row;
    const u32* mask = masks + share * v.n;
    FftNoise<LOGN> nz;
    cpx tw[G::COLS];
    fft_load(sm, key, xr, xi);
    fft_product_tmem(tm + (high ? G::WORDS : 0), xr, xi);
    fft_inverse<LOGN>(sm, v.fft, xr, xi, tw, [&] {
      if (high) nz.load(noise + ((share * 2 + comp) * v.n) / 16, v.chk);
    });
    fft_finish<LOGN>(sm, lt, lt.fft, tw, xr, xi, high, nz, [&](u32 j, u64 s) {
      if (!D2MHE_CHK(v.chk, j, v.n, SITE_STORE)) return;
      const u64 dm = shoup_u32(__ldg(mask + j), lt.delta, lt.delta_sh, lt.np);  // Lambda M_k, below 2p
      __stcs(out + j, fft_canon(s + (comp ? dm : lt.twop - dm), lt));
    });
    key = next;
    if (high) a += split;
    high = !high;
  }
  __syncthreads();
  if (tid == 0) sm.finish(v);
  if (tid < 32) tmem_free(tbase, G::tmem_cols(2));
}

template <int LOGN>
cudaError_t launch_boot(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, const u32* parties_dev,
                        u32 n_parties, u32 n_cts, u32 unit_first, u32 n_units, const u64* alpha, const void* noise,
                        const u32* masks, u64* shares) {
  using G = FftGeo<LOGN>;
  const FftDeal deal = fft_deal(v.sms * G::CTAS, n_units * v.L * 2, n_parties, FFT_WORK_BOOT);
  const auto kernel = deal.whole ? k_boot_fft<LOGN, true> : k_boot_fft<LOGN, false>;
  const cudaError_t e = set_smem(kernel, G::smem_bytes(1));
  if (e != cudaSuccess) return e;
  kernel<<<deal.blocks, G::T, G::smem_bytes(1), s>>>(
      v, lp, agg, parties_dev, n_parties, n_cts, unit_first, alpha, reinterpret_cast<const uint4*>(noise), masks, shares,
      deal);
  return cudaGetLastError();
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

// scratch: per unit 8 N L bytes (alpha) and 6 N bytes for each party (bytes of e_0, e_1, words of M_k)
cudaError_t boot_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, const u32* recipients_dev,
                     u32 n_rec, const u32* parties_dev, u32 n_parties, u32 ct_first, u32 n_cts, u64* shares,
                     void* scratch, size_t scratch_bytes, u32* launches) {
  const size_t poly_bytes_ = (size_t)v.L * v.n * sizeof(u64), per_unit = poly_bytes_ + (size_t)n_parties * 6 * v.n;
  const u32 n_units = n_rec * n_cts;
  u32 per_batch = (u32)std::min<size_t>(scratch_bytes / per_unit, n_units);
  if (per_batch == 0) return cudaErrorInvalidValue;
  per_batch = whole_wave_batch(v, per_batch, n_units, 2 * v.L);
  for (u32 first = 0; first < n_units; first += per_batch) {
    const u32 nu = std::min(per_batch, n_units - first);
    unsigned char* base = reinterpret_cast<unsigned char*>(scratch);
    u64* alpha = reinterpret_cast<u64*>(base);
    u32* masks = reinterpret_cast<u32*>(base + nu * poly_bytes_);
    unsigned char* noise = base + nu * (poly_bytes_ + (size_t)n_parties * 4 * v.n);
    cudaError_t e = sample_alpha(v, s, recipients_dev, ct_first, n_cts, first, nu, alpha);
    if (e != cudaSuccess) return e;
    e = sample_boot(v, s, recipients_dev, parties_dev, n_parties, ct_first, n_cts, first, nu, true, noise, masks, launches);
    if (e != cudaSuccess) return e;
    switch (v.logn) {
#define D2MHE_BOOT(LOGN_)                                                                                          \
  case LOGN_:                                                                                                      \
    e = launch_boot<LOGN_>(v, lp, s, agg, parties_dev, n_parties, n_cts, first, nu, alpha, noise, masks, shares);  \
    break
      D2MHE_BOOT(12);
      D2MHE_BOOT(13);
      D2MHE_BOOT(14);
#undef D2MHE_BOOT
      default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    *launches += 2;
  }
  return cudaSuccess;
}

}  // namespace D2MHE_LAUNCH_NS
