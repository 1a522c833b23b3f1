// Encryption and decryption shares on 32-bit words by double-precision FFT (see d2mhe_fft.cuh): a residue below 2^30
// is one part, so a product takes one transform instead of two, and nothing waits in shared memory.
// Used when the error bound there allows it: log2 N + bits <= 43, where it is 0.44 for any residues.  Seen: below 2^-11.
#include <algorithm>

#include "d2mhe_fft_block.cuh"

namespace {

__device__ __forceinline__ cpx centred_pair(u32 a, u32 b, const LimbTab& lt) {
  const u32 p = (u32)lt.p, half = p >> 1;
  return cpx{small_to_double((int)(a > half ? a - p : a)), small_to_double((int)(b > half ? b - p : b))};
}

// V + e mod p, below 3p, from the rounded result: s = V + e + a multiple of p is in [0, 2^45); the quotient from its
// bits above 14 and floor(2^46 / p) is at most two low.
__device__ __forceinline__ u32 fft_residue32(u64 bits, u32 e0, const LimbTab& lt) {
  const u64 s = (bits >> D2MHE_FFT32_F) + (lt.fft32_k + e0);
  return (u32)s - __umulhi((u32)(s >> 14), lt.fft32_mu) * (u32)lt.p;
}

// the end of an inverse transform: store(coefficient, value below 3p)
template <int LOGN, class Store>
__device__ __forceinline__ void fft_finish32(const FftSmem<LOGN, 0>& sm, const LimbTab& lt, const cpx (&tw)[FftGeo<LOGN>::COLS],
                                             double* xr, double* xi, const FftNoise<LOGN>& nz, Store store) {
  fft_results<LOGN>(sm, tw, xr, xi, D2MHE_FFT32_MAGIC, [&](auto, auto i_, auto rr_, const u64(&v)[4]) {
    static_for<4>([&](auto q_) {
      constexpr int q = decltype(q_)::value, i = fft_result_number<decltype(i_)::value, decltype(rr_)::value, q>();
      store(fft_coef<LOGN>(sm, i), fft_residue32(v[q], nz.template get<i>(), lt));
    });
  });
}

template <int LOGN>
constexpr size_t smem32() {
  return FftGeo<LOGN>::smem_bytes(0);
}

// One thread block = one (recipient, ciphertext, limb) and its part of the parties; as k_share_fft.
// grid: fft_deal, rows = n_units * L
template <int LOGN, bool MIXED>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_share32_fft(DevView v, const __grid_constant__ LimbParams lp, const u32* __restrict__ agg,
                  const u32* __restrict__ parties, u32 n_parties, u32 n_cts, u32 unit_first,
                  const uint4* __restrict__ noise, u32* __restrict__ shares, FftDeal deal) {
  using G = FftGeo<LOGN>;
  constexpr int n = G::n;
  u32 part, split;
  const u32 rest = fft_dealt<MIXED>(deal, blockIdx.x, part, split);
  const u32 l = rest % v.L, ulocal = rest / v.L, unit = unit_first + ulocal;
  if (part >= n_parties) return;
  const u32 irec = unit / n_cts, cl = unit % n_cts, tid = threadIdx.x;
  const LimbTab& lt = lp.limbs[l];
  const u32 p = (u32)lt.p;
  FftSmem<LOGN, 0> sm(v);
  if (tid == 0) sm.init();
  if (tid < 32) tmem_alloc(sm.slot, G::tmem_cols(1));
  __syncthreads();
  const u32 tbase = *sm.slot, tm = tmem_thread_base(tbase, G::WORDS);
  const size_t row = (size_t)l * v.n, poly = (size_t)v.L * v.n;
  const u32* c1 = agg + ((size_t)unit * 2 + 1) * poly + row;
  double xr[16], xi[16];
  fft_forward<LOGN>(sm, v.fft, xr, xi, [&](u32 j) {
    if (!D2MHE_CHK(v.chk, j + n, v.n, SITE_LOAD)) return cpx{0.0, 0.0};
    return centred_pair(__ldg(c1 + j), __ldg(c1 + j + n), lt);
  });
  fft_to_tmem(tm, xr, xi);
  tmem_store_done();
  auto key_of = [&](u32 a) {
    u32 party = parties[a];
    if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY)) party = 0;
    return v.s_fft + (size_t)party * n;
  };
  const double2* key = key_of(part);
#pragma unroll 1
  for (u32 a = part; a < n_parties; a += split) {
    const double2* next = a + split < n_parties ? key_of(a + split) : key;
    u32* out = shares + (((size_t)irec * n_parties + a) * n_cts + cl) * poly + row;
    FftNoise<LOGN> nz;
    cpx tw[G::COLS];
    fft_load(sm, key, xr, xi);
    fft_product_tmem(tm, xr, xi);
    fft_inverse<LOGN>(sm, v.fft, xr, xi, tw, [&] { nz.load(noise + (((size_t)ulocal * n_parties + a) * v.n) / 16, v.chk); });
    fft_finish32<LOGN>(sm, lt, tw, xr, xi, nz, [&](u32 j, u32 x) {
      if (D2MHE_CHK(v.chk, j, v.n, SITE_STORE)) __stcs(out + j, csub32(csub32(x, p), p));
    });
    key = next;
  }
  __syncthreads();
  if (tid == 0) sm.finish(v);
  if (tid < 32) tmem_free(tbase, G::tmem_cols(1));
}

// One thread block = one (party, ciphertext, limb), or one component of it; as k_encrypt_fft.
template <int LOGN>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_encrypt32_fft(DevView v, const __grid_constant__ LimbParams lp, u32 unit_first, const double2* __restrict__ u_fft,
                    const uint4* __restrict__ noise, const u32* __restrict__ plain, u32* __restrict__ ct, u32 split) {
  using G = FftGeo<LOGN>;
  constexpr int n = G::n;
  const u32 part = blockIdx.x % split, rest = blockIdx.x / split;
  const u32 l = rest % v.L, ulocal = rest / v.L, unit = unit_first + ulocal, tid = threadIdx.x;
  const LimbTab& lt = lp.limbs[l];
  const u32 p = (u32)lt.p, delta = (u32)lt.delta, delta_sh = (u32)(lt.delta_sh >> 32);
  FftSmem<LOGN, 0> sm(v);
  sm.announce = false;
  if (tid == 0) sm.init();
  if (tid < 32) tmem_alloc(sm.slot, G::tmem_cols(1));
  __syncthreads();
  const u32 tbase = *sm.slot, tm = tmem_thread_base(tbase, G::WORDS);
  double xr[16], xi[16];
  fft_load(sm, u_fft + (size_t)ulocal * n, xr, xi);
  fft_loaded_to_tmem(tm, xr, xi);
  tmem_store_done();
  const u32* m = plain + (size_t)unit * v.n;
  const u32 end = split > 1 ? part + 1 : 2;
#pragma unroll 1
  for (u32 comp = part; comp < end; ++comp) {
    u32* out = ct + (((size_t)unit * 2 + comp) * v.L + l) * v.n;
    FftNoise<LOGN> nz;
    cpx tw[G::COLS];
    fft_load(sm, v.pk_fft + ((size_t)comp * v.L + l) * n, xr, xi);
    fft_product_tmem(tm, xr, xi);
    fft_inverse<LOGN>(sm, v.fft, xr, xi, tw, [&] { nz.load(noise + (((size_t)ulocal * 3 + 1 + comp) * v.n) / 16, v.chk); });
    fft_finish32<LOGN>(sm, lt, tw, xr, xi, nz, [&](u32 j, u32 x) {
      if (!D2MHE_CHK(v.chk, j, v.n, SITE_STORE)) return;
      x = csub32(csub32(x, p), p);
      if (comp == 0) x = csub32(x + csub32(shoup32(__ldg(m + j), delta, delta_sh, p), p), p);  // Lambda m
      out[j] = x;
    });
  }
  __syncthreads();
  if (tid == 0) sm.finish(v);
  if (tid < 32) tmem_free(tbase, G::tmem_cols(1));
}

template <int LOGN>
cudaError_t launch_share32(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* agg, const u32* parties_dev,
                           u32 n_parties, u32 n_cts, u32 unit_first, u32 n_units, const void* noise, u32* shares) {
  using G = FftGeo<LOGN>;
  const FftDeal deal = fft_deal(v.sms * G::CTAS, n_units * v.L, n_parties, FFT_WORK_SHARE32);
  const auto kernel = deal.whole ? k_share32_fft<LOGN, true> : k_share32_fft<LOGN, false>;
  const cudaError_t e = set_smem(kernel, smem32<LOGN>());
  if (e != cudaSuccess) return e;
  kernel<<<deal.blocks, G::T, smem32<LOGN>(), s>>>(
      v, lp, agg, parties_dev, n_parties, n_cts, unit_first, reinterpret_cast<const uint4*>(noise), shares, deal);
  return cudaGetLastError();
}
template <int LOGN>
cudaError_t launch_encrypt32(const DevView& v, const LimbParams& lp, cudaStream_t s, u32 unit_first, u32 n_units,
                             const double2* u_fft, const void* noise, const u32* plain, u32* ct) {
  using G = FftGeo<LOGN>;
  cudaError_t e = set_smem(k_encrypt32_fft<LOGN>, smem32<LOGN>());
  if (e != cudaSuccess) return e;
  const u32 split = fft_component_split(v, n_units * v.L, G::CTAS);
  k_encrypt32_fft<LOGN><<<n_units * v.L * split, G::T, smem32<LOGN>(), s>>>(
      v, lp, unit_first, u_fft, reinterpret_cast<const uint4*>(noise), plain, ct, split);
  return cudaGetLastError();
}
#define D2MHE_BY_SIZE(FN, ...)                   \
  switch (v.logn) {                              \
    case 12: return FN<12>(__VA_ARGS__);         \
    case 13: return FN<13>(__VA_ARGS__);         \
    case 14: return FN<14>(__VA_ARGS__);         \
    default: return cudaErrorInvalidValue;       \
  }

}  // namespace

namespace D2MHE_LAUNCH_NS {

cudaError_t share32_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* agg, const u32* parties_dev,
                        u32 n_parties, u32 n_cts, u32 unit_first, u32 n_units, const void* noise, u32* shares) {
  D2MHE_BY_SIZE(launch_share32, v, lp, s, agg, parties_dev, n_parties, n_cts, unit_first, n_units, noise, shares)
}

// noise: the bytes of u, e_0, e_1 of every unit; u_fft: [n_units][n]
cudaError_t encrypt32_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, u32 unit_first, u32 n_units,
                          const double2* u_fft, const void* noise, const u32* plain, u32* ct) {
  D2MHE_BY_SIZE(launch_encrypt32, v, lp, s, unit_first, n_units, u_fft, noise, plain, ct)
}
}  // namespace D2MHE_LAUNCH_NS
