// Decryption shares h = s_k c_1 + e by double-precision FFT (see d2mhe_fft.cuh and DevView::fft_on).
#include <algorithm>

#include "d2mhe_fft_block.cuh"

namespace {

// One thread block = one (recipient, ciphertext, limb); it walks over the parties of the list.
// What bounds it: the double-precision pipe and the issue slots around it (42, 46 and 52 double-precision and as many other
// instructions per complex point and part at N = 4096, 8192 and 16384, in captures of whole waves; the pipe is busy 48, 47
// and 45 %, the load/store data pipe 65, 58 and 55 %), then shared memory (two exchanges per transform).  The transforms of
// both parts of c_1 stay in tensor memory (all 256 KB of an SM: 32 bytes per point), where neither the load/store
// pipe nor L2 sees them again; the key's transform does not depend on the limb (8 N bytes per party) and comes from
// L2, or from L1 when the other block of the SM has just read it.  (Fetching it point by point into the registers that
// the end of the previous transform frees was slower: 46.8 k instead of 40.0 k clocks per share and limb at N = 16384,
// 18.5 k instead of 17.3 k at N = 8192.)  The rounded low part waits in shared memory, thread by thread, for the high
// part.  The shares are written with a streaming hint, so that the keys stay in L2.
// grid: fft_deal, rows = n_units * L.
// OWN: the products c_1 sk_i with user i's own key instead (parties: the users of the units' rows, one to a unit, no
// noise), as BFV.Decrypt needs them.
template <int LOGN, bool OWN, bool MIXED>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_share_fft(DevView v, const __grid_constant__ LimbParams lp, const u64* __restrict__ agg,
                const u32* __restrict__ parties, u32 n_parties, u32 n_cts, u32 unit_first,
                const uint4* __restrict__ noise, u64* __restrict__ shares, FftDeal deal) {
  using G = FftGeo<LOGN>;
  constexpr int n = G::n;
  u32 part, split;
  const u32 rest = fft_dealt<MIXED>(deal, blockIdx.x, part, split);
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
  const u64* c1 = agg + ((size_t)unit * 2 + 1) * poly + row;
  double xr[16], xi[16];
#pragma unroll 1
  for (u32 half = 0; half < 2; ++half) {
    fft_forward<LOGN>(sm, v.fft, xr, xi, [&](u32 j) {
      if (!D2MHE_CHK(v.chk, j + n, v.n, SITE_LOAD)) return cpx{0.0, 0.0};
      return fft_split_pair(c1, j, n, half, lt.p, lt.fft.h);
    });
    fft_to_tmem(tm + half * G::WORDS, xr, xi);
  }
  tmem_store_done();
  // the stored transform of a party's key; a party number that fails the check reads row 0
  auto key_of = [&](u32 a) {
    u32 party = parties[OWN ? irec : a];
    if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY)) party = 0;
    return (OWN ? v.usk_fft : v.s_fft) + (size_t)party * n;
  };
  const double2* key = key_of(part);
  u32 a = part;
  bool high = false;
#pragma unroll 1
  while (a < n_parties) {
    const double2* next = high && a + split < n_parties ? key_of(a + split) : key;  // the address, a part ahead
    u64* out = shares + (((size_t)irec * n_parties + a) * n_cts + cl) * poly + row;
    typename std::conditional<OWN, FftNoNoise, FftNoise<LOGN>>::type nz;
    cpx tw[G::COLS];
    fft_load(sm, key, xr, xi);
    fft_product_tmem(tm + (high ? G::WORDS : 0), xr, xi);
    fft_inverse<LOGN>(sm, v.fft, xr, xi, tw, [&] {
      if constexpr (!OWN)
        if (high) nz.load(noise + (((size_t)ulocal * n_parties + a) * v.n) / 16, v.chk);
    });
    fft_finish<LOGN>(sm, lt, lt.fft, tw, xr, xi, high, nz, [&](u32 j, u64 s) {
      if (D2MHE_CHK(v.chk, j, v.n, SITE_STORE)) __stcs(out + j, fft_canon(s, lt));
    });
    key = next;
    if (high) a += split;
    high = !high;
  }
  __syncthreads();
  if (tid == 0) sm.finish(v);
  if (tid < 32) tmem_free(tbase, G::tmem_cols(2));
}

template <int LOGN, bool OWN>
cudaError_t launch_share(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, const u32* parties_dev,
                         u32 n_parties, u32 n_cts, u32 unit_first, u32 n_units, const void* noise, u64* shares) {
  using G = FftGeo<LOGN>;
  const FftDeal deal = fft_deal(v.sms * G::CTAS, n_units * v.L, n_parties, FFT_WORK_SHARE);
  auto kernel = k_share_fft<LOGN, OWN, false>;
  if constexpr (!OWN)  // one product a row: every row is whole
    if (deal.whole) kernel = k_share_fft<LOGN, OWN, true>;
  const cudaError_t e = set_smem(kernel, G::smem_bytes(1));
  if (e != cudaSuccess) return e;
  kernel<<<deal.blocks, G::T, G::smem_bytes(1), s>>>(v, lp, agg, parties_dev, n_parties, n_cts, unit_first,
                                                     reinterpret_cast<const uint4*>(noise), shares, deal);
  return cudaGetLastError();
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

cudaError_t share_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, const u32* parties_dev,
                      u32 n_parties, u32 n_cts, u32 unit_first, u32 n_units, const void* noise, u64* shares) {
  switch (v.logn) {
    case 12: return launch_share<12, false>(v, lp, s, agg, parties_dev, n_parties, n_cts, unit_first, n_units, noise, shares);
    case 13: return launch_share<13, false>(v, lp, s, agg, parties_dev, n_parties, n_cts, unit_first, n_units, noise, shares);
    case 14: return launch_share<14, false>(v, lp, s, agg, parties_dev, n_parties, n_cts, unit_first, n_units, noise, shares);
    default: return cudaErrorInvalidValue;
  }
}

// prod[i, c] = c_1 sk_i, canonical, for users[i] and ct[i, c]
cudaError_t secret_product_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* ct,
                               const u32* users_dev, u32 n_users, u32 n_cts, u64* prod) {
  const u32 n_units = n_users * n_cts;
  switch (v.logn) {
    case 12: return launch_share<12, true>(v, lp, s, ct, users_dev, 1, n_cts, 0, n_units, nullptr, prod);
    case 13: return launch_share<13, true>(v, lp, s, ct, users_dev, 1, n_cts, 0, n_units, nullptr, prod);
    case 14: return launch_share<14, true>(v, lp, s, ct, users_dev, 1, n_cts, 0, n_units, nullptr, prod);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace D2MHE_LAUNCH_NS
