// BFV.Encrypt under the collective key by double-precision FFT: ct = (Lambda m + u p_0 + e_0, u p_1 + e_1).
#include <algorithm>

#include "d2mhe_fft_block.cuh"

namespace {

// One thread block = one (party, ciphertext, limb), or one component of it (split = 2).  The transform of u does not
// depend on the limb: it is made once per (party, ciphertext) by k_fft_samples and comes from L2, or (OWN_U, calls of one
// wave of blocks) every block makes it from the samples; it stays in tensor memory for all four products (two components,
// two parts of the key).  Bound like the share kernel.
// noise: the bytes of u, e_0 and e_1, N each per unit.   grid = n_units * L * split
template <int LOGN, bool OWN_U>
__global__ void __launch_bounds__(FftGeo<LOGN>::T, FftGeo<LOGN>::CTAS)
    k_encrypt_fft(DevView v, const __grid_constant__ LimbParams lp, u32 unit_first, const double2* __restrict__ u_fft,
                  const uint4* __restrict__ noise, const u32* __restrict__ plain, u64* __restrict__ ct, u32 split) {
  using G = FftGeo<LOGN>;
  constexpr int n = G::n;
  const u32 part = blockIdx.x % split, rest = blockIdx.x / split;
  const u32 l = rest % v.L, ulocal = rest / v.L, unit = unit_first + ulocal, tid = threadIdx.x;
  const LimbTab& lt = lp.limbs[l];
  FftSmem<LOGN> sm(v);
  sm.announce = LOGN == 12;
  if (tid == 0) sm.init();
  if (tid < 32) tmem_alloc(sm.slot, G::tmem_cols(1));
  __syncthreads();
  const u32 tbase = *sm.slot, tm = tmem_thread_base(tbase, G::WORDS);
  double xr[16], xi[16];
  if (!OWN_U) {
    fft_load(sm, u_fft + (size_t)ulocal * n, xr, xi);
    fft_loaded_to_tmem(tm, xr, xi);
  } else {
    fft_samples_forward(sm, v.fft, noise + (size_t)ulocal * 3 * (v.n / 16), xr, xi);
    fft_to_tmem(tm, xr, xi);
  }
  tmem_store_done();
  const u32* m = plain + (size_t)unit * v.n;
  const u32 end = split > 1 ? 2 * part + 2 : 4;
#pragma unroll 1
  for (u32 i = 2 * part; i < end; ++i) {  // component i / 2, part i % 2 of the key
    const u32 comp = i >> 1;
    const bool high = (i & 1u) != 0;
    u64* out = ct + (((size_t)unit * 2 + comp) * v.L + l) * v.n;
    FftNoise<LOGN> nz;
    cpx tw[G::COLS];
    fft_load(sm, v.pk_fft + (((size_t)comp * v.L + l) * 2 + (high ? 1 : 0)) * n, xr, xi);
    fft_product_tmem(tm, xr, xi);
    fft_inverse<LOGN>(sm, v.fft, xr, xi, tw, [&] {
      if (high) nz.load(noise + (((size_t)ulocal * 3 + 1 + comp) * v.n) / 16, v.chk);
    });
    fft_finish<LOGN>(sm, lt, lt.fft, tw, xr, xi, high, nz, [&](u32 j, u64 s) {
      if (!D2MHE_CHK(v.chk, j, v.n, SITE_STORE)) return;
      if (comp == 0) s += shoup_u32(__ldg(m + j), lt.delta, lt.delta_sh, lt.np);  // Lambda m, below 2p
      out[j] = fft_canon(s, lt);
    });
  }
  __syncthreads();
  if (tid == 0) sm.finish(v);
  if (tid < 32) tmem_free(tbase, G::tmem_cols(1));
}

template <int LOGN>
cudaError_t launch_encrypt(const DevView& v, const LimbParams& lp, cudaStream_t s, u32 unit_first, u32 n_units,
                           const double2* u_fft, const void* noise, const u32* plain, u64* ct) {
  using G = FftGeo<LOGN>;
  const auto kernel = u_fft ? k_encrypt_fft<LOGN, false> : k_encrypt_fft<LOGN, true>;
  const cudaError_t e = set_smem(kernel, G::smem_bytes(1));
  if (e != cudaSuccess) return e;
  const u32 split = fft_component_split(v, n_units * v.L, G::CTAS);
  kernel<<<n_units * v.L * split, G::T, G::smem_bytes(1), s>>>(v, lp, unit_first, u_fft,
                                                               reinterpret_cast<const uint4*>(noise), plain, ct, split);
  return cudaGetLastError();
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

// scratch: at least 11 N bytes (the transform of u and the bytes of u, e_0, e_1 of a unit)
cudaError_t encrypt_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* parties_dev, u32 ct_first,
                        u32 n_cts, u32 n_units, const u32* plain, u64* ct, void* scratch, size_t scratch_bytes,
                        u32* launches) {
  const size_t per_unit = 11 * (size_t)v.n;
  u32 per_batch = (u32)std::min<size_t>(scratch_bytes / per_unit, n_units);
  if (per_batch == 0) return cudaErrorInvalidValue;
  per_batch = whole_wave_batch(v, per_batch, n_units, v.L);
  for (u32 first = 0; first < n_units; first += per_batch) {
    const u32 nu = std::min(per_batch, n_units - first);
    double2* u_fft = reinterpret_cast<double2*>(scratch);
    unsigned char* noise = reinterpret_cast<unsigned char*>(scratch) + (size_t)nu * 8 * v.n;
    cudaError_t e = sample_streams(v, s, nullptr, parties_dev, 1, ct_first, n_cts, first, nu, kSampleEncrypt, true, noise);
    if (e != cudaSuccess) return e;
    // One wave of blocks: each makes the transform of its u, which takes less time than a launch for it; more waves would make
    // it again and again.  Whole calls with it and with a launch for it, L = 4: N = 4096, 88 blocks 25.9 / 28.4 us, a full wave
    // (592) 54.9 / 56.5; N = 8192, 44 blocks 27.3 / 31.1, a full wave (296) 55.6 / 58.2; N = 16384, 20 blocks 37.3 / 42.4, a
    // full wave (148) 60.9 / 65.3; with L = 1 and L = 8 it saves 0.6 to 8 us everywhere, too.
    const u32 ctas = v.logn == 12 ? FftGeo<12>::CTAS : v.logn == 13 ? FftGeo<13>::CTAS : FftGeo<14>::CTAS;
    if (nu * v.L <= v.sms * ctas) {
      u_fft = nullptr;
    } else {
      e = fft_samples(v, s, noise, 3, nu, u_fft);
      if (e != cudaSuccess) return e;
    }
    switch (v.logn) {
      case 12: e = launch_encrypt<12>(v, lp, s, first, nu, u_fft, noise, plain, ct); break;
      case 13: e = launch_encrypt<13>(v, lp, s, first, nu, u_fft, noise, plain, ct); break;
      case 14: e = launch_encrypt<14>(v, lp, s, first, nu, u_fft, noise, plain, ct); break;
      default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
    *launches += u_fft ? 3 : 2;
  }
  return cudaSuccess;
}

}  // namespace D2MHE_LAUNCH_NS
