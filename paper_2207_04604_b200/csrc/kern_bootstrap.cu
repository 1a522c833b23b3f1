// MBFV.Bootstrap (Sec. 4.2 item 4, Eq. 4): collective noise refresh.
#include <algorithm>

#define D2MHE_SHIFT_AS_MULTIPLY 1  // as in the decryption-share kernel: measured 0.7-1 % faster here with both
#define D2MHE_LATE_BARRIER 1
#include "d2mhe_kernels_common.cuh"

namespace {

// e_{0,k}, e_{1,k} (one byte per coefficient) and the mask M_k (one 32-bit word per coefficient,
// uniform mod t) of a share do not depend on the limb: kernels of their own (kern_sample.cu) sample them once per
// share into scratch memory that the caller of the launcher lends (6 N bytes per (recipient, ciphertext) unit and
// party: all M_k, then all [e_0 | e_1]), so the share kernel needs no clusters.

// Shares (eta_0, eta_1) = (s_k c_1 - Lambda M_k + e_{0,k}, -s_k alpha + Lambda M_k + e_{1,k}).
// grid = n_units * L; units unit_first .. unit_first + n_units - 1 of the (recipient, ciphertext) grid.
// NTT(c_1) is parked in the eta_0 row and NTT(alpha) in the eta_1 row of the last share.
// Iterations -2 and -1 run the two forward transforms, iteration a >= 0 produces share a, so that
// one forward and one inverse call site serve the whole kernel.
template <int LOGN, int G, bool WIDE>
__global__ void __launch_bounds__(ntt_threads_ct(LOGN, G), ntt_minb_ct(LOGN, G))
    k_boot_share(DevView v, const __grid_constant__ LimbParams lp, const u64* __restrict__ agg,
                 const u32* __restrict__ recipients, const u32* __restrict__ parties, u32 n_parties,
                 u32 ct_first, u32 n_cts, u32 unit_first, const u32* __restrict__ noise, const u32* __restrict__ masks,
                 u64* shares) {
  const u32 l = blockIdx.x % v.L, ulocal = blockIdx.x / v.L, unit = unit_first + ulocal;
  const u32 irec = unit / n_cts, cl = unit % n_cts, c = ct_first + cl;
  const u32 recipient = recipients[irec];
  if (!D2MHE_CHK(v.chk, recipient, v.K, SITE_PARTY)) return;
  const LimbTab& lt = lp.limbs[l];
  signed char* small = bytes_smem();                        // e_0, e_1: N bytes each
  u32* mask = reinterpret_cast<u32*>(small + 2 * v.n);      // M_k: N words
  u64* sm = poly_smem(6 * v.n);
  const size_t row = (size_t)l * v.n, poly = (size_t)v.L * v.n;
  const u64* c1 = agg + ((size_t)unit * 2 + 1) * poly + row;
  u64* park = shares + ((((size_t)irec * n_parties + (n_parties - 1)) * n_cts + cl) * 2) * poly + row;
  const Stream sa(v.seed, TAG_BOOT_ALPHA, c, l, recipient);
  const u32 words = 2 * (v.n >> 2);
#pragma unroll 1
  for (int a = -2; a < (int)n_parties; ++a) {
    const u32 party = a < 0 ? 0u : parties[a];
    if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY)) continue;
    if (a >= 0) {
      __syncthreads();  // every thread is done with the previous share's samples
      const size_t share = (size_t)ulocal * n_parties + a;
      const u32 *src = noise + share * words, *src_m = masks + share * v.n - words;
      if (LOGN == 0) {  // rings up to 1024: one round of loads instead of two (N = 16, 30 parties: 170 -> 156 us)
        for (u32 w = threadIdx.x; w < words + v.n; w += blockDim.x)
          reinterpret_cast<u32*>(small)[w] = __ldg((w < words ? src : src_m) + w);
      } else {
        for (u32 w = threadIdx.x; w < words; w += blockDim.x) reinterpret_cast<u32*>(small)[w] = __ldg(src + w);
        for (u32 w = threadIdx.x; w < v.n; w += blockDim.x) mask[w] = __ldg(src_m + words + w);
      }
      // the barrier that opens the first inverse transform publishes the copy
    }
    u64* h0 = a < 0 ? park : shares + ((((size_t)irec * n_parties + a) * n_cts + cl) * 2) * poly + row;
    u64* h1 = h0 + poly;
    if (a < 0) {
      u64* dst = a == -2 ? park : park + poly;
      ntt_forward<LOGN, G, WIDE>(
          sm, lt, v.logn,
          [&](u32 j) { return a == -2 ? __ldg(c1 + j) : uniform_mod(sa, j, lt.p, lt.mask); },
          [&](int, u32 q, u64(&x)[8]) { store_octet_il(dst, q, v.n >> 3, x); });
      continue;
    }
    const u64* sk = v.s_mont + ((size_t)party * v.L + l) * v.n;
#pragma unroll 1
    for (u32 comp = 0; comp < 2; ++comp) {
      const u64* src = comp ? park + poly : park;
      u64* out = comp ? h1 : h0;
      const signed char* e = small + comp * v.n;
      ntt_inverse<LOGN, G, WIDE>(
          sm, lt, v.logn,
          [&](int, u32 q, u64(&x)[8]) {
            u64 a8[8];
            load_octet_rw_il(src, q, v.n >> 3, a8);
            load_octet_il(sk, q, v.n >> 3, x);
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = mont_lazy(a8[k], x[k], lt.p, lt.pinv);
          },
          [&](u32 j, u64 val) {
            const u64 dm = shoup_u32(mask[j], lt.delta, lt.delta_sh, lt.np);  // Lambda M_k, below 2p
            // eta_0 = val - dm + e,  eta_1 = -val + dm + e; both sums below 8p
            const u64 s = (comp ? (2 * lt.twop - val) + dm : val + (lt.twop - dm)) + lt.p + (u64)(long long)e[j];
            out[j] = canon8<WIDE>(s, lt);
          });
    }
  }
}

// ct' = (Lambda x + sum_k eta_{1,k}, alpha) with x the rounded plaintext of c_0 + eta_0.
// grid = (n_rec * n_cts, chunks); a pair of residues per thread and iteration.  Bound by HBM (8 N L bytes of every
// share): the loads of five shares are in flight before the first is added.
__global__ void __launch_bounds__(256)
    k_boot_finish(DevView v, const u32* __restrict__ x, const u64* __restrict__ shares,
                  const u32* __restrict__ recipients, u32 n_shares, u32 ct_first, u32 n_cts,
                  u64* __restrict__ out) {
  const u32 unit = blockIdx.x, irec = unit / n_cts, cl = unit % n_cts;
  const u32 recipient = recipients[irec];
  if (!D2MHE_CHK(v.chk, recipient, v.K, SITE_PARTY)) return;
  const size_t pairs = (size_t)v.L * v.n / 2, stride = (size_t)n_cts * 2 * pairs;  // stride: from share to share
  const ulonglong2* eta = reinterpret_cast<const ulonglong2*>(shares) + (((size_t)irec * n_shares * n_cts + cl) * 2 + 1) * pairs;
  const uint2* xs = reinterpret_cast<const uint2*>(x) + (size_t)unit * (v.n / 2);
  ulonglong2* o = reinterpret_cast<ulonglong2*>(out) + (size_t)unit * 2 * pairs;
  for (size_t e = (size_t)blockIdx.y * blockDim.x + threadIdx.x; e < pairs; e += (size_t)gridDim.y * blockDim.x) {
    const u32 l = (u32)((2 * e) >> v.logn), j = (u32)((2 * e) & (v.n - 1));
    const LimbTab* lt = v.limbs + l;
    const u64 p = lt->p;
    const uint2 xv = __ldg(xs + (j >> 1));
    ulonglong2 acc = make_ulonglong2(csub(shoup_u32(xv.x, lt->delta, lt->delta_sh, lt->np), p),
                                     csub(shoup_u32(xv.y, lt->delta, lt->delta_sh, lt->np), p));
    const ulonglong2* src = eta + e;
    for (u32 k = 0; k < n_shares; k += 5) {
      ulonglong2 h[5];
#pragma unroll
      for (u32 i = 0; i < 5; ++i)
        h[i] = k + i < n_shares ? __ldcs(src + (k + i) * stride) : make_ulonglong2(0, 0);
#pragma unroll
      for (u32 i = 0; i < 5; ++i) {
        acc.x = addmod(acc.x, h[i].x, p);
        acc.y = addmod(acc.y, h[i].y, p);
      }
    }
    o[e] = acc;
    const Stream sa(v.seed, TAG_BOOT_ALPHA, ct_first + cl, l, recipient);
    o[pairs + e] = make_ulonglong2(uniform_mod(sa, j, p, lt->mask), uniform_mod(sa, j + 1, p, lt->mask));
  }
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

static cudaError_t boot_share_units(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg,
                                    const u32* recipients_dev, const u32* parties_dev, u32 n_parties, u32 ct_first,
                                    u32 n_cts, u32 unit_first, u32 n_units, const u32* noise, const u32* masks,
                                    u64* shares) {
  D2MHE_DISPATCH_EX(k_boot_share, v, n_units * v.L, s, 6 * (size_t)v.n, 1, v, lp, agg, recipients_dev, parties_dev,
                    n_parties, ct_first, n_cts, unit_first, noise, masks, shares);
}

// scratch: at least n_parties * 6 N bytes; (recipient, ciphertext) units are processed in batches of as
// many as it holds.
cudaError_t boot_share(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg,
                       const u32* recipients_dev, u32 n_rec, const u32* parties_dev, u32 n_parties,
                       u32 ct_first, u32 n_cts, u64* shares, void* scratch, size_t scratch_bytes, u32* launches) {
  const size_t per_unit = (size_t)n_parties * 6 * v.n;
  const u32 n_units = n_rec * n_cts;
  // double-precision products; lists of parties too long for their samples take the modular transforms
  if (v.fft_on && launches && scratch_bytes >= (size_t)n_parties * 6 * v.n + (size_t)v.L * v.n * sizeof(u64)) {
    *launches = 0;
    return boot_fft(v, lp, s, agg, recipients_dev, n_rec, parties_dev, n_parties, ct_first, n_cts, shares, scratch,
                    scratch_bytes, launches);
  }
  u32 per_batch = (u32)std::min<size_t>(scratch_bytes / per_unit, n_units);
  if (launches) *launches = 0;
  if (per_batch == 0) return cudaErrorInvalidValue;
  per_batch = whole_wave_batch(v, per_batch, n_units, v.L);
  for (u32 first = 0; first < n_units; first += per_batch) {
    const u32 nu = std::min(per_batch, n_units - first);
    u32* masks = reinterpret_cast<u32*>(scratch);
    u32* noise = masks + (size_t)nu * n_parties * v.n;
    u32 sampling = 0;
    cudaError_t e = sample_boot(v, s, recipients_dev, parties_dev, n_parties, ct_first, n_cts, first, nu, false, noise, masks,
                                &sampling);
    if (e != cudaSuccess) return e;
    e = boot_share_units(v, lp, s, agg, recipients_dev, parties_dev, n_parties, ct_first, n_cts, first, nu, noise, masks,
                         shares);
    if (e != cudaSuccess) return e;
    if (launches) *launches += 1 + sampling;
  }
  return cudaSuccess;
}

cudaError_t boot_finish(const DevView& v, cudaStream_t s, const u32* x, const u64* shares,
                        const u32* recipients_dev, u32 n_rec, u32 n_shares, u32 ct_first, u32 n_cts, u64* out) {
  const size_t pairs = (size_t)v.L * v.n / 2;
  u32 by = (u32)((pairs + 255) / 256);
  if (by > 32768) by = 32768;
  dim3 grid(n_rec * n_cts, by);
  k_boot_finish<<<grid, 256, 0, s>>>(v, x, shares, recipients_dev, n_shares, ct_first, n_cts, out);
  return cudaGetLastError();
}

}  // namespace D2MHE_LAUNCH_NS
