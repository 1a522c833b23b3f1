// Small samples drawn ahead of the protocol kernels: error polynomials, u and mu_k, one byte per coefficient.
#include <algorithm>

#include "d2mhe_kernels_common.cuh"

namespace {

// A discrete Gaussian sample is a count of the thresholds at or below a 64-bit draw.  The table gives the count for
// the top 12 bits; bit 7 marks the 0.9 % of the buckets that hold a threshold, where the exact thresholds decide.
// (With 8 bits, one bucket in eight: nearly every warp walked the thresholds.)
__device__ __forceinline__ u32 gauss_count(const GaussFast& g, u32 o0, u32 o1, u32 cnt) {
  const u64 r = ((u64)o0 << 32) | o1;
  cnt &= 0x7fu;
  while (cnt < D2MHE_CDT_LEN && r >= g.cdt[cnt]) ++cnt;
  return cnt;
}

// Polynomial number p of this launch: sample kind tag[p % n_tags] of share p / n_tags; N bytes each, one after
// another.  A share is a (unit, party) pair (recipients != null) or a (party, ciphertext) unit.  A thread block works
// on one polynomial, so all of the counter but the coefficient is uniform over the block and the first two of the ten
// Philox rounds cost half.  What bounds it: the integer multiplier (17 widening multiplications per sample).
// ORDER = 0: byte j is the sample of coefficient j, signed.  ORDER = 12, 13, 14 (log2 N): samples + 19 in the order in
// which the threads of the double-precision kernels of that size need them (fft_coef): 32 for each of T = N / 32
// threads, as 16-byte slots [2][T].
// grid = polynomials * segs; a block draws words / segs packed words of its polynomial.
// Measured at N = 8192, 32 M samples: 154 us with a block-independent kernel and an 8-bit table, 110 us now.
template <int ORDER>
__global__ void __launch_bounds__(256)
    k_sample_streams(DevView v, const u32* __restrict__ recipients, const u32* __restrict__ parties, u32 n_parties,
                     u32 ct_first, u32 n_cts, u32 unit_first, SampleKinds kinds, u32 segs, u32* __restrict__ out) {
  __shared__ GaussFast gt;
  for (u32 i = threadIdx.x; i < sizeof(GaussFast) / 16; i += blockDim.x)
    reinterpret_cast<uint4*>(&gt)[i] = __ldg(reinterpret_cast<const uint4*>(v.gauss_fast) + i);
  __syncthreads();
  const u32 poly = blockIdx.x / segs, seg = blockIdx.x % segs;
  const u32 which = poly % kinds.n, share = poly / kinds.n;
  const u32 tag = which == 0 ? kinds.tag0 : which == 1 ? kinds.tag1 : kinds.tag2;
  const u32 unit = unit_first + (recipients ? share / n_parties : share);
  const u32 party = recipients ? parties[share % n_parties] : parties[unit / n_cts];
  const u32 recipient = recipients ? recipients[unit / n_cts] : 0u;
  if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY) || !D2MHE_CHK(v.chk, recipient, v.K, SITE_PARTY)) return;
  const u32 c1 = ct_first + unit % n_cts, c2 = party | (recipient << 16), k0 = (u32)v.seed, k1 = (u32)(v.seed >> 32);
  const u32 words = v.n >> 2, per = words / segs;
  u32* dst = out + (size_t)poly * words;
#pragma unroll 1
  for (u32 w = seg * per + threadIdx.x; w < (seg + 1) * per; w += blockDim.x) {
    u32 j0 = 4 * w;
    constexpr u32 step = ORDER ? 256u : 1u;
    if (ORDER) {
      constexpr u32 T = (1u << ORDER) / 32u;
      const u32 t = (w >> 2) & (T - 1), m = (w & 3u) + 4u * (w / (ORDER ? 4u * T : 1u));  // word m of thread t
      j0 = ORDER == 14   ? (t & 255u) + 2048u * (t >> 8) + 1024u * (m & 1u) + 4096u * (m >> 1)
           : ORDER == 13 ? t + 1024u * m
                         : t + 128u * (m >> 2) + 1024u * (m & 3u);
    }
    u32 o0[4], o1[4], e[4];
#pragma unroll
    for (u32 b = 0; b < 4; ++b) {
      u32 o2, o3;
      philox4x32_10(k0, k1, j0 + b * step, c1, c2, tag, o0[b], o1[b], o2, o3);
    }
    if (tag == TAG_ENC_U) {
#pragma unroll
      for (u32 b = 0; b < 4; ++b) e[b] = __umulhi(o0[b], 3u) + (D2MHE_GAUSS_B - 1);
    } else {
#pragma unroll
      for (u32 b = 0; b < 4; ++b) e[b] = gt.lut[o0[b] >> 20];
      if ((e[0] | e[1] | e[2] | e[3]) & 0x80u) {
#pragma unroll
        for (u32 b = 0; b < 4; ++b)
          if (e[b] & 0x80u) e[b] = gauss_count(gt, o0[b], o1[b], e[b]);
      }
    }
    u32 pack = e[0] | (e[1] << 8) | (e[2] << 16) | (e[3] << 24);
    if (!ORDER) pack = __vsub4(pack, 0x01010101u * D2MHE_GAUSS_B);
    dst[w] = pack;
  }
}

// The same in the order of the coefficients for rings below 256, whose polynomials do not fill a block: one word for each
// thread and step, whatever polynomial it belongs to, and behind them (masks != null) the words M_k of every share, so that
// a small refresh needs one launch.  A block for each polynomial cost 5 % on the shares of 400 parties at N = 64, and a
// launch of its own for the masks 10 to 19 % of a small refresh.
__global__ void __launch_bounds__(256)
    k_sample_small(DevView v, const u32* __restrict__ recipients, const u32* __restrict__ parties, u32 n_parties,
                   u32 ct_first, u32 n_cts, u32 unit_first, SampleKinds kinds, size_t shares, u32* __restrict__ out,
                   u32* __restrict__ masks) {
  __shared__ GaussFast gt;
  for (u32 i = threadIdx.x; i < sizeof(GaussFast) / 16; i += blockDim.x)
    reinterpret_cast<uint4*>(&gt)[i] = __ldg(reinterpret_cast<const uint4*>(v.gauss_fast) + i);
  __syncthreads();
  const size_t noise = shares * kinds.n << (v.logn - 2), total = noise + (masks ? shares << v.logn : 0);
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const bool mask = e >= noise;
    const size_t poly = mask ? (e - noise) >> v.logn : e >> (v.logn - 2), share = mask ? poly : poly / kinds.n;
    const u32 which = mask ? 3u : (u32)(poly % kinds.n);
    const u32 tag = which == 0 ? kinds.tag0 : which == 1 ? kinds.tag1 : which == 2 ? kinds.tag2 : TAG_BOOT_MASK;
    const u32 unit = unit_first + (u32)(recipients ? share / n_parties : share);
    const u32 party = recipients ? parties[share % n_parties] : parties[unit / n_cts];
    const u32 recipient = recipients ? recipients[unit / n_cts] : 0u;
    if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY) || !D2MHE_CHK(v.chk, recipient, v.K, SITE_PARTY)) continue;
    const Stream st(v.seed, tag, ct_first + unit % n_cts, party, recipient);
    if (mask) {
      const u32 t = (u32)v.round.t;
      masks[e - noise] = (u32)uniform_mod(st, (u32)(e - noise) & (v.n - 1), t, 0xffffffffu >> __clz(t));
      continue;
    }
    const u32 j0 = 4 * ((u32)e & ((v.n >> 2) - 1));
    u32 pack = 0;
#pragma unroll
    for (u32 b = 0; b < 4; ++b) {
      int x;
      if (tag == TAG_ENC_U) {
        x = st.ternary(j0 + b);
      } else {
        const u64 r = st.draw64(j0 + b);
        const u32 cnt = gt.lut[r >> 52];
        x = (int)(cnt & 0x80u ? gauss_count(gt, (u32)(r >> 32), (u32)r, cnt) : cnt) - D2MHE_GAUSS_B;
      }
      pack |= ((u32)x & 0xffu) << (8 * b);
    }
    out[e] = pack;
  }
}

// M_k uniform mod t by rejection on bitlen(t)-bit draws, N words per share.  Half of the draws are rejected for
// t = 65537, so what counts is that no lane waits for another's redraw: a warp draws once for each of its coefficients,
// packs the numbers of the rejected ones into a list in shared memory and goes over the list again, 32 at a time, until
// it is empty.  512 coefficients take 31 full draws and about five partly filled ones, where lanes that walk over 16
// coefficients of their own wait for the slowest of the 32 (46 draws).  The attempt is uniform over the warp.
// Bound by the integer multiplier and the logic pipe beside it, as above.  10.6 M masks mod 65537: 91 us (107 us with
// both words of every draw, 125 us without the lists); with 64 coefficients at a time, two draws to a lane, 20 % slower
// (twice as many partly filled draws).
// grid = shares * segs; each warp of a block has per <= MASKS_PER_WARP coefficients.
constexpr u32 MASKS_PER_WARP = 512;
__global__ void __launch_bounds__(128)
    k_sample_masks(DevView v, const u32* __restrict__ recipients, const u32* __restrict__ parties, u32 n_parties,
                   u32 ct_first, u32 n_cts, u32 unit_first, u32 segs, u32 per, u32* __restrict__ out) {
  __shared__ unsigned short lists[4][MASKS_PER_WARP];
  const u32 share = blockIdx.x / segs, seg = blockIdx.x % segs, lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const u32 unit = unit_first + share / n_parties, party = parties[share % n_parties], recipient = recipients[unit / n_cts];
  if (!D2MHE_CHK(v.chk, party, v.K, SITE_PARTY) || !D2MHE_CHK(v.chk, recipient, v.K, SITE_PARTY)) return;
  const Stream st(v.seed, TAG_BOOT_MASK, ct_first + unit % n_cts, party, recipient);
  const u32 t = (u32)v.round.t, tmask = 0xffffffffu >> __clz(t);
  const u32 first = (seg * (blockDim.x >> 5) + warp) * per;
  u32* dst = out + (size_t)share * v.n + first;
  unsigned short* list = lists[warp];
  u32 count = per;
#pragma unroll 1
  for (u32 attempt = 0; count; ++attempt) {  // the draw of attempt 255 is taken mod t: the list is empty after it
    u32 left = 0;
#pragma unroll 1
    for (u32 b = 0; b < count; b += 32) {
      const u32 at = b + lane;
      bool again = false;
      u32 j = at;
      if (at < count) {
        if (attempt) j = list[at];
        // the rule of uniform_mod; only the low word of the draw matters, but for the last attempt
        const u32 r = attempt < 255 ? (u32)st.draw64(first + j, attempt) & tmask
                                    : (u32)(st.draw64(first + j, attempt) % t);
        again = r >= t;
        if (!again) dst[j] = r;
      }
      // packed in place: left <= b, and what stands below b + 32 has been read
      const u32 votes = __ballot_sync(0xffffffffu, again);
      if (again) list[left + __popc(votes & ((1u << lane) - 1u))] = (unsigned short)j;
      left += __popc(votes);
    }
    __syncwarp();
    count = left;
  }
}

// The common polynomial alpha of every unit, all limbs: [units][L][N].
__global__ void __launch_bounds__(256)
    k_sample_alpha(DevView v, const u32* __restrict__ recipients, u32 ct_first, u32 n_cts, u32 unit_first, u32 rows,
                   u64* __restrict__ out) {
  const size_t total = (size_t)rows << v.logn, stride = (size_t)gridDim.x * blockDim.x;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += stride) {
    const u32 j = (u32)(e & (v.n - 1)), row = (u32)(e >> v.logn), l = row % v.L, unit = unit_first + row / v.L;
    const u32 recipient = recipients[unit / n_cts];
    if (!D2MHE_CHK(v.chk, recipient, v.K, SITE_PARTY)) continue;
    const Stream st(v.seed, TAG_BOOT_ALPHA, ct_first + unit % n_cts, l, recipient);
    out[e] = uniform_mod(st, j, v.limbs[l].p, v.limbs[l].mask);
  }
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

static cudaError_t sample_masks(const DevView& v, cudaStream_t s, const u32* recipients_dev, const u32* parties_dev,
                         u32 n_parties, u32 ct_first, u32 n_cts, u32 unit_first, u32 n_units, u32* out) {
  const u32 per = std::min(v.n, MASKS_PER_WARP), warps = std::min(v.n / per, 4u), segs = v.n / (per * warps);
  k_sample_masks<<<n_units * n_parties * segs, 32 * warps, 0, s>>>(v, recipients_dev, parties_dev, n_parties, ct_first,
                                                                   n_cts, unit_first, segs, per, out);
  return cudaGetLastError();
}

cudaError_t sample_alpha(const DevView& v, cudaStream_t s, const u32* recipients_dev, u32 ct_first, u32 n_cts,
                         u32 unit_first, u32 n_units, u64* out) {
  const size_t total = (size_t)n_units * v.L * v.n;
  const u32 blocks = (u32)std::min<size_t>((total + 255) / 256, (size_t)v.sms * 32);
  k_sample_alpha<<<blocks, 256, 0, s>>>(v, recipients_dev, ct_first, n_cts, unit_first, n_units * v.L, out);
  return cudaGetLastError();
}

static cudaError_t sample_small(const DevView& v, cudaStream_t s, const u32* recipients_dev, const u32* parties_dev,
                                u32 n_parties, u32 ct_first, u32 n_cts, u32 unit_first, u32 n_units, SampleKinds kinds,
                                void* out, u32* masks) {
  const size_t shares = (size_t)n_units * (recipients_dev ? n_parties : 1u);
  const size_t blocks = (shares * (kinds.n * (v.n >> 2) + (masks ? v.n : 0)) + 255) / 256;
  const unsigned grid = (unsigned)std::min(blocks, std::max((size_t)8 * v.sms, blocks / 8));  // the table once per 8 words
  k_sample_small<<<grid, 256, 0, s>>>(v, recipients_dev, parties_dev, n_parties, ct_first, n_cts, unit_first, kinds, shares,
                                      reinterpret_cast<u32*>(out), masks);
  return cudaGetLastError();
}

// e_0, e_1 and M_k of a refresh, for the modular kernels in one launch unless there are enough masks (2^20) for the lists
// of k_sample_masks to pay for theirs, and lists of 256 and more.  (N = 1024, ten parties: 40 indices, 4 M masks, one launch
// 546 us, two 511; 4 parties, two indices 73 / 83 us; N = 64, 400 parties: 3.47 / 3.59 ms.)
cudaError_t sample_boot(const DevView& v, cudaStream_t s, const u32* recipients_dev, const u32* parties_dev, u32 n_parties,
                        u32 ct_first, u32 n_cts, u32 unit_first, u32 n_units, bool fft_order, void* noise, u32* masks,
                        u32* launches) {
  if (v.n < 256 || (!fft_order && ((size_t)n_units * n_parties << v.logn) <= (size_t)1 << 20)) {
    *launches += 1;
    return sample_small(v, s, recipients_dev, parties_dev, n_parties, ct_first, n_cts, unit_first, n_units, kSampleBoot, noise,
                        masks);
  }
  *launches += 2;
  const cudaError_t e = sample_masks(v, s, recipients_dev, parties_dev, n_parties, ct_first, n_cts, unit_first, n_units, masks);
  if (e != cudaSuccess) return e;
  return sample_streams(v, s, recipients_dev, parties_dev, n_parties, ct_first, n_cts, unit_first, n_units, kSampleBoot,
                        fft_order, noise);
}

cudaError_t sample_streams(const DevView& v, cudaStream_t s, const u32* recipients_dev, const u32* parties_dev,
                           u32 n_parties, u32 ct_first, u32 n_cts, u32 unit_first, u32 n_units, SampleKinds kinds,
                           bool fft_order, void* out) {
  if (v.n < 256)
    return sample_small(v, s, recipients_dev, parties_dev, n_parties, ct_first, n_cts, unit_first, n_units, kinds, out, nullptr);
  const u32 words = v.n >> 2, threads = std::min(words, 256u);
  const size_t polys = (size_t)n_units * (recipients_dev ? n_parties : 1u) * kinds.n;
  // Eight words per thread, so that the table is fetched once for 8192 samples (2 % over two words on the share call);
  // when that does not fill the GPU (eight blocks per SM), down to one word per thread.
  u32 segs = std::max(1u, words / (8 * threads));
  while (segs * 2 * threads <= words && polys * segs < (size_t)8 * v.sms) segs *= 2;
  const unsigned grid = (unsigned)(polys * segs);
  u32* o = reinterpret_cast<u32*>(out);
  switch (fft_order ? v.logn : 0) {
#define D2MHE_SAMPLE(ORDER_)                                                                                         \
  k_sample_streams<ORDER_><<<grid, threads, 0, s>>>(v, recipients_dev, parties_dev, n_parties, ct_first, n_cts,       \
                                                    unit_first, kinds, segs, o)
    case 0: D2MHE_SAMPLE(0); break;
    case 12: D2MHE_SAMPLE(12); break;
    case 13: D2MHE_SAMPLE(13); break;
    case 14: D2MHE_SAMPLE(14); break;
    default: return cudaErrorInvalidValue;
#undef D2MHE_SAMPLE
  }
  return cudaGetLastError();
}

}  // namespace D2MHE_LAUNCH_NS
