// Packing at N = 4096, 8192, 16384: negacyclic transforms mod t with 16 values per thread.
#include "d2mhe_kernels_common.cuh"

namespace {

__device__ __forceinline__ u32 shoup32_lazy(u32 x, uint2 w, u32 t) { return x * w.x - __umulhi(x, w.y) * t; }
__device__ __forceinline__ u32 csub_t(u32 x, u32 t) { return x >= t ? x - t : x; }
// Gentleman-Sande / Cooley-Tukey butterflies mod t on lazily reduced 32-bit values (below 2t)
__device__ __forceinline__ void gs_t(u32& X, u32& Y, uint2 w, u32 t, u32 twot) {
  const u32 s = X + Y, d = X - Y + twot;
  X = csub_t(s, twot);
  Y = shoup32_lazy(d, w, t);
}
__device__ __forceinline__ void ct_t(u32& X, u32& Y, uint2 w, u32 t, u32 twot) {
  const u32 x = csub_t(X, twot), T = shoup32_lazy(Y, w, t);
  X = x + T;
  Y = x - T + twot;
}

// Both directions walk the address bits from the top down, four (the first pass: log2 N mod 4, or four) per pass, and
// end with the bit-reversed address as the index of the output:
//   decode  coefficient p at address p, forward transform; position p is slot brv(p).
//   encode  slot j at address j, which is transform position brv(j): the inverse transform's spans 1, 2, 4, .. are the
//           address bits from the top; address a ends as coefficient brv(a).
// In the pass over bits B .. B+3 thread x owns a = (hi << B+4) + (c << B) + a0, c = 0 .. 15, with a0 = x mod 2^B and
// hi = x >> B; in the last one hi = brv(x), so that the reads of the first pass and the writes of the last are
// coalesced.  Shared memory is swizzled by the top five address bits for that last pass.
// Twiddles come from one table per pass, [15][a0] (encode) or [15][hi] (decode; the last pass in the order of x),
// fetched before the barrier that ends the previous pass.
// What bounds it: latency (one block per ciphertext; calls of a few dozen blocks).  N = 8192, 70 blocks: encode 17.0 ->
// 9.6 us, decode 18.7 -> 9.7 us against passes of two stages on 1024 threads.
template <int LOGN>
struct PackGeo {
  static constexpr int r0 = LOGN % 4 ? LOGN % 4 : 4, passes = (LOGN + 3) / 4, T = (1 << LOGN) / 16;
  // lowest address bit of pass i
  __host__ __device__ static constexpr int low(int i) { return i == 0 ? LOGN - 4 : LOGN - r0 - 4 * i; }
  __host__ __device__ static constexpr int stages(int i) { return i == 0 ? r0 : 4; }
};
template <int LOGN>
__device__ __forceinline__ u32 pack_swz(u32 a) {
  return a ^ (a >> (LOGN - 5));
}

template <int LOGN, bool INV>
__global__ void __launch_bounds__(PackGeo<LOGN>::T)
    k_pack(DevView v, const u32* in, u32* out, u32 group, size_t group_stride) {
  using G = PackGeo<LOGN>;
  constexpr u32 N = 1u << LOGN, T = G::T;
  u32* sm = reinterpret_cast<u32*>(smem_raw);
  const PlainTab pt = v.plain;
  const u32 t = pt.t, twot = pt.twot, x = threadIdx.x;
  // the values of block b = (g, c), c < group, start at g * group_stride + c * N
  const size_t vals = (size_t)(blockIdx.x / group) * group_stride + (size_t)(blockIdx.x % group) * N;
  const u32* src = INV ? in + vals : in + (size_t)blockIdx.x * N;
  u32* dst = INV ? out + (size_t)blockIdx.x * N : out + vals;
  const uint2* tab = INV ? pt.enc_tw : pt.dec_tw;
  u32 z[16];
  // in and out may be the same storage: a block has read its whole row when it reaches the first barrier
#pragma unroll
  for (u32 c = 0; c < 16; ++c) z[c] = src[c * T + x];
  if (INV) {
    bool bad = false;
#pragma unroll
    for (u32 c = 0; c < 16; ++c) {
      const int val = (int)z[c];
      bad |= val > (int)pt.half || val < -(int)pt.half;
    }
    if (bad) {
      atomicOr(v.range_flag, RANGE_FLAG_VALUE);
#pragma unroll
      for (u32 c = 0; c < 16; ++c) z[c] = (u32)((int)z[c] % (int)t);
    }
#pragma unroll
    for (u32 c = 0; c < 16; ++c) z[c] += (int)z[c] < 0 ? t : 0u;
  }
#pragma unroll
  for (int p = 0; p < G::passes; ++p) {
    const int B = G::low(p), S = G::stages(p);
    const u32 nidx = INV ? 1u << B : T >> B;  // entries per twiddle of this pass
    const u32 idx = INV ? x & (nidx - 1) : (B == 0 ? x : x >> B);
    uint2 w[15];
#pragma unroll
    for (int i = 0; i < 15; ++i) {
      const bool used = INV ? i < 16 - (16 >> S) : i < (1 << S) - 1;
      if (used && D2MHE_CHK(v.chk, i * nidx + idx, 15 * nidx, SITE_TWIDDLE)) w[i] = __ldg(tab + i * nidx + idx);
    }
    tab += 15 * nidx;
    const u32 hi = B == 0 ? __brev(x) >> (32 - (LOGN - 4)) : x >> B;
    const u32 base = (hi << (B + 4)) + (x & ((1u << B) - 1));
    if (p > 0) {
      __syncthreads();
#pragma unroll
      for (u32 c = 0; c < 16; ++c) {
        const u32 a = pack_swz<LOGN>(base + (c << B));
        z[c] = D2MHE_CHK(v.chk, a, N, SITE_STAGED) ? sm[a] : 0;
      }
    }
#pragma unroll
    for (int e = 0; e < S; ++e) {
      const int half = 8 >> e;  // pairs c, c + half
#pragma unroll
      for (int c = 0; c < 16; ++c)
        if ((c & half) == 0) {
          if (INV)
            gs_t(z[c], z[c + half], w[16 - (16 >> e) + (c & (half - 1))], t, twot);
          else
            ct_t(z[c], z[c + half], w[(1 << e) - 1 + (c >> (4 - e))], t, twot);
        }
    }
    if (p + 1 < G::passes) {  // in place: this thread's own addresses
#pragma unroll
      for (u32 c = 0; c < 16; ++c) {
        const u32 a = pack_swz<LOGN>(base + (c << B));
        if (D2MHE_CHK(v.chk, a, N, SITE_STAGED)) sm[a] = z[c];
      }
    }
  }
  const uint2 ninv = make_uint2(pt.ninv, pt.ninv_sh);
#pragma unroll
  for (u32 c = 0; c < 16; ++c) {
    const u32 o = (__brev(c) >> 28) * T + x;
    if (INV) {
      dst[o] = csub_t(shoup32_lazy(z[c], ninv, t), t);
    } else {
      const u32 y = csub_t(csub_t(z[c], twot), t);
      dst[o] = y > pt.half ? y - t : y;
    }
  }
}

template <bool INV>
cudaError_t launch_pack(const DevView& v, cudaStream_t s, const u32* in, u32* out, u32 blocks, u32 group,
                        size_t group_stride) {
  const size_t smem = (size_t)v.n * 4;
#define D2MHE_PACK(LOGN_)                                                                             \
  case LOGN_: {                                                                                       \
    cudaError_t e_ = set_smem(k_pack<LOGN_, INV>, smem);                                              \
    if (e_ != cudaSuccess) return e_;                                                                 \
    k_pack<LOGN_, INV><<<blocks, PackGeo<LOGN_>::T, smem, s>>>(v, in, out, group, group_stride);      \
    break;                                                                                            \
  }
  switch (v.logn) {
    D2MHE_PACK(12)
    D2MHE_PACK(13)
    D2MHE_PACK(14)
    default: return cudaErrorInvalidValue;
  }
#undef D2MHE_PACK
  return cudaGetLastError();
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

cudaError_t encode16(const DevView& v, cudaStream_t s, const int32_t* values, u32 n_groups, u32 group,
                     size_t group_stride, u32* plain) {
  return launch_pack<true>(v, s, reinterpret_cast<const u32*>(values), plain, n_groups * group, group, group_stride);
}
cudaError_t decode16(const DevView& v, cudaStream_t s, const u32* plain, u32 n_groups, u32 group, size_t group_stride,
                     int32_t* values) {
  return launch_pack<false>(v, s, plain, reinterpret_cast<u32*>(values), n_groups * group, group, group_stride);
}

}  // namespace D2MHE_LAUNCH_NS
