// Streaming kernels: RNS multiply-add, neighbour sums, combine + exact scale-and-round, packing.
#include "d2mhe_kernels_common.cuh"

namespace {

// d = a (.) b + c per residue; two residues per thread (16-byte accesses).
__global__ void __launch_bounds__(256) k_muladd(DevView v, const u64* __restrict__ a,
                                                const u64* __restrict__ b,
                                                const u64* __restrict__ c, u64* __restrict__ d,
                                                size_t n_pairs) {
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < n_pairs; e += stride) {
    const u32 l = (u32)(((e * 2) >> v.logn) % v.L);
    if (!D2MHE_CHK(v.chk, e, n_pairs, SITE_ELEMENT) || !D2MHE_CHK(v.chk, l, v.L, SITE_LIMB)) continue;
    const LimbTab* lt = v.limbs + l;
    const u64 p = lt->p, pinv = lt->pinv, r = lt->rmod, rs = lt->rmod_sh;
    const ulonglong2 av = reinterpret_cast<const ulonglong2*>(a)[e];
    const ulonglong2 bv = reinterpret_cast<const ulonglong2*>(b)[e];
    const ulonglong2 cv = reinterpret_cast<const ulonglong2*>(c)[e];
    ulonglong2 o;
    o.x = addmod(shoup_full(mont_lazy(av.x, bv.x, p, pinv), r, rs, p), cv.x, p);
    o.y = addmod(shoup_full(mont_lazy(av.y, bv.y, p, pinv), r, rs, p), cv.y, p);
    reinterpret_cast<ulonglong2*>(d)[e] = o;
  }
}

// ---------------------------------------------------------------------------
// BFV.Add over neighbour lists.  grid = (n_out * n_cts, chunks); two residues per thread.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256)
    k_aggregate(DevView v, const u64* __restrict__ ct, u32 n_cts, const u32* __restrict__ offsets,
                const u32* __restrict__ rows, u64* __restrict__ agg) {
  const u32 unit = blockIdx.x, i = unit / n_cts, c = unit % n_cts;
  const size_t ct_pairs = (size_t)v.L * v.n;  // 2*L*N residues = L*N pairs
  const u32 beg = offsets[i], end = offsets[i + 1];
  const bool lazy = v.wide != 0 && end - beg < 64;
  ulonglong2* out = reinterpret_cast<ulonglong2*>(agg) + (size_t)unit * ct_pairs;
  for (size_t e = (size_t)blockIdx.y * blockDim.x + threadIdx.x; e < ct_pairs;
       e += (size_t)gridDim.y * blockDim.x) {
    // a block of 256 pairs lies inside one limb row whenever N >= 512: take the row from a
    // block-uniform index so that the division runs on the uniform datapath
    const size_t e_row = v.n >= 512 ? e - threadIdx.x : e;
    const u32 l = (u32)(((e_row * 2) >> v.logn) % v.L);
    if (!D2MHE_CHK(v.chk, e, ct_pairs, SITE_ELEMENT) || !D2MHE_CHK(v.chk, l, v.L, SITE_LIMB)) continue;
    const u64 p = v.limbs[l].p;
    ulonglong2 acc = make_ulonglong2(0, 0);
    if (lazy) {
      // primes below 2^56 and fewer than 64 addends: the plain 64-bit sums cannot overflow, so the
      // loads are independent (several in flight per thread) and one reduction at the end replaces
      // one per addend
#pragma unroll 4
      for (u32 a = beg; a < end; ++a) {
        const ulonglong2 x =
            __ldg(reinterpret_cast<const ulonglong2*>(ct) + ((size_t)rows[a] * n_cts + c) * ct_pairs + e);
        acc.x += x.x;
        acc.y += x.y;
      }
      const u64 one_sh = v.limbs[l].one_sh;
      acc.x = shoup_full(acc.x, 1, one_sh, p);
      acc.y = shoup_full(acc.y, 1, one_sh, p);
    } else {
      for (u32 a = beg; a < end; ++a) {
        const ulonglong2 x =
            __ldg(reinterpret_cast<const ulonglong2*>(ct) + ((size_t)rows[a] * n_cts + c) * ct_pairs + e);
        acc.x = addmod(acc.x, x.x, p);
        acc.y = addmod(acc.y, x.y, p);
      }
    }
    out[e] = acc;
  }
}

// The same with every ciphertext read once: a block keeps COLS columns of 16 bytes of all n_rows ciphertexts of index c in
// shared memory and adds them up list by list.  What the kernel above spends its time on is one L2 read per list entry
// (70 sums of five at N = 8192, L = 4: 26.6 -> 20.4 us; MNIST-shaped round 527 -> 504 us).  The sums are a chain of
// shared-memory reads (entry, then residues), and columns of many rows leave room for few threads to hide it, so GROUPS
// groups of COLS threads share the columns and each takes every GROUPS-th list (N = 16384, L = 8, one group of 128 ->
// four of 32: 20 rows, lists of 7, 11 indices 227 -> 207 us; 50 rows, lists of 9, four indices 363 -> 223 us).
// Chosen when the lists together name more rows than there are, the columns of four blocks fit an SM's shared memory
// (200 rows, columns of two blocks: 349 us against 242 without columns; 100 rows: 231 against 262), and there are
// 512 columns for every SM (a tiny round is 2 us slower).
// grid = (n_cts, ciphertext bytes / 16 / COLS); shared memory: columns [n_rows][COLS], then offsets and rows.
template <class W, u32 COLS, u32 GROUPS>
__global__ void __launch_bounds__(COLS * GROUPS)
    k_aggregate_columns(DevView v, const W* __restrict__ ct, u32 n_rows, u32 n_cts, const u32* __restrict__ offsets,
                        const u32* __restrict__ rows, u32 n_out, u32 nnz, W* __restrict__ agg) {
  constexpr u32 PER = 16 / sizeof(W);  // residues per vector
  const u32 tx = threadIdx.x % COLS, group = threadIdx.x / COLS;
  uint4* col = reinterpret_cast<uint4*>(smem_raw) + tx;
  u32* off = reinterpret_cast<u32*>(smem_raw + (size_t)n_rows * COLS * 16);
  u32* lst = off + n_out + 1;
  for (u32 i = threadIdx.x; i <= n_out; i += COLS * GROUPS) off[i] = offsets[i];
  for (u32 i = threadIdx.x; i < nnz; i += COLS * GROUPS) lst[i] = rows[i];
  const u32 c = blockIdx.x, vecs = 2 * v.L * v.n / PER, e = blockIdx.y * COLS + tx;
  const u32 l = ((e * PER) >> v.logn) % v.L;
  const bool in = e < vecs;
  const uint4* src = reinterpret_cast<const uint4*>(ct) + (size_t)c * vecs + e;
  if (in) {
    // global -> shared without passing through registers: all rows in flight at once
    const u32 dst = (u32)__cvta_generic_to_shared(col);
#pragma unroll 4
    for (u32 r = group; r < n_rows; r += GROUPS)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + r * (COLS * 16)),
                   "l"(src + (size_t)r * n_cts * vecs)
                   : "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  __syncthreads();
  if (!in) return;
  const u64 p = v.limbs[l].p, one_sh = v.limbs[l].one_sh;
  uint4* out = reinterpret_cast<uint4*>(agg) + (size_t)c * vecs + e;
  for (u32 i = group; i < n_out; i += GROUPS) {
    const u32 beg = off[i], end = off[i + 1];
    uint4 o;
    if (sizeof(W) == 8) {
      u64 a0 = 0, a1 = 0;
      const bool lazy = v.wide != 0 && end - beg < 64;  // plain 64-bit sums of primes below 2^56, one reduction
      for (u32 a = beg; a < end; ++a) {
        const u32 r = lst[a];
        if (!D2MHE_CHK(v.chk, r, n_rows, SITE_PARTY)) continue;
        const uint4 x = col[r * COLS];
        a0 += join64(x.x, x.y);
        a1 += join64(x.z, x.w);
        if (!lazy) a0 = csub(a0, p), a1 = csub(a1, p);
      }
      if (lazy) a0 = shoup_full(a0, 1, one_sh, p), a1 = shoup_full(a1, 1, one_sh, p);
      o = make_uint4((u32)a0, (u32)(a0 >> 32), (u32)a1, (u32)(a1 >> 32));
    } else {
      const u32 q = (u32)p;
      o = make_uint4(0, 0, 0, 0);
      for (u32 a = beg; a < end; ++a) {
        const u32 r = lst[a];
        if (!D2MHE_CHK(v.chk, r, n_rows, SITE_PARTY)) continue;
        const uint4 x = col[r * COLS];
        o.x += x.x, o.y += x.y, o.z += x.z, o.w += x.w;
        o.x = min(o.x, o.x - q), o.y = min(o.y, o.y - q), o.z = min(o.z, o.z - q), o.w = min(o.w, o.w - q);
      }
    }
    out[(size_t)i * n_cts * vecs] = o;
  }
}

// ---------------------------------------------------------------------------
// Combine + exact scale-and-round.
//   v_l = c_0 + sum_k h_k mod q_l;  y_l = v_l (q / q_l)^-1 mod q_l;
//   t v / q = sum_l t y_l / q_l  (mod t),  x = round(that) mod t.
// Every term is rounded down to F fraction bits (59 - bitlen(t): 42 for t = 65537), two units low at most, so the sum
// is at most 2L units low, and x is exact unless the fraction of sum + 1/2 lies within 2L units below a whole number:
// then (once in 2^38 for random input, never for a ciphertext with noise to spare) the mixed-radix conversion below
// decides.  L + 1 products per coefficient instead of L (L + 7) / 2 and no array of digits: the kernel is left with its
// loads.  (The digits for every coefficient, one coefficient per thread: 48 us for 70 units of 10 shares at N = 8192,
// L = 4 and 73 us for 40 of one share at N = 16384, L = 8; 42 and 46 us now.)
// grid = n_rec * n_cts * N / 32 V, 32 L threads: the blocks of a unit side by side, so that the loads in flight fall into
// long runs of a few units' rows (with the units side by side 81.7 us for 99 units of nine shares at N = 8192, L = 6, now
// 78.0; 130 units of ten, L = 4: 76.1 and 71.6).  Words of 32 bits four at a time, 16 bytes as for 64 bits: 130 units of ten,
// L = 7: 91.6 and 74.5 us, in an instance for blocks of at most eight warps, 64 registers a thread (for twelve warps it took
// 122 registers, and that round 67 us more); combine_words has the rule.
// ---------------------------------------------------------------------------

// mixed-radix (Garner) digits d_i of w' = t v + (q-1)/2 in [0, q);  w' mod t = sum d_i prod_{j<i} q_j mod t;
// x = ((q-1)/2 - w') q^-1 mod t.  acc(l): v_l, any 64-bit representative.
template <class Acc>
__device__ __noinline__ u32 round_exact(const DevView& v, Acc acc) {
  const u32 L = v.L;
  u64 d[D2MHE_MAX_LIMBS];
  const u64 t = v.round.t, tsh = v.round.t_sh;
  u64 sum = 0;
  for (u32 i = 0; i < L; ++i) {
    const LimbTab* lt = v.limbs + i;
    u64 tmp = addmod(shoup_full(acc(i), lt->tmod, lt->tmod_sh, lt->p), lt->half, lt->p);
    for (u32 j = 0; j < i; ++j) {
      const ulonglong2 gi = __ldg(v.round.ginv + i * L + j);
      tmp = shoup_full(tmp + lt->cq - d[j], gi.x, gi.y, lt->p);
    }
    d[i] = tmp;
    sum = shoup_full(sum + shoup_full(tmp, 1, tsh, t) * v.round.prefix_mod_t[i], 1, tsh, t);
  }
  const u64 diff = v.round.half_mod_t + t - sum;  // in (0, 2t)
  return (u32)shoup_full(diff * v.round.qinv_mod_t, 1, tsh, t);
}

// V residues of W as one load
template <class W, u32 V>
struct Residues;
template <>
struct Residues<u64, 2> {
  ulonglong2 q = {0, 0};
  __device__ __forceinline__ u64 get(u32 i) const { return i ? q.y : q.x; }
};
template <>
struct Residues<u32, 2> {
  uint2 q = {0, 0};
  __device__ __forceinline__ u64 get(u32 i) const { return i ? q.y : q.x; }
};
template <>
struct Residues<u32, 4> {
  uint4 q = {0, 0, 0, 0};
  __device__ __forceinline__ u64 get(u32 i) const { return i == 0 ? q.x : i == 1 ? q.y : i == 2 ? q.z : q.w; }
};

// W = u64, or u32 for the 32-bit-word messages (same arithmetic on the loaded residues).
// One warp per limb, at most LIMBS of them: a thread sums the shares of V coefficients of its limb, all of its loads independent of one
// another, and the block adds up the limbs' terms through shared memory.  (All limbs in one thread, one after another,
// had too few loads in flight: 59 us for the 70 units above.)
template <class W, u32 V, int LIMBS>
__global__ void __launch_bounds__(32 * LIMBS)
    k_combine(const __grid_constant__ DevView v, const W* __restrict__ agg, const W* __restrict__ shares, u32 n_shares,
              u32 share_comps, u32 n_cts, u32* __restrict__ plain) {
  typedef Residues<W, V> R;
  constexpr u32 COLS = 32 * V;
  __shared__ u64 terms[LIMBS][COLS];
  const u32 chunks = (v.n + COLS - 1) / COLS, unit = blockIdx.x / chunks, irec = unit / n_cts, cl = unit % n_cts;
  const u32 lane = threadIdx.x & 31u, wl = threadIdx.x >> 5, L = v.L, j0 = blockIdx.x % chunks * COLS, jj = j0 + V * lane;
  const size_t poly = (size_t)L * v.n;
  const W* c0 = agg + (size_t)unit * 2 * poly;
  const W* sh = shares + ((size_t)irec * n_shares * n_cts + cl) * share_comps * poly;
  const size_t kstride = (size_t)n_cts * share_comps * poly;
  // primes below 2^56 and fewer than 120 shares: the plain 64-bit sum cannot overflow and the multiplication by the
  // CRT factor reduces any 64-bit value, so the loads are all independent
  const bool lazy = (v.wide != 0 || sizeof(W) == 4) && n_shares < 120;
  if (jj < v.n && D2MHE_CHK(v.chk, wl, L, SITE_LIMB)) {
    const LimbTab* lt = v.limbs + wl;
    const u64 p = lt->p, w = lt->crt, ws = lt->crt_sh, fr = lt->frac;
    const u32 fs = lt->frac_shift;
    const size_t at = (size_t)wl * v.n + jj;
    auto load = [](const W* p) {
      R r;
      r.q = __ldg(reinterpret_cast<const decltype(r.q)*>(p));
      return r;
    };
    const R c = load(c0 + at);
    u64 a[V];
#pragma unroll
    for (u32 i = 0; i < V; ++i) a[i] = c.get(i);
    const W* s = sh + at;
    // Ten shares at a time, predicated, so that the loads of a remainder are in flight together too.  (Four at a time from 120
    // shares on: 130 recipients of 130 shares at N = 2048, L = 2 100 us, 92 us like this.)
    auto add = [&](auto sum) {
      for (u32 k0 = 0; k0 < n_shares; k0 += 10) {
        R h[10];
#pragma unroll
        for (u32 k = 0; k < 10; ++k)
          if (k0 + k < n_shares) h[k] = load(s + (k0 + k) * kstride);
#pragma unroll
        for (u32 k = 0; k < 10; ++k)
#pragma unroll
          for (u32 i = 0; i < V; ++i) a[i] = sum(a[i], h[k].get(i));
      }
    };
    if (lazy)
      add([](u64 x, u64 y) { return x + y; });
    else
      add([p](u64 x, u64 y) { return addmod(x, y, p); });
#pragma unroll
    for (u32 i = 0; i < V; ++i) terms[wl][V * lane + i] = mulhi_u64(shoup_full(a[i], w, ws, p) << fs, fr);
  }
  __syncthreads();
  for (u32 i = threadIdx.x; i < COLS && j0 + i < v.n; i += blockDim.x) {
    const u32 F = v.round.frac_bits;
    u64 sum = (u64)1 << (F - 1);
    for (u32 l = 0; l < L; ++l) sum += terms[l][i];
    u32 x = (u32)shoup_full(sum >> F, 1, v.round.t_sh, v.round.t);
    if ((sum & (((u64)1 << F) - 1)) >= ((u64)1 << F) - 2 * L)
      x = round_exact(v, [&](u32 l) {
        const size_t at = (size_t)l * v.n + j0 + i;
        const u64 p = v.limbs[l].p;
        u64 acc = c0[at];
        for (u32 k = 0; k < n_shares; ++k) acc = addmod(acc, sh[k * kstride + at], p);
        return acc;
      });
    plain[(size_t)unit * v.n + j0 + i] = x;
  }
}

// ---------------------------------------------------------------------------
// Packing: negacyclic transforms mod t in shared memory (32-bit arithmetic).
// Slot j sits at transform position brv(j).  grid = n_cts
// ---------------------------------------------------------------------------
__device__ __forceinline__ u32 shoup32_lazy(u32 x, uint2 w, u32 t) {
  return x * w.x - __umulhi(x, w.y) * t;
}
__device__ __forceinline__ u32 csub32(u32 x, u32 t) { return x >= t ? x - t : x; }

// Gentleman-Sande / Cooley-Tukey butterflies mod t on lazily reduced 32-bit values (below 2t)
__device__ __forceinline__ void gs32(u32& X, u32& Y, uint2 w, u32 t, u32 twot) {
  const u32 s = X + Y, d = X - Y + twot;
  X = csub32(s, twot);
  Y = shoup32_lazy(d, w, t);
}
__device__ __forceinline__ void ct32(u32& X, u32& Y, uint2 w, u32 t, u32 twot) {
  const u32 x = csub32(X, twot), T = shoup32_lazy(Y, w, t);
  X = x + T;
  Y = x - T + twot;
}

// encode: values -> slots at bit-reversed positions -> inverse transform, two stages per barrier
// values and plain may be the same storage (every CTA reads its whole row into shared memory before
// it writes the row back), so neither pointer is declared __restrict__
__global__ void __launch_bounds__(1024)
    k_encode(DevView v, const int32_t* values, u32* plain, u32 group, size_t group_stride) {
  u32* sm = reinterpret_cast<u32*>(smem_raw);
  const PlainTab pt = v.plain;
  const u32 n = v.n, logn = v.logn, t = pt.t, twot = pt.twot;
  // the values of block b = (g, c), c < group, start at g * group_stride + c * N: contiguous rows when
  // group_stride = group * N, a slice of a larger [.., n_cts, N] array otherwise
  const int32_t* in = values + (size_t)(blockIdx.x / group) * group_stride + (size_t)(blockIdx.x % group) * n;
  u32* out = plain + (size_t)blockIdx.x * n;
  bool bad = false;
  for (u32 j = threadIdx.x; j < n; j += blockDim.x) {
    const int32_t val = in[j];
    bad |= (val > (int32_t)pt.half) || (val < -(int32_t)pt.half);
    int32_t r = val % (int32_t)t;
    if (r < 0) r += (int32_t)t;
    const u32 pos = __brev(j) >> (32 - logn);
    if (D2MHE_CHK(v.chk, pos, n, SITE_STAGED)) sm[pos] = (u32)r;
  }
  if (bad) atomicOr(v.range_flag, RANGE_FLAG_VALUE);
  __syncthreads();
  u32 lt = 0;  // log2 of the butterfly span of the next stage
  for (; lt + 1 < logn; lt += 2) {
    const u32 span = 1u << lt, m = n >> (lt + 1);
    for (u32 b = threadIdx.x; b < (n >> 2); b += blockDim.x) {
      const u32 i2 = b >> lt, jj = b & (span - 1);
      const u32 base = (i2 << (lt + 2)) + jj;
      if (!D2MHE_CHK(v.chk, base + 3 * span, n, SITE_STAGED) || !D2MHE_CHK(v.chk, m + 2 * i2 + 1, n, SITE_TWIDDLE)) continue;
      u32 x0 = sm[base], x1 = sm[base + span], x2 = sm[base + 2 * span], x3 = sm[base + 3 * span];
      gs32(x0, x1, __ldg(pt.IW + m + 2 * i2), t, twot);
      gs32(x2, x3, __ldg(pt.IW + m + 2 * i2 + 1), t, twot);
      const uint2 w = __ldg(pt.IW + (m >> 1) + i2);
      gs32(x0, x2, w, t, twot);
      gs32(x1, x3, w, t, twot);
      sm[base] = x0;
      sm[base + span] = x1;
      sm[base + 2 * span] = x2;
      sm[base + 3 * span] = x3;
    }
    __syncthreads();
  }
  if (lt < logn) {  // odd number of stages: the last one (m = 1)
    const u32 span = 1u << lt;
    const uint2 w = __ldg(pt.IW + 1);
    for (u32 b = threadIdx.x; b < (n >> 1); b += blockDim.x) {
      u32 x0 = sm[b], x1 = sm[b + span];
      gs32(x0, x1, w, t, twot);
      sm[b] = x0;
      sm[b + span] = x1;
    }
    __syncthreads();
  }
  const uint2 ninv = make_uint2(pt.ninv, pt.ninv_sh);
  for (u32 j = threadIdx.x; j < n; j += blockDim.x) out[j] = csub32(shoup32_lazy(sm[j], ninv, t), t);
}

// decode: forward transform (two stages per barrier), slots read back from bit-reversed positions
// plain and values may be the same storage (see k_encode)
__global__ void __launch_bounds__(1024)
    k_decode(DevView v, const u32* plain, int32_t* values, u32 group, size_t group_stride) {
  u32* sm = reinterpret_cast<u32*>(smem_raw);
  const PlainTab pt = v.plain;
  const u32 n = v.n, logn = v.logn, t = pt.t, twot = pt.twot;
  const u32* in = plain + (size_t)blockIdx.x * n;
  int32_t* out = values + (size_t)(blockIdx.x / group) * group_stride + (size_t)(blockIdx.x % group) * n;  // as in k_encode
  for (u32 j = threadIdx.x; j < n; j += blockDim.x) sm[j] = in[j];
  __syncthreads();
  int lt = (int)logn - 1;  // log2 span of the next stage (m = n >> (lt + 1) groups)
  if (logn & 1u) {  // odd number of stages: do the first one (m = 1) alone
    const u32 span = 1u << lt;
    const uint2 w = __ldg(pt.W + 1);
    for (u32 b = threadIdx.x; b < (n >> 1); b += blockDim.x) {
      u32 x0 = sm[b], x1 = sm[b + span];
      ct32(x0, x1, w, t, twot);
      sm[b] = x0;
      sm[b + span] = x1;
    }
    __syncthreads();
    --lt;
  }
  for (; lt >= 1; lt -= 2) {
    // stages with spans 2^lt (m2 groups) then 2^(lt-1) (2 m2 groups)
    const u32 span = 1u << (lt - 1), m2 = n >> (lt + 1);
    for (u32 b = threadIdx.x; b < (n >> 2); b += blockDim.x) {
      const u32 i2 = b >> (lt - 1), jj = b & (span - 1);
      const u32 base = (i2 << (lt + 1)) + jj;
      if (!D2MHE_CHK(v.chk, base + 3 * span, n, SITE_STAGED) || !D2MHE_CHK(v.chk, 2 * m2 + 2 * i2 + 1, n, SITE_TWIDDLE)) continue;
      u32 x0 = sm[base], x1 = sm[base + span], x2 = sm[base + 2 * span], x3 = sm[base + 3 * span];
      const uint2 w = __ldg(pt.W + m2 + i2);
      ct32(x0, x2, w, t, twot);
      ct32(x1, x3, w, t, twot);
      ct32(x0, x1, __ldg(pt.W + 2 * m2 + 2 * i2), t, twot);
      ct32(x2, x3, __ldg(pt.W + 2 * m2 + 2 * i2 + 1), t, twot);
      sm[base] = x0;
      sm[base + span] = x1;
      sm[base + 2 * span] = x2;
      sm[base + 3 * span] = x3;
    }
    __syncthreads();
  }
  for (u32 j = threadIdx.x; j < n; j += blockDim.x) {
    const u32 pos = __brev(j) >> (32 - logn);
    if (!D2MHE_CHK(v.chk, pos, n, SITE_STAGED)) continue;
    const u32 y = csub32(csub32(sm[pos], twot), t);
    out[j] = y > pt.half ? (int32_t)y - (int32_t)t : (int32_t)y;
  }
}

}  // namespace

namespace D2MHE_LAUNCH_NS {

cudaError_t muladd(const DevView& v, cudaStream_t s, const u64* a, const u64* b, const u64* c,
                   u64* d, u32 batch) {
  const size_t n_pairs = (size_t)batch * v.L * v.n / 2;
  size_t blocks = (n_pairs + 255) / 256;
  if (blocks > 148 * 32) blocks = 148 * 32;
  k_muladd<<<(u32)blocks, 256, 0, s>>>(v, a, b, c, d, n_pairs);
  return cudaGetLastError();
}

template <class W>
static cudaError_t columns_launch(const DevView& v, cudaStream_t s, const W* ct, u32 n_rows, u32 n_cts,
                                  const u32* offsets_dev, const u32* rows_dev, u32 n_out, u32 nnz, W* agg, bool* done) {
  // groups of 32 threads but for few rows (N = 8192, L = 4, one group of 128 / four of 32: 9 rows 43.0 / 48.1 us, 10 rows
  // 41.0 / 43.9, 13 rows 41.0 / 39.8, 16 rows 56.0 / 51.2, 30 rows 73.7 / 51.2)
  const u32 cols = n_rows < 12 ? 128 : 32;
  const size_t smem = (size_t)n_rows * cols * 16 + ((size_t)n_out + 1 + nnz) * 4, most = 56 * 1024;
  const u32 blocks = (u32)((2 * (size_t)v.L * v.n * sizeof(W) / 16 + cols - 1) / cols);
  *done = nnz > n_rows && smem <= most && blocks <= 65535 && (size_t)n_cts * blocks * cols >= 512 * (size_t)v.sms;
  if (!*done) return cudaSuccess;
  const auto kernel = cols == 128 ? k_aggregate_columns<W, 128, 1> : k_aggregate_columns<W, 32, 4>;
  // The limit is one value per kernel and device: always the same one, so that a call with fewer rows on another host
  // thread cannot lower it between this call's two steps.
  cudaError_t e = set_smem(kernel, most);
  if (e != cudaSuccess) return e;
  kernel<<<dim3(n_cts, blocks), 128, smem, s>>>(v, ct, n_rows, n_cts, offsets_dev, rows_dev, n_out, nnz, agg);
  return cudaGetLastError();
}
// neighbour sums by columns where that is the better kernel (*done)
cudaError_t aggregate_columns32(const DevView& v, cudaStream_t s, const u32* ct, u32 n_rows, u32 n_cts,
                                const u32* offsets_dev, const u32* rows_dev, u32 n_out, u32 nnz, u32* agg, bool* done) {
  return columns_launch(v, s, ct, n_rows, n_cts, offsets_dev, rows_dev, n_out, nnz, agg, done);
}

cudaError_t aggregate(const DevView& v, cudaStream_t s, const u64* ct, u32 n_rows, u32 n_cts,
                      const u32* offsets_dev, const u32* rows_dev, u32 n_out, u32 nnz, u64* agg) {
  bool done = false;
  const cudaError_t e = columns_launch(v, s, ct, n_rows, n_cts, offsets_dev, rows_dev, n_out, nnz, agg, &done);
  if (e != cudaSuccess || done) return e;
  const size_t ct_pairs = (size_t)v.L * v.n;
  u32 by = (u32)((ct_pairs + 255) / 256);
  if (by > 32768) by = 32768;
  dim3 grid(n_out * n_cts, by);
  k_aggregate<<<grid, 256, 0, s>>>(v, ct, n_cts, offsets_dev, rows_dev, agg);
  return cudaGetLastError();
}

template <class W>
static cudaError_t combine_words(const DevView& v, cudaStream_t s, const W* agg, const W* shares, u32 n_rec,
                                 u32 n_shares, u32 share_comps, u32 n_cts, u32* plain) {
  const u32 units = n_rec * n_cts;
  auto launch = [&](auto kernel, u32 cols) {
    kernel<<<units * ((v.n + cols - 1) / cols), 32 * v.L, 0, s>>>(v, agg, shares, n_shares, share_comps, n_cts, plain);
    return cudaGetLastError();
  };
  // Four words to a thread leave half the blocks, which pays once the launch fills the chip: from a dozen warps per
  // multiprocessor on (four units of twenty, N = 8192, L = 8, 14 warps: 6.5 and 4.7 us; 40 of ten, L = 7: 28.6 and 23.4; eight
  // of ten, L = 3, 10 warps: 3.8 and 3.8; nine of fifty at N = 2048, L = 3, 3 warps: 4.9 and 5.9; one of ten at N = 8192,
  // L = 3: 2.5 and 3.0).  Below N = 128 half the lanes would idle (1600 units of four at N = 64: 4.6 and 5.8 us).
  if constexpr (sizeof(W) == 4)
    if (v.L <= 8 && v.n >= 128 && (u64)units * (v.n / 128) * v.L >= 12 * (u64)v.sms) return launch(k_combine<W, 4, 8>, 128);
  return launch(k_combine<W, 2, D2MHE_MAX_LIMBS>, 64);
}
cudaError_t combine(const DevView& v, cudaStream_t s, const u64* agg, const u64* shares, u32 n_rec,
                    u32 n_shares, u32 share_comps, u32 n_cts, u32* plain) {
  return combine_words<u64>(v, s, agg, shares, n_rec, n_shares, share_comps, n_cts, plain);
}
cudaError_t combine32(const DevView& v, cudaStream_t s, const u32* agg, const u32* shares, u32 n_rec, u32 n_shares,
                      u32 n_cts, u32* plain) {
  return combine_words<u32>(v, s, agg, shares, n_rec, n_shares, 1, n_cts, plain);
}

// values: n_groups groups of `group` rows of N values, group g starting at values + g * group_stride
// (elements); plain: [n_groups * group, N] contiguous
cudaError_t encode_strided(const DevView& v, cudaStream_t s, const int32_t* values, u32 n_groups, u32 group,
                           size_t group_stride, u32* plain) {
  if (v.logn >= 12 && v.logn <= 14) return encode16(v, s, values, n_groups, group, group_stride, plain);
  const size_t smem = (size_t)v.n * 4;
  cudaError_t e = set_smem(k_encode, smem);
  if (e != cudaSuccess) return e;
  u32 threads = v.n / 4 < 1024 ? (v.n / 4 < 32 ? 32 : v.n / 4) : 1024;
  k_encode<<<n_groups * group, threads, smem, s>>>(v, values, plain, group, group_stride);
  return cudaGetLastError();
}
cudaError_t encode(const DevView& v, cudaStream_t s, const int32_t* values, u32 n_cts, u32* plain) {
  return encode_strided(v, s, values, 1, n_cts, (size_t)n_cts * v.n, plain);
}

cudaError_t decode_strided(const DevView& v, cudaStream_t s, const u32* plain, u32 n_groups, u32 group,
                           size_t group_stride, int32_t* values) {
  if (v.logn >= 12 && v.logn <= 14) return decode16(v, s, plain, n_groups, group, group_stride, values);
  const size_t smem = (size_t)v.n * 4;
  cudaError_t e = set_smem(k_decode, smem);
  if (e != cudaSuccess) return e;
  u32 threads = v.n / 4 < 1024 ? (v.n / 4 < 32 ? 32 : v.n / 4) : 1024;
  k_decode<<<n_groups * group, threads, smem, s>>>(v, plain, values, group, group_stride);
  return cudaGetLastError();
}
cudaError_t decode(const DevView& v, cudaStream_t s, const u32* plain, u32 n_cts, int32_t* values) {
  return decode_strided(v, s, plain, 1, n_cts, (size_t)n_cts * v.n, values);
}

}  // namespace D2MHE_LAUNCH_NS
