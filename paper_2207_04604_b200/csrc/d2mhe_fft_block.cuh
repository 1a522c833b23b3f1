// Block-level pieces of the double-precision ring products (see d2mhe_fft.cuh): transforms of one
// polynomial held in the registers of a thread block, tensor memory as the home of the transform that
// stays with the block, and the rounding to residues.
#pragma once
#include "d2mhe_fft.cuh"
#include "d2mhe_kernels_common.cuh"

namespace {

// GR groups of TG = 16 R threads, n = 256 R GR points, 16 per thread; COLS columns r = tg + c TG of R points each
// in pass C (tg = thread of the group).  CTAS: thread blocks per SM, 512 threads of 128 registers in all.
template <int LOGN>
struct FftGeo {
  static constexpr int R = LOGN == 12 ? 8 : 16, GR = LOGN == 14 ? 2 : 1;
  static constexpr int TG = 16 * R, T = TG * GR, NG = 256 * R, n = NG * GR, COLS = 16 / R;
  static constexpr int CTAS = 512 / T;
  // Shared memory: per group NG complex numbers in rows of 256 (kC) with a stride of 271, which leaves room for the
  // 16 x 17 layout of the exchange inside a row; the low part's results (stash: 0 none, 1 a word and a byte for each of
  // 2n, 2 half a byte more).
  static constexpr int RS = 271;
  static constexpr size_t ex_bytes = (size_t)GR * R * RS * 16;
  __host__ __device__ static constexpr size_t smem_bytes(int stash) {
    // 16: the word of tcgen05.alloc, one for a wait that ran out, and the barrier
    return ex_bytes + (stash ? (size_t)n * (9 + stash) : 0) + 16;
  }
  // Words of tensor memory per thread for one transform, and columns for `k` of them: warp w of a block
  // reaches the lanes 32 (w mod 4) .. + 31 only, so warps w, w + 4, .. share lanes and split the columns.
  static constexpr int WORDS = 64;
  __host__ __device__ static constexpr u32 tmem_cols(int k) { return (u32)(WORDS * k * (T / 128)); }
};

// the block's shared memory and this thread's place in it (STASH: as in FftGeo::smem_bytes)
template <int LOGN, int STASH = 1>
struct FftSmem {
  using G = FftGeo<LOGN>;
  double2* ex;     // of this thread's group
  double2* other;  // of the other group (GR = 2)
  u32 *words, *bytes, *slot;
  unsigned short* nibbles;
  u32* chk;  // device check words (read by the checked kernel build only)
  u32 tg;
  static constexpr int WAIT_TRIES = 1 << 18;
  u32 phase = 0;           // of the barrier in the last transform
  int tries = WAIT_TRIES;  // left to this thread's waits
  bool announce = true;    // false: a block barrier instead (a constant in every kernel)
  __device__ __forceinline__ explicit FftSmem(const DevView& v) {
    chk = v.chk;
    const u32 g = group();
    tg = G::GR > 1 ? threadIdx.x % G::TG : threadIdx.x;
    double2* base = reinterpret_cast<double2*>(smem_raw);
    ex = base + g * (G::R * G::RS);
    other = base + (1u - g) * (G::R * G::RS);
    words = reinterpret_cast<u32*>(smem_raw + G::ex_bytes);
    bytes = words + 2 * G::n;
    nibbles = reinterpret_cast<unsigned short*>(bytes + G::n / 2);
    slot = reinterpret_cast<u32*>(smem_raw + G::smem_bytes(STASH) - 16);
  }
  // element i of the exchange area behind e
  __device__ __forceinline__ void put(double2* e, u32 i, double r, double im) const {
    if (D2MHE_CHK(chk, (u32)(e - reinterpret_cast<double2*>(smem_raw)) + i, G::GR * G::R * G::RS, SITE_STAGED))
      e[i] = make_double2(r, im);
  }
  __device__ __forceinline__ double2 get(const double2* e, u32 i) const {
    if (!D2MHE_CHK(chk, (u32)(e - reinterpret_cast<const double2*>(smem_raw)) + i, G::GR * G::R * G::RS, SITE_STAGED))
      return make_double2(0.0, 0.0);
    return e[i];
  }
  // The exchange area is free for the next transform when every warp has read the last one's columns.  A warp arrives
  // when it has, and waits only when it writes there again, most of a transform later: nothing stalls where a block
  // barrier made every warp wait for the slowest one.  Shares at N = 8192 716 -> 679 us, at N = 16384 1852 -> 1709 us,
  // Conversion at N = 16384 4247 -> 3888 us (1480 rows of ten parties); not in the encryption kernels from N = 8192
  // on, whose two to four transforms a block don't repay it (370 ciphertexts, L = 4, block barriers against this: N = 4096
  // 83.9 / 77.0 us, N = 8192 153.8 / 161.8, N = 16384 352 / 359), nor in the one for 32-bit words with its one or two
  // (N = 4096, L = 7, 370 ciphertexts 63.9 / 62.7 us).
  __device__ __forceinline__ void init() const {  // one thread, ahead of a block barrier
    slot[1] = 0;
    asm volatile("mbarrier.init.shared.b64 [%0], %1;" ::"r"(bar()), "r"(G::T / 32) : "memory");
  }
  __device__ __forceinline__ u32 bar() const { return (u32)__cvta_generic_to_shared(slot) + 8; }
  __device__ __forceinline__ void finish(const DevView& v) const {  // one thread, behind the last block barrier
    if (slot[1]) atomicOr(v.range_flag, RANGE_FLAG_WAIT);
  }
  __device__ __forceinline__ void release() const {
    if (!announce) return;
    __syncwarp();
    // one lane, by a predicate: with a branch the warp would not be known to be converged at the tensor-memory loads that follow
    asm volatile("{.reg .b64 t; .reg .pred p; setp.eq.u32 p, %1, 0; @p mbarrier.arrive.shared.b64 t, [%0];}" ::"r"(bar()),
                 "r"(threadIdx.x & 31u) : "memory");
  }
  // A try that fails takes 4 us on this GPU (5000 of them in the self-test's kernel 20 ms, with and without a time hint), and
  // all the waits of a thread have WAIT_TRIES failing ones between them: a block loses about a second, whatever is wrong, and
  // its call is reported as failed (finish).
  __device__ __forceinline__ void acquire() {
    if (!announce) {
      __syncthreads();
      return;
    }
    u32 done = 0;
#pragma unroll 1  // refresh shares at N = 4096 737 -> 730 us, receiving call of 594 rows of nine 262.6 -> 260.9
    for (; !done && tries; --tries)
      asm volatile("{.reg .pred p; mbarrier.try_wait.parity.shared.b64 p, [%1], %2; selp.u32 %0, 1, 0, p;}"
                   : "=r"(done) : "r"(bar()), "r"(phase ^ 1u) : "memory");
    tries += (int)done;  // the one that succeeded
    if (!done) slot[1] = 1;
    phase ^= 1u;
  }
  __device__ __forceinline__ u32 group() const { return G::GR > 1 ? threadIdx.x / G::TG : 0u; }
  __device__ __forceinline__ void group_sync() const {
    if (G::GR == 1)
      __syncthreads();
    else
      asm volatile("bar.sync %0, %1;" ::"r"(1u + group()), "n"(G::TG) : "memory");
  }
};

// ---- tensor memory --------------------------------------------------------------------------------
// One warp allocates; every thread then owns `words` 32-bit words at the returned address.  All tcgen05 instructions here
// are .aligned: a warp has to be converged at them, which __syncwarp guarantees after the branches of single threads (the
// loads and stores of transforms come behind the exchanges, which have theirs).
__device__ __forceinline__ void tmem_alloc(u32* slot_smem, u32 cols) {
  __syncwarp();
  const u32 a = (u32)__cvta_generic_to_shared(slot_smem);
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(a), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(u32 base, u32 cols) {
  __syncwarp();
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols));
}
__device__ __forceinline__ u32 tmem_thread_base(u32 base, u32 words) {
  const u32 w = threadIdx.x >> 5;
  return base + ((w & 3u) << 21) + (w >> 2) * words;
}
__device__ __forceinline__ void tmem_store4(u32 addr, const cpx (&c)[4]) {
  u32 w[16];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    w[4 * i] = (u32)__double2loint(c[i].r), w[4 * i + 1] = (u32)__double2hiint(c[i].r);
    w[4 * i + 2] = (u32)__double2loint(c[i].i), w[4 * i + 3] = (u32)__double2hiint(c[i].i);
  }
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(addr),
      "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7]), "r"(w[8]), "r"(w[9]),
      "r"(w[10]), "r"(w[11]), "r"(w[12]), "r"(w[13]), "r"(w[14]), "r"(w[15])
      : "memory");
}
__device__ __forceinline__ void tmem_store_done() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
// issues the load of four points; the words are valid after tmem_wait
struct TmemQuad {
  u32 w[16];
  __device__ __forceinline__ void issue(u32 addr) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
        : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]), "=r"(w[8]),
          "=r"(w[9]), "=r"(w[10]), "=r"(w[11]), "=r"(w[12]), "=r"(w[13]), "=r"(w[14]), "=r"(w[15])
        : "r"(addr));
  }
  // ties the words to a wait issued before: nothing that uses them can move above it
  __device__ __forceinline__ void get(cpx (&c)[4]) {
    asm volatile("" : "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3]), "+r"(w[4]), "+r"(w[5]), "+r"(w[6]), "+r"(w[7]),
                      "+r"(w[8]), "+r"(w[9]), "+r"(w[10]), "+r"(w[11]), "+r"(w[12]), "+r"(w[13]), "+r"(w[14]), "+r"(w[15]));
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      c[i].r = __hiloint2double((int)w[4 * i + 1], (int)w[4 * i]);
      c[i].i = __hiloint2double((int)w[4 * i + 3], (int)w[4 * i + 2]);
    }
  }
};
__device__ __forceinline__ void tmem_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---- exchanges through shared memory: 16-byte accesses, eight lanes to a wavefront ----------------------------------
// Inside the 16 threads of a row: element k of lane a goes to element a of lane k, through a 16 x 17 layout (both
// directions without bank conflicts, constant offsets).  Rows belong to one warp: no block barrier.
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_swap_row(const FftSmem<LOGN, STASH>& sm, double* xr, double* xi) {
  using G = FftGeo<LOGN>;
  const u32 l16 = sm.tg & 15u;
  double2* e = sm.ex + (sm.tg >> 4) * G::RS;
  static_for<16>([&](auto k_) {
    constexpr int k = decltype(k_)::value, i = brev_c<16>(k);
    sm.put(e, l16 + k * 17, xr[i], xi[i]);
  });
  __syncwarp();
  static_for<16>([&](auto k_) {
    constexpr int k = brev_c<16>(decltype(k_)::value);  // in the order in which the next pass uses them
    const double2 t = sm.get(e, l16 * 17 + k);
    xr[k] = t.x;
    xi[k] = t.y;
  });
  __syncwarp();
}
// the 16 results of a row pass -> row-major, and back; own rows only
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_put_rows(const FftSmem<LOGN, STASH>& sm, const double* xr, const double* xi) {
  double2* e = sm.ex + (sm.tg >> 4) * FftGeo<LOGN>::RS + (sm.tg & 15u);
  static_for<16>([&](auto k_) {
    constexpr int k = decltype(k_)::value, i = brev_c<16>(k);
    sm.put(e, 16 * k, xr[i], xi[i]);
  });
}
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_get_rows(const FftSmem<LOGN, STASH>& sm, double* xr, double* xi) {
  const double2* e = sm.ex + (sm.tg >> 4) * FftGeo<LOGN>::RS + (sm.tg & 15u);
  static_for<16>([&](auto k_) {
    constexpr int k = brev_c<16>(decltype(k_)::value);
    const double2 t = sm.get(e, 16 * k);
    xr[k] = t.x;
    xi[k] = t.y;
  });
}
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_put_cols(const FftSmem<LOGN, STASH>& sm, const double* xr, const double* xi) {
  using G = FftGeo<LOGN>;
#pragma unroll
  for (int c = 0; c < G::COLS; ++c)
    static_for<G::R>([&](auto k_) {
      constexpr int k = decltype(k_)::value, i = brev_c<G::R>(k);
      sm.put(sm.ex, sm.tg + k * G::RS + c * G::TG, xr[c * G::R + i], xi[c * G::R + i]);
    });
}
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_get_cols(const FftSmem<LOGN, STASH>& sm, double* xr, double* xi) {
  using G = FftGeo<LOGN>;
#pragma unroll
  for (int c = 0; c < G::COLS; ++c)
    static_for<G::R>([&](auto k_) {
      constexpr int k = brev_c<G::R>(decltype(k_)::value);
      const double2 t = sm.get(sm.ex, sm.tg + k * G::RS + c * G::TG);
      xr[c * G::R + k] = t.x;
      xi[c * G::R + k] = t.y;
    });
}

// A 16-byte load that stays where it is written (a table entry that is read again in every transform instead of
// living in registers, or a batch of loads that is issued as a whole).
__device__ __forceinline__ cpx ld_here(const double2* p) {
  cpx c;
  asm volatile("ld.global.nc.v2.f64 {%0, %1}, [%2];" : "=d"(c.r), "=d"(c.i) : "l"(p));
  return c;
}
__device__ __forceinline__ cpx ld_cpx(const double2* p) {
  const double2 t = __ldg(p);
  return cpx{t.x, t.y};
}
// entry i of a table of `limit`
template <int LOGN, int STASH>
__device__ __forceinline__ cpx tw_cpx(const FftSmem<LOGN, STASH>& sm, const double2* table, u32 i, u32 limit) {
  return D2MHE_CHK(sm.chk, i, limit, SITE_TWIDDLE) ? ld_cpx(table + i) : cpx{0.0, 0.0};
}
template <int LOGN, int STASH>
__device__ __forceinline__ cpx tw_here(const FftSmem<LOGN, STASH>& sm, const double2* table, u32 i, u32 limit) {
  return D2MHE_CHK(sm.chk, i, limit, SITE_TWIDDLE) ? ld_here(table + i) : cpx{0.0, 0.0};
}

// Forward transform.  in(c, jC, h): the coefficients j and j + n as a complex number, j = r + 256 jC + h n/2 with
// r = tg + c TG (h = 0 for one group).  Leaves Z_k, k = kC + R kB + 16 R kA, in x[brev(kA)] of thread (kC, kB) of its group.
template <int LOGN, int STASH, class In>
__device__ __forceinline__ void fft_forward_at(const FftSmem<LOGN, STASH>& sm, const FftTab& ft, double* xr, double* xi, In in) {
  using G = FftGeo<LOGN>;
  constexpr int R = G::R;
  const u32 g = sm.group();
  static_for<G::COLS>([&](auto c_) {
    constexpr int c = decltype(c_)::value;
    const cpx t = tw_cpx(sm, ft.twist, 256 * g + sm.tg + (u32)(c * G::TG), 256 * G::GR);
    static_for<R>([&](auto j_) {
      constexpr int j = decltype(j_)::value;
      cpx z = in(c_, j_, std::integral_constant<int, 0>{});
      if constexpr (G::GR == 2) {  // z_j +- q z_(j + n/2)
        const cpx y = in(c_, j_, std::integral_constant<int, 1>{});
        const double h = g ? -root_c<16>() : root_c<16>();
        z = cpx{D2MHE_FMA(h, y.r - y.i, z.r), D2MHE_FMA(h, y.r + y.i, z.i)};
      }
      const cpx p = fft_twist<G::R, G::GR, j>(t, g);
      z = cmul(z, cpx{p.r, -p.i});
      xr[c * R + j] = z.r;
      xi[c * R + j] = z.i;
    });
    fft_eval<R, 1, 0>(xr + c * R, xi + c * R, TwNone());
  });
  __syncthreads();  // previous users of ex are done
  fft_put_cols<LOGN>(sm, xr, xi);
  sm.group_sync();
  fft_get_rows<LOGN>(sm, xr, xi);
  const u32 l16 = sm.tg & 15u, row = sm.tg >> 4;
  {
    const cpx t[2] = {tw_cpx(sm, ft.fwd2, row, R), tw_cpx(sm, ft.fwd2, R + row, 2 * R)};
    fft_eval<16, 1, 0>(xr, xi, TwDerived<16, 1>(t));
  }
  __syncwarp();  // the rows have been read by their own warp only
  fft_swap_row<LOGN>(sm, xr, xi);
  {
    const u32 k = row + (u32)R * l16;
    const cpx t[2] = {tw_cpx(sm, ft.fwd3, k, 16 * R), tw_cpx(sm, ft.fwd3, 16 * R + k, 32 * R)};
    fft_eval<16, 1, 0>(xr, xi, TwDerived<16, 1>(t));
  }
}

// in(j): the same by coefficient number, j < n
template <int LOGN, int STASH, class In>
__device__ __forceinline__ void fft_forward(const FftSmem<LOGN, STASH>& sm, const FftTab& ft, double* xr, double* xi, In in) {
  using G = FftGeo<LOGN>;
  fft_forward_at<LOGN>(sm, ft, xr, xi, [&](auto c_, auto j_, auto h_) {
    return in(sm.tg + (u32)(c_.value * G::TG + 256 * j_.value + h_.value * G::NG));
  });
}

// A transform in tensor memory: four points (k, k + 8, k + 4, k + 12) after one another, as fft_product4 takes them.
__device__ __forceinline__ void fft_to_tmem(u32 addr, const double* xr, const double* xi) {
  static_for<4>([&](auto q_) {
    cpx c[4];
    static_for<4>([&](auto i_) {
      constexpr int k = brev_c<16>(decltype(q_)::value + 4 * brev_c<4>(decltype(i_)::value));
      c[i_.value] = cpx{xr[k], xi[k]};
    });
    tmem_store4(addr + q_.value * 16, c);
  });
}

// the same for the points of a stored transform as fft_load leaves them
__device__ __forceinline__ void fft_loaded_to_tmem(u32 addr, const double* xr, const double* xi) {
  static_for<4>([&](auto q_) {
    cpx c[4];
    static_for<4>([&](auto i_) {
      constexpr int k = decltype(q_)::value + 4 * brev_c<4>(decltype(i_)::value);
      c[i_.value] = cpx{xr[k], xi[k]};
    });
    tmem_store4(addr + q_.value * 16, c);
  });
}

// A stored transform (a row of n points): point kA of a thread in slot kA T + thread.
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_load(const FftSmem<LOGN, STASH>& sm, const double2* row, double* xr, double* xi) {
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const cpx s = tw_here(sm, row, threadIdx.x + k * FftGeo<LOGN>::T, FftGeo<LOGN>::n);
    xr[k] = s.r;
    xi[k] = s.i;
  }
}
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_store(const FftSmem<LOGN, STASH>& sm, double2* row, const double* xr, const double* xi) {
  static_for<16>([&](auto k_) {
    constexpr int k = decltype(k_)::value, i = brev_c<16>(k);
    const u32 at = threadIdx.x + k * FftGeo<LOGN>::T;
    if (D2MHE_CHK(sm.chk, at, FftGeo<LOGN>::n, SITE_STORE)) row[at] = make_double2(xr[i], xi[i]);
  });
}

// Products of the points in registers with a transform in tensor memory (with the first two stages of pass A).
__device__ __forceinline__ void fft_product_tmem(u32 addr, double* xr, double* xi) {
  TmemQuad buf[2];
  buf[0].issue(addr);
  static_for<4>([&](auto q_) {
    constexpr int q = decltype(q_)::value;
    tmem_wait();
    cpx c[4];
    buf[q & 1].get(c);
    if constexpr (q + 1 < 4) buf[(q + 1) & 1].issue(addr + (q + 1) * 16);
    fft_product4<-1>(xr, xi, q, c);
  });
}

// The same with a stored transform instead of the one in tensor memory.
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_product_row(const FftSmem<LOGN, STASH>& sm, const double2* row, double* xr, double* xi) {
  static_for<4>([&](auto q_) {
    constexpr int q = decltype(q_)::value;
    cpx c[4];
    static_for<4>([&](auto i_) {
      c[i_.value] = tw_cpx(sm, row, threadIdx.x + (q + 4 * brev_c<4>(decltype(i_)::value)) * FftGeo<LOGN>::T, FftGeo<LOGN>::n);
    });
    fft_product4<-1>(xr, xi, q, c);
  });
}
// Sums of two products: registers by tensor memory, and two stored transforms.
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_product_sum(const FftSmem<LOGN, STASH>& sm, u32 addr, const double2* row_a,
                                                const double2* row_b, double* xr, double* xi) {
  static_for<4>([&](auto q_) {
    constexpr int q = decltype(q_)::value;
    TmemQuad quad;
    quad.issue(addr + q * 16);
    cpx a[4], b[4], c[4];
    static_for<4>([&](auto i_) {
      constexpr int k = q + 4 * brev_c<4>(decltype(i_)::value);
      a[i_.value] = tw_cpx(sm, row_a, threadIdx.x + k * FftGeo<LOGN>::T, FftGeo<LOGN>::n);
      b[i_.value] = tw_cpx(sm, row_b, threadIdx.x + k * FftGeo<LOGN>::T, FftGeo<LOGN>::n);
    });
    tmem_wait();
    quad.get(c);
    fft_product4_sum<-1>(xr, xi, q, c, a, b);
  });
}

// Inverse transform of what the products left, up to the twist: digit jC of column r = tg + c TG is left in
// x[c R + brev(jC)]; tw: the columns' twist.  before_last(): called ahead of the arithmetic of pass C.
// Table entries are fetched a pass ahead of their use (they come from L2 as often as not).
template <int LOGN, int STASH, class Hook>
__device__ __forceinline__ void fft_inverse(FftSmem<LOGN, STASH>& sm, const FftTab& ft, double* xr, double* xi,
                                            cpx (&tw)[FftGeo<LOGN>::COLS], Hook before_last) {
  using G = FftGeo<LOGN>;
  const cpx t2[2] = {tw_here(sm, ft.inv2, sm.tg & 15u, 16), tw_here(sm, ft.inv2, 16 + (sm.tg & 15u), 32)};
  fft_eval<16, -1, 2>(xr, xi, TwNone());
  sm.acquire();  // previous users of ex are done
  fft_swap_row<LOGN>(sm, xr, xi);
  cpx t[G::COLS][2];
#pragma unroll
  for (int c = 0; c < G::COLS; ++c)
#pragma unroll
    for (int i = 0; i < 2; ++i) t[c][i] = tw_here(sm, ft.inv3, 256 * i + sm.tg + c * G::TG, 256 * (i + 1));
  fft_eval<16, -1, 0>(xr, xi, TwDerived<16, -1>(t2));
  fft_put_rows<LOGN>(sm, xr, xi);
#pragma unroll
  for (int c = 0; c < G::COLS; ++c) tw[c] = tw_here(sm, ft.twist, 256 * sm.group() + sm.tg + c * G::TG, 256 * G::GR);
  sm.group_sync();
  fft_get_cols<LOGN>(sm, xr, xi);
  if (G::GR == 1) sm.release();
  before_last();
#pragma unroll
  for (int c = 0; c < G::COLS; ++c) fft_eval<G::R, -1, 0>(xr + c * G::R, xi + c * G::R, TwDerived<G::R, -1>(t[c]));
}

// Result number i of a thread (below 32) belongs to this coefficient.
template <int LOGN, int STASH>
__device__ __forceinline__ u32 fft_coef(const FftSmem<LOGN, STASH>& sm, int i) {
  using G = FftGeo<LOGN>;
  if (G::GR == 2) return sm.tg + 256u * (8u * sm.group() + (u32)(i & 7)) + 4096u * (u32)(i >> 3);
  if (G::R == 8) return sm.tg + 128u * (u32)(i >> 4) + 256u * (u32)(i & 15);
  return sm.tg + 256u * (u32)i;
}
// fft_twist's constants of two groups, by group and digit.  Selected instead, they were kept across the loop and spilled:
// shares at N = 16384 1868 us, Conversion 4505 us, with two copies of the end of a part, 1852 and 4247 us like this.
struct FftDigits {
  double2 c[32];
  constexpr FftDigits() : c() {
    for (int g = 0; g < 2; ++g)
      for (int j = 0; j < 16; ++j) c[16 * g + j].x = fft_digit(g, j).r, c[16 * g + j].y = fft_digit(g, j).i;
  }
};
static __device__ __constant__ FftDigits c_digit;
// The last step of an inverse transform: twists, joins the groups and hands the 32 results of this thread over in
// eight portions of four, rounded: out(m, first number, R or 0 (see fft_result_number), v[4]) with v = bits of
// M + value, M = 1.5 * 2^(52 - f) + 1/2, so that bits >> f is floor(value + 1/2) plus a constant.
template <int LOGN, int STASH, class Out>
__device__ __forceinline__ void fft_results(const FftSmem<LOGN, STASH>& sm, const cpx (&tw)[FftGeo<LOGN>::COLS], double* xr,
                                            double* xi, double magic, Out out) {
  using G = FftGeo<LOGN>;
  constexpr int R = G::R;
  if constexpr (G::GR == 1) {
    // portion: digits j, j + 1 of a column; results (column c) i = 2R c + j, + 1 (real) and + R (imaginary)
    static_for<8>([&](auto m_) {
      constexpr int m = decltype(m_)::value, c = 2 * m / R, j = 2 * m % R, i0 = c * R + brev_c<R>(j), i1 = c * R + brev_c<R>(j + 1);
      const cpx p0 = fft_twist<G::R, G::GR, j>(tw[c], 0), p1 = fft_twist<G::R, G::GR, j + 1>(tw[c], 0);
      u64 v[4];
      v[0] = (u64)__double_as_longlong(__fma_rn(xr[i0], p0.r, __fma_rn(-xi[i0], p0.i, magic)));
      v[1] = (u64)__double_as_longlong(__fma_rn(xr[i1], p1.r, __fma_rn(-xi[i1], p1.i, magic)));
      v[2] = (u64)__double_as_longlong(__fma_rn(xr[i0], p0.i, __fma_rn(xi[i0], p0.r, magic)));
      v[3] = (u64)__double_as_longlong(__fma_rn(xr[i1], p1.i, __fma_rn(xi[i1], p1.r, magic)));
      out(m_, std::integral_constant<int, 2 * R * c + j>{}, std::integral_constant<int, R>{}, v);
    });
  } else {
    // Group g finishes the digits 8 g .. 8 g + 7 and sends the others; column r of ex is this thread's own until the
    // block barrier.  z_j = y0 + y1, z_(j + 4096) = (y0 - y1) e^(-i pi / 4); the group signs make both sides equal.
    const u32 g = sm.group();
    u32 step = g;  // not known to be the same in every transform: the constants are read where they are used
    asm volatile("" : "+r"(step));
    static_for<16>([&](auto j_) {
      constexpr int j = decltype(j_)::value, i = brev_c<16>(j);
      const double2 c = c_digit.c[step * 16 + j];
      const cpx z = cmul(cpx{xr[i], xi[i]}, cmul(tw[0], cpx{c.x, c.y}));
      xr[i] = z.r;
      xi[i] = z.i;
    });
    static_for<8>([&](auto j_) {
      constexpr int j = decltype(j_)::value, lo = brev_c<16>(j), hi = brev_c<16>(j + 8);
      sm.put(sm.ex, sm.tg + j * G::RS, g ? xr[lo] : xr[hi], g ? xi[lo] : xi[hi]);
      if (g) xr[lo] = xr[hi], xi[lo] = xi[hi];
    });
    __syncthreads();
    const double s = g ? -root_c<16>() : root_c<16>();
    static_for<8>([&](auto j_) {
      constexpr int j = decltype(j_)::value, lo = brev_c<16>(j), hi = brev_c<16>(j + 8);
      const double2 o = sm.get(sm.other, sm.tg + j * G::RS);
      if constexpr (j == 7) sm.release();
      const double dr = xr[lo] - o.x, di = xi[lo] - o.y;  // group 1: the negative, undone by s
      u64 v[4];
      v[0] = (u64)__double_as_longlong((xr[lo] + o.x) + magic);
      v[1] = (u64)__double_as_longlong(__fma_rn(s, dr + di, magic));
      v[2] = (u64)__double_as_longlong((xi[lo] + o.y) + magic);
      v[3] = (u64)__double_as_longlong(__fma_rn(s, di - dr, magic));
      out(j_, j_, std::integral_constant<int, 0>{}, v);
    });
  }
}
// number (fft_coef's i) of result B of the portion whose first is I0: one group: I0, I0 + 1, I0 + R, I0 + R + 1;
// two groups: I0 + 8 B
template <int I0, int RR, int B>
__device__ __forceinline__ constexpr int fft_result_number() {
  return RR ? I0 + (B & 1) + (B >> 1) * RR : I0 + 8 * B;
}

// The low part's result V_lo waits for the high part: with 8 fraction bits V_lo + 2^39 is bytes 1 .. 5 of the rounded
// value (|V_lo| <= 2^39: ternary factors), V_lo + 2^43 is these and the low half of byte 6 (Conversion: below 2^43).
#define D2MHE_FFT_MAGIC_LO (1.5 * 17592186044416.0 + 549755813888.0 + 0.5) /* 1.5 * 2^44 + 2^39 + 1/2 */
#define D2MHE_FFT_MAGIC_LO44 (1.5 * 17592186044416.0 + 0.5)                /* 1.5 * 2^44 + 1/2 */
__device__ __forceinline__ u32 lo_word(u64 bits) { return __byte_perm((u32)bits, (u32)(bits >> 32), 0x4321); }
__device__ __forceinline__ u32 lo_bytes(u64 a, u64 b, u64 c, u64 d) {  // byte 5 of four rounded values
  return __byte_perm(__byte_perm((u32)(a >> 32), (u32)(b >> 32), 0x0051),
                     __byte_perm((u32)(c >> 32), (u32)(d >> 32), 0x0051), 0x5410);
}

// 2^b + 64 p + V_lo + 2^h V_hi + e0 - 19, between 2^b and 2^b + 129 p, for fft_canon and nothing else (any other reduction
// would be off by d for the 2^b): the multiples of d below add up to less than 61 p (d N / 2 with ternary factors, where
// 256 d < 2^b is enough; FFT_CONV_V times that in Conversion, which the host tests).  low: V_lo plus
// its offset; hi: the rounded high part with f fraction bits, f = 32 - (b - h) and p = 2^b - d: its low word holds
// V_hi mod 2^(b-h) above the fraction, its high word floor(V_hi / 2^(b-h)) plus a constant, which counts multiples of
// 2^b = d (mod p).  The constants are collected in k0.
__device__ __forceinline__ u64 fft_sum(u64 low, u64 hi, u32 e0, const FftSplit& sp, const LimbTab& lt) {
  u32 hl, hh;
  split64(hi, hl, hh);
  u64 s = madwide(hl & sp.fmask, 1u << lt.sf_shift, sp.k0 + e0);
  s = madwide(hh, lt.sf_d, s);
  return s + low;
}

// The canonical residue of s = 2^b + a value in [0, 256 p) (fft_sum and what a store adds: below 132 p): with s = (k + 1) 2^b + rem, u = rem + (k + 1) d = r + d for
// r = s - 2^b mod p below 2p, and bit b of u says whether r >= p = 2^b - d: then r - p is u without that bit, else r = u - d.
// (The subtraction by a multiple of that bit goes to the multiplier; a comparison and two selections cost two more
// instructions on the logic pipe, which this part of the kernels keeps busy: refresh shares at N = 8192 1604 -> 1568 us, shares
// at N = 16384 1710 -> 1702 us, at N = 4096 331 -> 328 us.)
__device__ __forceinline__ u64 fft_canon(u64 s, const LimbTab& lt) {
  u32 s0, s1, u0, u1;
  split64(s, s0, s1);
  const u32 mask = (1u << lt.sf_shift) - 1u;
  split64(madwide(s1 >> lt.sf_shift, lt.sf_d, join64(s0, s1 & mask)), u0, u1);
  return join64(u0, u1 & mask) - madlo(u1 >> lt.sf_shift, 0u - lt.sf_d, lt.sf_d);
}

__device__ __forceinline__ u32 lo_nibbles(u64 a, u64 b, u64 c, u64 d) {  // low half of byte 6 of four rounded values
  return ((u32)(a >> 48) & 15u) | ((u32)(b >> 44) & 0xf0u) | ((u32)(c >> 40) & 0xf00u) | ((u32)(d >> 36) & 0xf000u);
}

// Noise bytes (e + 19) of a polynomial, 32 per thread in the order of fft_coef: 16-byte slots [2][T].
template <int LOGN>
struct FftNoise {
  u32 w[8];
  __device__ __forceinline__ void load(const uint4* poly, u32* chk) {
    if (!D2MHE_CHK(chk, 16 * (threadIdx.x + FftGeo<LOGN>::T) + 15, 2 * FftGeo<LOGN>::n, SITE_LOAD)) return;
    // volatile: a plain load is moved down to its first use, and its latency costs 7-12 % of the share kernel
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                 : "l"(poly + threadIdx.x));
    asm volatile("ld.global.nc.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "l"(poly + threadIdx.x + FftGeo<LOGN>::T));
  }
  template <int I>
  __device__ __forceinline__ u32 get() const {
    return __byte_perm(w[I / 4], 0, 0x4440 | (I % 4));
  }
};

struct FftNoNoise {
  template <int I>
  __device__ __forceinline__ u32 get() const {
    return D2MHE_GAUSS_B;
  }
};

__device__ __forceinline__ double small_to_double(int v) {  // exact for any 32-bit integer
  return __hiloint2double(0x43300000, v ^ (int)0x80000000u) - __hiloint2double(0x43300000, (int)0x80000000u);
}

// The transform of a sampled polynomial, from its bytes in the order of the double-precision kernels.
template <int LOGN, int STASH>
__device__ __forceinline__ void fft_samples_forward(const FftSmem<LOGN, STASH>& sm, const FftTab& ft, const uint4* poly,
                                                    double* xr, double* xi) {
  using G = FftGeo<LOGN>;
  // number i of thread t is coefficient fft_coef(i): a column's coefficients are this thread's, or (two groups) this
  // thread's and the one's at the same place of the other group
  u32 w[G::GR * 8];
#pragma unroll
  for (int g = 0; g < G::GR; ++g)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const uint4 a = __ldg(poly + sm.tg + g * G::TG + h * G::T);
      w[8 * g + 4 * h] = a.x, w[8 * g + 4 * h + 1] = a.y, w[8 * g + 4 * h + 2] = a.z, w[8 * g + 4 * h + 3] = a.w;
    }
  auto value = [&](int word, int byte) {
    return small_to_double((int)__byte_perm(w[word], 0, 0x4440 | byte) - D2MHE_GAUSS_B);
  };
  fft_forward_at<LOGN>(sm, ft, xr, xi, [&](auto c_, auto j_, auto h_) {
    // digit j of column c; h: the upper half of the coefficients below n (two groups)
    constexpr int j = decltype(j_)::value;
    if constexpr (G::GR == 2) {  // i = (j & 7) + 8 (h + 2 imaginary) of group j / 8
      constexpr int base = 8 * (j / 8) + 2 * decltype(h_)::value + (j & 7) / 4;
      return cpx{value(base, j & 3), value(base + 4, j & 3)};
    } else {  // i = 2R c + j + R imaginary
      constexpr int i = 2 * G::R * decltype(c_)::value + j;
      return cpx{value(i / 4, i & 3), value((i + G::R) / 4, i & 3)};
    }
  });
}

// How many thread blocks share the two components of a ciphertext: two when that is no more work for the slowest SM.
inline u32 fft_component_split(const DevView& v, u32 base, u32 ctas) {
  const u32 resident = v.sms * ctas;
  return (2 * base + resident - 1) / resident < 2 * ((base + resident - 1) / resident) ? 2 : 1;
}

// Nothing computed from the columns' twist before this point is kept for after it (and the other way round).
template <int COLS>
__device__ __forceinline__ void fft_fence(const cpx (&tw)[COLS], cpx (&out)[COLS]) {
#pragma unroll
  for (int c = 0; c < COLS; ++c) {
    out[c] = tw[c];
    asm volatile("" : "+d"(out[c].r), "+d"(out[c].i));
  }
}

// The end of a part's inverse transform.  Low part (high = false): the rounded results are kept in shared memory.
// High part: store(coefficient, sum) gets fft_sum's 2^b + 64 p + product + noise for every coefficient of the thread, and
// may add a few p more before fft_canon.  Each part has a
// copy of the code of its own, so that the loads and the arithmetic of several portions overlap (with one copy and a
// branch in every portion the end of a high part took 5.3 k clocks of a transform's 10.2 k at N = 8192; refresh shares there
// 1789 -> 1630 us, encryption at N = 16384 459 -> 353 us); the fences keep the copies from sharing subexpressions, 300 bytes
// of which were spilled.
template <int LOGN, int STASH, class Noise, class Store>
__device__ __forceinline__ void fft_finish(const FftSmem<LOGN, STASH>& sm, const LimbTab& lt, const FftSplit& sp,
                                           const cpx (&tw)[FftGeo<LOGN>::COLS], double* xr, double* xi, bool high,
                                           const Noise& nz, Store store) {
  using G = FftGeo<LOGN>;
  cpx t[G::COLS];
  if (high) {
    fft_fence(tw, t);
    fft_results<LOGN>(sm, t, xr, xi, sp.magic, [&](auto m_, auto i_, auto rr_, const u64(&v)[4]) {
      constexpr int m = decltype(m_)::value;
      const u32* w = sm.words + threadIdx.x + 4 * m * G::T;
      if (!D2MHE_CHK(sm.chk, threadIdx.x + (4 * m + 3) * G::T, 2 * G::n, SITE_STAGED)) return;
      const u32 bytes = sm.bytes[threadIdx.x + m * G::T], nibbles = STASH == 2 ? sm.nibbles[threadIdx.x + m * G::T] : 0u;
      static_for<4>([&](auto q_) {
        constexpr int q = decltype(q_)::value, i = fft_result_number<decltype(i_)::value, decltype(rr_)::value, q>();
        u32 top = __byte_perm(bytes, 0, 0x4440 | q);
        if (STASH == 2) top |= (q < 3 ? nibbles << (8 - 4 * (q < 3 ? q : 0)) : nibbles >> 4) & 0xf00u;
        store(fft_coef<LOGN>(sm, i), fft_sum(join64(w[q * G::T], top), v[q], nz.template get<i>(), sp, lt));
      });
    });
  } else {
    fft_fence(tw, t);
    fft_results<LOGN>(sm, t, xr, xi, STASH == 2 ? D2MHE_FFT_MAGIC_LO44 : D2MHE_FFT_MAGIC_LO,
                      [&](auto m_, auto, auto, const u64(&v)[4]) {
      constexpr int m = decltype(m_)::value;
      u32* w = sm.words + threadIdx.x + 4 * m * G::T;
      if (!D2MHE_CHK(sm.chk, threadIdx.x + (4 * m + 3) * G::T, 2 * G::n, SITE_STAGED)) return;
#pragma unroll
      for (int i = 0; i < 4; ++i) w[i * G::T] = lo_word(v[i]);
      sm.bytes[threadIdx.x + m * G::T] = lo_bytes(v[0], v[1], v[2], v[3]);
      if (STASH == 2) sm.nibbles[threadIdx.x + m * G::T] = (unsigned short)lo_nibbles(v[0], v[1], v[2], v[3]);
    });
  }
}

// part `half` of coefficients j and j + n of a residue row mod p, split at 2^h
__device__ __forceinline__ cpx fft_split_pair(const u64* row, u32 j, u32 n, u32 half, u64 p, u32 h) {
  int a0, a1, b0, b1;
  fft_split(__ldg(row + j), p, h, a0, a1);
  fft_split(__ldg(row + j + n), p, h, b0, b1);
  return cpx{small_to_double(half ? a1 : a0), small_to_double(half ? b1 : b0)};
}

}  // namespace
