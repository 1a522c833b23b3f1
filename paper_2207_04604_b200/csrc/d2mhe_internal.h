// Host-side view of the context and the kernel launch entry points.
#pragma once
#include <cstddef>
#include <cstdint>
#include <cuda_runtime.h>

#include "d2mhe_device.cuh"
#include "d2mhe_fft.cuh"

#define D2MHE_MAX_LIMBS 24
#define D2MHE_MAX_SMEM_LOGN 14  // largest polynomial that fits one CTA's shared memory

// Constants for the plaintext-modulus transforms (32-bit arithmetic).
struct PlainTab {
  u32 t, twot;
  u32 ninv, ninv_sh;   // N^-1 mod t with 32-bit Shoup companion
  u32 half;            // (t-1)/2
  const uint2* W;      // [N] psi_t^brv(i) as {w, floor(w 2^32 / t)}
  const uint2* IW;     // [N] inverses
  const uint2* enc_tw; // the same by passes (kern_pack.cu), N = 4096 .. 16384
  const uint2* dec_tw;
};

// Constants of the exact scale-and-round (mixed-radix conversion).
struct RoundTab {
  const ulonglong2* ginv;  // [L*L]: entry i*L+j (j < i) = q_j^-1 mod q_i with Shoup companion
  const u64* prefix_mod_t; // [L]: prod_{j<i} q_j mod t
  u64 t, t_sh;             // t and floor(2^64 / t)
  u64 half_mod_t;          // (q-1)/2 mod t
  u64 qinv_mod_t;          // q^-1 mod t
  u32 frac_bits;           // fraction bits F of the fixed-point sum of t y_l / q_l
};

// Twiddle factors of the double-precision ring products: groups of m = 256 R points (w_k = e^(2 pi i / k)).
struct FftTab {
  const double2* twist;  // [groups][256]  psi_g^-r: psi = e^(i pi / 2m), or psi_0 = e^(i pi / 4m) and psi_1 = e^(-3 i pi / 4m)
  const double2* fwd2;   // [2][R]         w_(16R)^(4^i k)
  const double2* fwd3;   // [2][m/16]      w_m^(4^i k)
  const double2* inv2;   // [2][16]        w_256^(-4^i k)
  const double2* inv3;   // [2][256]       w_m^(-4^i r)
  const ddc* roots;      // roots of unity of order 8m: every 256th, then the first 256 (dd_root)
};

// The per-limb constants travel as a kernel parameter (constant bank): indexed by the
// CTA-uniform limb number they are read through the uniform datapath instead of occupying
// vector registers in every thread.
struct LimbParams {
  LimbTab limbs[D2MHE_MAX_LIMBS];
};

enum : u32 { RANGE_FLAG_VALUE = 1 /* a value out of range */, RANGE_FLAG_WAIT = 2 /* a wait inside a kernel ran out */ };

// Everything a kernel needs, passed by value.
struct DevView {
  const LimbTab* limbs;
  const GaussTab* gauss;
  const GaussFast* gauss_fast;
  PlainTab plain;
  RoundTab round;
  u64 seed;
  u32 logn, n, L, K;
  u32 sms;       // multiprocessors of the device (launch shaping only)
  u32 wide;      // 1 if every q_l < 2^56: lazy-reduction policy with no conditional subtractions
  u32 below60;   // 1 if every q_l < 2^60
  u64* s_mont;   // [K][L][N]  NTT(s_k) * N^-1 in Montgomery form
  u64* pk_mont;  // [2][L][N]  NTT(p_0), NTT(p_1) * N^-1 in Montgomery form
  u64* pk_coef;  // [2][L][N]  (p_0, p_1), coefficient domain
  u64* usk_mont;  // [K][L][N]     NTT(sk_i) * N^-1 (Montgomery form) of the users' own keys
  u64* upk_mont;  // [K][2][L][N]  NTT(p_{0,i}), NTT(p_{1,i}) * N^-1 (Montgomery form)
  u64* upk_coef;  // [K][2][L][N]  pk_i, coefficient domain
  // only when every prime is below 2^30 (the 32-bit-word protocol calls): the same keys as words
  // {residue out of Montgomery form, its 32-bit Shoup companion}
  u64* s32;       // [K][L][N]
  u64* pk32;      // [2][L][N]
  // ring products in double precision (set when the sizes are inside the bounds of d2mhe_fft.cuh and the device has room
  // for the keys; usk_fft and upk_fft, null without room, serve BFV.Decrypt and Conversion)
  u32 fft_on;    // the 64-bit calls
  u32 fft32_on;  // the 32-bit-word calls
  FftTab fft;
  double2* s_fft;   // [K][n]        transforms of s_k, times 1/n
  double2* pk_fft;  // [2][L][2][n]  both parts of p_0, p_1, times 1/n (fft32_on: [2][L][n], whole)
  double2* usk_fft;  // [K][n]            the same of the users' own keys
  double2* upk_fft;  // [K][2][L][2][n]
  u32* range_flag;  // bits RANGE_FLAG_*, read and cleared by d2mhe_sync
  u32* chk;       // four check words {site, index, limit, block} of the checked build
};

// What is sampled for a share or ciphertext, in order: stream tags (TAG_ENC_U is ternary, the others Gaussian).
struct SampleKinds {
  u32 n, tag0, tag1, tag2;
};
static const SampleKinds kSampleShare = {1, TAG_DEC_ERR, 0, 0};
static const SampleKinds kSampleEncrypt = {3, TAG_ENC_U, TAG_ENC_E0, TAG_ENC_E1};
static const SampleKinds kSampleBoot = {2, TAG_BOOT_E0, TAG_BOOT_E1, 0};
static const SampleKinds kSampleConvert = {3, TAG_CONV_MU, TAG_CONV_E0, TAG_CONV_E1};

// ---- host-side context (shared by the translation units that implement the C ABI) ----
#include <vector>

#include "../../include/d2mhe.h"

static const size_t kIdxSlotWords = (size_t)1 << 21;  // u32 words per staging slot (8 MiB)
static const int kIdxSlots = 4;
// Sample scratch of a context (for the single calls): 64 MiB, or what two waves of thread blocks of the share kernel with
// the largest samples need (build_tables), up to 512 MiB.
static const size_t kNoiseScratchBytes = (size_t)64 << 20;
static const size_t kNoiseScratchMaxBytes = (size_t)512 << 20;
#ifndef D2MHE_ROUND_LANES
#define D2MHE_ROUND_LANES 2
#endif
#ifndef D2MHE_ROUND_LANES_HOST
#define D2MHE_ROUND_LANES_HOST 3
#endif
// Internal streams of the whole-round entry points: two for device buffers (ten users, N = 8192, L = 4, 13 indices 499 us,
// with three and one 558 and 549), three when the call also copies from and to host buffers (the same round 748 us, 755 with
// two; 40 indices 1678 and 1763; twenty users, 40 indices 4995 and 5056; six users, L = 5, 30 indices 984 and 1069; thirty
// users, N = 4096, 12 indices 1328 and 1267: one more stream hides the copies of longer rounds better).
static const int kRoundLanesDevice = D2MHE_ROUND_LANES;
static const int kRoundLanesHost = D2MHE_ROUND_LANES_HOST;
static const int kRoundLanes = kRoundLanesDevice > kRoundLanesHost ? kRoundLanesDevice : kRoundLanesHost;

struct d2mhe_ctx {
  d2mhe_params params;
  std::vector<u64> moduli;
  std::vector<u64> roots;
  u64 psi_t = 0;
  bool can_pack = false;
  bool narrow = false;  // every prime below 2^30: the 32-bit-word calls are available
  int device = 0;
  cudaStream_t stream = nullptr;
  DevView view;
  LimbParams limb_params;
  std::vector<void*> allocs;        // device allocations to free
  unsigned char* arena = nullptr;   // rest of the last allocation that small blocks share
  size_t arena_left = 0;
  std::vector<bool> has_share;
  std::vector<bool> has_user_key;
  std::vector<u32> pk_parties;      // party set of the last collective_pk
  std::vector<u32> all_parties;     // 0 .. K-1 (the users of a whole-round call)
  bool has_pk = false;
  u64 launches = 0;
  // index staging: pinned host ring + device ring, one event per slot
  u32* idx_host = nullptr;
  u32* idx_dev = nullptr;
  cudaEvent_t idx_event[kIdxSlots] = {};
  bool idx_event_valid[kIdxSlots] = {};
  int idx_next = 0;
  // the four index lists of the whole-round calls: kept on the device from one call to the next and
  // uploaded again only when they change
  u32* round_lists_host = nullptr;        // pinned
  u32* round_lists_dev = nullptr;
  std::vector<u32> round_lists_cache;     // what round_lists_dev holds
  cudaEvent_t round_lists_event = nullptr;  // after the last upload
  bool round_lists_valid = false;
  cudaStream_t lane_stream[kRoundLanes] = {};
  cudaEvent_t lane_event[kRoundLanes] = {};
  cudaEvent_t fork_event = nullptr;
  unsigned char* noise_scratch = nullptr;  // device: noise bytes of the shares of one d2mhe_partial_decrypt batch
  size_t noise_scratch_bytes = 0;
  cudaError_t last_cuda = cudaSuccess;
  bool checked = false;             // launches the checked kernel build
  u32 last_check[4] = {};           // the last violation that d2mhe_sync reported
};

// The kernel translation units are compiled twice: as they are into namespace d2mhe_launch, and
// with D2MHE_CHECKED (index checks in every kernel, see d2mhe_device.cuh) into d2mhe_launch_chk.
// A context created with D2MHE_FLAG_DEVICE_CHECKS launches the second set.
#ifdef D2MHE_CHECKED
#define D2MHE_LAUNCH_NS d2mhe_launch_chk
#else
#define D2MHE_LAUNCH_NS d2mhe_launch
#endif

// Launchers (one per kernel or kernel sequence).  Notes: encrypt and partial_decrypt_scratch sample
// u, e_0, e_1 / the shares' noise ahead into caller-lent scratch (at least 3 N / n_parties N bytes; with
// 11 N bytes encrypt takes the double-precision products, which keep the transform of u there too)
// and report their number of launches, and so do convert_share (n_parties 3 N bytes, double precision from
// n_parties 11 N) and boot_share (n_parties 6 N bytes, double precision from
// n_parties 6 N + 8 N L); combine sums the first of share_comps polynomials per
// (recipient, party, ciphertext); int_probe synchronises the stream; export_secret turns key rows
// [L][N] (transform domain, Montgomery form) into int8 coefficients [L][N] (127 = not ternary);
// check_selftest makes one thread of the checked build raise SITE_SELFTEST (no memory access);
// wait_selftest runs one block whose waits for its exchange area run into the limit.
#define D2MHE_LAUNCHER_DECLS \
cudaError_t keygen(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* parties_dev, u32 n_parties); \
cudaError_t collective_pk(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* parties_dev, u32 n_parties, \
                          u64* shares_out); \
cudaError_t int_probe(const DevView& v, const LimbParams& lp, cudaStream_t s, u32 kind, u32 iters, u32* sink, \
                      float* ms, double* lane_ops); \
cudaError_t export_secret(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* key, signed char* out); \
cudaError_t encode(const DevView& v, cudaStream_t s, const int32_t* values, u32 n_cts, u32* plain); \
cudaError_t decode(const DevView& v, cudaStream_t s, const u32* plain, u32 n_cts, int32_t* values); \
cudaError_t encode16(const DevView& v, cudaStream_t s, const int32_t* values, u32 n_groups, u32 group, \
                     size_t group_stride, u32* plain); \
cudaError_t decode16(const DevView& v, cudaStream_t s, const u32* plain, u32 n_groups, u32 group, size_t group_stride, \
                     int32_t* values); \
cudaError_t encode_strided(const DevView& v, cudaStream_t s, const int32_t* values, u32 n_groups, u32 group, \
                           size_t group_stride, u32* plain); \
cudaError_t decode_strided(const DevView& v, cudaStream_t s, const u32* plain, u32 n_groups, u32 group, \
                           size_t group_stride, int32_t* values); \
cudaError_t encrypt(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* parties_dev, u32 n_parties, \
                    u32 ct_first, u32 n_cts, const u32* plain, u64* ct, void* scratch, size_t scratch_bytes, \
                    u32* launches); \
cudaError_t aggregate(const DevView& v, cudaStream_t s, const u64* ct, u32 n_rows, u32 n_cts, \
                      const u32* offsets_dev, const u32* rows_dev, u32 n_out, u32 nnz, u64* agg); \
cudaError_t aggregate_columns32(const DevView& v, cudaStream_t s, const u32* ct, u32 n_rows, u32 n_cts, \
                                const u32* offsets_dev, const u32* rows_dev, u32 n_out, u32 nnz, u32* agg, bool* done); \
cudaError_t partial_decrypt_scratch(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, \
                                    const u32* recipients_dev, u32 n_rec, const u32* parties_dev, \
                                    u32 n_parties, u32 ct_first, u32 n_cts, u64* shares, void* scratch, \
                                    size_t scratch_bytes, u32* launches); \
cudaError_t combine(const DevView& v, cudaStream_t s, const u64* agg, const u64* shares, u32 n_rec, \
                    u32 n_shares, u32 share_comps, u32 n_cts, u32* plain); \
cudaError_t boot_share(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, \
                       const u32* recipients_dev, u32 n_rec, const u32* parties_dev, u32 n_parties, \
                       u32 ct_first, u32 n_cts, u64* shares, void* scratch, size_t scratch_bytes, u32* launches); \
cudaError_t boot_finish(const DevView& v, cudaStream_t s, const u32* x, const u64* shares, \
                        const u32* recipients_dev, u32 n_rec, u32 n_shares, u32 ct_first, u32 n_cts, u64* out); \
cudaError_t ntt(const DevView& v, const LimbParams& lp, cudaStream_t s, u64* polys, u32 batch, bool inverse); \
cudaError_t ntt32(const DevView& v, const LimbParams& lp, cudaStream_t s, u32* polys, u32 batch, bool inverse); \
cudaError_t muladd32(const DevView& v, cudaStream_t s, const u32* a, const u32* b, const u32* c, u32* d, \
                     u32 batch); \
cudaError_t user_keygen(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* users_dev, \
                        u32 n_users); \
cudaError_t convert_share(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, \
                          const u32* recipients_dev, u32 n_rec, const u32* parties_dev, u32 n_parties, \
                          u32 ct_first, u32 n_cts, u64* shares, void* scratch, size_t scratch_bytes, u32* launches); \
cudaError_t convert_combine(const DevView& v, cudaStream_t s, const u64* agg, const u64* shares, u32 n_rec, \
                            u32 n_shares, u32 n_cts, u64* out); \
cudaError_t secret_product(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* ct, \
                           const u32* users_dev, u32 n_users, u32 n_cts, u64* prod); \
cudaError_t muladd(const DevView& v, cudaStream_t s, const u64* a, const u64* b, const u64* c, \
                   u64* d, u32 batch); \
cudaError_t check_selftest(const DevView& v, cudaStream_t s); \
cudaError_t wait_selftest(const DevView& v, cudaStream_t s, u32 tries); \
cudaError_t sample_streams(const DevView& v, cudaStream_t s, const u32* recipients_dev, const u32* parties_dev, \
                           u32 n_parties, u32 ct_first, u32 n_cts, u32 unit_first, u32 n_units, SampleKinds kinds, \
                           bool fft_order, void* out); \
cudaError_t share_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, const u32* parties_dev, \
                      u32 n_parties, u32 n_cts, u32 unit_first, u32 n_units, const void* noise, u64* shares); \
cudaError_t encrypt_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* parties_dev, u32 ct_first, \
                        u32 n_cts, u32 n_units, const u32* plain, u64* ct, void* scratch, size_t scratch_bytes, \
                        u32* launches); \
cudaError_t fft_samples(const DevView& v, cudaStream_t s, const void* src, u32 stride, u32 polys, double2* dst); \
cudaError_t fft_rows(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* src, const u32* users_dev, \
                     u32 rows, bool whole, double2* dst); \
cudaError_t share32_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* agg, const u32* parties_dev, \
                        u32 n_parties, u32 n_cts, u32 unit_first, u32 n_units, const void* noise, u32* shares); \
cudaError_t encrypt32_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, u32 unit_first, u32 n_units, \
                          const double2* u_fft, const void* noise, const u32* plain, u32* ct); \
cudaError_t convert_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, \
                        const u32* recipients_dev, u32 n_rec, const u32* parties_dev, u32 n_parties, u32 ct_first, \
                        u32 n_cts, u64* shares, void* scratch, size_t scratch_bytes, u32* launches); \
cudaError_t boot_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* agg, const u32* recipients_dev, \
                     u32 n_rec, const u32* parties_dev, u32 n_parties, u32 ct_first, u32 n_cts, u64* shares, \
                     void* scratch, size_t scratch_bytes, u32* launches); \
cudaError_t sample_boot(const DevView& v, cudaStream_t s, const u32* recipients_dev, const u32* parties_dev, \
                        u32 n_parties, u32 ct_first, u32 n_cts, u32 unit_first, u32 n_units, bool fft_order, void* noise, \
                        u32* masks, u32* launches); \
cudaError_t sample_alpha(const DevView& v, cudaStream_t s, const u32* recipients_dev, u32 ct_first, u32 n_cts, \
                         u32 unit_first, u32 n_units, u64* out); \
cudaError_t secret_product_fft(const DevView& v, const LimbParams& lp, cudaStream_t s, const u64* ct, \
                               const u32* users_dev, u32 n_users, u32 n_cts, u64* prod); \
cudaError_t fft_secret(const DevView& v, cudaStream_t s, const u32* parties_dev, u32 n_parties, u32 tag, double2* dst); \
cudaError_t make_tab32(const DevView& v, cudaStream_t s, const u64* src, u64* dst, size_t rows); \
cudaError_t encrypt32(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* parties_dev, u32 n_parties, \
                      u32 ct_first, u32 n_cts, const u32* plain, u32* ct, void* scratch, size_t scratch_bytes, \
                      u32* launches); \
cudaError_t aggregate32(const DevView& v, cudaStream_t s, const u32* ct, u32 n_rows, u32 n_cts, const u32* offsets_dev, \
                        const u32* rows_dev, u32 n_out, u32 nnz, u32* agg); \
cudaError_t partial_decrypt32(const DevView& v, const LimbParams& lp, cudaStream_t s, const u32* agg, \
                              const u32* recipients_dev, u32 n_rec, const u32* parties_dev, u32 n_parties, \
                              u32 ct_first, u32 n_cts, u32* shares, void* scratch, size_t scratch_bytes, \
                              u32* launches); \
cudaError_t combine32(const DevView& v, cudaStream_t s, const u32* agg, const u32* shares, u32 n_rec, u32 n_shares, \
                      u32 n_cts, u32* plain);

namespace d2mhe_launch {
D2MHE_LAUNCHER_DECLS
}
namespace d2mhe_launch_chk {
D2MHE_LAUNCHER_DECLS
}

