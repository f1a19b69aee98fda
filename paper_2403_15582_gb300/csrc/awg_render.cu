// Render kernels for multi-tone additive synthesis on sm_103a.
//
//   x[n] = sum_k A_k sin(2 pi Phi_k(n) / 2^64)       (Eq. main / Eq. dynamicandstatic)
//
// Phase words.  Static tones: Phi(n) = phi_ref + n F.  Chirps (Eq. freqchirp, linear or
// minimum-jerk): Phi(n_s + m) = Phi(n_s) + top64(sum_k d_k C(m,k)) with the 192-bit forward
// differences d_k set up on the host; evaluated here exactly by the closed form
// (exact_chirp_word), which is what a sequential 192-bit cascade would produce.  Exponential
// chirps: Phi(n_s) + C (e^(alpha m) - 1) in FP64.
//
// Work decomposition (see awg_internal.h): a CTA renders one tile of TILE = 4096 absolute-aligned
// samples (or a half or a quarter of it, see Geo); thread j owns the run of RUN = 32 samples starting
// at T0 + 32 j (or a half or a quarter of a run) and keeps its partial sums in registers; the tones are
// split over `split` CTAs, whose partial tiles are added in rank order (through L2 scratch by the last
// CTA of the tile to finish, or through distributed shared memory in a thread-block cluster), then
// scaled, rounded and stored by the same kernel.
//
// Per (tone, run) the phase is set up once and then stepped per sample in 32-bit fixed point
// (units of 2^-32 turn):
//   static runs   p_r = p_0 + r f                                  (p_0 from the exact word)
//   chirp runs    p_r = p_0 + r f + C(r,2) g + C(r,3) h            (32-bit difference cascade)
// where (p_0, f, g, h) come from a per-(chirp, tile) record of stride-32 forward differences
// (prep_kernel) evaluated at the run index j.  The sine takes the top 23 bits of p_r as a
// signed fraction of a turn (round to nearest) and runs on the SFU (__sinf in [-pi, pi)).
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <algorithm>
#include <atomic>
#include <cstdint>

#include "awg_internal.h"

namespace cg = cooperative_groups;

namespace awgk {

namespace {

constexpr int STATUS_TIMEOUT = -4;   // AWG_ETIMEOUT

// ------------------------------------------------------------------------------------------
// 192-bit integers, arithmetic mod 2^192 (two's complement for signed values)
// ------------------------------------------------------------------------------------------
struct U192 {
  uint64_t w0, w1, w2;
};

__device__ __forceinline__ U192 from_s64(int64_t a) {
  uint64_t s = (uint64_t)(a >> 63);
  return {(uint64_t)a, s, s};
}

__device__ __forceinline__ U192 add192(U192 a, U192 b) {
  U192 r;
  unsigned __int128 t = (unsigned __int128)a.w0 + b.w0;
  r.w0 = (uint64_t)t;
  t = (unsigned __int128)a.w1 + b.w1 + (uint64_t)(t >> 64);
  r.w1 = (uint64_t)t;
  r.w2 = a.w2 + b.w2 + (uint64_t)(t >> 64);
  return r;
}

__device__ __forceinline__ U192 mul192(U192 a, U192 b) {
  unsigned __int128 p00 = (unsigned __int128)a.w0 * b.w0;
  unsigned __int128 p01 = (unsigned __int128)a.w0 * b.w1;
  unsigned __int128 p10 = (unsigned __int128)a.w1 * b.w0;
  unsigned __int128 mid = (p00 >> 64) + (uint64_t)p01 + (uint64_t)p10;
  U192 r;
  r.w0 = (uint64_t)p00;
  r.w1 = (uint64_t)mid;
  r.w2 = (uint64_t)(mid >> 64) + (uint64_t)(p01 >> 64) + (uint64_t)(p10 >> 64) + a.w0 * b.w2 +
         a.w1 * b.w1 + a.w2 * b.w0;
  return r;
}

__device__ __forceinline__ U192 sar192(U192 a, int v) {
  if (v == 0) return a;
  U192 r;
  r.w0 = (a.w0 >> v) | (a.w1 << (64 - v));
  r.w1 = (a.w1 >> v) | (a.w2 << (64 - v));
  r.w2 = (uint64_t)((int64_t)a.w2 >> v);
  return r;
}


// C(m, j) for j = 0..6 and signed m (|m| < 2^30): the product of j consecutive integers is
// below 2^180 in magnitude, so it is exact mod 2^192; dividing by j! = 2^v * odd is a
// multiplication by the inverse of the odd part mod 2^192 and an arithmetic shift.
__device__ __forceinline__ void binomials(int64_t m, const uint64_t (*inv)[3], U192 c[7]) {
  U192 p = {1, 0, 0};
  c[0] = p;
#pragma unroll
  for (int j = 1; j <= 6; ++j) {
    p = mul192(p, from_s64(m - (j - 1)));
    U192 q = p;
    if (j == 3 || j == 4) q = mul192(q, U192{inv[0][0], inv[0][1], inv[0][2]});   // 1/3
    if (j == 5) q = mul192(q, U192{inv[1][0], inv[1][1], inv[1][2]});              // 1/15
    if (j == 6) q = mul192(q, U192{inv[2][0], inv[2][1], inv[2][2]});              // 1/45
    const int v = (j == 2 || j == 3) ? 1 : (j == 4 || j == 5) ? 3 : (j == 6) ? 4 : 0;
    c[j] = sar192(q, v);
  }
}

__device__ __forceinline__ U192 dword(const ChirpRec& c, int i) {
  return U192{c.d[3 * i], c.d[3 * i + 1], c.d[3 * i + 2]};
}

// x 2^64 rounded to an integer, mod 2^128 (two's complement): the double's exact value M 2^e
// (M its 53-bit integer mantissa) shifted into Q64.64.  Zero for |x| < 2^-65.
__device__ __forceinline__ unsigned __int128 q64_of(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0) return 0;
  const uint64_t M = (b & 0xFFFFFFFFFFFFFull) | (1ull << 52);
  const int sh = ex - 1075 + 64;
  unsigned __int128 v;
  if (sh >= 128) v = 0;
  else if (sh >= 0) v = (unsigned __int128)M << sh;
  else if (sh > -54) v = ((unsigned __int128)M + ((unsigned __int128)1 << (-sh - 1))) >> (-sh);
  else v = 0;
  return (b >> 63) ? (unsigned __int128)0 - v : v;
}

// Exponential chirp (TONE_EXP): the phase offset R(m) = C (e^(alpha m) - 1) words (the integral of
// the frequency F_start e^(alpha t)), FP64, rounded to the word.
__device__ __forceinline__ uint64_t exp_chirp_offset(const ChirpRec& c, int64_t m) {
  const double alpha = __longlong_as_double((long long)c.d[2]);
  const double C = __longlong_as_double((long long)c.d[3]);
  return (uint64_t)((q64_of(C * expm1(alpha * (double)m)) + ((unsigned __int128)1 << 63)) >> 64);
}

// Exact phase word of a chirp at offset m from its start: Phi(n_s) + top64(sum_i d_i C(m, i)).
// d_0 carries the 2^127 rounding offset.  (Exponential chirps: Phi(n_s) + R(m).)
__device__ uint64_t exact_chirp_word(const ChirpRec& c, int64_t m, const uint64_t (*inv)[3]) {
  if (c.flags & TONE_EXP) return c.phi_start + exp_chirp_offset(c, m);
  U192 b[7];
  binomials(m, inv, b);
  U192 s = {0, 0, 0};
#pragma unroll
  for (int i = 0; i < 7; ++i) s = add192(s, mul192(dword(c, i), b[i]));
  return c.phi_start + s.w2;
}

__device__ __forceinline__ uint64_t exact_word(const ToneRec& t, const ChirpRec* chirps, int64_t n,
                                               const uint64_t (*inv)[3]) {
  if (t.slot < 0 || n < t.n_s) return t.phi_ref + (uint64_t)n * t.F;
  if (n > t.n_e) return t.phi_post_ref + (uint64_t)n * t.F_end;
  return exact_chirp_word(chirps[t.slot], n - t.n_s, inv);
}

// ------------------------------------------------------------------------------------------
// 32-bit run phases
// ------------------------------------------------------------------------------------------
constexpr uint64_t P_OFFSET = 1ull << 40;   // makes the 23-bit truncation of p round to nearest
constexpr uint64_t HALF32 = 1ull << 31;
// P_OFFSET plus half a turn: folded into the records' B_0 (stride_records)
constexpr uint64_t B0_OFFSET = P_OFFSET + (1ull << 63);

// A run's 32-bit cascade state: p is the run-start phase plus half a turn (the centred form that
// sin_pair takes), f, g, h its first three differences.
struct RunPoly {
  uint32_t p, f, g, h;
};

// C(j, q) for the run index j (0 <= j < RUNS = 128): q <= 5 fit in 32 bits, C(j, 6) needs 33.
struct RunBin {
  uint32_t c1, c2, c3, c4, c5;
  uint64_t c6;
};

__device__ __forceinline__ RunBin run_binomials(int j) {
  RunBin b;
  const uint64_t u = (uint64_t)j;
  const uint64_t c2 = u * (u - 1) / 2, c3 = c2 * (u - 2) / 3, c4 = c3 * (u - 3) / 4, c5 = c4 * (u - 4) / 5;
  b.c1 = (uint32_t)j;
  b.c2 = (uint32_t)c2;
  b.c3 = (uint32_t)c3;
  b.c4 = (uint32_t)c4;
  b.c5 = (uint32_t)c5;
  b.c6 = c5 * (u - 5) / 6;
  // a factor (u - i) is zero for j = i, so every product with q > j vanishes; j < q wraps (u - i)
  // but the zero factor comes first, so the products above are already 0 for those j.
  return b;
}

// acc + x * c (mod 2^64) for a 32-bit c: one wide and one narrow integer multiply-add
__device__ __forceinline__ uint64_t mac_u32(uint64_t acc, uint64_t x, uint32_t c) {
  const uint64_t lo = (uint64_t)(uint32_t)x * c;
  const uint32_t hi = (uint32_t)(x >> 32) * c;
  return acc + lo + ((uint64_t)hi << 32);
}

// The top 32 bits of a sum of 64-bit words times small integers, (sum_q x_q c_q mod 2^64) >> 32,
// accumulated as a 64-bit sum of the low halves' products plus a 32-bit sum of the high halves'
// products: S = 2^32 sum hi32(x_q) c_q + sum lo32(x_q) c_q, so bits 32..63 of S are the high sum
// plus bits 32..63 of the low sum, whatever wraps above bit 63.  Two integer multiply-adds per
// term; the same integers as the full 64-bit sum.
struct Top32 {
  uint64_t lo;
  uint32_t hi;
};
// start from word x (the records carry the rounding offsets in their order-0 words)
__device__ __forceinline__ Top32 top_init(uint64_t x) {
  return Top32{(uint64_t)(uint32_t)x, (uint32_t)(x >> 32)};
}
__device__ __forceinline__ void top_mac(Top32& t, uint64_t x, uint32_t c) {
  t.lo += (uint64_t)(uint32_t)x * c;
  t.hi += (uint32_t)(x >> 32) * c;
}
// x c mod 2^64 for a 64-bit c: lo32(x) lo32(c) + 2^32 (hi32(x) lo32(c) + lo32(x) hi32(c))
__device__ __forceinline__ void top_mac64(Top32& t, uint64_t x, uint64_t c) {
  t.lo += (uint64_t)(uint32_t)x * (uint32_t)c;
  t.hi += (uint32_t)(x >> 32) * (uint32_t)c + (uint32_t)x * (uint32_t)(c >> 32);
}
__device__ __forceinline__ uint32_t top_get(const Top32& t) { return t.hi + (uint32_t)(t.lo >> 32); }

constexpr uint64_t HALF32_OFF = 1ull << 31;

// (p, f, g, h) at run j from the stride-RUN records: p = sum_q B_q C(j,q), f = sum_q E_q C(j,q),
// g = sum_q G_q C(j,q), h = sum_q H_q C(j,q), all mod 2^64, then the top 32 bits.  The records'
// order-0 words carry the offsets (stride_records): B_0 the 2^8 offset of the sine argument and
// half a turn, so p is floor((phase + 2^40) / 2^32) + 2^31; E_0, G_0, H_0 half a unit, so f, g, h
// round to nearest.
__device__ __forceinline__ RunPoly poly_state(const TileRec& rc, const RunBin& b, bool linear) {
  RunPoly r;
  if (linear) {   // B_q (q >= 3), E_q (q >= 2), G_q (q >= 1) and H are exactly zero
    Top32 p = top_init(rc.w[rec_b(0)]);
    top_mac(p, rc.w[rec_b(1)], b.c1);
    top_mac(p, rc.w[rec_b(2)], b.c2);
    Top32 f = top_init(rc.w[rec_e(0)]);
    top_mac(f, rc.w[rec_e(1)], b.c1);
    r.p = top_get(p);
    r.f = top_get(f);
    r.g = (uint32_t)(rc.w[rec_g(0)] >> 32);
    r.h = 0;
    return r;
  }
  Top32 p = top_init(rc.w[rec_b(0)]);
  top_mac(p, rc.w[rec_b(1)], b.c1);
  top_mac(p, rc.w[rec_b(2)], b.c2);
  top_mac(p, rc.w[rec_b(3)], b.c3);
  top_mac(p, rc.w[rec_b(4)], b.c4);
  top_mac(p, rc.w[rec_b(5)], b.c5);
  top_mac64(p, rc.w[rec_b(6)], b.c6);
  Top32 f = top_init(rc.w[rec_e(0)]);
  top_mac(f, rc.w[rec_e(1)], b.c1);
  top_mac(f, rc.w[rec_e(2)], b.c2);
  top_mac(f, rc.w[rec_e(3)], b.c3);
  top_mac(f, rc.w[rec_e(4)], b.c4);
  top_mac(f, rc.w[rec_e(5)], b.c5);
  Top32 g = top_init(rc.w[rec_g(0)]);
  top_mac(g, rc.w[rec_g(1)], b.c1);
  top_mac(g, rc.w[rec_g(2)], b.c2);
  top_mac(g, rc.w[rec_g(3)], b.c3);
  top_mac(g, rc.w[rec_g(4)], b.c4);
  Top32 h = top_init(rc.w[rec_h(0)]);
  top_mac(h, rc.w[rec_h(1)], b.c1);
  top_mac(h, rc.w[rec_h(2)], b.c2);
  top_mac(h, rc.w[rec_h(3)], b.c3);
  r.p = top_get(p);
  r.f = top_get(f);
  r.g = top_get(g);
  r.h = top_get(h);
  return r;
}

// poly_state for a degree-6 chirp whose h is known to round to 0 (TONE_FLAT3): no H polynomial.
__device__ __forceinline__ RunPoly poly_state_flat3(const TileRec& rc, const RunBin& b) {
  Top32 p = top_init(rc.w[rec_b(0)]);
  top_mac(p, rc.w[rec_b(1)], b.c1);
  top_mac(p, rc.w[rec_b(2)], b.c2);
  top_mac(p, rc.w[rec_b(3)], b.c3);
  top_mac(p, rc.w[rec_b(4)], b.c4);
  top_mac(p, rc.w[rec_b(5)], b.c5);
  top_mac64(p, rc.w[rec_b(6)], b.c6);
  Top32 f = top_init(rc.w[rec_e(0)]);
  top_mac(f, rc.w[rec_e(1)], b.c1);
  top_mac(f, rc.w[rec_e(2)], b.c2);
  top_mac(f, rc.w[rec_e(3)], b.c3);
  top_mac(f, rc.w[rec_e(4)], b.c4);
  top_mac(f, rc.w[rec_e(5)], b.c5);
  Top32 g = top_init(rc.w[rec_g(0)]);
  top_mac(g, rc.w[rec_g(1)], b.c1);
  top_mac(g, rc.w[rec_g(2)], b.c2);
  top_mac(g, rc.w[rec_g(3)], b.c3);
  top_mac(g, rc.w[rec_g(4)], b.c4);
  return RunPoly{top_get(p), top_get(f), top_get(g), 0u};
}

// poly_state for a TONE_LOW6 chirp: FLAT3, and the set-up bounds B_6, E_5 and G_2..G_4 below 64
// units of 2^-32 turn of phase over a run, so they are left out.
__device__ __forceinline__ RunPoly poly_state_low6(const TileRec& rc, const RunBin& b) {
  Top32 p = top_init(rc.w[rec_b(0)]);
  top_mac(p, rc.w[rec_b(1)], b.c1);
  top_mac(p, rc.w[rec_b(2)], b.c2);
  top_mac(p, rc.w[rec_b(3)], b.c3);
  top_mac(p, rc.w[rec_b(4)], b.c4);
  top_mac(p, rc.w[rec_b(5)], b.c5);
  Top32 f = top_init(rc.w[rec_e(0)]);
  top_mac(f, rc.w[rec_e(1)], b.c1);
  top_mac(f, rc.w[rec_e(2)], b.c2);
  top_mac(f, rc.w[rec_e(3)], b.c3);
  top_mac(f, rc.w[rec_e(4)], b.c4);
  Top32 g = top_init(rc.w[rec_g(0)]);
  top_mac(g, rc.w[rec_g(1)], b.c1);
  return RunPoly{top_get(p), top_get(f), top_get(g), 0u};
}

// poly_state for a TONE_LOW3 chirp: LOW6, and B_5, E_3, E_4 left out as well (the set-up bounds all
// left-out terms below 256 units of 2^-32 turn over a two-run cascade).
__device__ __forceinline__ RunPoly poly_state_low3(const TileRec& rc, const RunBin& b) {
  Top32 p = top_init(rc.w[rec_b(0)]);
  top_mac(p, rc.w[rec_b(1)], b.c1);
  top_mac(p, rc.w[rec_b(2)], b.c2);
  top_mac(p, rc.w[rec_b(3)], b.c3);
  top_mac(p, rc.w[rec_b(4)], b.c4);
  Top32 f = top_init(rc.w[rec_e(0)]);
  top_mac(f, rc.w[rec_e(1)], b.c1);
  top_mac(f, rc.w[rec_e(2)], b.c2);
  Top32 g = top_init(rc.w[rec_g(0)]);
  top_mac(g, rc.w[rec_g(1)], b.c1);
  return RunPoly{top_get(p), top_get(f), top_get(g), 0u};
}


__device__ __forceinline__ uint32_t static_p0(uint64_t phi_ref, uint64_t F, int64_t n0) {
  return (uint32_t)((phi_ref + (uint64_t)n0 * F + P_OFFSET) >> 32);
}
__device__ __forceinline__ uint32_t static_f(uint64_t F) { return (uint32_t)((F + HALF32) >> 32); }

// Tile classification of a tone against a tile [T0, T0 + TILE).
enum { TILE_PRE = 0, TILE_POST = 1, TILE_CHIRP = 2 };
__device__ __forceinline__ int classify_tile(const ToneRec& t, int64_t T0) {
  if (t.slot < 0 || T0 + TILE - 1 < t.n_s) return TILE_PRE;
  if (T0 > t.n_e) return TILE_POST;
  return TILE_CHIRP;
}

// The sine takes a phase already offset by half a turn (pc = p + 2^31, added once per run, not per
// sample; sin_pair): the float v = 1.m with the 23-bit fraction m = pc >> 9 (exponent field of [1, 2)).
constexpr uint32_t HALF_TURN = 1u << 31;
__device__ __forceinline__ float mantissa_float(uint32_t pc) { return __uint_as_float((pc >> 9) + 0x3F800000u); }

// ------------------------------------------------------------------------------------------
// TMA bulk copies and mbarriers (inline PTX)
// ------------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: gives up after ~2 s of wall time.
__device__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_ns() - t0 > 2000000000ull) return false;
  }
  return true;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_addr(dst)),
      "l"(src), "r"(bytes), "r"(smem_addr(bar))
      : "memory");
}

// ------------------------------------------------------------------------------------------
// prep: per (active chirp, tile) stride-RUN forward differences at the tile start
// ------------------------------------------------------------------------------------------
// a * b mod 2^192 for a signed 64-bit b: a (b mod 2^64) - [b < 0] a 2^64
__device__ __forceinline__ U192 mul192_s64(U192 a, int64_t bs) {
  const uint64_t b = (uint64_t)bs;
  unsigned __int128 p0 = (unsigned __int128)a.w0 * b;
  unsigned __int128 p1 = (unsigned __int128)a.w1 * b + (uint64_t)(p0 >> 64);
  U192 r;
  r.w0 = (uint64_t)p0;
  r.w1 = (uint64_t)p1;
  r.w2 = a.w2 * b + (uint64_t)(p1 >> 64);
  if (bs < 0) {
    unsigned __int128 t = (unsigned __int128)r.w1 - a.w0;
    r.w1 = (uint64_t)t;
    r.w2 = r.w2 - a.w1 - (uint64_t)((t >> 64) & 1);
  }
  return r;
}

// C(m, j), j = 0..DEG, signed m, exact (see binomials())
template <int DEG>
__device__ __forceinline__ void binomials_deg(int64_t m, const uint64_t (*inv)[3], U192 c[DEG + 1]) {
  U192 p = {1, 0, 0};
  c[0] = p;
#pragma unroll
  for (int j = 1; j <= DEG; ++j) {
    p = mul192_s64(p, m - (j - 1));
    U192 q = p;
    if (j == 3 || j == 4) q = mul192(q, U192{inv[0][0], inv[0][1], inv[0][2]});
    if (j == 5) q = mul192(q, U192{inv[1][0], inv[1][1], inv[1][2]});
    if (j == 6) q = mul192(q, U192{inv[2][0], inv[2][1], inv[2][2]});
    const int v = (j == 2 || j == 3) ? 1 : (j == 4 || j == 5) ? 3 : (j == 6) ? 4 : 0;
    c[j] = sar192(q, v);
  }
}

// Upper 128 bits of a 192-bit value (units of 2^64 of the Q64.128 word, i.e. Q64.64).
__device__ __forceinline__ unsigned __int128 hi128(U192 a) {
  return ((unsigned __int128)a.w2 << 64) | a.w1;
}
// Q64.64 -> word, rounded to nearest (mod 2^64)
__device__ __forceinline__ uint64_t round_q64(unsigned __int128 v) {
  return (uint64_t)((v + ((unsigned __int128)1 << 63)) >> 64);
}

// The stride-RUN records of a tile from the unit-stride forward differences h[1..DEG] of the
// chirp phase at the tile start (Q64.64 words, mod 2^128) and its phase word B0: the first WORDS
// words of the record.  The order-0 words take the run set-up's rounding offsets (poly_state):
// B_0 + 2^40 + 2^63, E_0, G_0 and H_0 + 2^31.
template <int DEG, int WORDS, class Args>
__device__ __forceinline__ void stride_records(const unsigned __int128* h, uint64_t B0, const Args& a,
                                               TileRec& out) {
  // sum over i >= q of h[i + k] W[q][i]: order q of the k-th unit difference
  auto word = [&](int q, int k) -> uint64_t {
    if (q + k > DEG) return 0;
    unsigned __int128 s = 0;
#pragma unroll
    for (int i = 0; i <= 6; ++i)
      if (i >= q && i + k <= DEG) s += h[i + k] * (unsigned __int128)a.W[q][i];
    return round_q64(s);
  };
#pragma unroll
  for (int q = 0; q < 7; ++q)
    if (rec_b(q) < WORDS) out.w[rec_b(q)] = q == 0 ? B0 + B0_OFFSET : word(q, 0);
#pragma unroll
  for (int q = 0; q < 6; ++q)
    if (rec_e(q) < WORDS) out.w[rec_e(q)] = word(q, 1) + (q == 0 ? HALF32_OFF : 0);
#pragma unroll
  for (int q = 0; q < 5; ++q)
    if (rec_g(q) < WORDS) out.w[rec_g(q)] = word(q, 2) + (q == 0 ? HALF32_OFF : 0);
#pragma unroll
  for (int q = 0; q < 4; ++q)
    if (rec_h(q) < WORDS) out.w[rec_h(q)] = word(q, 3) + (q == 0 ? HALF32_OFF : 0);
}

// d c mod 2^192 for a multiplier c whose 64-bit limbs above the first L are zero: the partial
// products of those limbs are left out (the same value as mul192).
template <int L>
__device__ __forceinline__ U192 mul192_limbs(U192 d, U192 c) {
  const unsigned __int128 p00 = (unsigned __int128)d.w0 * c.w0;
  const unsigned __int128 p10 = (unsigned __int128)d.w1 * c.w0;
  unsigned __int128 mid = (p00 >> 64) + (uint64_t)p10;
  uint64_t top = (uint64_t)(p10 >> 64) + d.w2 * c.w0;
  if (L >= 2) {
    const unsigned __int128 p01 = (unsigned __int128)d.w0 * c.w1;
    mid += (uint64_t)p01;
    top += (uint64_t)(p01 >> 64) + d.w1 * c.w1;
  }
  if (L >= 3) top += d.w0 * c.w2;
  return U192{(uint64_t)p00, (uint64_t)mid, top + (uint64_t)(mid >> 64)};
}

// Inverses of 3 and 5 modulo 2^128 / 2^192 (3 * 0xA..AB = 1 and 5 * 0xC..CD = 1 modulo the power of
// two): an exact quotient by 3 or 5 is a product with the inverse.
constexpr uint64_t INV3_W = 0xAAAAAAAAAAAAAAAAull, INV3_W0 = 0xAAAAAAAAAAAAAAABull;
constexpr uint64_t INV5_W = 0xCCCCCCCCCCCCCCCCull, INV5_W0 = 0xCCCCCCCCCCCCCCCDull;

// C(m, j), j = 0..DEG, for 0 <= m < 2^29 (every tile a chirp covers), each from the one before:
// C(m, j) = C(m, j-1) (m - j + 1) / j.  C(m, 1), C(m, 2) < 2^57 fit one 64-bit limb, C(m, 3) and
// C(m, 4) < 2^112 two, C(m, 5), C(m, 6) < 2^165 three; the quotients are exact, so a division by 3
// or 5 is a product with the inverse modulo 2^128 or 2^192 and a division by 2 or 4 a shift.
template <int DEG>
__device__ __forceinline__ void binomials_pos(uint64_t m, U192 c[DEG + 1]) {
  c[0] = U192{1, 0, 0};
  c[1] = U192{m, 0, 0};
  const uint64_t c2 = (m * (m - 1)) >> 1;
  c[2] = U192{c2, 0, 0};
  if (DEG >= 3) {
    unsigned __int128 t = (unsigned __int128)c2 * (m - 2);                 // 3 C(m, 3) < 2^86
    t *= ((unsigned __int128)INV3_W << 64) | INV3_W0;
    c[3] = U192{(uint64_t)t, (uint64_t)(t >> 64), 0};
    t = (t * (unsigned __int128)(m - 3)) >> 2;                              // C(m, 4) < 2^112
    c[4] = U192{(uint64_t)t, (uint64_t)(t >> 64), 0};
    U192 u = mul192_limbs<1>(c[4], U192{m - 4, 0, 0});                      // 5 C(m, 5)
    c[5] = mul192(u, U192{INV5_W0, INV5_W, INV5_W});
    u = mul192_limbs<1>(c[5], U192{m - 5, 0, 0});                           // 6 C(m, 6)
    u = mul192(u, U192{INV3_W0, INV3_W, INV3_W});                           // 2 C(m, 6)
    c[6] = U192{(u.w0 >> 1) | (u.w1 << 63), (u.w1 >> 1) | (u.w2 << 63), u.w2 >> 1};
  }
}

// acc[k] = sum over i >= k of d_i C(m, i - k), k = 0..DEG, the products by C(m, j) taking its limb
// count.  Each d_i is loaded once and added into every acc[k] it contributes to (the sums are
// exact mod 2^192, so their order does not matter).
template <int DEG>
__device__ __forceinline__ void newton_shift_pos(const ChirpRec& c, const U192* bin, U192* acc) {
#pragma unroll
  for (int i = 0; i <= DEG; ++i) {
    const U192 d = dword(c, i);
    acc[i] = d;
#pragma unroll
    for (int k = 0; k < i; ++k) {
      const int j = i - k;
      if (j <= 2) acc[k] = add192(acc[k], mul192_limbs<1>(d, bin[j]));
      else if (j <= 4) acc[k] = add192(acc[k], mul192_limbs<2>(d, bin[j]));
      else acc[k] = add192(acc[k], mul192_limbs<3>(d, bin[j]));
    }
  }
}

// DEG = 2 (linear chirps) or 6 (minimum-jerk).  The unit-stride differences at the tile start
// are exact (192-bit); the stride-RUN transform that follows only needs the word-level result,
// so it runs on the upper 128 bits (error < W 2^-64 word per term, below 2^-20 word).  Tiles
// from the chirp's start on (0 <= m < 2^29) take the binomials' limb counts into account; a tile
// that begins before the chirp (m < 0) takes signed binomials (both the same integers).
// the unit-stride differences at a tile that begins before the chirp (signed binomials)
template <int DEG>
__device__ __forceinline__ void newton_shift_signed(const ChirpRec& c, int64_t m, const uint64_t (*inv)[3], U192* acc) {
  U192 bin[DEG + 1];
  binomials_deg<DEG>(m, inv, bin);
#pragma unroll
  for (int k = 0; k <= DEG; ++k) {
    U192 s = {0, 0, 0};
#pragma unroll
    for (int i = k; i <= DEG; ++i) s = add192(s, mul192(dword(c, i), bin[i - k]));
    acc[k] = s;
  }
}

template <int DEG, int WORDS, class Args>
__device__ __forceinline__ void prep_one(const ChirpRec& c, int64_t m, const Args& a, TileRec& out) {
  U192 acc[DEG + 1];
  if (m >= 0 && m < ((int64_t)1 << 29)) {
    U192 bin[DEG + 1];
    binomials_pos<DEG>((uint64_t)m, bin);
    newton_shift_pos<DEG>(c, bin, acc);
  } else {
    newton_shift_signed<DEG>(c, m, a.inv_odd, acc);
  }
  unsigned __int128 h[DEG + 1];
#pragma unroll
  for (int k = 0; k <= DEG; ++k) h[k] = hi128(acc[k]);
  stride_records<DEG, WORDS>(h, c.phi_start + acc[0].w2, a, out);   // acc_0 holds 2^127
}

// Exponential chirps: the unit forward differences of R(m) = C (e^(alpha m) - 1) at the tile
// start are C e^(alpha m) q^k (k >= 1, q = e^alpha - 1), in FP64 (a few 1e-10 turn), cut after
// order 6: the set-up gives a chirp a per-sample table instead when the dropped orders could
// reach 2^-26 turn over a tile.
template <int WORDS, class Args>
__device__ __forceinline__ void prep_exp(const ChirpRec& c, int64_t m, const Args& a, TileRec& out) {
  const double alpha = __longlong_as_double((long long)c.d[2]);
  const double C = __longlong_as_double((long long)c.d[3]);
  const double q = __longlong_as_double((long long)c.d[4]);
  const double e1 = expm1(alpha * (double)m);
  unsigned __int128 h[7];
  h[0] = q64_of(C * e1);
  double g = C * (e1 + 1.0) * q;
#pragma unroll
  for (int k = 1; k <= 6; ++k) {
    h[k] = q64_of(g);
    g *= q;
  }
  stride_records<6, WORDS>(h, c.phi_start + (uint64_t)((h[0] + ((unsigned __int128)1 << 63)) >> 64), a, out);
}

// Programmatic dependent launch (pipelined chunk sequences): the next kernel in the stream may
// start once every CTA of this one has passed launch_dependents; wait blocks until the preceding
// kernel has completed and its memory is visible.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// Device times of a handle's last render (awg_last_render_ms): the first kernel of a call writes the
// start, every CTA raises the end once its samples are stored (time only grows, so the largest is
// the last render's).  Events in the stream would serve too, but a timed event between two kernels
// keeps the second from starting before the first has ended: 6.6 us between kernels with the
// events, 2.3 without, none with the kernels overlapping.
__device__ __forceinline__ void mark_start(unsigned long long* t) {
  if (t && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *t = global_ns();   // (the replay's grid has rows)
}
__device__ __forceinline__ void mark_end(unsigned long long* t) {
  if (t && threadIdx.x == 0) atomicMax(t, (unsigned long long)global_ns());
}

// Bounded wait (limit_ns of wall time) until a device counter reaches target; false on timeout.
__device__ bool wait_counter(const unsigned long long* ctr, unsigned long long target, uint64_t limit_ns) {
  const volatile unsigned long long* v = ctr;
  if (*v >= target) return true;
  const uint64_t t0 = global_ns();
  while (*v < target) {
    if (global_ns() - t0 > limit_ns) return false;
    __nanosleep(256);
  }
  return true;
}

// Words of a record that the render reads: the run set-up of a linear chirp takes 6 in every tile;
// one in LOW3 form takes 10 in the tiles that it covers without an amplitude ramp (tile_kind,
// kind_state); every other takes all.
__device__ __forceinline__ int rec_words(const ChirpRec& c, const ToneRec& t, int64_t T0) {
  if (c.flags & TONE_LINEAR) return REC_WORDS_LINEAR;
  const bool ramp = (t.flags & TONE_AMP_RAMP) && T0 + TILE - 1 > t.a_ns && T0 < t.a_ns + t.a_L;
  const bool inside = T0 >= c.n_s && T0 + TILE - 1 <= c.n_s + c.L;
  return (c.flags & TONE_LOW3) && inside && !ramp ? REC_WORDS_LOW3 : REC_WORDS;
}
template <int WORDS>
__device__ __forceinline__ void store_record(TileRec* out, const TileRec& r) {
  static_assert(WORDS % 2 == 0, "16-byte stores");
  uint4* o = reinterpret_cast<uint4*>(out);
#pragma unroll
  for (int i = 0; i < WORDS / 2; ++i)
    o[i] = make_uint4((uint32_t)r.w[2 * i], (uint32_t)(r.w[2 * i] >> 32), (uint32_t)r.w[2 * i + 1], (uint32_t)(r.w[2 * i + 1] >> 32));
}

// The record of chirp c (of tone t) at tile T0, handed to put(record, its word count as a constant).
template <int N>
struct Count {
  static constexpr int value = N;
};
template <class Args, class Put>
__device__ __forceinline__ void form_record(const ChirpRec& c, const ToneRec& t, int64_t T0, const Args& a, Put put) {
  const int words = rec_words(c, t, T0);
  TileRec r;
  if (words == REC_WORDS_LINEAR) {
    prep_one<2, REC_WORDS_LINEAR>(c, T0 - c.n_s, a, r);
    put(r, Count<REC_WORDS_LINEAR>());
  } else if (words == REC_WORDS_LOW3) {
    if (c.flags & TONE_EXP) prep_exp<REC_WORDS_LOW3>(c, T0 - c.n_s, a, r);
    else prep_one<6, REC_WORDS_LOW3>(c, T0 - c.n_s, a, r);
    put(r, Count<REC_WORDS_LOW3>());
  } else {
    if (c.flags & TONE_EXP) prep_exp<REC_WORDS>(c, T0 - c.n_s, a, r);
    else prep_one<6, REC_WORDS>(c, T0 - c.n_s, a, r);
    put(r, Count<REC_WORDS>());
  }
}

template <class Args>
__global__ void __launch_bounds__(128, 5) prep_kernel(const __grid_constant__ Args a) {
  mark_start(a.start);
  // A render behind this kernel starts when it is complete: one that started earlier would put its
  // CTAs on the SMs that happen to have room, not evenly (1000-chirp 2^18 chunk: 109 against 96 us)
  if (a.more) pdl_launch_dependents();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t total = (int64_t)a.n_active * a.n_tiles;
  if (idx >= total) return;
  const int ai = (int)(idx / a.n_tiles);
  const int t = (int)(idx - (int64_t)ai * a.n_tiles);
  const int slot = a.slots[ai];
  const ChirpRec& c = a.chirps[slot];
  const int64_t T0 = (a.tile0 + t) * (int64_t)TILE;
  TileRec* out = a.recs + (int64_t)t * a.rec_stride + a.act_base + ai;
  // the preceding kernel of the stream may be a render that reads the buffers written here: it has
  // to be complete before the first write, not before the arithmetic
  form_record(c, a.tones[c.tone], T0, a, [&](const TileRec& r, auto words) {
    pdl_wait();
    store_record<decltype(words)::value>(out, r);
  });
  if (t == 0) a.act_of_slot[slot] = a.act_base + ai;
}

// ------------------------------------------------------------------------------------------
// render
// ------------------------------------------------------------------------------------------
// Geometry of a render CTA: RT = 128 threads take SPT consecutive samples each, RT x SPT samples of
// one tile: the whole tile (SPT 32) or one of PARTS = RUN / SPT equal parts of it.  A run of RUN
// samples belongs to PARTS neighbouring lanes; the run cascade is an exact integer recurrence, so
// a lane that starts r0 samples into its run advances the run's state by r0 in closed form and
// takes the same integers.  Parts cut the work of a window finer without a change in any sum:
// see render_parts in the host code for where each form is used.
template <int SPT>
struct Geo {
  static constexpr int PARTS = RUN / SPT;
  static constexpr int PSAMP = RT * SPT;       // samples of a part
  static constexpr int PRUNS = RUNS / PARTS;   // runs of a part
  static constexpr int RW = 32 / PARTS;        // runs of a warp
};

// Accumulators: a thread's SPT partial sums as SPT / 2 pairs of consecutive samples (float2).
// The loops compute the sine arguments and the multiply-adds of two samples as packed FP32 pairs
// (each component rounds as fmaf, so the sums are the same bits as with scalar fmaf).
template <int SPT>
using Acc = float2[SPT / 2];

constexpr float TWO_PI_F = 6.28318530717958647692f;
constexpr float THREE_PI_F = 9.42477796076937971538f;

// sin(2 pi p / 2^32) of two phases already offset by half a turn: 2 pi (v - 3/2) of their mantissa floats
// v lies in [-pi, pi) and is congruent to the phase
__device__ __forceinline__ float2 sin_pair(uint32_t p0, uint32_t p1) {
  const float2 v = make_float2(mantissa_float(p0), mantissa_float(p1));
  const float2 x = __ffma2_rn(v, make_float2(TWO_PI_F, TWO_PI_F), make_float2(-THREE_PI_F, -THREE_PI_F));
  return make_float2(__sinf(x.x), __sinf(x.y));
}
// acc += A (sin(p0), sin(p1))
__device__ __forceinline__ void acc_pair(float2& acc, float A, uint32_t p0, uint32_t p1) {
  acc = __ffma2_rn(make_float2(A, A), sin_pair(p0, p1), acc);
}

// Static segment: p += f per sample.
template <int SPT>
__device__ __forceinline__ void static_loop(uint32_t p, uint32_t f, float A, Acc<SPT>& acc) {
#pragma unroll
  for (int r = 0; r < SPT; r += 2) {
    const uint32_t p1 = p + f;
    acc_pair(acc[r / 2], A, p, p1);
    p = p1 + f;
  }
}

// Chirp cascade p += f, f += g (and g += h with WITH_H).
template <int SPT, bool WITH_H>
__device__ __forceinline__ void cascade(const RunPoly& q, float A, Acc<SPT>& acc) {
  uint32_t p = q.p, f = q.f, g = q.g;
  const uint32_t h = q.h;
#pragma unroll
  for (int r = 0; r < SPT; r += 2) {
    const uint32_t p1 = p + f;
    const uint32_t f1 = f + g;
    if (WITH_H) g += h;
    acc_pair(acc[r / 2], A, p, p1);
    p = p1 + f1;
    f = f1 + g;
    if (WITH_H) g += h;
  }
}

// The state r0 samples later (exact mod 2^32).
__device__ __forceinline__ RunPoly advance(const RunPoly& q, uint32_t r0) {
  const uint32_t c2 = r0 * (r0 - 1) / 2, c3 = r0 >= 3 ? r0 * (r0 - 1) * (r0 - 2) / 6 : 0u;
  RunPoly n;
  n.p = q.p + r0 * q.f + c2 * q.g + c3 * q.h;
  n.f = q.f + r0 * q.g + c2 * q.h;
  n.g = q.g + r0 * q.h;
  n.h = q.h;
  return n;
}

// The same with h = 0.
__device__ __forceinline__ RunPoly advance3(const RunPoly& q, uint32_t r0) {
  return RunPoly{q.p + r0 * q.f + (r0 * (r0 - 1) / 2) * q.g, q.f + r0 * q.g, q.g, 0u};
}

// Amplitude a(n) of a ramping tone (TONE_AMP_RAMP): A before a_ns, A_end from a_ns + a_L on, and
// A + (A_end - A) s(tau) between, tau = (n - a_ns) / a_L, s linear or minimum-jerk
// (10 tau^3 - 15 tau^4 + 6 tau^5).  FP32 (tau as m times the rounded 1 / a_L); error
// <= 6e-7 |A_end - A|.
struct Ramp {
  int32_t m0;       // the thread's first sample - a_ns, clamped to -RUN .. a_L (beyond, a is constant)
  int32_t L;
  float inv_L, A, A_end, dA;
  bool minjerk;
};
__device__ __forceinline__ Ramp ramp_setup(const ToneRec& t, int64_t n) {
  Ramp rr;
  rr.L = t.a_L;
  rr.m0 = (int32_t)max((int64_t)-RUN, min((int64_t)t.a_L, n - t.a_ns));
  rr.inv_L = 1.0f / (float)t.a_L;
  rr.A = t.A;
  rr.A_end = t.A_end;
  rr.dA = t.A_end - t.A;
  rr.minjerk = (t.flags & TONE_AMP_MINJERK) != 0;
  return rr;
}
// a(n) at the offsets m (mf: m as floats), two samples as packed pairs
__device__ __forceinline__ float2 ramp_curve(const Ramp& rr, float2 mf, bool minjerk) {
  const float2 tau = __fmul2_rn(mf, make_float2(rr.inv_L, rr.inv_L));
  float2 s = tau;
  if (minjerk) {
    const float2 poly = __ffma2_rn(tau, __ffma2_rn(make_float2(6.f, 6.f), tau, make_float2(-15.f, -15.f)),
                                   make_float2(10.f, 10.f));
    s = __fmul2_rn(__fmul2_rn(__fmul2_rn(tau, tau), tau), poly);
  }
  return __ffma2_rn(make_float2(rr.dA, rr.dA), s, make_float2(rr.A, rr.A));
}
__device__ __forceinline__ float2 ramp_amp_pair(const Ramp& rr, int r) {
  const int m = rr.m0 + r;
  float2 a = ramp_curve(rr, make_float2((float)m, (float)(m + 1)), rr.minjerk);
  a.x = m <= 0 ? rr.A : (m >= rr.L ? rr.A_end : a.x);
  a.y = m + 1 <= 0 ? rr.A : (m + 1 >= rr.L ? rr.A_end : a.y);
  return a;
}

// A ramping tone whose phase follows one cascade over the thread's samples (CHIRP: a chirp, else a
// static segment).  Where the ramp covers all the samples of the warp and m < 2^24, the sample
// offsets are stepped in FP32 (exact integers, so the same tau, s and a) and the amplitudes come in
// packed pairs without selects: 3 (linear) or 8 instructions per two samples.  A warp whose
// amplitudes are constant takes the plain loop.  (Per sample before: 64-bit compares, a 64-bit
// conversion and a branch: 600 tones, 500 of them ramping, 200,000 samples took 255 us.)
template <int SPT, bool CHIRP>
__device__ __forceinline__ void ramp_loop(RunPoly q, const Ramp& rr, Acc<SPT>& acc) {
  const bool before = rr.m0 + (SPT - 1) <= 0, after = rr.m0 >= rr.L;
  if (__all_sync(0xffffffffu, before || after)) {
    const float A = before ? rr.A : rr.A_end;
    if constexpr (CHIRP) cascade<SPT, true>(q, A, acc);
    else static_loop<SPT>(q.p, q.f, A, acc);
    return;
  }
  auto step = [&](uint32_t& p0, uint32_t& p1) {   // the next two phases
    p0 = q.p;
    p1 = q.p + q.f;
    if constexpr (CHIRP) {
      const uint32_t f1 = q.f + q.g;
      q.g += q.h;
      q.p = p1 + f1;
      q.f = f1 + q.g;
      q.g += q.h;
    } else {
      q.p = p1 + q.f;
    }
  };
  const bool inside = rr.m0 > 0 && rr.m0 + (SPT - 1) < rr.L && rr.L <= (1 << 24);
  uint32_t p0, p1;
  if (!__all_sync(0xffffffffu, inside)) {
#pragma unroll
    for (int r = 0; r < SPT; r += 2) {
      step(p0, p1);
      acc[r / 2] = __ffma2_rn(ramp_amp_pair(rr, r), sin_pair(p0, p1), acc[r / 2]);
    }
    return;
  }
  const float mf = (float)rr.m0;
  auto run = [&](bool minjerk) {
#pragma unroll
    for (int r = 0; r < SPT; r += 2) {
      step(p0, p1);
      const float2 m = __fadd2_rn(make_float2(mf, mf), make_float2((float)r, (float)(r + 1)));
      acc[r / 2] = __ffma2_rn(ramp_curve(rr, m, minjerk), sin_pair(p0, p1), acc[r / 2]);
    }
  };
  if (rr.minjerk) run(true);
  else run(false);
}

// Tile kinds of a tone.  The chirp kinds cover the tile from start to end.
enum { DESC_STATIC = 0, DESC_STATIC_ROT = 1,
       DESC_RAMP_STATIC = 2,    // a static segment with an amplitude ramp in the tile
       DESC_RAMP_CHIRP = 3,     // a chirp that covers the tile, with an amplitude ramp in it
       DESC_MIXED = 4,          // a chirp boundary or a per-sample phase table in the tile
       DESC_SKIP = 5,           // a static segment the tensor-core engine sums
       DESC_LINEAR = 8, DESC_MINJERK = 9,
       DESC_FLAT3 = 10,         // a degree-6 chirp whose h is 0 in every run (TONE_FLAT3)
       DESC_LOW6 = 11,          // FLAT3 without the negligible high orders (TONE_LOW6)
       DESC_LOW3 = 12 };        // LOW6 without B_5, E_3, E_4 (TONE_LOW3)

// Per-stage tone descriptor, built by warp 0 once per (tone, tile) so that the other threads
// skip the classification and the 64-bit phase set-up of static segments.
struct alignas(16) Desc {
  uint64_t p0;    // static: phase word at the tile start of the segment covering the tile
  uint64_t F;     // static: its frequency word
  float A;
  int32_t rec;    // the tone's record in the stage (chirp kinds, DESC_RAMP_CHIRP, DESC_MIXED)
  float c, s;     // DESC_STATIC_ROT: cos and sin of the per-sample phase step
};

// Kind of a chirp tile that the chirp covers from start to end (no table, no ramp in the tile).
__device__ __forceinline__ int chirp_inside_kind(int32_t flags) {
  return (flags & TONE_LINEAR) ? DESC_LINEAR : (flags & TONE_LOW3) ? DESC_LOW3 : (flags & TONE_LOW6) ? DESC_LOW6
         : (flags & TONE_FLAT3) ? DESC_FLAT3 : DESC_MINJERK;
}

// Descriptor kind of a tone in the tile [T0, T0 + TILE) (the stage turns DESC_STATIC into
// DESC_STATIC_ROT under the rotator sine).
__device__ __forceinline__ int tile_kind(const ToneRec& tr, int64_t T0, bool skip_static) {
  if (skip_static && tile_static(tr, T0)) return DESC_SKIP;
  const int tcls = classify_tile(tr, T0);
  const bool ramp = (tr.flags & TONE_AMP_RAMP) && T0 + TILE - 1 > tr.a_ns && T0 < tr.a_ns + tr.a_L;
  if (tcls != TILE_CHIRP) return ramp ? DESC_RAMP_STATIC : DESC_STATIC;
  const bool inside = T0 >= tr.n_s && T0 + TILE - 1 <= tr.n_e;
  if (!inside || (tr.flags & TONE_EXACT)) return DESC_MIXED;
  return ramp ? DESC_RAMP_CHIRP : chirp_inside_kind(tr.flags);
}

// Visit group of a stage's tone: chirps in linear form that may share their run set-up (TONE_PAIR),
// the other linear ones, chirps in LOW3 form that may share it, the same two for LOW6 form, static
// segments, then the rest (every tone in plain order; LOW3 chirps that may not share).  Shared set-ups
// only in renders without the tensor-core engine (pair false).
enum { GRP_LIN_PAIR = 0, GRP_LIN = 1, GRP_LOW3_PAIR = 2, GRP_LOW6_PAIR = 3, GRP_LOW6 = 4, GRP_STATIC = 5, GRP_REST = 6,
       N_GRP = 7 };
__device__ __forceinline__ int visit_group(int kind, bool plain, bool pair) {
  if (plain) return GRP_REST;
  if (kind == DESC_LINEAR) return pair ? GRP_LIN_PAIR : GRP_LIN;
  if (kind == DESC_LOW3) return pair ? GRP_LOW3_PAIR : GRP_REST;
  if (kind == DESC_LOW6) return pair ? GRP_LOW6_PAIR : GRP_LOW6;
  return (kind == DESC_STATIC || kind == DESC_STATIC_ROT) ? GRP_STATIC : GRP_REST;
}

// Run set-up shared by a lane pair.  Lanes 2m and 2m + 1 (runs j and j + 1) take two tones of a
// group: each evaluates one tone's set-up exactly (the even run's lane the first tone's, the odd
// run's the second's) and takes the other tone's from its partner, moved by one run with the
// cascade's own integer steps (h = 0): forward from run j - 1, p + 32 f + 496 g and f + 32 g (the
// state the partner's cascade reaches after 32 samples); backward from run j + 1, p - 32 f + 528 g
// and f - 32 g (C(-32, 2) = 528).  The moved state's error is the cascade's over up to 63 steps
// (pair_setup_ok on the host bounds it).  Every lane of the warp takes part.
__device__ __forceinline__ RunPoly partner_state(const RunPoly& own, bool odd) {
  const uint32_t p = __shfl_xor_sync(0xffffffffu, own.p, 1);
  const uint32_t f = __shfl_xor_sync(0xffffffffu, own.f, 1);
  const uint32_t g = __shfl_xor_sync(0xffffffffu, own.g, 1);
  RunPoly q;
  if (odd) {
    q.p = p + 32u * f + 496u * g;
    q.f = f + 32u * g;
  } else {
    q.p = p - 32u * f + 528u * g;
    q.f = f - 32u * g;
  }
  q.g = g;
  q.h = 0;
  return q;
}

// A tile with a chirp boundary or a per-sample table (DESC_MIXED): the thread's samples n0s ..
// n0s + SPT - 1, the first of them r0 samples into the run that starts at n0.  Sample r takes the
// static phase before the chirp (r < n_s - n0), the one after it (r > n_e - n0), else the chirp's
// cascade (or its table entry); the amplitude is the ramp's where one is under way.  The warp that holds
// the boundary sets the tile's time: its samples take one static segment, picked by a bit mask (two
// segments and two comparisons per sample: 6699 chirps over 28.6 tiles that end in the last 612 -> 561 us,
// 1.5e6 samples of them in chunks 2693 -> 2547; the engine's 100 chirps in 10,000 tones 217 -> 210).
template <int SPT>
__device__ __forceinline__ void mixed_run(const ToneRec& tr, const TileRec* rec, const RunBin& rb, Acc<SPT>& acc,
                                          int64_t n0, int r0, const uint32_t* exact_tab) {
  const int64_t n0s = n0 + r0, last = n0s + SPT - 1;
  const bool ramp = (tr.flags & TONE_AMP_RAMP) != 0;
  const bool exact = (tr.flags & TONE_EXACT) != 0;
  const bool ramp_run = ramp && last > tr.a_ns && n0s < tr.a_ns + tr.a_L;   // a(n) varies here
  const float A = (ramp && n0s >= tr.a_ns + tr.a_L) ? tr.A_end : tr.A;
  const bool pre = last < tr.n_s, post = n0s > tr.n_e;
  const uint32_t ur0 = (uint32_t)r0;
  if (__all_sync(0xffffffffu, (pre || post) && !ramp_run)) {
    const uint64_t phi = pre ? tr.phi_ref : tr.phi_post_ref;
    const uint64_t F = pre ? tr.F : tr.F_end;
    const uint32_t f = static_f(F);
    static_loop<SPT>(static_p0(phi, F, n0) + HALF_TURN + ur0 * f, f, A, acc);
    return;
  }
  RunPoly st = {0, 0, 0, 0};
  if (!exact) st = advance(poly_state(*rec, rb, (tr.flags & TONE_LINEAR) != 0), ur0);
  if (__all_sync(0xffffffffu, !exact && !ramp_run && n0s >= tr.n_s && last <= tr.n_e)) {
    if (__all_sync(0xffffffffu, st.h == 0)) cascade<SPT, false>(st, A, acc);
    else cascade<SPT, true>(st, A, acc);
    return;
  }
  // i1, i2: the chirp's samples i1 <= r <= i2 of the thread, clamped to [-1, SPT]
  const int i1 = (int)max((int64_t)-1, min((int64_t)SPT, tr.n_s - n0s));
  const int i2 = (int)max((int64_t)-1, min((int64_t)SPT, tr.n_e - n0s));
  const bool begins = i1 > 0, ends = i2 < SPT - 1;
  if (!__any_sync(0xffffffffu, exact || ramp_run || (begins && ends))) {
    // one boundary at most in each thread's samples: one static segment, its samples as a bit mask
    const uint32_t fs = static_f(begins ? tr.F : tr.F_end);
    uint32_t qs = static_p0(begins ? tr.phi_ref : tr.phi_post_ref, begins ? tr.F : tr.F_end, n0) + HALF_TURN + ur0 * fs;
    const uint32_t m = begins ? (i1 < 32 ? (1u << i1) - 1u : ~0u) : ends ? ~0u << (i2 + 1) : 0u;
    auto next = [&](int r) {
      const uint32_t ph = (m & (1u << r)) ? qs : st.p;
      qs += fs;
      st.p += st.f;
      st.f += st.g;
      st.g += st.h;
      return ph;
    };
#pragma unroll
    for (int r = 0; r < SPT; r += 2) {
      const uint32_t ph0 = next(r);
      const uint32_t ph1 = next(r + 1);
      acc_pair(acc[r / 2], A, ph0, ph1);
    }
    return;
  }
  // table chirps, ramps, chirps that begin and end within a thread's samples: the phases one by one into
  // local memory, then the sums
  const uint32_t fa = static_f(tr.F), fb = static_f(tr.F_end);
  const uint32_t qa = static_p0(tr.phi_ref, tr.F, n0) + HALF_TURN + ur0 * fa;
  const uint32_t qb = static_p0(tr.phi_post_ref, tr.F_end, n0) + HALF_TURN + ur0 * fb;
  const Ramp rr = ramp_setup(tr, n0s);
  uint32_t col[SPT];
  const uint32_t* tab = exact ? exact_tab + tr.tab_off : nullptr;
  const int32_t t0 = (int32_t)(n0s - tr.n_s);   // table index of sample 0 (negative before the chirp)
#pragma unroll 4
  for (int r = 0; r < SPT; ++r) {
    uint32_t ph;
    if (r < i1) ph = qa + (uint32_t)r * fa;
    else if (r > i2) ph = qb + (uint32_t)r * fb;
    else ph = exact ? tab[t0 + r] + HALF_TURN : st.p;
    col[r] = ph;
    st.p += st.f;
    st.f += st.g;
    st.g += st.h;
  }
  if (ramp_run) {
#pragma unroll
    for (int r = 0; r < SPT; r += 2)
      acc[r / 2] = __ffma2_rn(ramp_amp_pair(rr, r), sin_pair(col[r], col[r + 1]), acc[r / 2]);
  } else {
#pragma unroll
    for (int r = 0; r < SPT; r += 2) acc_pair(acc[r / 2], A, col[r], col[r + 1]);
  }
}

// Scale, round half to even, clamp and store sample n (inside the window), after adding the
// tensor-core engine's static sum when there is one.
__device__ __forceinline__ void store_sample(const RenderArgs& a, int64_t n, float x) {
  if (n < a.win_start || n >= a.win_end) return;
  if (a.base) x += a.base[n - a.win_start];
  float q = rintf(x * a.scale);
  q = fminf(fmaxf(q, -32767.f), 32767.f);
  if (a.out_q) a.out_q[(n - a.win_start) * (a.q_stride ? a.q_stride : 1)] = (int16_t)q;
  if (a.out_f) a.out_f[n - a.win_start] = x;
}

// Whether 8-sample groups (first sample a multiple of 8) of the int16 and FP32 outputs start on
// 16-byte boundaries: sample n sits at out + (n - win_start), so this holds for every group at
// once when out - win_start is 16-byte aligned.
__device__ __forceinline__ bool q_vec_ok(const RenderArgs& a) {
  return a.out_q && a.q_stride <= 1 && (((uintptr_t)a.out_q - 2u * (uint64_t)a.win_start) & 15u) == 0;
}
__device__ __forceinline__ bool f_vec_ok(const RenderArgs& a) {
  return !a.out_f || (((uintptr_t)a.out_f - 4u * (uint64_t)a.win_start) & 15u) == 0;
}

// Store the 8 samples n .. n + 7 (n a multiple of 8) of a group inside the window, the outputs aligned
// (q_vec_ok, f_vec_ok): one 16-byte vector of int16 codes and, where asked for, two of FP32 sums.
__device__ __forceinline__ void store_group(const RenderArgs& a, int64_t n, const float (&xv)[8]) {
  const int64_t o = n - a.win_start;
  float x[8];
#pragma unroll
  for (int u = 0; u < 8; ++u) x[u] = a.base ? xv[u] + a.base[o + u] : xv[u];
  uint32_t w[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float q0 = fminf(fmaxf(rintf(x[2 * u] * a.scale), -32767.f), 32767.f);
    const float q1 = fminf(fmaxf(rintf(x[2 * u + 1] * a.scale), -32767.f), 32767.f);
    w[u] = (uint32_t)(uint16_t)(int16_t)q0 | ((uint32_t)(uint16_t)(int16_t)q1 << 16);
  }
  if (a.out_q) *reinterpret_cast<uint4*>(a.out_q + o) = make_uint4(w[0], w[1], w[2], w[3]);
  if (a.out_f) {
    float4* f4 = reinterpret_cast<float4*>(a.out_f + o);
    f4[0] = make_float4(x[0], x[1], x[2], x[3]);
    f4[1] = make_float4(x[4], x[5], x[6], x[7]);
  }
}

// Samples of a part that go through shared memory at a time.
constexpr int OUT_STAGE = 4096;

// Sum over the split without clusters.  The thread holds samples at .. at + SPT - 1 of the part
// in acc.  With split 1 it stores them; otherwise the CTA writes them to its partial part
// a.part[(unit split + crank) PSAMP ...] (unit: the part's index in the launch) and counts itself in
// on a.tile_ctr[unit]; the CTA that brings the count to split - 1 (mod split) is the last of the
// part: it sums the split's partials in rank order (as the cluster reduction does: the same FP32
// sums) and stores the part, thread t taking the 8-sample groups t, t + RT, ... (coalesced
// 16-byte stores).  A part at the window's edge, an output off the vectors' alignment or with a stride
// goes through s_out, OUT_STAGE samples at a time, so that a warp stores 32 consecutive samples; eight
// by one thread, one after another, met a cache line per lane and store (80 tones x 1,000,001 samples
// from sample 12345, FP32 and int16: 41.8 -> 18.6 us; eight multiplexed channels of 100 chirps x 50,001
// 21.2 -> 18.7; two of 60 static tones x 2^20, at the stores' rate either way, 29.6 -> 30.4).
// The loads of several ranks are in flight at a time: one rank at a time left the last CTA of a tile
// waiting for the L2 `split` times in a row (12 us at split 11).
// The preceding kernel of the stream is complete before the first write to global memory (in a
// sequence: before the first write to the split scratch).
template <int SPT>
__device__ __forceinline__ void tile_epilogue_split(const RenderArgs& a, int unit, int crank, int split, int64_t P0,
                                                    int at, const Acc<SPT>& acc, float* s_out) {
  constexpr int PSAMP = Geo<SPT>::PSAMP;
  const int tid = threadIdx.x;
  __shared__ int s_last;
  const bool vec = q_vec_ok(a) && f_vec_ok(a) && P0 >= a.win_start && P0 + PSAMP <= a.win_end;
  auto store_out = [&](int64_t n0, int count) {   // s_out[0 .. count): samples n0 ..
    __syncthreads();
    for (int i = tid; i < count; i += RT) store_sample(a, n0 + i, s_out[i]);
    __syncthreads();
  };
  if (a.pdl != PDL_NONE && (a.pdl != PDL_SEQUENCE || split > 1)) pdl_wait();
  if (split == 1) {
    if (vec) {
#pragma unroll
      for (int g = 0; g < SPT / 8; ++g) {
        float xv[8];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          xv[2 * u] = 0.f + acc[4 * g + u].x;
          xv[2 * u + 1] = 0.f + acc[4 * g + u].y;
        }
        store_group(a, P0 + at + 8 * g, xv);
      }
    } else {
      __syncthreads();   // s_out is free
      for (int b = 0; b < PSAMP; b += OUT_STAGE) {
        if (at >= b && at < b + OUT_STAGE) {
          float4* d = reinterpret_cast<float4*>(s_out + (at - b));
#pragma unroll
          for (int j = 0; j < SPT / 4; ++j)
            d[j] = make_float4(0.f + acc[2 * j].x, 0.f + acc[2 * j].y, 0.f + acc[2 * j + 1].x, 0.f + acc[2 * j + 1].y);
        }
        store_out(P0 + b, PSAMP < OUT_STAGE ? PSAMP : OUT_STAGE);
      }
    }
  } else {
    float4* dst = reinterpret_cast<float4*>(a.part + ((int64_t)unit * split + crank) * PSAMP + at);
#pragma unroll
    for (int j = 0; j < SPT / 4; ++j)
      __stcg(dst + j, make_float4(acc[2 * j].x, acc[2 * j].y, acc[2 * j + 1].x, acc[2 * j + 1].y));
    __threadfence();
    __syncthreads();
    if (tid == 0) s_last = atomicAdd(&a.tile_ctr[unit], 1ull) % (unsigned long long)split == (unsigned long long)(split - 1);
    __syncthreads();
    if (s_last) {
      __threadfence();
      constexpr int G = SPT / 8;             // 8-sample groups per thread
      constexpr int H = G > 2 ? 2 : G;       // groups summed at a time
      constexpr int CU = 4 / H;              // ranks in flight
      const float4* src = reinterpret_cast<const float4*>(a.part + (int64_t)unit * split * PSAMP) + 2 * tid;
#pragma unroll
      for (int v0 = 0; v0 < G; v0 += H) {
        float xs[H][8];
#pragma unroll
        for (int v = 0; v < H; ++v)
#pragma unroll
          for (int u = 0; u < 8; ++u) xs[v][u] = 0.f;
        for (int c = 0; c < split; c += CU) {
          float4 lo[CU][H], hi[CU][H];
#pragma unroll
          for (int k = 0; k < CU; ++k)
#pragma unroll
            for (int v = 0; v < H; ++v)
              if (c + k < split) {
                lo[k][v] = __ldcg(src + (int64_t)(c + k) * (PSAMP / 4) + 2 * RT * (v0 + v));
                hi[k][v] = __ldcg(src + (int64_t)(c + k) * (PSAMP / 4) + 2 * RT * (v0 + v) + 1);
              }
#pragma unroll
          for (int k = 0; k < CU; ++k)
            if (c + k < split) {
#pragma unroll
              for (int v = 0; v < H; ++v) {
                xs[v][0] += lo[k][v].x;
                xs[v][1] += lo[k][v].y;
                xs[v][2] += lo[k][v].z;
                xs[v][3] += lo[k][v].w;
                xs[v][4] += hi[k][v].x;
                xs[v][5] += hi[k][v].y;
                xs[v][6] += hi[k][v].z;
                xs[v][7] += hi[k][v].w;
              }
            }
        }
        if (vec) {
#pragma unroll
          for (int v = 0; v < H; ++v) store_group(a, P0 + 8 * ((int64_t)tid + RT * (v0 + v)), xs[v]);
        } else {
          static_assert(8 * RT * H <= OUT_STAGE, "the groups summed at a time fit s_out");
#pragma unroll
          for (int v = 0; v < H; ++v) {
            float4* d = reinterpret_cast<float4*>(s_out + 8 * (tid + RT * v));
            d[0] = make_float4(xs[v][0], xs[v][1], xs[v][2], xs[v][3]);
            d[1] = make_float4(xs[v][4], xs[v][5], xs[v][6], xs[v][7]);
          }
          store_out(P0 + 8 * RT * v0, 8 * RT * H);
        }
      }
    }
  }
  if (a.exit_ctr) {   // this CTA's samples (if any) are stored and visible
    __threadfence();
    __syncthreads();
    if (tid == 0) atomicAdd(a.exit_ctr, 1ull);
  }
  mark_end(a.end);
}

// One CTA's share of one part of a tile: tones [K crank / split, K (crank+1) / split) of window tile
// unit / PARTS of the render described by `a` (or the listed tones of its bounds), then the sum over
// the split and the store.  CLUSTER: the split's CTAs form a thread-block cluster, sum through
// distributed shared memory in rank order and each stores a slice.  Otherwise each CTA writes its
// partial sums to a.part and the last of the split to finish (a counter per part) sums the partials
// in rank order and stores the whole part: the same sums, and no CTA waits for the others.
//
// The tones go through in stages of STAGE, in the stage's visit order: the groups of visit_group, each
// in a loop of its own without a per-tone dispatch, then the rest.
// MODE_ONCE: RenderArgs::once; MODE_LIST: a tone list, if a.tone_list is set, and renders for the tensor-core
// engine; MODE_ALL: all tones, no engine (with the engine's test for plain order in it 4770 chirps x 3829
// samples take 126.7 us, 124.6 without; 10,000 chirping tones on the engine 977 and, in MODE_LIST's kernel, 992).
enum { MODE_ALL = 0, MODE_LIST = 1, MODE_ONCE = 2, N_MODES = 3 };
template <int SPT, bool CLUSTER, int MODE>
__device__ __forceinline__ void render_tile(const RenderArgs& a, const int unit, const int crank, const int split) {
  using G = Geo<SPT>;
  constexpr int PARTS = G::PARTS, RW = G::RW;
  constexpr bool ONCE = MODE == MODE_ONCE;
  static_assert(!CLUSTER || SPT == RUN, "cluster sums take whole tiles");
  constexpr int NBUF = ONCE ? ONCE_TONES / STAGE : 2;   // stage buffers
  static_assert(!ONCE || NBUF <= RT / 32, "a warp prepares a stage");
  // The stage buffers in one object: one base address and constant offsets.  As variables of their own
  // (and with the output's stores not in a common loop) the 35 ms record took 2622 us, so 2524; one
  // object per stage, with the descriptors in visit order, costs static tones more registers (1000
  // tones x 2^19 118 against 113 us).  The epilogue stages the output in it.
  struct StageBuf {
    alignas(16) ToneRec tone[NBUF][STAGE];
    alignas(16) TileRec rec[NBUF][STAGE];
    alignas(16) Desc desc[NBUF][STAGE];
    uint8_t order[NBUF][STAGE];
    uint8_t kind[NBUF][STAGE];
    int ngrp[NBUF][N_GRP];
  };
  __shared__ StageBuf s_buf;
  auto& s_tone = s_buf.tone;
  auto& s_rec = s_buf.rec;
  auto& s_desc = s_buf.desc;
  auto& s_order = s_buf.order;
  auto& s_kind = s_buf.kind;
  auto& s_ngrp = s_buf.ngrp;
  // cluster sums through distributed shared memory: [i][thread]
  __shared__ alignas(16) float s_red[CLUSTER ? TILE : 4];
  __shared__ alignas(8) uint64_t s_bar[4];        // tones[0], tones[1], records[0], records[1]

  cg::cluster_group cluster = cg::this_cluster();
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int tile = unit / PARTS, part = unit % PARTS;
  const int64_t T0 = (a.tile0 + tile) * (int64_t)TILE;
  const int64_t P0 = T0 + (int64_t)part * G::PSAMP;   // the part's first sample
  // the thread's run of the tile and its first sample in the run (lanes l, l + RW, ... of a warp
  // share a run, neighbouring lanes have neighbouring runs)
  const int run = part * G::PRUNS + warp * RW + lane % RW;
  const uint32_t r0 = (uint32_t)(lane / RW * SPT);
  // positions [l_begin, l_end) of the visit: the CTA's range of tones, or of the tone list
  int l_begin = (int)((int64_t)a.K * crank / split);
  int l_end = (int)((int64_t)a.K * (crank + 1) / split);
  const int32_t* list = MODE == MODE_LIST ? a.tone_list : nullptr;
  if (MODE != MODE_LIST) {
  } else if (a.tile_first) {
    const int32_t* first = a.tile_first + (int64_t)(a.rec_tile0 + tile) * (split + 1);
    list += (int64_t)(a.rec_tile0 + tile) * a.n_list;
    l_begin = first[crank];
    l_end = first[crank + 1];
  } else if (list) {
    const int k_begin = a.bounds[crank], k_end = a.bounds[crank + 1];
    auto lower = [&](int key) {
      int lo = 0, hi = a.n_list;
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (list[mid] < key) lo = mid + 1;
        else hi = mid;
      }
      return lo;
    };
    l_begin = lower(k_begin);
    l_end = lower(k_end);
  }
  const int n_stages = (l_end - l_begin + STAGE - 1) / STAGE;

  Acc<SPT> acc;
#pragma unroll
  for (int r = 0; r < SPT / 2; ++r) acc[r] = make_float2(0.f, 0.f);

  if (a.pdl == PDL_SETUP_FIRST) {   // the records' set-up (the preceding kernel) is complete before
    pdl_wait();                      // the next render may start (it relies on the same set-up)
    pdl_launch_dependents();
  } else if (a.pdl != PDL_NONE) {
    pdl_launch_dependents();
  }
  if (tid == 0) {
#pragma unroll
    for (int b = 0; b < 4; ++b) mbar_init(&s_bar[b], 1);
    fence_mbar_init();
  }
  __syncthreads();

  // thread 0 issues the copies and counts the issues per barrier (for a bounded drain)
  uint32_t issued = 0;   // 8-bit issue count per barrier
  // warp 0: one bulk copy of the stage's contiguous tone records, or one per listed tone
  auto issue_tones = [&](int st) {
    const int lb = l_begin + st * STAGE;
    const int cnt = min(STAGE, l_end - lb);
    fence_proxy_async();
    if (tid == 0) {
      mbar_arrive_expect_tx(&s_bar[st & 1], (uint32_t)cnt * (uint32_t)sizeof(ToneRec));
      issued += 1u << (8 * (st & 1));
    }
    __syncwarp();
    if (!list) {
      if (tid == 0) bulk_g2s(&s_tone[st & 1][0], a.tones + lb, (uint32_t)cnt * (uint32_t)sizeof(ToneRec), &s_bar[st & 1]);
    } else if (tid < cnt) {
      bulk_g2s(&s_tone[st & 1][tid], a.tones + list[lb + tid], (uint32_t)sizeof(ToneRec), &s_bar[st & 1]);
    }
  };
  // One warp (warp 0, or warp st with ONCE), once the stage's tones have landed: descriptors, visit
  // order, and the records of tones that chirp inside this tile.  ONCE forms them here, a tone per
  // lane; otherwise the set-up kernel did: the window's active chirps are numbered in tone order, so
  // the records of a stage's consecutive tones lie one after another and come in one bulk copy.
  auto prepare_stage = [&](int st) {
    const int b = ONCE ? st : st & 1;
    const int cnt = min(STAGE, l_end - (l_begin + st * STAGE));
    bool need = false, pairable = false;
    int kind = DESC_SKIP, act = 0;
    if (lane < cnt) {
      const ToneRec& tr = s_tone[b][lane];
      const int tcls = classify_tile(tr, T0);
      need = tcls == TILE_CHIRP && !(tr.flags & TONE_EXACT);
      if (!ONCE && need) act = a.act_of_slot[tr.slot];
      Desc d;
      const bool ramp = (tr.flags & TONE_AMP_RAMP) != 0;
      d.A = (ramp && T0 >= tr.a_ns + tr.a_L) ? tr.A_end : tr.A;
      d.c = d.s = 0.f;
      d.F = 0;
      d.p0 = 0;
      d.rec = lane;
      if (tcls == TILE_PRE || tcls == TILE_POST) {
        const bool pre = tcls == TILE_PRE;
        d.F = pre ? tr.F : tr.F_end;
        d.p0 = (pre ? tr.phi_ref : tr.phi_post_ref) + (uint64_t)T0 * d.F;
        if (a.sine_mode == SINE_ROTATOR) {
          d.c = pre ? tr.rot_c : tr.rot_c_end;
          d.s = pre ? tr.rot_s : tr.rot_s_end;
        }
      }
      kind = tile_kind(tr, T0, a.skip_static != 0);
      if (kind == DESC_STATIC && a.sine_mode == SINE_ROTATOR) kind = DESC_STATIC_ROT;
      s_desc[b][lane] = d;
      pairable = (tr.flags & TONE_PAIR) && !a.skip_static;
    }
    // visit order: the chirps that cover the tile in linear form, those in LOW3 and LOW6 form, the
    // static tones (SFU or rotator), then the rest; tone order within each group.  The order of the
    // FP32 sums then depends on which tones share a stage; with a tone list (the window's listed
    // tones) that changes with the window.  So a render for the tensor-core engine keeps plain tone
    // order in every tile that some window may take with a list: all but those in which every tone
    // chirps (full0 .. full1; there the groups save 5 to 8 %: 10,000 chirping tones x 2^18 samples 992
    // us, 1068 in plain order).  Every window cut gives the same bits.  Skipped tones are left out.
    const bool plain = MODE != MODE_ALL && (list != nullptr || (a.skip_static && (T0 < a.full0 || T0 > a.full1)));
    const int grp = kind == DESC_SKIP ? -1 : visit_group(kind, plain, pairable);
    const unsigned below = (1u << lane) - 1u;
    int pos = 0, end = 0;
#pragma unroll
    for (int g = 0; g < N_GRP; ++g) {
      const unsigned m = __ballot_sync(0xffffffffu, grp == g);
      if (grp == g) pos = end + __popc(m & below);
      end += __popc(m);
      if (lane == 0) s_ngrp[b][g] = end;
    }
    if (grp >= 0) {
      s_order[b][pos] = (uint8_t)lane;
      s_kind[b][pos] = (uint8_t)kind;
    }
    if constexpr (ONCE) {
      if (need) {
        const ToneRec& tr = s_tone[b][lane];
        form_record(a.chirps[tr.slot], tr, T0, a, [&](const TileRec& r, auto words) {
#pragma unroll
          for (int i = 0; i < decltype(words)::value; ++i) s_rec[b][lane].w[i] = r.w[i];
        });
      }
      return;
    }
    const unsigned mask = __ballot_sync(0xffffffffu, need);
    const int first = __shfl_sync(0xffffffffu, act, mask ? __ffs(mask) - 1 : 0);
    const int last = __shfl_sync(0xffffffffu, act, mask ? 31 - __clz(mask) : 0);
    // (the tones left out of a sifted list leave gaps: then one copy per record)
    const bool dense = MODE != MODE_LIST || (unsigned)(last - first) < (unsigned)STAGE;
    if (need) s_desc[b][lane].rec = dense ? act - first : tid;
    const TileRec* recs = a.recs + (int64_t)(a.rec_tile0 + tile) * a.rec_stride;
    if (tid == 0) {
      const uint32_t n_rec = !mask ? 0u : dense ? (uint32_t)(last - first + 1) : (uint32_t)__popc(mask);
      fence_proxy_async();
      mbar_arrive_expect_tx(&s_bar[2 + b], n_rec * (uint32_t)sizeof(TileRec));
      issued += 1u << (8 * (2 + b));
      if (dense && n_rec) bulk_g2s(&s_rec[b][0], recs + first, n_rec * (uint32_t)sizeof(TileRec), &s_bar[2 + b]);
    }
    __syncwarp();
    if (!dense && need) bulk_g2s(&s_rec[b][tid], recs + act, (uint32_t)sizeof(TileRec), &s_bar[2 + b]);
    __syncwarp();
  };

  bool ok = true;
  if constexpr (ONCE) {
    if (n_stages > 0) {
      if (tid == 0) {
        const uint32_t bytes = (uint32_t)(l_end - l_begin) * (uint32_t)sizeof(ToneRec);
        mbar_arrive_expect_tx(&s_bar[0], bytes);
        issued = 1u;
        bulk_g2s(&s_tone[0][0], a.tones + l_begin, bytes, &s_bar[0]);
      }
      ok = mbar_wait(&s_bar[0], 0);
      ok = __syncthreads_and(ok) != 0;
      if (ok && warp < n_stages) prepare_stage(warp);
      __syncthreads();
    }
  } else if (n_stages > 0) {
    if (tid < 32) {
      issue_tones(0);
      if (n_stages > 1) issue_tones(1);
      if (a.pdl == PDL_AFTER_SETUP) pdl_wait();   // the records' set-up is complete
      ok &= mbar_wait(&s_bar[0], 0);
      prepare_stage(0);
    }
    __syncthreads();   // stage-0 descriptors visible
  }
  int fail_stage = ONCE && !ok ? 0 : -1;
  const RunBin rb = run_binomials(run);
  for (int st = 0; st < n_stages; ++st) {
    const int b = ONCE ? st : st & 1;
    if constexpr (!ONCE) {
      const uint32_t par = (uint32_t)((st >> 1) & 1);
      if (tid < 32 && st + 1 < n_stages) {
        ok &= mbar_wait(&s_bar[(st + 1) & 1], (uint32_t)(((st + 1) >> 1) & 1));
        prepare_stage(st + 1);
      }
      ok &= mbar_wait(&s_bar[b], par);
      ok &= mbar_wait(&s_bar[2 + b], par);
      // the same decision in every lane of the warp: the loops below exchange values between lanes
      ok = __all_sync(0xffffffffu, ok);
    }
    if (ok) {
      const int e_lp = s_ngrp[b][GRP_LIN_PAIR], e_lin = s_ngrp[b][GRP_LIN], e_l3p = s_ngrp[b][GRP_LOW3_PAIR],
                e_l6p = s_ngrp[b][GRP_LOW6_PAIR], e_low6 = s_ngrp[b][GRP_LOW6], e_static = s_ngrp[b][GRP_STATIC],
                n_vis = s_ngrp[b][GRP_REST];
      auto record = [&](int i) -> const TileRec& { return s_rec[b][s_desc[b][i].rec]; };
      // a chirp run with h = 0 from its run state
      auto chirp = [&](const RunPoly& q, int i) {
        cascade<SPT, false>(PARTS > 1 ? advance3(q, r0) : q, s_desc[b][i].A, acc);
      };
      auto linear = [&](int i) { chirp(poly_state(record(i), rb, true), i); };
      auto low6 = [&](int i) { chirp(poly_state_low6(record(i), rb), i); };
      auto low3 = [&](int i) { chirp(poly_state_low3(record(i), rb), i); };
      auto flat3 = [&](int i) { chirp(poly_state_flat3(record(i), rb), i); };
      auto static_state = [&](const Desc& d) {   // the thread's first sample
        const uint32_t f = static_f(d.F);
        const uint32_t p = (uint32_t)((mac_u32(d.p0 + P_OFFSET, d.F, (uint32_t)(run * RUN))) >> 32) + HALF_TURN;
        return RunPoly{PARTS > 1 ? p + r0 * f : p, f, 0u, 0u};
      };
      auto static_sfu = [&](int i) {
        const RunPoly q = static_state(s_desc[b][i]);
        static_loop<SPT>(q.p, q.f, s_desc[b][i].A, acc);
      };
      // the exact phase word at the run start, SFU sine and cosine once, then 31 rotations by the
      // per-sample step on the FP32 pipe (amplitude folded into the phasor).  Whole tiles only: a
      // rotation cannot enter its run in the middle, so the rotator's renders have no parts
      // (render_parts).  The branches stay in the kernels of parts all the same: without them the
      // halves' static loop comes out slower (comb of 100 tones x 2^20 24.39 -> 24.52 us).
      auto phasor = [&](const Desc& d, float& re, float& im) {
        const uint64_t w = d.p0 + (uint64_t)(uint32_t)(run * RUN) * d.F;
        float sn, cs;
        __sincosf((float)(int32_t)(w >> 32) * 1.46291807926715968e-9f, &sn, &cs);   // 2 pi / 2^32
        im = d.A * sn;
        re = d.A * cs;
      };
      auto rotate = [](float& re, float& im, float c, float s) {
        const float t = fmaf(re, c, -im * s);
        im = fmaf(re, s, im * c);
        re = t;
      };
      auto static_rot = [&](int i) {
        const Desc& d = s_desc[b][i];
        float re, im;
        phasor(d, re, im);
        const float c = d.c, s = d.s;
#pragma unroll
        for (int r = 0; r < SPT; ++r) {
          if (r & 1) acc[r / 2].y += im;
          else acc[r / 2].x += im;
          rotate(re, im, c, s);
        }
      };
      // the sharing groups two tones at a time: one set-up per lane, the other tone's state from the
      // partner lane (partner_state); per sample the first tone's multiply-add, then the second's,
      // as in two single loops; an odd group's last tone alone
      const bool odd = (run & 1) != 0;
      auto pair = [&](const RunPoly& own, int i, int k) {
        const RunPoly oth = partner_state(own, odd);
        chirp(odd ? oth : own, i);
        chirp(odd ? own : oth, k);
      };
      for (int o = 0; o + 1 < e_lp; o += 2) {
        const int i = s_order[b][o], k = s_order[b][o + 1];
        pair(poly_state(record(odd ? k : i), rb, true), i, k);
      }
      for (int o = e_lp & ~1; o < e_lin; ++o) linear(s_order[b][o]);
      for (int o = e_lin; o + 1 < e_l3p; o += 2) {
        const int i = s_order[b][o], k = s_order[b][o + 1];
        pair(poly_state_low3(record(odd ? k : i), rb), i, k);
      }
      if ((e_l3p - e_lin) & 1) low3(s_order[b][e_l3p - 1]);
      for (int o = e_l3p; o + 1 < e_l6p; o += 2) {
        const int i = s_order[b][o], k = s_order[b][o + 1];
        pair(poly_state_low6(record(odd ? k : i), rb), i, k);
      }
      for (int o = e_l3p + ((e_l6p - e_l3p) & ~1); o < e_low6; ++o) low6(s_order[b][o]);
      if (a.sine_mode == SINE_ROTATOR) {
        for (int o = e_low6; o < e_static; ++o) static_rot(s_order[b][o]);
      } else {
        // the next tone's set-up before this tone's loop
        RunPoly nx = {0, 0, 0, 0};
        float nA = 0.f;
        if (e_low6 < e_static) {
          const Desc& d = s_desc[b][s_order[b][e_low6]];
          nx = static_state(d);
          nA = d.A;
        }
        for (int o = e_low6; o < e_static; ++o) {
          const RunPoly q = nx;
          const float A = nA;
          const Desc& d = s_desc[b][s_order[b][min(o + 1, e_static - 1)]];
          nx = static_state(d);
          nA = d.A;
          static_loop<SPT>(q.p, q.f, A, acc);
        }
      }
      for (int o = e_static; o < n_vis; ++o) {
        const int i = s_order[b][o], kind = s_kind[b][o];
        if (kind == DESC_STATIC) {
          static_sfu(i);
        } else if (kind == DESC_STATIC_ROT) {
          static_rot(i);
        } else if (kind == DESC_LINEAR) {
          linear(i);
        } else if (kind == DESC_LOW6) {
          low6(i);
        } else if (kind == DESC_LOW3) {
          low3(i);
        } else if (kind == DESC_FLAT3) {
          flat3(i);
        } else if (kind == DESC_MINJERK) {
          // third difference below 2^-33 turn (long ramps): g is constant over the run, the same
          // integers as the loop with h
          const RunPoly q0 = poly_state(record(i), rb, false);
          if (__all_sync(0xffffffffu, q0.h == 0)) chirp(q0, i);
          else cascade<SPT, true>(PARTS > 1 ? advance(q0, r0) : q0, s_desc[b][i].A, acc);
        } else {
          const ToneRec& tr = s_tone[b][i];
          const int64_t n0 = T0 + (int64_t)run * RUN;
          if (kind == DESC_RAMP_STATIC) {
            ramp_loop<SPT, false>(static_state(s_desc[b][i]), ramp_setup(tr, n0 + r0), acc);
          } else if (kind == DESC_RAMP_CHIRP) {
            const RunPoly q = poly_state(record(i), rb, (tr.flags & TONE_LINEAR) != 0);
            ramp_loop<SPT, true>(advance(q, r0), ramp_setup(tr, n0 + r0), acc);
          } else {
            mixed_run<SPT>(tr, &record(i), rb, acc, n0, (int)r0, a.exact_tab);
          }
        }
      }
    }
    if constexpr (!ONCE) {
      if (!__syncthreads_and(ok)) {   // stage buffers free, next stage's descriptors visible
        fail_stage = st;
        break;
      }
      if (tid < 32 && st + 2 < n_stages) issue_tones(st + 2);
    }
  }
  if (fail_stage >= 0) {
    // report, then let every copy still in flight land (bounded) before shared memory goes away
    if (tid == 0) {
      atomicExch(a.status, STATUS_TIMEOUT);
      for (int bb = 0; bb < 4; ++bb) {
        const uint32_t cnt_b = (issued >> (8 * bb)) & 0xffu;
        if (cnt_b > 0) (void)mbar_wait(&s_bar[bb], (cnt_b - 1) & 1u);
      }
    }
    __syncthreads();
  }

  if constexpr (!CLUSTER) {
    static_assert(sizeof(StageBuf) >= OUT_STAGE * sizeof(float), "the stage buffers hold the staged samples");
    tile_epilogue_split<SPT>(a, unit, crank, split, P0, (run - part * G::PRUNS) * RUN + (int)r0, acc,
                             reinterpret_cast<float*>(&s_buf));
  } else {
    // partial sums -> shared memory ([i][thread], sample RUN thread + i), then the cluster-wide
    // sum in rank order
#pragma unroll
    for (int r = 0; r < RUN / 2; ++r) {
      s_red[(2 * r) * RT + tid] = acc[r].x;
      s_red[(2 * r + 1) * RT + tid] = acc[r].y;
    }
    cluster.sync();

    // this CTA reduces and stores samples [lo, hi) of the tile; thread t takes `per` consecutive ones
    const int lo = (int)((int64_t)TILE * crank / split), hi = (int)((int64_t)TILE * (crank + 1) / split);
    const int per = (hi - lo + RT - 1) / RT;
    const int s_first = lo + tid * per;
    float xs[RUN];
#pragma unroll
    for (int u = 0; u < RUN; ++u) xs[u] = 0.f;
    for (int c = 0; c < split; ++c) {
      const float* rem = cluster.map_shared_rank(s_red, c);
#pragma unroll
      for (int u = 0; u < RUN; ++u) {
        const int sidx = s_first + u;
        if (u < per && sidx < hi) xs[u] += rem[(sidx % RUN) * RT + sidx / RUN];
      }
    }
    cluster.sync();   // remote reads done before any CTA of the cluster exits

    // scale, round half to even, clamp, store the window part
#pragma unroll
    for (int u = 0; u < RUN; ++u) {
      const int sidx = s_first + u;
      if (u < per && sidx < hi) store_sample(a, T0 + sidx, xs[u]);
    }
    mark_end(a.end);
  }
}

// Register budgets, by CTAs per SM.  Whole tiles: six (80 registers, 52 bytes of spill loads); the
// 1000-chirp 35 ms record takes 2524 us at six, 2599 at seven (72 registers), 2587 at five; the batched
// and cluster renders keep five (no spills).  Parts need fewer accumulators: eight, but six where the
// CTA forms its records (at eight 1.2 KB of spills).  A kernel per mode: with the list's code in it the
// plain render's record takes 2539 us where it takes 2534 without (before the stage buffers lay in one
// object 2640 and 2616).
#define AWG_RENDER_MIN_BLOCKS 5
#define AWG_RENDER_SPLIT_MIN_BLOCKS 6
#define AWG_RENDER_PART_MIN_BLOCKS 8
__global__ void __launch_bounds__(RT, AWG_RENDER_MIN_BLOCKS) render_kernel(const __grid_constant__ RenderArgs a) {
  mark_start(a.start);
  cg::cluster_group cluster = cg::this_cluster();
  render_tile<RUN, true, MODE_ALL>(a, blockIdx.x / a.split, (int)cluster.block_rank(), a.split);
}

// The same without clusters (a.part set when split > 1): CTA blockIdx.x takes rank blockIdx.x % split.
template <int SPT, int MODE>
__global__ void __launch_bounds__(RT, SPT == RUN || MODE == MODE_ONCE ? AWG_RENDER_SPLIT_MIN_BLOCKS : AWG_RENDER_PART_MIN_BLOCKS)
    render_split_kernel(const __grid_constant__ RenderArgs a) {
  mark_start(a.start);
  render_tile<SPT, false, MODE>(a, blockIdx.x / a.split, blockIdx.x % a.split, a.split);
}

// All channels of a multiplexed render in one grid (the channels' arguments differ, so the kernel reads
// them by channel; the loops are render_split_kernel's).
template <int SPT, int MODE>
__global__ void __launch_bounds__(RT, SPT == RUN || MODE == MODE_ONCE ? AWG_RENDER_SPLIT_MIN_BLOCKS : AWG_RENDER_PART_MIN_BLOCKS)
    render_mux_kernel(const __grid_constant__ MuxArgs m) {
  int c = 0;
  while (c + 1 < m.n && (int)blockIdx.x >= m.first[c + 1]) ++c;
  const RenderArgs& a = m.a[c];
  const int i = (int)blockIdx.x - m.first[c];
  if (a.start && i == 0 && threadIdx.x == 0) *a.start = global_ns();
  render_tile<SPT, false, MODE>(a, i / a.split, i % a.split, a.split);
}

// Several renders in one grid (continuous batching): CTA group i (split CTAs) renders window tile
// items[i].y of request items[i].x; every request of the launch has the same tone split.  The
// split sums through each request's scratch (reqs[i].part and .tile_ctr, counters zero at
// launch); CTA blockIdx.x takes rank blockIdx.x % split.
__global__ void __launch_bounds__(RT, AWG_RENDER_MIN_BLOCKS) render_batch_split_kernel(const RenderArgs* __restrict__ reqs,
                                                                                       const int2* __restrict__ items,
                                                                                       int split) {
  const int2 it = items[blockIdx.x / split];
  render_tile<RUN, false, MODE_LIST>(reqs[it.x], it.y, (int)(blockIdx.x % split), split);
}

// The 32-bit phase the render feeds to the sine for sample s of the tile [T0, T0 + TILE) (any
// segment), by the same integer steps as the render's loops: run j = s / RUN, sample r = s % RUN.
// role: 0 the tone's own run set-up, 1 / 2 the first / second tone of a lane pair sharing its
// set-up (the first tone's state is the odd lanes' partner state, the second's the even lanes').
__device__ __noinline__ uint32_t phase32_at(const ToneRec& t, const TileRec* rec, const ChirpRec* chirps, int64_t T0,
                                            int s, const uint64_t (*inv)[3], int role = 0) {
  const int j = s / RUN, r = s % RUN;
  const int64_t n0 = T0 + (int64_t)j * RUN, n = T0 + s;
  const uint32_t ur = (uint32_t)r;
  const uint32_t c2 = ur * (ur - 1) / 2, c3 = (r >= 3) ? ur * (ur - 1) * (ur - 2) / 6 : 0u;
  if (t.slot < 0 || n < t.n_s) return static_p0(t.phi_ref, t.F, n0) + ur * static_f(t.F);
  if (n > t.n_e) return static_p0(t.phi_post_ref, t.F_end, n0) + ur * static_f(t.F_end);
  if (t.flags & TONE_EXACT) return (uint32_t)((exact_chirp_word(chirps[t.slot], n - t.n_s, inv) + P_OFFSET) >> 32);
  const bool ramp_in_tile = (t.flags & TONE_AMP_RAMP) && T0 + TILE - 1 > t.a_ns && T0 < t.a_ns + t.a_L;
  const bool inside = T0 >= t.n_s && T0 + TILE - 1 <= t.n_e;
  RunPoly q;
  if (!ramp_in_tile && inside) {   // the tile's kind decides the set-up (LOW6 leaves terms out)
    const int kind = chirp_inside_kind(t.flags);
    const bool odd = (j & 1) != 0;
    // a shared set-up: the lane of the other parity evaluated it one run away
    const bool moved = (role == 1 && odd) || (role == 2 && !odd);
    const int js = moved ? (odd ? j - 1 : j + 1) : j;
    const RunBin b = run_binomials(js);
    q = kind == DESC_LOW3 ? poly_state_low3(*rec, b)
        : kind == DESC_LOW6 ? poly_state_low6(*rec, b)
        : kind == DESC_FLAT3 ? poly_state_flat3(*rec, b) : poly_state(*rec, b, kind == DESC_LINEAR);
    if (moved) {
      if (odd) {
        q.p = q.p + 32u * q.f + 496u * q.g;
        q.f = q.f + 32u * q.g;
      } else {
        q.p = q.p - 32u * q.f + 528u * q.g;
        q.f = q.f - 32u * q.g;
      }
    }
  } else {
    const RunBin b = run_binomials(j);
    q = poly_state(*rec, b, (t.flags & TONE_LINEAR) != 0);
  }
  return q.p - HALF_TURN + ur * q.f + c2 * q.g + c3 * q.h;
}

// Exact phase words of the first n tones at one sample (test hook).
__global__ void phase_words_kernel(const __grid_constant__ PhaseArgs a) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= a.n) return;
  a.out[k] = exact_word(a.tones[k], a.chirps, a.sample, a.inv_odd);
}

// Exact per-sample 32-bit phases of a short chirp (TONE_EXACT), m = 0..L.
__global__ void exact_table_kernel(const __grid_constant__ TableArgs a, int64_t L) {
  const int64_t m = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (m > L) return;
  a.out[m] = (uint32_t)((exact_chirp_word(a.chirps[a.slot], m, a.inv_odd) + P_OFFSET) >> 32);
}

// Whether tone k shares its run set-up in tile T0 of a render without a tone list or the tensor-
// core engine, by the render's own visit: the CTA whose tone range [K c / split, K (c + 1) / split)
// holds k, its stage of STAGE tones, and k's place among the stage's tones of its sharing group
// (in tone order, taken two at a time).  0: own set-up, 1 / 2: first / second tone of a pair.
__device__ __noinline__ int pair_role(const TraceArgs& a, int k, int64_t T0) {
  if (a.listed || !(a.tones[k].flags & TONE_PAIR)) return 0;
  const int g = visit_group(tile_kind(a.tones[k], T0, false), false, true);
  if (g != GRP_LIN_PAIR && g != GRP_LOW3_PAIR && g != GRP_LOW6_PAIR) return 0;
  const int64_t K = a.K, S = a.split;
  int c = (int)((int64_t)k * S / K);
  while (c + 1 < S && K * (c + 1) / S <= k) ++c;
  while (c > 0 && K * c / S > k) --c;
  const int lb = (int)(K * c / S), le = (int)(K * (c + 1) / S);
  const int s0 = lb + (k - lb) / STAGE * STAGE, s1 = min(s0 + STAGE, le);
  int pos = 0, n = 0;
  for (int u = s0; u < s1; ++u) {
    const ToneRec& t = a.tones[u];
    if (visit_group(tile_kind(t, T0, false), false, (t.flags & TONE_PAIR) != 0) != g) continue;
    if (u == k) pos = n;
    ++n;
  }
  if (pos & 1) return 2;
  return pos + 1 < n ? 1 : 0;
}

// The render's per-sample 32-bit phases of one tone (test hook).
__global__ void trace_kernel(const __grid_constant__ TraceArgs a) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= a.count) return;
  const int64_t n = a.n0 + i;
  const int64_t tile_abs = n / TILE;
  const int64_t T0 = tile_abs * TILE;
  const ToneRec t = a.tones[a.tone];
  const TileRec* rec = nullptr;
  if (classify_tile(t, T0) == TILE_CHIRP && !(t.flags & TONE_EXACT))
    rec = a.recs + (tile_abs - a.tile0);   // the one active chirp of the window
  a.out[i] = phase32_at(t, rec, a.chirps, T0, (int)(n - T0), a.inv_odd, pair_role(a, a.tone, T0));
}

}  // namespace

int device_sm_count() {
  constexpr int MAX_DEV = 64;
  static std::atomic<int> cache[MAX_DEV];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEV) return 1;
  int n = cache[dev].load(std::memory_order_relaxed);
  if (n > 0) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) return 1;
  cache[dev].store(n, std::memory_order_relaxed);
  return n;
}

// The render kernel that cuts a tile over `parts` CTAs.
typedef void (*SplitKernel)(const RenderArgs);
template <int MODE>
static SplitKernel split_kernel_of(int parts) {
  return parts == 4 ? render_split_kernel<8, MODE> : parts == 2 ? render_split_kernel<16, MODE> : render_split_kernel<32, MODE>;
}
static SplitKernel split_kernel(int parts, int mode) {
  return mode == MODE_ONCE ? split_kernel_of<MODE_ONCE>(parts)
         : mode == MODE_LIST ? split_kernel_of<MODE_LIST>(parts) : split_kernel_of<MODE_ALL>(parts);
}

typedef void (*MuxKernel)(const MuxArgs);
static MuxKernel mux_kernel(int parts, bool once) {
  if (once)
    return parts == 4 ? render_mux_kernel<8, MODE_ONCE> : parts == 2 ? render_mux_kernel<16, MODE_ONCE> : render_mux_kernel<32, MODE_ONCE>;
  return parts == 4 ? render_mux_kernel<8, MODE_ALL> : parts == 2 ? render_mux_kernel<16, MODE_ALL> : render_mux_kernel<32, MODE_ALL>;
}

cudaError_t render_setup_attributes() {
  cudaError_t e = cudaFuncSetAttribute(render_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  // shared memory before L1 for AWG_RENDER_SPLIT_MIN_BLOCKS CTAs
  for (int parts = 1; parts <= MAX_PARTS; parts *= 2)
    for (int mode = 0; mode < N_MODES; ++mode)
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(split_kernel(parts, mode), cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  for (int parts = 1; parts <= MAX_PARTS; parts *= 2)
    for (bool once : {false, true})
      if (e == cudaSuccess)
        e = cudaFuncSetAttribute(mux_kernel(parts, once), cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  return e;
}

cudaError_t launch_render_batch_split(const RenderArgs* reqs, const int2* items, int n_items, int split,
                                      cudaStream_t s) {
  if (n_items == 0) return cudaSuccess;
  render_batch_split_kernel<<<(unsigned)(n_items * split), RT, 0, s>>>(reqs, items, split);
  return cudaGetLastError();
}

// A launch configuration with programmatic stream serialisation: the kernel may start before the
// preceding one of the stream has completed (it then waits where it has to, pdl_wait).
struct PdlLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  PdlLaunch(unsigned grid, unsigned block, cudaStream_t s) {
    cfg.gridDim = dim3(grid, 1, 1);
    cfg.blockDim = dim3(block, 1, 1);
    cfg.stream = s;
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
  }
};

cudaError_t launch_prep(const PrepArgs& a, cudaStream_t s) {
  const int64_t total = (int64_t)a.n_active * a.n_tiles;
  if (total == 0) return cudaSuccess;
  const PdlLaunch l((unsigned)((total + 127) / 128), 128, s);
  if (a.n_active <= SMALL_PREP) {   // the small parameter form: fewer bytes copied with the launch
    PrepArgsT<SMALL_PREP> b;
    b.chirps = a.chirps;
    b.tones = a.tones;
    b.recs = a.recs;
    b.act_of_slot = a.act_of_slot;
    b.tile0 = a.tile0;
    b.n_tiles = a.n_tiles;
    b.n_active = a.n_active;
    b.act_base = a.act_base;
    b.rec_stride = a.rec_stride;
    b.start = a.start;
    b.more = a.more;
    for (int q = 0; q < 7; ++q)
      for (int i = 0; i < 7; ++i) b.W[q][i] = a.W[q][i];
    for (int q = 0; q < 3; ++q)
      for (int i = 0; i < 3; ++i) b.inv_odd[q][i] = a.inv_odd[q][i];
    for (int i = 0; i < a.n_active; ++i) b.slots[i] = a.slots[i];
    return cudaLaunchKernelEx(&l.cfg, prep_kernel<PrepArgsT<SMALL_PREP>>, b);
  }
  return cudaLaunchKernelEx(&l.cfg, prep_kernel<PrepArgs>, a);
}

// Replay of a periodic record of 2^log2 samples, written at a stride (multiplexed channels):
// out[i * stride] = table[(c + i) mod period].
__global__ void replay_strided_kernel(const int16_t* __restrict__ tab, uint64_t mask, int64_t c, int64_t n,
                                      int16_t* __restrict__ out, int32_t stride, unsigned long long* start,
                                      unsigned long long* end) {
  mark_start(start);
  pdl_wait();
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += step)
    out[i * stride] = tab[((uint64_t)c + (uint64_t)i) & mask];
  mark_end(end);
}

// The same for a plain output, bound by the samples written (2 bytes each).  `out` is the first 16-byte
// boundary of the output, `head` samples into it; its vector v (8 samples) is the table's samples
// 8 (v0 + v) + SHIFT .. + 7 mod period, SHIFT = shift samples.  A thread takes vectors u of one period
// and writes each to its REPS repeats u, u + P, u + 2 P ... (P vectors per period), so a record that
// repeats is read from the L2 once per REPS writes: 2^27 samples of a 2^24 table 52 -> 45.6 us among others
// (58.5 while timed events stood between the kernels; reading the table for every vector ran at 5.4 TB/s
// written, plain fills at 6.9).  Streaming stores keep the
// table in the L2.  Samples before `out` and after its last whole vector are copied one by one.
constexpr int REPLAY_VEC = 2, REPLAY_REPS = 8;
__global__ void __launch_bounds__(256) replay_kernel(const int16_t* __restrict__ tab, uint64_t mask, int64_t c, int64_t n,
                                                     int16_t* __restrict__ out, int head, unsigned long long* start,
                                                     unsigned long long* end) {
  mark_start(start);
  const uint64_t P = (mask + 1) >> 3;
  const int64_t nv = (n - head) >> 3;
  const uint64_t c1 = (uint64_t)c + (uint64_t)head, v0 = c1 >> 3;
  const int shift = (int)(c1 & 7);
  const int64_t span = min((int64_t)P, nv);   // vectors of the first period
  const uint4* t4 = reinterpret_cast<const uint4*>(tab);
  const int64_t u0 = (int64_t)blockIdx.x * (blockDim.x * REPLAY_VEC) + threadIdx.x;
  uint4 x[REPLAY_VEC];
#pragma unroll
  for (int j = 0; j < REPLAY_VEC; ++j) {
    const int64_t u = u0 + (int64_t)j * blockDim.x;
    if (u >= span) continue;
    x[j] = __ldg(t4 + ((v0 + (uint64_t)u) & (P - 1)));
    if (shift) {   // the vector straddles two of the table's
      const uint4 y = __ldg(t4 + ((v0 + (uint64_t)u + 1) & (P - 1)));
      const uint32_t w[8] = {x[j].x, x[j].y, x[j].z, x[j].w, y.x, y.y, y.z, y.w};
      uint32_t o[5];
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        o[i] = w[i];
        if (i + 1 < 8 && (shift >> 1) >= 1) o[i] = w[i + 1 < 8 ? i + 1 : 7];
        if (i + 2 < 8 && (shift >> 1) >= 2) o[i] = w[i + 2 < 8 ? i + 2 : 7];
        if ((shift >> 1) >= 3) o[i] = w[i + 3 < 8 ? i + 3 : 7];
      }
      if (shift & 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) o[i] = __funnelshift_r(o[i], o[i + 1], 16);
      }
      x[j] = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
  pdl_wait();
  uint4* o4 = reinterpret_cast<uint4*>(out);
  for (int64_t r0 = (int64_t)blockIdx.y * REPLAY_REPS; r0 * (int64_t)P < nv; r0 += (int64_t)gridDim.y * REPLAY_REPS) {
#pragma unroll
    for (int r = 0; r < REPLAY_REPS; ++r) {
#pragma unroll
      for (int j = 0; j < REPLAY_VEC; ++j) {
        const int64_t u = u0 + (int64_t)j * blockDim.x, v = u + (r0 + r) * (int64_t)P;
        if (u < span && v < nv) __stcs(o4 + v, x[j]);
      }
    }
  }
  if (blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x < 16) {   // up to 7 samples at either end
    const int64_t tail = n - head - 8 * nv;
    const int t = (int)threadIdx.x;
    if (t < head) out[t - head] = tab[((uint64_t)c + (uint64_t)t) & mask];
    else if (t >= 8 && t - 8 < tail) out[8 * nv + t - 8] = tab[(c1 + 8 * (uint64_t)nv + (uint64_t)(t - 8)) & mask];
  }
  mark_end(end);
}

cudaError_t launch_replay(const int16_t* tab, int32_t log2_len, int64_t c, int64_t n, int16_t* out, int32_t stride,
                          unsigned long long* start, unsigned long long* end, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const uint64_t mask = ((uint64_t)1 << log2_len) - 1;
  if (stride != 1) {
    const int64_t blocks = std::min<int64_t>((n + 255) / 256, (int64_t)device_sm_count() * 16);
    const PdlLaunch l((unsigned)blocks, 256, s);
    return cudaLaunchKernelEx(&l.cfg, replay_strided_kernel, tab, mask, c, n, out, stride, start, end);
  }
  const int head = (int)std::min<int64_t>(n, (int64_t)((16 - ((uintptr_t)out & 15)) & 15) / 2);
  const int64_t P = (int64_t)(mask + 1) / 8, nv = (n - head) / 8, span = std::max<int64_t>(1, std::min(P, nv));
  PdlLaunch l((unsigned)((span + 256 * REPLAY_VEC - 1) / (256 * REPLAY_VEC)), 256, s);
  l.cfg.gridDim.y = (unsigned)std::max<int64_t>(1, std::min<int64_t>(65535, (nv + P * REPLAY_REPS - 1) / (P * REPLAY_REPS)));
  return cudaLaunchKernelEx(&l.cfg, replay_kernel, tab, mask, c, n, out + head, head, start, end);
}

// The tensor-core engine's two sums of a window, formed side by side (awg_host.cpp, render_engine):
// the render's (part) plus the GEMM's (base), quantised and stored as the render's own epilogue
// would.  10 bytes per sample; 8 samples per thread, 16-byte accesses where the outputs allow.
__global__ void __launch_bounds__(256) combine_kernel(const float* __restrict__ part, const float* __restrict__ base,
                                                      int64_t n, float scale, int16_t* __restrict__ out_q, int32_t q_stride,
                                                      float* __restrict__ out_f, int vec, unsigned long long* end) {
  const int64_t i0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 8;
  if (vec && i0 + 8 <= n) {
    float x[8];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 p = __ldg(reinterpret_cast<const float4*>(part + i0) + h), b = __ldg(reinterpret_cast<const float4*>(base + i0) + h);
      x[4 * h] = p.x + b.x;
      x[4 * h + 1] = p.y + b.y;
      x[4 * h + 2] = p.z + b.z;
      x[4 * h + 3] = p.w + b.w;
    }
    if (out_f) {
#pragma unroll
      for (int h = 0; h < 2; ++h)
        reinterpret_cast<float4*>(out_f + i0)[h] = make_float4(x[4 * h], x[4 * h + 1], x[4 * h + 2], x[4 * h + 3]);
    }
    if (out_q) {
      uint32_t w[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float q0 = fminf(fmaxf(rintf(x[2 * u] * scale), -32767.f), 32767.f);
        const float q1 = fminf(fmaxf(rintf(x[2 * u + 1] * scale), -32767.f), 32767.f);
        w[u] = (uint32_t)(uint16_t)(int16_t)q0 | ((uint32_t)(uint16_t)(int16_t)q1 << 16);
      }
      *reinterpret_cast<uint4*>(out_q + i0) = make_uint4(w[0], w[1], w[2], w[3]);
    }
  } else {
    for (int64_t i = i0; i < min(i0 + 8, n); ++i) {
      const float x = part[i] + base[i];
      if (out_f) out_f[i] = x;
      if (out_q) out_q[i * q_stride] = (int16_t)fminf(fmaxf(rintf(x * scale), -32767.f), 32767.f);
    }
  }
  mark_end(end);
}

cudaError_t launch_combine(const float* part, const float* base, int64_t n, float scale, int16_t* out_q, int32_t q_stride,
                           float* out_f, unsigned long long* end, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  const int vec = (!out_q || (q_stride <= 1 && ((uintptr_t)out_q & 15) == 0)) && ((uintptr_t)out_f & 15) == 0;
  combine_kernel<<<(unsigned)((n + 2047) / 2048), 256, 0, s>>>(part, base, n, scale, out_q, q_stride > 1 ? q_stride : 1, out_f,
                                                              vec, end);
  return cudaGetLastError();
}

// End of a pipelined sequence: returns once every render CTA of the sequence has stored its
// samples (*exit_ctr >= target), so that later work in the stream sees all of them.  Gives up after
// limit_ns, sets the status word to AWG_ETIMEOUT and returns.  The end of the call's device time is the
// join's: a CTA that has counted itself in may still be on its way to a stamp of its own.
__global__ void join_kernel(const unsigned long long* exit_ctr, unsigned long long target, int32_t* status,
                            uint64_t limit_ns, unsigned long long* end) {
  if (!wait_counter(exit_ctr, target, limit_ns)) atomicExch(status, STATUS_TIMEOUT);
  __threadfence();
  mark_end(end);
}

cudaError_t launch_join(const unsigned long long* exit_ctr, unsigned long long target, int32_t* status,
                        uint64_t limit_ns, unsigned long long* end, cudaStream_t s) {
  join_kernel<<<1, 1, 0, s>>>(exit_ctr, target, status, limit_ns, end);
  return cudaGetLastError();
}

cudaError_t launch_render(const RenderArgs& a, cudaStream_t s) {
  if (a.n_tiles == 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  const int parts = a.cluster ? 1 : a.parts;
  cfg.gridDim = dim3((unsigned)(a.n_tiles * parts * a.split), 1, 1);
  cfg.blockDim = dim3(RT, 1, 1);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)a.split;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  if (!a.cluster) {   // the split sums through the scratch partials
    cfg.attrs = attr + 1;
    cfg.numAttrs = a.pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, split_kernel(parts, a.once ? MODE_ONCE : a.tone_list || a.skip_static ? MODE_LIST : MODE_ALL), a);
  }
  cfg.attrs = attr;
  cfg.numAttrs = a.pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, render_kernel, a);
}

// A list covers its whole window, but groups of tones that chirp in turn are live in a few tiles each:
// one CTA per tile keeps the listed tones that are not static there, in order, and notes where each
// rank's share begins.  Without it every render CTA searched the list (4 us) and staged all its
// listed tones to skip most of them.
__global__ void __launch_bounds__(128) sift_kernel(const __grid_constant__ SiftArgs a) {
  __shared__ int s_live[4];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t T0 = (a.tile0 + blockIdx.x) * (int64_t)TILE;
  int32_t* row = a.rows + (int64_t)blockIdx.x * a.n_list;
  int32_t* first = a.first + (int64_t)blockIdx.x * (a.split + 1);
  int count = 0;     // live tones so far
  for (int i0 = 0; i0 < a.n_list; i0 += 128) {
    const int i = i0 + tid;
    const int k = i < a.n_list ? a.list[i] : -1;
    const bool live = k >= 0 && !tile_static(a.tones[k], T0);
    const unsigned m = __ballot_sync(0xffffffffu, live);
    if (lane == 0) s_live[warp] = __popc(m);
    __syncthreads();
    int at = count + __popc(m & ((1u << lane) - 1u));
    for (int w = 0; w < 4; ++w) {
      if (w < warp) at += s_live[w];
      count += s_live[w];
    }
    if (live) row[at] = k;
    __syncthreads();
  }
  // rank boundaries (the row is ascending, its entries visible after the last barrier)
  const int key = tid <= a.split ? a.bounds[tid] : 0;
  int lo = 0, hi = count;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (row[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  if (tid <= a.split) first[tid] = lo;
}

cudaError_t launch_sift(const SiftArgs& a, cudaStream_t s) {
  if (a.n_tiles == 0) return cudaSuccess;
  sift_kernel<<<(unsigned)a.n_tiles, 128, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_render_mux(const MuxArgs& m, bool once, cudaStream_t s) {
  const PdlLaunch l((unsigned)m.first[m.n], RT, s);
  return cudaLaunchKernelEx(&l.cfg, mux_kernel(m.a[0].parts, once), m);
}

cudaError_t launch_exact_table(const TableArgs& a, int64_t L, cudaStream_t s) {
  const int64_t n = L + 1;
  exact_table_kernel<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(a, L);
  return cudaGetLastError();
}

cudaError_t launch_phase_words(const PhaseArgs& a, cudaStream_t s) {
  if (a.n == 0) return cudaSuccess;
  phase_words_kernel<<<(a.n + 127) / 128, 128, 0, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_trace(const TraceArgs& a, cudaStream_t s) {
  if (a.count == 0) return cudaSuccess;
  trace_kernel<<<(a.count + 127) / 128, 128, 0, s>>>(a);
  return cudaGetLastError();
}

// The rate the SFU sustains in the render's own static loop (a measured ceiling for the sine
// roofline): every thread runs `runs` runs of RUN samples of one static tone through static_loop,
// with no staging, set-up or split sum, and writes the sum of its partial sums (so that nothing
// is optimised away).  One sine per sample: blocks x RT x runs x RUN sines per launch.
__global__ void __launch_bounds__(RT, AWG_RENDER_MIN_BLOCKS) sfu_rate_kernel(float* __restrict__ out, int runs) {
  const uint32_t id = blockIdx.x * RT + threadIdx.x;
  uint32_t p = id * 0x9E3779B9u;
  const uint32_t f = (id * 0x85EBCA6Bu) | 1u;
  const float A = 1e-3f;
  Acc<RUN> acc;
#pragma unroll
  for (int r = 0; r < RUN / 2; ++r) acc[r] = make_float2(0.f, 0.f);
  for (int k = 0; k < runs; ++k) {
    static_loop<RUN>(p, f, A, acc);
    p += (uint32_t)RUN * f;
  }
  float t = 0.f;
#pragma unroll
  for (int r = 0; r < RUN / 2; ++r) t += acc[r].x + acc[r].y;
  out[id] = t;
}

cudaError_t launch_sfu_rate(float* out, int blocks, int runs, cudaStream_t s) {
  sfu_rate_kernel<<<blocks, RT, 0, s>>>(out, runs);
  return cudaGetLastError();
}

// The same for the render's chirp loop (cascade without h, the loop of linear and LOW6 chirps):
// each run takes a chirp state (p, f, g) from the thread's id, one sine per sample.
__global__ void __launch_bounds__(RT, AWG_RENDER_MIN_BLOCKS) chirp_rate_kernel(float* __restrict__ out, int runs) {
  const uint32_t id = blockIdx.x * RT + threadIdx.x;
  RunPoly q;
  q.p = id * 0x9E3779B9u;
  q.f = (id * 0x85EBCA6Bu) | 1u;
  q.g = (id * 0xC2B2AE35u) >> 8;
  q.h = 0;
  const float A = 1e-3f;
  Acc<RUN> acc;
#pragma unroll
  for (int r = 0; r < RUN / 2; ++r) acc[r] = make_float2(0.f, 0.f);
  for (int k = 0; k < runs; ++k) {
    cascade<RUN, false>(q, A, acc);
    q.p += 32u * q.f + 496u * q.g;   // the state after the run
    q.f += 32u * q.g;
  }
  float t = 0.f;
#pragma unroll
  for (int r = 0; r < RUN / 2; ++r) t += acc[r].x + acc[r].y;
  out[id] = t;
}

cudaError_t launch_chirp_rate(float* out, int blocks, int runs, cudaStream_t s) {
  chirp_rate_kernel<<<blocks, RT, 0, s>>>(out, runs);
  return cudaGetLastError();
}

}  // namespace awgk
