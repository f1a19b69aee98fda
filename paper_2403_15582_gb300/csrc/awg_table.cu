// Periodic multi-tone table as a split-precision tensor-core GEMM (tcgen05, sm_103a).
//
// For tones on the f_s / 2^log2_len grid (Eq. freqapprox) the record of N = 2^log2_len samples is
// periodic.  With n = n1 * NB + n2 (NB = 256) and the angle-addition identity,
//   x[n] = sum_k A_k sin(a_k(n1) + b_k(n2))
//        = sum_k [A_k sin a_k(n1)] cos b_k(n2) + [A_k cos a_k(n1)] sin b_k(n2),
// a_k(n1) = 2 pi (Phi0_k + n1 NB F_k) / 2^64 and b_k(n2) = 2 pi n2 F_k / 2^64 from exact 64-bit
// phase words.  That is a GEMM X[M = N/NB, NB] = Aop[M, 2K] * Bop[2K, NB].  Each operand is split
// into hi + lo in BF16 (or FP16); the kernel accumulates hi*hi + hi*lo + lo*hi in FP32 in tensor
// memory and quantises in the epilogue.
//
// Kernel structure: a cluster of S CTAs per 128-row tile of X splits the K dimension (fewer FP32
// accumulations per chain); each CTA (320 threads) has a 2-stage ring of
// {A_hi, A_lo (128 x 64), B_hi, B_lo (256 x 64)} tiles in the 128-byte-swizzled K-major layout:
//   warp 0   TMA producer of the B tiles (prepared once per call, 256 x 2K, L2-resident),
//            mbarrier transaction counts
//   warp 1   allocates 512 TMEM columns; lane 0 issues tcgen05.mma (M 128, N 256, K 16) x 3 passes
//            x 4 k-steps per stage, commits each stage back to the producers
//   warps 2-9 generate the A tiles in shared memory (one tone per lane, every eighth row per warp:
//            A_k sin a_k(n1), A_k cos a_k(n1) from the exact phase word, SFU sine and cosine, hi + lo
//            split), so the M x 2K A
//            operand never exists in HBM; then the epilogue: tcgen05.ld 32x32b of both
//            accumulators (warp w reads TMEM lane quarter w mod 4, half of the columns) into a
//            padded FP32 partial tile in shared memory; the cluster sums the S
//            partial tiles through distributed shared memory in rank order, and each CTA scales,
//            rounds, clamps and stores its rows.
// Every wait is bounded (about 2 s); on a timeout the CTA records AWG_ETIMEOUT, lets in-flight
// copies and MMAs drain (bounded), frees its TMEM and exits.
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>

#include "awg_internal.h"

namespace cg = cooperative_groups;

namespace awgk {

namespace {

constexpr int TM = 128;               // rows of X per CTA (UMMA M)
constexpr int TN = 256;               // NB: columns of X (UMMA N)
constexpr int TK = 64;                // K elements per stage (128 bytes of 16-bit values)
constexpr int NSTAGE = 2;
// A-operand generator warps (rows g, g + NGEN, ...): eight keep the tensor pipe fed (four left the
// MMAs waiting for the A tiles: 1.44 -> 1.29 ms on the 10,000-tone 2^24 table; sixteen, no faster)
constexpr int NGEN = 8;
constexpr int GEMM_THREADS = 32 * (2 + NGEN);
static_assert(NGEN % 4 == 0 && TM % NGEN == 0, "generator warps cover every TMEM lane quarter and every row");
constexpr uint32_t A_TILE = TM * TK * 2;   // 16 KB
constexpr uint32_t B_TILE = TN * TK * 2;   // 32 KB
constexpr uint32_t STAGE_BYTES = 2 * A_TILE + 2 * B_TILE;   // 96 KB
constexpr int STATUS_TIMEOUT = -4;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ uint64_t now_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  if (mbar_try(bar, parity)) return true;
  const uint64_t t0 = now_ns();
  while (!mbar_try(bar, parity))
    if (now_ns() - t0 > 2000000000ull) return false;
  return true;
}

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(map), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor: K-major tile with 128-byte rows, 128-byte swizzle, 8-row groups
// 1024 bytes apart (stride byte offset), descriptor version 1.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)1 << 16;                 // leading byte offset (unused for swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;       // stride byte offset
  d |= (uint64_t)1 << 46;                 // version
  d |= (uint64_t)2 << 61;                 // 128-byte swizzle
  return d;
}

__device__ __forceinline__ void mma_f16(uint32_t tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

constexpr int PART_STRIDE = TN + 1;   // padded row of a partial tile (conflict-free column writes)

struct TableGemmArgs {
  int32_t n_kb;          // K blocks of TK (all CTAs of a cluster together)
  int16_t* out_q;
  float* out_f;
  float scale;           // 32767 / FS
  int32_t* status;
  uint32_t idesc;
  const ToneRec* tones;  // A operand source: phase word, frequency word, amplitude
  int32_t K;
  int32_t nb_log2;       // row n1 starts at sample n1 << nb_log2
  int64_t row_base;      // absolute row of tile row 0 of tile 0
  int64_t win_start, win_end;
  int32_t window_mode;
  float a_scale, inv_a_scale;   // A operand scaling (a power of two) and its inverse
  unsigned long long* end;      // device time of the call's end (null: not taken)
};

template <typename T>
__device__ __forceinline__ uint32_t pack2(float lo, float hi);
template <>
__device__ __forceinline__ uint32_t pack2<__nv_bfloat16>(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
template <>
__device__ __forceinline__ uint32_t pack2<__half>(float lo, float hi) {
  const __half2 v = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
template <typename T>
__device__ __forceinline__ float2 unpack2(uint32_t u);
template <>
__device__ __forceinline__ float2 unpack2<__nv_bfloat16>(uint32_t u) {
  return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xFFFF0000u));
}
template <>
__device__ __forceinline__ float2 unpack2<__half>(uint32_t u) {
  const __half2 v = *reinterpret_cast<const __half2*>(&u);
  return __half22float2(v);
}

// The static engine's A tile of one stage: 16 tones, four columns each (sine and cosine for the
// segment before the tone's chirp, the same for the one after it), 128 rows.  A segment's columns are
// zero in the 4096-sample tiles where the tone is not static in it (tile_segment_static), so every
// (row, tone) holds at most one live segment: one sine and cosine per (row, tone), and one 8-byte
// store per half, a row of 128 bytes per half warp.  Warp g takes the rows 16 g .. 16 g + 15, lane l
// tone l mod 16 and every second row.  (Before, each segment had a lane of its own with 64-bit tile
// compares per row, and the tone records were read after the wait for the stage: 270 us for 10,000
// tones x 2^20; now 177.  At the table's rate the MMAs over 40,000 columns take about 155 of them, and
// half of that multiplies zeros where few tones have a second segment: with 400 chirping tones 20,800
// columns would do.)
//
// The rows of a tone where a segment is live, as rows of this CTA's tile (clamped to 0 .. TM): segment
// 0 in rows < pre, segment 1 in rows >= post, neither in the rows ramp_lo .. ramp_hi - 1 of an
// amplitude ramp; the amplitude is amp before the ramp, amp_end from ramp_hi on.
struct WindowTone {
  uint64_t phi0, F0, phi1, F1;
  int32_t pre, post, ramp_lo, ramp_hi;
  float amp, amp_end;
};
// The first row of a tile (given by its absolute index), relative to the CTA's first row R0.
__device__ __forceinline__ int32_t clamp_row(int64_t tile, int64_t R0) {
  return (int32_t)max((int64_t)0, min((int64_t)TM, tile * (TILE / TN) - R0));
}
__device__ __forceinline__ WindowTone window_tone(const ToneRec* t, float a_scale, int64_t R0) {
  WindowTone w;
  w.phi0 = w.F0 = w.phi1 = w.F1 = 0;
  w.pre = TM;
  w.post = TM;
  w.ramp_lo = w.ramp_hi = TM;
  w.amp = w.amp_end = 0.f;
  if (t) {
    const int32_t flags = t->flags;
    w.phi0 = t->phi_ref;
    w.F0 = t->F;
    w.amp = t->A * a_scale;
    w.amp_end = w.amp;
    if (t->slot >= 0) {
      w.phi1 = t->phi_post_ref;
      w.F1 = t->F_end;
      w.pre = clamp_row(t->n_s / TILE, R0);           // T0 + TILE - 1 < n_s
      w.post = clamp_row(t->n_e / TILE + 1, R0);      // T0 > n_e
    }
    if (flags & TONE_AMP_RAMP) {                      // T0 + TILE - 1 > a_ns and T0 < a_ns + a_L
      w.ramp_lo = clamp_row((t->a_ns + 1) / TILE, R0);
      w.ramp_hi = clamp_row((t->a_ns + t->a_L + TILE - 1) / TILE, R0);
      w.amp_end = t->A_end * a_scale;
    }
  }
  return w;
}

// (a sin, a cos) of phase word w as packed hi and lo halves.  The sine and cosine take the top 32
// bits of the phase word as a signed turn on the SFU (|error| < 5e-7).
template <typename T>
__device__ __forceinline__ void sincos_halves(uint64_t w, float a, uint32_t* hv, uint32_t* lv) {
  float sn, cs;
  __sincosf((float)(int32_t)(w >> 32) * 1.46291807926715968e-9f, &sn, &cs);   // 2 pi / 2^32
  const float sv = a * sn, cv = a * cs;
  *hv = pack2<T>(sv, cv);
  const float2 h = unpack2<T>(*hv);
  *lv = pack2<T>(sv - h.x, cv - h.y);
}

template <typename T>
__device__ __forceinline__ void gen_a_window(const TableGemmArgs& a, const WindowTone& t, int64_t R0, int g, int lane,
                                             uint32_t tile_hi, uint32_t tile_lo) {
  constexpr int ROWS = TM / NGEN;   // rows of a warp
  static_assert(ROWS == 16 && TK / 4 == 16, "a half warp holds the stage's tones");
  const uint32_t r_first = (uint32_t)(ROWS * g + (lane >> 4));
  const uint32_t chunk = (uint32_t)((lane & 15) >> 1), col = (uint32_t)(lane & 1) * 8u;
  const uint64_t f0 = t.F0 << a.nb_log2;
  uint64_t w0 = t.phi0 + (uint64_t)(R0 + r_first) * f0;
  // one live segment and one amplitude in all rows of the tile (a tone whose chirp and ramp lie
  // elsewhere), or none: segment and amplitude are chosen once
  const bool ramp_out = t.ramp_lo >= TM || t.ramp_hi <= 0;
  const bool plain = ramp_out && (t.pre >= TM || t.post <= 0 || (t.pre <= 0 && t.post >= TM));
  auto store = [&](uint32_t r, uint32_t h0, uint32_t h1, uint32_t l0, uint32_t l1) {
    const uint32_t off = r * 128u + ((chunk ^ (r & 7u)) << 4) + col;
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(tile_hi + off), "r"(h0), "r"(h1) : "memory");
    asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(tile_lo + off), "r"(l0), "r"(l1) : "memory");
  };
  if (__all_sync(0xffffffffu, plain)) {
    const bool second = t.post <= 0, live = second || t.pre >= TM;
    const uint64_t f = second ? t.F1 << a.nb_log2 : f0;
    uint64_t w = second ? t.phi1 + (uint64_t)(R0 + r_first) * f : w0;
    const uint64_t step = 2 * f;
    const float amp = live ? (t.ramp_hi <= 0 ? t.amp_end : t.amp) : 0.f;
#pragma unroll
    for (int i = 0; i < ROWS / 2; ++i) {
      uint32_t hv, lv;
      sincos_halves<T>(w, amp, &hv, &lv);
      store(r_first + 2 * i, second ? 0u : hv, second ? hv : 0u, second ? 0u : lv, second ? lv : 0u);
      w += step;
    }
    return;
  }
  const uint64_t f1 = t.F1 << a.nb_log2;
  uint64_t w1 = t.phi1 + (uint64_t)(R0 + r_first) * f1;
#pragma unroll 2
  for (int i = 0; i < ROWS / 2; ++i) {
    const int r = (int)r_first + 2 * i;
    const bool second = r >= t.post;
    const bool live = (second || r < t.pre) && !(r >= t.ramp_lo && r < t.ramp_hi);
    uint32_t hv, lv;
    sincos_halves<T>(second ? w1 : w0, live ? (r >= t.ramp_hi ? t.amp_end : t.amp) : 0.f, &hv, &lv);
    store((uint32_t)r, second ? 0u : hv, second ? hv : 0u, second ? 0u : lv, second ? lv : 0u);
    w0 += 2 * f0;
    w1 += 2 * f1;
  }
}

// Table mode: the A tile of one stage for one generator warp.  Lane j holds tone kt0 + j (its phase
// word, frequency word and scaled amplitude, loaded before; zero amplitude past K), warp g the rows g,
// g + NGEN, ...; for each row n1 it forms the hi and lo halves of (A_k sin a, A_k cos a), a = 2 pi
// (Phi0_k + n1 NB F_k) / 2^64, stepping the exact phase word by NGEN NB F_k from row to row.  The
// pair is one 32-bit word at byte 4 (j mod 4) of 16-byte chunk j / 4 of the row, which the 128-byte
// swizzle moves to chunk (j / 4) ^ (row mod 8).
template <typename T>
__device__ __forceinline__ void gen_a_rows(const TableGemmArgs& a, uint64_t phi, uint64_t F, float A, uint32_t row0,
                                           int g, int lane, uint32_t tile_hi, uint32_t tile_lo) {
  const uint64_t f8 = F << a.nb_log2;
  uint64_t w = phi + (uint64_t)(a.row_base + (int64_t)row0 + g) * f8;
  const uint64_t step = f8 * (uint64_t)NGEN;
  const uint32_t col = (uint32_t)(lane & 3) * 4u;
  const uint32_t chunk = (uint32_t)(lane >> 2);
#pragma unroll 8
  for (int i = 0; i < TM / NGEN; ++i) {
    const uint32_t r = (uint32_t)(g + NGEN * i);
    uint32_t hv, lv;
    sincos_halves<T>(w, A, &hv, &lv);
    const uint32_t off = r * 128u + ((chunk ^ (r & 7u)) << 4) + col;
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(tile_hi + off), "r"(hv) : "memory");
    asm volatile("st.shared.b32 [%0], %1;" ::"r"(tile_lo + off), "r"(lv) : "memory");
    w += step;
  }
}

template <typename T, bool WINDOW>
__global__ void __launch_bounds__(GEMM_THREADS, 1)
    table_gemm_kernel(const __grid_constant__ CUtensorMap mB_hi, const __grid_constant__ CUtensorMap mB_lo,
                      const __grid_constant__ TableGemmArgs a) {
  extern __shared__ uint8_t dyn_smem[];
  __shared__ alignas(8) uint64_t bars[2 * NSTAGE + 1];   // full[2], empty[2], done
  __shared__ uint32_t s_tmem;
  __shared__ volatile int s_fail;

  cg::cluster_group cluster = cg::this_cluster();
  const int split = (int)cluster.num_blocks();
  const int crank = (int)cluster.block_rank();
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const uint32_t base = (smem_u32(dyn_smem) + 1023u) & ~1023u;   // 1024-byte aligned stages
  float* part = reinterpret_cast<float*>(dyn_smem + (base - smem_u32(dyn_smem)));   // reuses the stages
  const uint32_t full0 = smem_u32(&bars[0]), empty0 = smem_u32(&bars[NSTAGE]), done = smem_u32(&bars[2 * NSTAGE]);
  const int row0 = (blockIdx.x / split) * TM;
  const int kb0 = (int)((int64_t)a.n_kb * crank / split), kb1 = (int)((int64_t)a.n_kb * (crank + 1) / split);
  const int n_kb = kb1 - kb0;

  if (threadIdx.x == 0) {
    for (int s = 0; s < NSTAGE; ++s) {
      mbar_init(full0 + 8 * s, 1 + NGEN);   // the B copies' transaction arrive + one per generator warp
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(done, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {   // whole warp: 512 TMEM columns, two 128 x 256 FP32 accumulators
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(2 * TN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = s_tmem;

  if (warp == 0 && lane == 0) {
    // ---------------- TMA producer ----------------
    int issued = 0;
    for (int kb = 0; kb < n_kb; ++kb) {
      const int s = kb % NSTAGE;
      if (kb >= NSTAGE && !mbar_wait(empty0 + 8 * s, (uint32_t)(((kb / NSTAGE) - 1) & 1))) {
        s_fail = 1;
        break;
      }
      if (s_fail) break;
      const uint32_t st = base + (uint32_t)s * STAGE_BYTES;
      mbar_expect_tx(full0 + 8 * s, 2 * B_TILE);
      const int kx = (kb0 + kb) * TK;
      tma_load_2d(st + 2 * A_TILE, &mB_hi, kx, 0, full0 + 8 * s);
      tma_load_2d(st + 2 * A_TILE + B_TILE, &mB_lo, kx, 0, full0 + 8 * s);
      issued = kb + 1;
    }
    if (s_fail) {   // let the copies already issued land (bounded) before the CTA exits
      for (int kb = (issued > NSTAGE ? issued - NSTAGE : 0); kb < issued; ++kb)
        (void)mbar_wait(full0 + 8 * (kb % NSTAGE), (uint32_t)((kb / NSTAGE) & 1));
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------- MMA issuer ----------------
    bool ok = true;
    for (int kb = 0; kb < n_kb && ok; ++kb) {
      const int s = kb % NSTAGE;
      if (!mbar_wait(full0 + 8 * s, (uint32_t)((kb / NSTAGE) & 1)) || s_fail) {
        ok = false;
        s_fail = 1;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t st = base + (uint32_t)s * STAGE_BYTES;
      const uint32_t a_hi = st, a_lo = st + A_TILE, b_hi = st + 2 * A_TILE, b_lo = st + 2 * A_TILE + B_TILE;
#pragma unroll
      for (int j = 0; j < TK / 16; ++j) {   // K = 16 per instruction: +32 bytes inside the swizzle atom
        const uint32_t off = 32u * (uint32_t)j;
        const uint32_t first = (kb == 0 && j == 0) ? 0u : 1u;
        // the large products and the small corrections accumulate separately, so the large
        // accumulator takes one rounding per k-step instead of three
        mma_f16(tmem, sw128_desc(a_hi + off), sw128_desc(b_hi + off), a.idesc, first);
        mma_f16(tmem + TN, sw128_desc(a_hi + off), sw128_desc(b_lo + off), a.idesc, first);
        mma_f16(tmem + TN, sw128_desc(a_lo + off), sw128_desc(b_hi + off), a.idesc, 1u);
      }
      mma_commit(empty0 + 8 * s);   // stage free once these MMAs have read it
    }
    mma_commit(done);               // all MMAs issued so far complete -> epilogue (also on abort)
  } else if (warp >= 2) {
    // ---------------- A operand generation ----------------
    {
      const int g = warp - 2;
      const int64_t R0 = a.row_base + row0;   // absolute row of the CTA's first row
      for (int kb = 0; kb < n_kb; ++kb) {
        const int s = kb % NSTAGE;
        // this k-block's tone words are loaded before the wait for the stage, so their latency hides
        // under it
        uint64_t phi = 0, F = 0;
        float A = 0.f;
        WindowTone wt;
        if (WINDOW) {
          const int k = (kb0 + kb) * (TK / 4) + (lane & 15);
          wt = window_tone(k < a.K ? a.tones + k : nullptr, a.a_scale, R0);
        } else {
          const int k = (kb0 + kb) * (TK / 2) + lane;
          if (k < a.K) {
            phi = __ldg(&a.tones[k].phi_ref);
            F = __ldg(&a.tones[k].F);
            A = __ldg(&a.tones[k].A) * a.a_scale;
          }
        }
        if (kb >= NSTAGE && !mbar_wait(empty0 + 8 * s, (uint32_t)(((kb / NSTAGE) - 1) & 1))) {
          s_fail = 1;
          break;
        }
        if (s_fail) break;
        const uint32_t st = base + (uint32_t)s * STAGE_BYTES;
        if (WINDOW) gen_a_window<T>(a, wt, R0, g, lane, st, st + A_TILE);
        else gen_a_rows<T>(a, phi, F, A, (uint32_t)row0, g, lane, st, st + A_TILE);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // visible to the tensor cores
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(full0 + 8 * s) : "memory");
      }
    }
    // ---------------- epilogue ----------------
    const bool ok = mbar_wait(done, 0);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const int lane_base = 32 * (warp % 4);          // TMEM lanes this warp may read
    const int row = lane_base + lane;                // row of the tile = TMEM lane
    const bool go = __all_sync(0xffffffffu, ok && !s_fail);   // warp-uniform: tcgen05.ld is .aligned
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // stage memory becomes the partial tile
    // warps with the same lane quarter take consecutive column ranges of the tile
    constexpr int COLS = TN / (NGEN / 4);
    const int c_begin = ((warp - 2) / 4) * COLS;
    if (go) {
#pragma unroll 1
      for (int c0 = c_begin; c0 < c_begin + COLS; c0 += 32) {
        uint32_t v[32], w[32];
        const uint32_t taddr = tmem + ((uint32_t)lane_base << 16) + (uint32_t)c0;
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
            "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
              "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
              "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
            : "r"(taddr));
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
            "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
            : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7]),
              "=r"(w[8]), "=r"(w[9]), "=r"(w[10]), "=r"(w[11]), "=r"(w[12]), "=r"(w[13]), "=r"(w[14]), "=r"(w[15]),
              "=r"(w[16]), "=r"(w[17]), "=r"(w[18]), "=r"(w[19]), "=r"(w[20]), "=r"(w[21]), "=r"(w[22]), "=r"(w[23]),
              "=r"(w[24]), "=r"(w[25]), "=r"(w[26]), "=r"(w[27]), "=r"(w[28]), "=r"(w[29]), "=r"(w[30]), "=r"(w[31])
            : "r"(taddr + (uint32_t)TN));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = __float_as_uint(__uint_as_float(v[i]) + __uint_as_float(w[i]));
#pragma unroll
        for (int i = 0; i < 32; ++i) part[row * PART_STRIDE + c0 + i] = __uint_as_float(v[i]);
      }
    }
    if (!ok) s_fail = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && s_fail) atomicExch(a.status, STATUS_TIMEOUT);
  if (warp == 1) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2 * TN) : "memory");
  }
  cluster.sync();   // every partial tile of the cluster is in shared memory

  // this CTA sums rows [r_lo, r_hi) of the S partial tiles in rank order, then quantises and stores
  const int r_lo = TM * crank / split, r_hi = TM * (crank + 1) / split;
  const int n_el = (r_hi - r_lo) * TN;
  for (int e = threadIdx.x; e < n_el; e += blockDim.x) {
    const int row = r_lo + e / TN, col = e % TN;
    float x = 0.f;
    for (int c = 0; c < split; ++c) x += cluster.map_shared_rank(part, c)[row * PART_STRIDE + col];
    x *= a.inv_a_scale;   // exact: a power of two
    const int64_t n = (a.row_base + row0 + row) * TN + col;   // absolute sample
    if (n < a.win_start || n >= a.win_end) continue;
    if (a.out_q) a.out_q[n - a.win_start] = (int16_t)fminf(fmaxf(rintf(x * a.scale), -32767.f), 32767.f);
    if (a.out_f) a.out_f[n - a.win_start] = x;
  }
  cluster.sync();   // remote reads done before any CTA of the cluster exits
  if (a.end && threadIdx.x == 0) atomicMax(a.end, (unsigned long long)now_ns());
}

// ---------------------------------------------------------------------------------------------
// operand preparation
// ---------------------------------------------------------------------------------------------
// sin and cos of 2 pi w / 2^64 for a 64-bit phase word, accurate to a few 1e-8: sincospi of the
// word's top bits (exactly representable), corrected to first order by the remaining bits.
__device__ __forceinline__ void sincos_word(uint64_t w, float* s, float* c) {
  const int32_t hi = (int32_t)(w >> 32);                 // half-turns x 2^31
  const int32_t h1 = hi & ~0xFF;                         // <= 23 significant bits: exact in float
  const float x1 = (float)h1 * 4.656612873077392578125e-10f;   // 2^-31
  const float x2 = ((float)(hi - h1) + (float)(uint32_t)w * 2.3283064365386963e-10f) * 4.656612873077392578125e-10f;
  float s1, c1;
  sincospif(x1, &s1, &c1);
  const float d = 3.14159265358979323846f * x2;
  *s = fmaf(c1, d, s1);
  *c = fmaf(-s1, d, c1);
}

// (c, s) as packed hi and lo halves
template <typename T>
__device__ __forceinline__ void split_pair(float c, float s, uint32_t* hi, uint32_t* lo) {
  *hi = pack2<T>(c, s);
  const float2 h = unpack2<T>(*hi);
  *lo = pack2<T>(c - h.x, s - h.y);
}

// Bt[n2][2k] = cos b_k(n2), Bt[n2][2k+1] = sin b_k(n2) (the B operand stored K-major); static engine:
// four columns per tone, its two segments' frequency words.  A thread holds one tone and PREP_ROWS
// rows n2, stepping the phase word by the frequency word; a warp stores 32 neighbouring tones (128
// or 256 bytes).  10,000 tones: 15.3 -> 8.7 us (two columns), 26.7 -> 13.5 us (four), from a 64-bit
// division and four 2-byte stores per element.  A tone without a chirp has no second segment (its A columns are zero).
constexpr int PREP_ROWS = 16;
template <typename T, bool WINDOW>
__global__ void __launch_bounds__(128) prep_b_kernel(const ToneRec* tones, int K, int64_t Kp, uint32_t* hi, uint32_t* lo,
                                                     unsigned long long* start) {
  if (start && blockIdx.x == 0 && blockIdx.y == 0 && threadIdx.x == 0) *start = now_ns();
  constexpr int PAIRS = WINDOW ? 2 : 1;   // column pairs per tone
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= Kp / (2 * PAIRS)) return;
  const bool in = k < K, second = WINDOW && in && tones[k].slot >= 0;
  const uint64_t F0 = in ? tones[k].F : 0, F1 = second ? tones[k].F_end : 0;
  const int n0 = (int)blockIdx.y * PREP_ROWS;
  uint64_t w0 = (uint64_t)n0 * F0, w1 = (uint64_t)n0 * F1;
  for (int n2 = n0; n2 < n0 + PREP_ROWS; ++n2) {
    float s = 0.f, c = 0.f;
    uint32_t h[2] = {0, 0}, l[2] = {0, 0};
    if (in) {
      sincos_word(w0, &s, &c);
      split_pair<T>(c, s, &h[0], &l[0]);
    }
    if (second) {
      sincos_word(w1, &s, &c);
      split_pair<T>(c, s, &h[1], &l[1]);
    }
    const int64_t at = (int64_t)n2 * (Kp / 2) + PAIRS * k;
    if (WINDOW) {
      *reinterpret_cast<uint2*>(hi + at) = make_uint2(h[0], h[1]);
      *reinterpret_cast<uint2*>(lo + at) = make_uint2(l[0], l[1]);
    } else {
      hi[at] = h[0];
      lo[at] = l[0];
    }
    w0 += F0;
    w1 += F1;
  }
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                   const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                   CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

cudaError_t encode_2d(EncodeTiledFn enc, CUtensorMap* m, CUtensorMapDataType dt, void* base, uint64_t inner,
                      uint64_t outer, uint32_t box_inner, uint32_t box_outer) {
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {inner * 2};
  const cuuint32_t box[2] = {box_inner, box_outer};
  const cuuint32_t estr[2] = {1, 1};
  CUresult r = enc(m, dt, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                   CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

float table_amp_scale(double amax) {
  if (!(amax > 0) || !std::isfinite(amax)) return 1.f;
  int e = 0;
  (void)std::frexp(amax, &e);                 // amax = m 2^e, m in [0.5, 1)
  e = std::max(-100, std::min(100, e));
  return (float)std::ldexp(1.0, 1 - e);      // amax a_scale in [1, 2)
}

size_t table_kp(int K) { return (((size_t)2 * K + TK - 1) / TK) * TK; }
size_t table_kp_window(int K) { return (((size_t)4 * K + TK - 1) / TK) * TK; }

cudaError_t launch_table_prep(const TableArgs2& t, cudaStream_t s) {
  const int64_t Kp = (int64_t)(t.window_mode ? table_kp_window(t.K) : table_kp(t.K));
  const int64_t per_row = Kp / (t.window_mode ? 4 : 2);
  const dim3 grid((unsigned)((per_row + 127) / 128), TN / PREP_ROWS);
  auto kern = t.window_mode ? (t.precision == 0 ? prep_b_kernel<__nv_bfloat16, true> : prep_b_kernel<__half, true>)
                            : (t.precision == 0 ? prep_b_kernel<__nv_bfloat16, false> : prep_b_kernel<__half, false>);
  kern<<<grid, 128, 0, s>>>(t.tones, t.K, Kp, (uint32_t*)t.b_hi, (uint32_t*)t.b_lo, t.start);
  return cudaGetLastError();
}

cudaError_t launch_table_gemm(const TableArgs2& t, cudaStream_t s) {
  const int64_t M = t.M;
  const int64_t Kp = (int64_t)(t.window_mode ? table_kp_window(t.K) : table_kp(t.K));
  const bool bf16 = (t.precision == 0);
  cudaError_t e;
  static EncodeTiledFn enc = nullptr;
  if (!enc) {
    cudaDriverEntryPointQueryResult q;
    void* fn = nullptr;
    e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
    if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
    enc = (EncodeTiledFn)fn;
  }
  const CUtensorMapDataType dt = bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16;
  CUtensorMap mBh, mBl;
  if ((e = encode_2d(enc, &mBh, dt, t.b_hi, (uint64_t)Kp, (uint64_t)TN, TK, TN)) != cudaSuccess) return e;
  if ((e = encode_2d(enc, &mBl, dt, t.b_lo, (uint64_t)Kp, (uint64_t)TN, TK, TN)) != cudaSuccess) return e;

  TableGemmArgs ga;
  ga.n_kb = (int32_t)(Kp / TK);
  ga.out_q = t.out_q;
  ga.out_f = t.out_f;
  ga.scale = t.scale;
  ga.status = t.status;
  ga.tones = t.tones;
  ga.K = t.K;
  ga.nb_log2 = t.nb_log2;
  ga.row_base = t.row_base;
  ga.win_start = t.win_start;
  ga.win_end = t.win_end;
  ga.window_mode = t.window_mode;
  ga.a_scale = t.a_scale > 0.f ? t.a_scale : 1.f;
  ga.inv_a_scale = 1.f / ga.a_scale;
  ga.end = t.end;
  // instruction descriptor: FP32 accumulate, A/B BF16 (1) or FP16 (0), both K-major, N/8, M/16
  const uint32_t fmt = bf16 ? 1u : 0u;
  ga.idesc = (1u << 4) | (fmt << 7) | (fmt << 10) | ((uint32_t)(TN >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
  const size_t smem = (size_t)NSTAGE * STAGE_BYTES + 1024;
  static_assert((size_t)TM * PART_STRIDE * 4 <= (size_t)NSTAGE * STAGE_BYTES, "partial tile fits in the stages");
  // the static engine's window mode is a separate instantiation, so that the table keeps its lean
  // A-operand generator
  auto kern = t.window_mode ? (bf16 ? table_gemm_kernel<__nv_bfloat16, true> : table_gemm_kernel<__half, true>)
                            : (bf16 ? table_gemm_kernel<__nv_bfloat16, false> : table_gemm_kernel<__half, false>);
  e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  // all of the SM's shared memory, not the smallest split that holds a CTA (196 KB): what is left
  // over takes a render CTA beside it (render_engine)
  if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  if (e != cudaSuccess) return e;
  // K split over a cluster of 1, 2 or 4 CTAs per 128-row tile (periodic tables), whichever finishes first by a
  // simple model: waves of co-resident clusters (a cluster of 4 leaves SMs of some GPCs idle: 36
  // clusters = 144 CTAs at once on 152 SMs, against 76 clusters of 2) times the K blocks per CTA
  // plus an epilogue worth about 8 K blocks
  const int64_t tiles = (M + TM - 1) / TM;
  static int active[5] = {0, 0, 0, 0, 0};
  unsigned split = 1;
  double best = 1e300;
  for (unsigned c = 1; c <= 4; c *= 2) {
    if ((int)c > ga.n_kb) break;
    // the static engine sums each sample over a K split that must not depend on the window's
    // length (chunk invariance): always the largest split there
    if (t.invariant && c < 4 && 4 <= ga.n_kb) continue;
    if (!active[c]) {
      cudaLaunchConfig_t q = {};
      q.gridDim = dim3(c, 1, 1);
      q.blockDim = dim3(GEMM_THREADS, 1, 1);
      q.dynamicSmemBytes = smem;
      cudaLaunchAttribute qa[1];
      qa[0].id = cudaLaunchAttributeClusterDimension;
      qa[0].val.clusterDim.x = c;
      qa[0].val.clusterDim.y = 1;
      qa[0].val.clusterDim.z = 1;
      q.attrs = qa;
      q.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, (const void*)kern, &q) != cudaSuccess || n < 1) {
        cudaGetLastError();
        n = 1;
      }
      active[c] = n;
    }
    const double waves = (double)((tiles + active[c] - 1) / active[c]);
    const double cost = waves * ((double)ga.n_kb / c + 8.0);
    if (cost < best) {
      best = cost;
      split = c;
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)tiles * split, 1, 1);
  cfg.blockDim = dim3(GEMM_THREADS, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = split;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, mBh, mBl, ga);
}

}  // namespace awgk
