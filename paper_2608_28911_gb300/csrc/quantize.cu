// quantize.cu — token-wise mixed-precision quantization and mixed-radix packing
// (Eq. 7; Sec. 4.1 affine base and its Hadamard-rotated form; Sec. 4.9 TurboQuant-MSE
// base with the randomized Hadamard or a dense random rotation), and fake quantization.
//
// Records are built by destination slot: after a slot -> token map (scatter_tok_kernel),
// the affine kernel gives a warp 4 consecutive slots of one pool (lanes own quarter rows),
// the rotated bases 8 (two lanes per row, half a row in registers).  Either way the level
// count is uniform and the record writes are contiguous.  The dense rotation takes 64 slots
// per group of four warps and runs its 128 x 128 product on tcgen05.
//
// Arithmetic (binary32, round to nearest even, no contraction), per row x:
//  affine: s = fp16((max-min)/(L-1)) limited to 65504, z = fp16(min);
//          c = clamp(rint((x - z) * fl(1/s)), 0, L-1)   (all 0 when s == 0)
//  rotated affine: u = fl(1/sqrt 128) * FWHT(x * sign); z = fp16 of min u rounded
//          toward -inf (limited to -65504); s and c as affine on u (all 0 unless s > 0)
//  TQ:     w = FWHT(x * sign) with butterflies h = 1..64; n = fp16(sqrt(sum x^2))
//          with the sum taken as 32 in-order partials of 4 squares then pairwise
//          stages 16, 8, 4, 2, 1; u = w * fl(1/n); c = #{k: u > t_k}
#include <cuda.h>
#include <cudaTypedefs.h>

#include "common.cuh"
#include "kernels.h"

namespace semkv {

namespace {

constexpr int kWarpsPerBlock = 8;

// ------------------------------------------------- affine pools, by slot -----
// Affine records are built by destination slot: a warp takes units of 4 consecutive
// slots of one pool of one (sequence, layer, KV head), so the level count is uniform
// across the warp and the records it writes are contiguous.  Lane 8i + 4r + q handles
// quarter q (dims 32q..32q+31) of row r (0 = K, 1 = V) of the i-th slot's token: 64 bytes
// in, one quarter bit field out.  The same arithmetic as the header states, and symbols
// beta = ceil(t 2^W / L^G) (the record format).
//
// Each warp has a two-stage ring: while a unit is quantized, the next one's rows come by
// cp.async, 256 contiguous bytes of K and of V per instruction, and the one after's token
// indices are read.  Quarters are staged 80 bytes apart, and the records leave through the
// stage in 16-byte stores.
//
// Bound by memory: the 4 x 64K prompt's kernel takes 217 us, 5.8 TB/s (85% of the measured
// copy rate), at 76% issue activity and 90 warp instructions per token and head.  It took 260
// with 119 instructions, a 64-byte quarter per lane in four loads (which kept the load/store
// pipe 74% busy), every code clamped and records put together by atomics and 4-byte stores.

constexpr int kAffineSlots = 4;
// resident CTAs of 8 warps per SM (64 registers; at 5 and 48 registers the 4 x 64K prompt takes
// 321 us against 314, at 6 with spills 338)
constexpr int kAffineCtas = 4;

constexpr int kQuarterStride = 80;  // bytes per staged quarter: 64 + 16 (5 x 16 B: the 8 lanes of a
                                    // quarter warp reach distinct banks)
constexpr int kAffineStage = 32 * kQuarterStride;

// The symbol beta = ceil(t 2^W / M) of a radix value t < M at bit pos of a 3-word field that is
// zero there (pos a compile-time value after unrolling); t arrives as t + off modulo 2^32.
// Without a division: beta = floor((t K + 2^16 - 1) / 2^16) with K = floor(2^(W+16) / M), and
// the multiplier takes the shift to the symbol's place along, so most symbols cost a
// multiply-add and a masked OR.  For M = 7776 (W = 13) that product passes 32 bits:
// beta = t + floor((t K + 2^23 - 1) / 2^23) with K = floor(2^23 (2^13 - M) / M); 13 / 243 is
// (2^13 - 7776) / 7776.  Both hold for every t (symbol_exact).
template <uint32_t M, int W>
struct Symbol {
  static constexpr bool kWide = W > 8;
  static constexpr int S = kWide ? 23 : 16;
  static constexpr uint32_t K = kWide ? (uint32_t)((13ull << S) / 243) : (uint32_t)((1ull << (W + S)) / M);
  static constexpr uint32_t C = (1u << S) - 1u;
};
template <uint32_t M, int W>
constexpr bool symbol_exact() {
  using Y = Symbol<M, W>;
  for (uint32_t t = 0; t < M; ++t) {
    const uint32_t q = (t * Y::K + Y::C) >> Y::S, beta = (uint32_t)((((uint64_t)t << W) + M - 1) / M);
    if ((uint64_t)t * Y::K + Y::C > 0xFFFFFFFFull || (Y::kWide ? t + q : q) != beta) return false;
  }
  return true;
}
static_assert(symbol_exact<7776, 13>() && symbol_exact<125, 7>() && symbol_exact<243, 8>() &&
                  symbol_exact<36, 6>() && symbol_exact<25, 5>() && symbol_exact<9, 4>() &&
                  symbol_exact<7, 3>(),
              "every group and tail of the record format");
template <uint32_t M, int W>
__device__ __forceinline__ void put_symbol(uint32_t (&w)[3], int pos, uint32_t t, uint32_t off) {
  using Y = Symbol<M, W>;
  const int wd = pos >> 5, sh = pos & 31;
  const uint32_t c = Y::C - off * Y::K, mask = ((1u << W) - 1u) << sh;
  if constexpr (Y::kWide) {
    const uint32_t q = t + ((t * Y::K + c) >> Y::S);  // beta + off
    if (sh + W <= 32) {
      w[wd] += (q << sh) - (off << sh);
    } else {
      const uint32_t beta = q - off;
      w[wd] += beta << sh;
      w[wd + 1] += beta >> (32 - sh);
    }
  } else if (sh < 16) {
    w[wd] |= ((t * Y::K + c) >> (16 - sh)) & mask;
  } else {
    w[wd] |= (t * (Y::K << (sh - 16)) + (c << (sh - 16))) & mask;
    if (sh + W > 32) w[wd + 1] |= (t * Y::K + c) >> (48 - sh);
  }
}

// One code of a quarter's field, streamed in order (j = 0..31, compile-time after
// unrolling): m is the code plus OFF (1.5 * 2^23 for magic-number patterns, or 0), t the
// running radix value of the open symbol (sums of L-weighted terms modulo 2^32); each
// completed symbol goes into the field.
template <int L, uint32_t OFF = 0x4B400000u>
__device__ __forceinline__ void field_push(uint32_t (&w)[3], uint32_t& t, int j, uint32_t m) {
  using F = Fmt<L>;
  if constexpr (F::G == 1 && F::LG == (1u << F::W)) {
    // L = 2, 4, 8: the code is its symbol; the offsets add up to one constant per word
    const int wd = (j * F::W) >> 5, sh = (j * F::W) & 31;
    w[wd] += (m << sh) - (OFF << sh);
    if (sh + F::W > 32) w[wd + 1] += (m - OFF) >> (32 - sh);
  } else {
    const bool tail = j >= F::NG * F::G;
    const int k = tail ? j - F::NG * F::G : j % F::G, len = tail ? F::R : F::G;
    t = (k == 0 ? 0u : t * (uint32_t)L) + m;
    if (k == len - 1) {
      uint32_t wsum = 0;
      for (int q = 0; q < len; ++q) wsum = wsum * (uint32_t)L + 1u;
      if constexpr (F::R > 0)
        if (tail) {
          put_symbol<F::LR, F::WT>(w, F::NG * F::W, t, wsum * OFF);
          return;
        }
      put_symbol<F::LG, F::W>(w, (j / F::G) * F::W, t, wsum * OFF);
    }
  }
}

// ---- shared addresses and mbarriers
__device__ __forceinline__ uint32_t dsmem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void dbar_init(uint64_t* bar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(dsmem_u32(bar)) : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dsmem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async8(void* dst, const void* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dsmem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// packed binary32 pairs (two independent IEEE operations, rounded to nearest)
__device__ __forceinline__ unsigned long long f2_add(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long f2_sub(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long f2_pack(float lo, float hi) {
  return (unsigned long long)__float_as_uint(lo) | ((unsigned long long)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ float f2_lo(unsigned long long v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ float f2_hi(unsigned long long v) {
  return __uint_as_float((uint32_t)(v >> 32));
}

// OR the 96-bit field v at bit pos (compile-time after unrolling) of a row's words
template <int N>
__device__ __forceinline__ void or_field(uint32_t (&w)[N], int pos, const uint32_t (&v)[3]) {
  const int wd = pos >> 5, sh = pos & 31;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const uint32_t lo = k < 3 ? v[k] : 0u, prev = k > 0 ? v[k - 1] : 0u;
    const uint32_t part = sh == 0 ? lo : (lo << sh) | (prev >> (32 - sh));
    if (wd + k < N) w[wd + k] |= part;
  }
}

// packed binary32 multiply and fused multiply-add (one rounding each).  The code
// generator may fuse a packed multiply into a packed add or subtract that consumes it,
// .rn notwithstanding (measured), so bit-exact paths use f2_mul only where the product
// is exact (squares of fp16 values) and the scalar __fmul_rn (never fused) elsewhere.
__device__ __forceinline__ unsigned long long f2_mul(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long f2_fma(unsigned long long a, unsigned long long b,
                                                     unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// a * b in a form that is not fused into the operation that takes the result: a * b + -0
// is the rounded product, signed zeros included.  nz must reach the code generator as a
// run-time value (opaque_neg_zero): it turns a constant -0 back into a multiply, and fuses.
__device__ __forceinline__ unsigned long long f2_mul_only(unsigned long long a, unsigned long long b,
                                                          unsigned long long nz) {
  return f2_fma(a, b, nz);
}
__device__ __forceinline__ unsigned long long opaque_neg_zero(uint32_t* scratch) {
  *reinterpret_cast<volatile uint32_t*>(scratch) = 0x80000000u;
  const uint32_t z = *reinterpret_cast<volatile uint32_t*>(scratch);
  return (unsigned long long)z | ((unsigned long long)z << 32);
}

// the larger of a and b, NaN if either is
__device__ __forceinline__ float fmax_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
// the parameters of an affine row from its minimum and maximum
struct AffineParams {
  float s, z, inv;  // inv: 1/s, or 0 when s == 0 (then every value rounds to code 0)
  uint32_t bits;    // s and z as fp16
};
__device__ __forceinline__ AffineParams affine_params(float mn, float mx, int L) {
  // a zero extreme is taken as +0 (min/max may return either signed zero)
  if (mn == 0.0f) mn = 0.0f;
  if (mx == 0.0f) mx = 0.0f;
  const uint16_t s16 = f16_param(__fdiv_rn(__fsub_rn(mx, mn), (float)(L - 1)));
  const uint16_t z16 = __half_as_ushort(__float2half_rn(mn));
  AffineParams p;
  p.s = f16_to_f32(s16);
  p.z = f16_to_f32(z16);
  p.inv = p.s != 0.0f ? __frcp_rn(p.s) : 0.0f;
  p.bits = (uint32_t)s16 | ((uint32_t)z16 << 16);
  return p;
}
// x - z of an fp16 x and a binary32 z, rounded once: one mixed-precision add instead of a
// conversion and a subtraction
__device__ __forceinline__ float sub_mixed(uint16_t x, float neg_z) {
  float d;
  asm("add.rn.f32.f16 %0, %1, %2;" : "=f"(d) : "h"(x), "f"(neg_z));
  return d;
}

// the codes of a quarter (32 fp16 values in hv) as its bit field: rint((x - z) * inv),
// clamped to L - 1 where CLAMP.  x - z >= 0 (z is the row minimum); adding 1.5 * 2^23 rounds
// to nearest even and leaves the code in the low bits of the pattern.
template <int L, bool CLAMP>
__device__ __forceinline__ void affine_field(const uint32_t (&hv)[16], float z, float inv,
                                             unsigned long long nz, uint32_t (&w)[3]) {
  const unsigned long long inv2 = f2_pack(inv, inv);
  const unsigned long long mg2 = f2_pack(12582912.0f, 12582912.0f);
  uint32_t t = 0u;
  w[0] = w[1] = w[2] = 0u;
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    unsigned long long y = f2_mul_only(
        f2_pack(sub_mixed((uint16_t)(hv[j] & 0xFFFFu), -z), sub_mixed((uint16_t)(hv[j] >> 16), -z)), inv2, nz);
    if constexpr (CLAMP) y = f2_pack(fminf(f2_lo(y), (float)(L - 1)), fminf(f2_hi(y), (float)(L - 1)));
    y = f2_add(y, mg2);
    field_push<L>(w, t, 2 * j, (uint32_t)y);
    field_push<L>(w, t, 2 * j + 1, (uint32_t)(y >> 32));
  }
}

template <int L, bool VEC16>
__device__ void affine_units(const QuantArgs& a, int b, int l, int h, bool hi, int64_t n_pool,
                             int u_begin, int step, uint8_t* stages,
                             unsigned long long nz) {
  using F = Fmt<L>;
  constexpr int kRecW = (2 * F::RB + 8) / 4;
  static_assert(F::QB >= 32 && F::QB <= 96, "a quarter fits three words, and a word two quarters");
  const int lane = threadIdx.x & 31;
  const int ti = lane >> 3, row = (lane >> 2) & 1, qd = lane & 3;
  const int64_t cap = hi ? a.hi_cap : a.lo_cap;
  const int64_t base = hi ? a.hi_base : a.lo_base;
  const int64_t bh = ((int64_t)b * a.NL + l) * a.H + h;
  const int32_t* tokmap = (hi ? a.hi_tok : a.lo_tok) + (int64_t)b * cap + base;
  // copies go row by row, 256 contiguous bytes of K and of V per instruction: chunk ch of 16
  // bytes of slot i's row (K: lanes 0..15) to the lane slot of its quarter
  const int ch = lane & 15;
  const uint16_t* src = (lane < 16 ? a.k : a.v) + (bh * a.Tsrc - a.tok_base) * kHeadDim + 8 * ch;
  const int at = (4 * (lane >> 4) + (ch >> 2)) * kQuarterStride + (ch & 3) * 16;
  uint32_t* recs = reinterpret_cast<uint32_t*>(hi ? a.hi_pool : a.lo_pool) + (bh * cap + base) * kRecW;
  const bool st16 = (reinterpret_cast<uintptr_t>(recs) & 15u) == 0;  // (so is every unit then)
  // this lane's bits in a record: the quarter starts at bit off, in word wd0; the word it
  // shares with the next quarter (the next lane) takes that one's first word, which then is
  // not written again
  constexpr int kSpan = (31 + F::QB + 31) / 32;
  const int off = row * 8 * F::RB + qd * F::QB, wd0 = off >> 5, sh = off & 31;
  const int cnt = ((off + F::QB + 31) >> 5) - wd0;
  const int nxt = (lane & 7) == 3 ? 8 * F::RB : (lane & 7) == 7 ? 16 * F::RB : off + F::QB;
  constexpr int kMin = F::QB / 32;  // words every quarter touches at least
  uint32_t take[kSpan];             // the neighbour's first word goes into this word
#pragma unroll
  for (int k = 0; k < kSpan; ++k)
    take[k] = (nxt >> 5) < wd0 + cnt && k == cnt - 1 ? 0xFFFFFFFFu : 0u;
  const int prev_end = row && qd == 0 ? 4 * F::QB - 1 : off - 1;
  const bool own_first = (lane & 7) == 0 || (prev_end >> 5) != wd0;
  const int units = (int)((n_pool + kAffineSlots - 1) / kAffineSlots);
  if (u_begin >= units) return;
  // this lane's token of unit u (lanes past the pool's slots take the last one's; nothing of
  // theirs is written)
  const int last = (int)n_pool - 1;
  auto token = [&](int u) { return tokmap[min(u * kAffineSlots + ti, last)]; };
  auto issue = [&](int32_t tok, int st) {
    uint8_t* dst = stages + st * kAffineStage + at;
#pragma unroll
    for (int i = 0; i < kAffineSlots; ++i) {
      const uint16_t* p = src + (int64_t)__shfl_sync(0xffffffffu, tok, 8 * i) * kHeadDim;
      uint8_t* d = dst + 8 * i * kQuarterStride;
      if constexpr (VEC16) {
        cp_async16(d, p);
      } else {
        cp_async8(d, p);
        cp_async8(d + 8, p + 4);
      }
    }
    cp_async_commit();
  };
  int32_t tok = token(u_begin);
  issue(tok, 0);
  if (u_begin + step < units) tok = token(u_begin + step);
  int st = 0;
  for (int u = u_begin; u < units; u += step, st ^= 1) {
    const int64_t s0 = (int64_t)u * kAffineSlots;
    const int nslots = min(kAffineSlots, (int)(n_pool - s0));
    cp_async_wait<0>();
    __syncwarp();  // the unit has landed; the other stage's image has been stored
    if (u + step < units) {
      issue(tok, st ^ 1);
      if (u + 2 * step < units) tok = token(u + 2 * step);
    }
    uint8_t* stage = stages + st * kAffineStage;
    uint32_t* img = reinterpret_cast<uint32_t*>(stage);
    uint32_t hv[16];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const uint4 x = *reinterpret_cast<const uint4*>(stage + lane * kQuarterStride + 16 * j);
      hv[4 * j] = x.x; hv[4 * j + 1] = x.y; hv[4 * j + 2] = x.z; hv[4 * j + 3] = x.w;
    }
    // row minimum and maximum: fp16 pairs (exact), then the row's other quarters
    // (a NaN in the row makes the maximum, and so s, NaN: the slow path below)
    __half2 mn2 = *reinterpret_cast<const __half2*>(&hv[0]), mx2 = mn2;
#pragma unroll
    for (int j = 1; j < 16; ++j) {
      const __half2 x2 = *reinterpret_cast<const __half2*>(&hv[j]);
      mn2 = __hmin2(mn2, x2);
      mx2 = __hmax2_nan(mx2, x2);
    }
    float mn = fminf(__low2float(mn2), __high2float(mn2));
    float mx = fmax_nan(__low2float(mx2), __high2float(mx2));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 1));
    mx = fmax_nan(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 2));
    mx = fmax_nan(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
    AffineParams pr = affine_params(mn, mx, L);
    // The bound L - 1 cannot be reached when s is a normal fp16 value that was not limited:
    // it is then within 2^-11 of (max - min) / (L - 1), so (x - z) / s < L - 1/2.  s = 0 gives
    // zeros either way.
    uint32_t w[3];
    if (__all_sync(0xffffffffu, (pr.s >= 0x1p-14f && pr.s < 65504.0f) || pr.s == 0.0f)) {
      affine_field<L, false>(hv, pr.z, pr.inv, nz, w);
    } else {
      // the maximum without NaNs, and the codes clamped
      mx2 = *reinterpret_cast<const __half2*>(&hv[0]);
#pragma unroll
      for (int j = 1; j < 16; ++j) mx2 = __hmax2(mx2, *reinterpret_cast<const __half2*>(&hv[j]));
      mx = fmaxf(__low2float(mx2), __high2float(mx2));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      pr = affine_params(mn, mx, L);
      affine_field<L, true>(hv, pr.z, pr.inv, nz, w);
    }
    uint32_t v[kSpan];
#pragma unroll
    for (int k = 0; k < kSpan; ++k)
      v[k] = __funnelshift_l(k > 0 ? w[k - 1] : 0u, k < 3 ? w[k] : 0u, sh);
    const uint32_t first = __shfl_down_sync(0xffffffffu, v[0], 1);
#pragma unroll
    for (int k = kMin - 1; k < kSpan; ++k) v[k] |= first & take[k];
    __syncwarp();  // every quarter has been read: the stage takes the records
    uint32_t* r = img + ti * kRecW + wd0;
#pragma unroll
    for (int k = 0; k < kSpan; ++k)
      if (k == 0 ? own_first : (k < kMin || k < cnt)) r[k] = v[k];
    if (qd == 0) img[ti * kRecW + (2 * F::RB) / 4 + row] = pr.bits;
    __syncwarp();
    // the unit's records are contiguous: 16 bytes per lane where the pool position allows
    uint32_t* dst = recs + s0 * kRecW;
    const int words = nslots * kRecW;
    if (st16 && nslots == kAffineSlots) {
      static_assert(kAffineSlots * kRecW % 4 == 0 && kAffineSlots * kRecW / 4 <= 32, "one pass");
      if (lane < kAffineSlots * kRecW / 4)
        reinterpret_cast<uint4*>(dst)[lane] = reinterpret_cast<const uint4*>(img)[lane];
    } else {
      for (int i = lane; i < words; i += 32) dst[i] = img[i];
    }
  }
}

// slot -> token maps of the tokens quantized by this call
__global__ void scatter_tok_kernel(QuantArgs a) {
  pdl_wait();  // the flags and slots come from earlier work on the stream
  pdl_trigger();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)a.B * a.n) return;
  const int b = (int)(i / a.n), j = (int)(i % a.n);
  const bool hi = a.is_high[(int64_t)b * a.n + j] != 0;
  const int64_t s = (hi ? a.hi_base : a.lo_base) + a.slot[(int64_t)b * a.n + j];
  const int64_t cap = hi ? a.hi_cap : a.lo_cap;
  if (s >= cap) {  // cannot happen after the host's capacity check
    raise_error(a.err, kDevCapacity);
    return;
  }
  (hi ? a.hi_tok : a.lo_tok)[(int64_t)b * cap + s] = (int32_t)(a.tok_base + j);
}

// grid (x, sequence*layer*head): x < bx_hi on the high pool, the rest on the low one, each
// warp striding over its pool's units
template <bool VEC16>  // rows on 16-byte boundaries (else 8)
__global__ void __launch_bounds__(kWarpsPerBlock * 32, kAffineCtas)
    quantize_affine_kernel(QuantArgs a, int64_t n_hi, int64_t n_lo, int bx_hi) {
  __shared__ __align__(128) uint8_t stage_sm[kWarpsPerBlock][2 * kAffineStage];
  // (the same in every lane: what follows from it stays in uniform registers)
  const int wib = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
  uint8_t* stages = stage_sm[wib];
  const unsigned long long nz = opaque_neg_zero(reinterpret_cast<uint32_t*>(stages));
  pdl_wait();  // the slot maps and the rows come from earlier work on the stream
  pdl_trigger();
  const bool hi = (int)blockIdx.x < bx_hi;
  const int64_t n_pool = hi ? n_hi : n_lo;
  const int x = (int)blockIdx.x - (hi ? 0 : bx_hi), bx = hi ? bx_hi : (int)gridDim.x - bx_hi;
  const int u_begin = x * kWarpsPerBlock + wib, step = bx * kWarpsPerBlock;
  const int bhs = a.B * a.NL * a.H;
  for (int bhi = blockIdx.y; bhi < bhs; bhi += gridDim.y) {
    const int h = bhi % a.H, l = (bhi / a.H) % a.NL, b = bhi / (a.H * a.NL);
    __syncwarp();  // (the last head's records have left the stages)
    switch (hi ? a.L_hi : a.L_lo) {
      case 2: affine_units<2, VEC16>(a, b, l, h, hi, n_pool, u_begin, step, stages, nz); break;
      case 3: affine_units<3, VEC16>(a, b, l, h, hi, n_pool, u_begin, step, stages, nz); break;
      case 4: affine_units<4, VEC16>(a, b, l, h, hi, n_pool, u_begin, step, stages, nz); break;
      case 5: affine_units<5, VEC16>(a, b, l, h, hi, n_pool, u_begin, step, stages, nz); break;
      case 6: affine_units<6, VEC16>(a, b, l, h, hi, n_pool, u_begin, step, stages, nz); break;
      case 7: affine_units<7, VEC16>(a, b, l, h, hi, n_pool, u_begin, step, stages, nz); break;
      case 8: affine_units<8, VEC16>(a, b, l, h, hi, n_pool, u_begin, step, stages, nz); break;
      default: break;
    }
  }
}

// ------------------------------ rotated bases by slot, two threads per row -----
// TQ and rotated affine records built by destination slot, as for the affine base: a warp
// takes tiles of 8 consecutive slots of one pool of one (sequence, layer, KV head), so the
// level count is uniform.  Lane 4i + 2r + f holds half f (dims 64f .. 64f + 63, quarters
// 2f and 2f + 1) of row r (0 = K, 1 = V) of slot i, in registers as 32 packed pairs
// (x_j, x_{j+32}).  The Walsh-Hadamard butterflies run in the quantizer's stage order
// (the same roundings as any other evaluation of them): stages 1..16 as packed
// operations across pairs, stage 32 inside each pair, stage 64 with the partner lane.
// Then the norm or the min/max (combined across the two halves), the codes, the two
// quarters' bit fields; each lane puts its half's bits into the tile's record image, which
// leaves in order with 16-byte stores.
constexpr int kRowSlots = 64;
constexpr int kRowStride = 272;  // bytes per staged row: 256 + 16 spreads the banks
constexpr int kTileSlots = 8;    // slots of a warp's tile
constexpr int kHalfStride = 144;  // bytes per half-row slot: 128 + 16 (9 x 16 B: the 8 lanes
                                  // of a quarter warp reach distinct banks)
constexpr int kWarpStageBytes = 32 * kHalfStride;
// The quantizer: CTAs of 128 threads, 5 per SM (96 registers, 20 warps).  At 6 per SM (80
// registers) the pairs spill (at 5 the TQ ones by 48 bytes) and at 4 fewer warps hide the shuffles: the 32K TQ prompt takes
// 87 us at 5, 103 at 6 and 92 at 4, the 3 x 20011 rotated one 133, 139 and 136.
constexpr int kRowsThreads = 128;
constexpr int kRowsCtas = 5;
// Fake quantization: 4 per SM (rotated affine: 127 registers, at 5 the two transforms spill, 144
// against 128 us for 4 layers x 16384 tokens, and at 3 fewer warps hide latency, 138; TQ: 128
// registers and 60 bytes spilled).
constexpr int kFakeCtas = 4;

// Butterfly stages 1, 2, 4, 8, 16 and 32 of the row transform over one half of the row,
// held as packed pairs xp[j] = (x_j, x_{j+32}) (half-local indices): stages 1..16 pair
// registers j and j + hs and so run packed, stage 32 works inside each register.  Each
// butterfly is (a + b, a - b), rounded to nearest.
__device__ __forceinline__ void fwht_half(unsigned long long (&xp)[32]) {
#pragma unroll
  for (int hs = 1; hs < 32; hs <<= 1) {
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      if (j & hs) continue;
      const unsigned long long p0 = xp[j], p1 = xp[j + hs];
      xp[j] = f2_add(p0, p1);
      xp[j + hs] = f2_sub(p0, p1);
    }
  }
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const float lo = f2_lo(xp[j]), hi = f2_hi(xp[j]);
    xp[j] = f2_pack(__fadd_rn(lo, hi), __fsub_rn(lo, hi));
  }
}

// Stage 64 across the two halves of a row (f: this lane's half, the partner is the lane
// beside it).  Half 0 keeps a + b and half 1 a - b (a from half 0): fma(own, +-1, partner),
// whose product is exact, rounds partner +- own once, which is that sum or difference.
__device__ __forceinline__ void fwht_stage64(unsigned long long (&xp)[32], int f) {
  const float sg = f ? -1.0f : 1.0f;
  const unsigned long long sg2 = f2_pack(sg, sg);
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const float plo = __shfl_xor_sync(0xffffffffu, f2_lo(xp[j]), 1);
    const float phi = __shfl_xor_sync(0xffffffffu, f2_hi(xp[j]), 1);
    xp[j] = f2_fma(xp[j], sg2, f2_pack(plo, phi));
  }
}

// TQ codes of both quarters of a half, straight into their bit fields.  u2[j] holds the
// pair (u of quarter 0, u of quarter 1) at dim j of the quarters; t2[k] the pair
// (thr_k, thr_k), ascending, with a zero threshold taken as +0.  d = thr_k - u rounds to
// a value below zero exactly when u > thr_k (binary32 subtraction of unequal values is
// never zero, and with +0 thresholds an equal pair gives +0), so bit 31 of d is the
// comparison, and c = sum_k [u > thr_k] is a thermometer code: c = 1 + ... + 1.
//   L = 2, 4, 8: the code's binary digits from those bits (parities and middles of the
//   thermometer), shifted into the field most significant bit first, one funnel shift
//   per bit (code j occupies bits jW .. jW + W - 1 of the field);
//   other L: c as a sum of the bits, radix groups as field_push.
template <int L>
__device__ __forceinline__ void tq_fields(const unsigned long long (&u2)[32],
                                          const unsigned long long (&t2)[7],
                                          uint32_t (&w0)[3], uint32_t (&w1)[3]) {
  using F = Fmt<L>;
  w0[0] = w0[1] = w0[2] = 0u;
  w1[0] = w1[1] = w1[2] = 0u;
  if constexpr (F::G == 1 && F::LG == (1u << F::W)) {
    constexpr int W = F::W;
    uint32_t a0 = 0u, a1 = 0u;
#pragma unroll
    for (int j = 31; j >= 0; --j) {
      uint32_t dl[7], dh[7];
#pragma unroll
      for (int k = 0; k < L - 1; ++k) {
        const unsigned long long d = f2_sub(t2[k], u2[j]);
        dl[k] = (uint32_t)d;
        dh[k] = (uint32_t)(d >> 32);
      }
#pragma unroll
      for (int b = W - 1; b >= 0; --b) {
        uint32_t bl, bh;
        if constexpr (L == 2) {
          bl = dl[0]; bh = dh[0];
        } else if constexpr (L == 4) {
          if (b == 1) { bl = dl[1]; bh = dh[1]; }
          else { bl = dl[0] ^ dl[1] ^ dl[2]; bh = dh[0] ^ dh[1] ^ dh[2]; }
        } else {
          if (b == 2) { bl = dl[3]; bh = dh[3]; }
          else if (b == 1) { bl = dl[1] ^ dl[3] ^ dl[5]; bh = dh[1] ^ dh[3] ^ dh[5]; }
          else {
            bl = dl[0] ^ dl[1] ^ dl[2] ^ dl[3] ^ dl[4] ^ dl[5] ^ dl[6];
            bh = dh[0] ^ dh[1] ^ dh[2] ^ dh[3] ^ dh[4] ^ dh[5] ^ dh[6];
          }
        }
        a0 = __funnelshift_l(bl, a0, 1);
        a1 = __funnelshift_l(bh, a1, 1);
        const int pbit = j * W + b;
        if ((pbit & 31) == 0) {
          w0[pbit >> 5] = a0;
          w1[pbit >> 5] = a1;
        }
      }
    }
  } else {
    // c = sum of the comparison bits
    uint32_t t0 = 0u, t1 = 0u;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      uint32_t cl = 0u, ch = 0u;
#pragma unroll
      for (int k = 0; k < L - 1; ++k) {
        const unsigned long long d = f2_sub(t2[k], u2[j]);
        cl += (uint32_t)d >> 31;
        ch += (uint32_t)(d >> 32) >> 31;
      }
      field_push<L, 0u>(w0, t0, j, cl);
      field_push<L, 0u>(w1, t1, j, ch);
    }
  }
}

// One tile: 8 slots of one pool, the warp's lanes 4i .. 4i + 3 on slot i (K dims 0..63, K
// dims 64..127, V likewise), in two parts so that the first is compiled once for all level
// counts: the body is straight-line code of several hundred instructions, and two copies of
// it in use at once do not stay in the instruction cache.
//
// rows_front: the rotated half row as pairs (u for the rotated affine base, w for TQ) and
// the row's parameters.  stage: the lane's 128 bytes at lane * kHalfStride; smask: the
// (layer, head)'s sign masks, one word per fp16 pair of dims (0x8000 in a half whose sign
// is -1).
template <int BASE>
__device__ __forceinline__ void rows_front(int L, const uint8_t* stage, const uint32_t* smask,
                                           unsigned long long nz, unsigned long long (&xp)[32],
                                           uint32_t& param, float& invq, float& zq, bool& live) {
  const int lane = threadIdx.x & 31, f = lane & 1;
  // ---- the half, sign-flipped on its fp16 bits (the signs are +-1), as pairs
  {
    const uint4* src = reinterpret_cast<const uint4*>(stage + lane * kHalfStride);
    const uint4* msk = reinterpret_cast<const uint4*>(smask + 32 * f);
    uint32_t wv[32];
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      const uint4 u = src[c], m = msk[c];
      wv[4 * c] = u.x ^ m.x; wv[4 * c + 1] = u.y ^ m.y;
      wv[4 * c + 2] = u.z ^ m.z; wv[4 * c + 3] = u.w ^ m.w;
    }
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const uint32_t lo = wv[j >> 1], hi2 = wv[16 + (j >> 1)];
      const int sh = 16 * (j & 1);
      xp[j] = f2_pack(f16_to_f32((uint16_t)(lo >> sh)), f16_to_f32((uint16_t)(hi2 >> sh)));
    }
  }
  if constexpr (BASE == SEMKV_BASE_TQ) {
    // the norm's fixed tree: 32 in-order partials of 4 squares (this half holds partials
    // 16f + g in the low lanes, 16f + g + 8 in the high ones), then the pairwise stages
    // 16 (across the halves), 8, 4, 2, 1
    // (a square of an fp16 value is exact in binary32, so a fused x * x + v rounds as
    // the separate multiply and add do)
    float pn[8];
#pragma unroll
    for (int g = 0; g < 8; ++g) {
      unsigned long long v = f2_mul(xp[4 * g], xp[4 * g]);
#pragma unroll
      for (int k = 1; k < 4; ++k) v = f2_add(v, f2_mul(xp[4 * g + k], xp[4 * g + k]));
      const float plo = __shfl_xor_sync(0xffffffffu, f2_lo(v), 1);
      const float phi = __shfl_xor_sync(0xffffffffu, f2_hi(v), 1);
      // partials g + (g + 16) and (g + 8) + (g + 24): the same sums in both halves
      const unsigned long long sp = f2_add(v, f2_pack(plo, phi));
      pn[g] = __fadd_rn(f2_lo(sp), f2_hi(sp));
    }
#pragma unroll
    for (int off = 4; off >= 1; off >>= 1)
#pragma unroll
      for (int g = 0; g < off; ++g) pn[g] = __fadd_rn(pn[g], pn[g + off]);
    const uint16_t n16 = f16_param(__fsqrt_rn(pn[0]));
    param = n16;
    const float n = f16_to_f32(n16);
    live = n != 0.0f;
    invq = live ? __fdiv_rn(1.0f, n) : 0.0f;
  }
  // ---- butterflies: stages 1..32 in the thread, stage 64 with the partner half
  fwht_half(xp);
  fwht_stage64(xp, f);
  if constexpr (BASE == SEMKV_BASE_AFFINE_HAD) {
    float mn = INFINITY, mx = -INFINITY;
    const unsigned long long rs2 = f2_pack(kInvSqrtD, kInvSqrtD);
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      xp[j] = f2_mul_only(xp[j], rs2, nz);
      mn = fminf(mn, fminf(f2_lo(xp[j]), f2_hi(xp[j])));
      mx = fmaxf(mx, fmaxf(f2_lo(xp[j]), f2_hi(xp[j])));
    }
    mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, 1));
    mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
    // a zero extreme is taken as +0 (min/max may return either signed zero)
    if (mn == 0.0f) mn = 0.0f;
    if (mx == 0.0f) mx = 0.0f;
    uint16_t z16 = __half_as_ushort(__float2half_rd(mn));
    if (z16 == 0xFC00u) z16 = 0xFBFFu;
    zq = f16_to_f32(z16);
    const uint16_t s16 = f16_param(__fdiv_rn(__fsub_rn(mx, zq), (float)(L - 1)));
    const float sv = f16_to_f32(s16);
    live = sv > 0.0f;
    // 1/s, or 0 when s == 0: then every (u - z) * 0 clamps and rounds to code 0
    invq = live ? __fdiv_rn(1.0f, sv) : 0.0f;
    param = (uint32_t)s16 | ((uint32_t)z16 << 16);
  }
}

// rows_back: the codes, the record image in the stage and the records (rec: the first one
// in the pool).
template <int BASE, int L>
__device__ __forceinline__ void rows_back(const float* thr, uint8_t* stage, uint8_t* rec, int ns,
                                          unsigned long long nz, unsigned long long (&xp)[32],
                                          uint32_t param, float invq, float zq, bool live) {
  using F = Fmt<L>;
  constexpr int kRecW = (2 * F::RB + (BASE == SEMKV_BASE_TQ ? 4 : 8)) / 4;
  constexpr int kBits = 2 * F::QB;             // a half's bits
  constexpr int kW0 = (kBits + 31) / 32;
  static_assert(F::QB <= 96 && 8 * kRecW * 4 <= 32 * kHalfStride, "the image fits the stage");
  const int lane = threadIdx.x & 31, f = lane & 1;
  const bool active = (lane >> 2) < ns;
  // ---- codes, quarter 2f from the low lanes, then quarter 2f + 1 from the high ones
  uint32_t lw[kW0];
#pragma unroll
  for (int k = 0; k < kW0; ++k) lw[k] = 0u;
  if constexpr (BASE == SEMKV_BASE_TQ) {
    // c = #{k : u > thr_k} (ties go low); a zero-norm row compares against +inf
    unsigned long long t2[7];
#pragma unroll
    for (int k = 0; k < L - 1; ++k) {
      const float tk = live ? thr[k] : INFINITY;
      t2[k] = f2_pack(tk, tk);
    }
    // u = y * fl(1/n), rounded before the comparisons subtract it
    const unsigned long long inv2 = f2_pack(invq, invq);
#pragma unroll
    for (int j = 0; j < 32; ++j) xp[j] = f2_mul_only(xp[j], inv2, nz);
    uint32_t fw0[3], fw1[3];
    tq_fields<L>(xp, t2, fw0, fw1);
    or_field<kW0>(lw, 0, fw0);
    or_field<kW0>(lw, F::QB, fw1);
  } else {
    // rint(clamp((u - z) / s)) = clamp(rint(...)) for integer bounds; + 1.5 * 2^23 rounds
    // to nearest even and leaves the code in the low bits of the pattern
    const unsigned long long z2 = f2_pack(zq, zq), inv2 = f2_pack(invq, invq);
    const unsigned long long mg2 = f2_pack(12582912.0f, 12582912.0f);
    // Neither bound can be reached when z was not limited (u >= z) and s is a normal fp16
    // value that was not limited either: s is then within 2^-11 of (max u - z) / (L - 1),
    // so (u - z) / s < L - 1/2.  NaN rows and s = 0 fail the test.
    const float sv = f16_to_f32((uint16_t)(param & 0xFFFFu));
    const bool plain = zq > -65504.0f && sv >= 0x1p-14f && sv < 65504.0f;
#pragma unroll
    for (int j = 0; j < 32; ++j) xp[j] = f2_mul_only(f2_sub(xp[j], z2), inv2, nz);
    if (!__all_sync(0xffffffffu, plain || !active)) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        xp[j] = f2_pack(fminf(fmaxf(f2_lo(xp[j]), 0.0f), (float)(L - 1)),
                        fminf(fmaxf(f2_hi(xp[j]), 0.0f), (float)(L - 1)));
    }
    uint32_t w0[3] = {0u, 0u, 0u}, w1[3] = {0u, 0u, 0u}, t0 = 0u, t1 = 0u;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const unsigned long long y = f2_add(xp[j], mg2);
      field_push<L>(w0, t0, j, (uint32_t)y);
      field_push<L>(w1, t1, j, (uint32_t)(y >> 32));
    }
    or_field<kW0>(lw, 0, w0);
    or_field<kW0>(lw, F::QB, w1);
  }
  // ---- the record image.  A half starts at bit `off` of its record; the word it shares
  // with the next half (the next lane) takes that half's first word, which then is not
  // written again.
  constexpr int kSpan = (31 + kBits + 31) / 32;  // words a half touches at most
  const int q = lane & 3;
  const int off = (q >> 1) * 8 * F::RB + f * kBits;
  const int wd0 = off >> 5, sh = off & 31;
  const int cnt = ((off + kBits + 31) >> 5) - wd0;
  const int next = q == 0 ? kBits : q == 1 ? 8 * F::RB : q == 2 ? 8 * F::RB + kBits : 16 * F::RB;
  const bool share_next = (next >> 5) < wd0 + cnt;
  const int prev_end = q == 0 ? -1 : q == 1 ? kBits - 1 : q == 2 ? 2 * kBits - 1 : 8 * F::RB + kBits - 1;
  const bool share_prev = (prev_end >> 5) == wd0 && q != 0;
  uint32_t v[kSpan];
#pragma unroll
  for (int k = 0; k < kSpan; ++k)
    v[k] = __funnelshift_l(k > 0 && k - 1 < kW0 ? lw[k - 1] : 0u, k < kW0 ? lw[k] : 0u, sh);
  const uint32_t first = __shfl_down_sync(0xffffffffu, v[0], 1);
#pragma unroll
  for (int k = kBits / 32 > 0 ? kBits / 32 - 1 : 0; k < kSpan; ++k)
    v[k] |= (share_next && k == cnt - 1) ? first : 0u;
  uint32_t* img = reinterpret_cast<uint32_t*>(stage);
  __syncwarp();  // every half row has been read
  if (active) {
    uint32_t* r = img + (lane >> 2) * kRecW;
#pragma unroll
    for (int k = 0; k < kSpan; ++k)
      if (k < cnt && (k > 0 || !share_prev)) r[wd0 + k] = v[k];
    if (f == 0) {
      if constexpr (BASE == SEMKV_BASE_TQ)
        reinterpret_cast<uint16_t*>(r + (2 * F::RB) / 4)[q >> 1] = (uint16_t)param;
      else
        r[(2 * F::RB) / 4 + (q >> 1)] = param;
    }
  }
  __syncwarp();
  // ---- the records are contiguous: 16 bytes per lane where the pool position allows
  const int words = ns * kRecW;
  int done = 0;
  if ((reinterpret_cast<uintptr_t>(rec) & 15u) == 0) {
    for (int i = lane; i < words / 4; i += 32)
      reinterpret_cast<uint4*>(rec)[i] = reinterpret_cast<const uint4*>(img)[i];
    done = words & ~3;
  }
  for (int i = done + lane; i < words; i += 32) reinterpret_cast<uint32_t*>(rec)[i] = img[i];
}

// A position in the tiles: tile r of (sequence, layer, head) bhi, the high pool's tiles
// before the low one's.
struct RowsPos {
  uint32_t bhi, r;
};
// Warps over tiles of 8 slots: a CTA takes a contiguous range, its warps the tiles in turn,
// each warp with its own two-stage pipeline.  While a tile is quantized, the next one's
// rows (8 cp.async of 16 bytes per lane) and the one after's token indices are on their way.
// No warp waits for another.  The positions stay in uniform registers, which leaves room for the
// pairs: the rotated affine instance does not spill (92 registers), the TQ one 48 bytes
// (96 registers).
//
// Bound by instruction issue: 75 (rotated affine) and 80 (TQ 4/3) warp instructions per row
// at 63% issue activity, against 97 and 95 at 53% for the CTA-wide 64-slot blocks with a
// barrier each, clamps on every code and records assembled word by word: the 32K prompt's
// kernel 81.8 -> 56.6 us (rotated affine, 2.8 TB/s) and 83.9 -> 61.3 us (TQ).  What is left is the butterflies (14 packed adds per row), conversions,
// radix groups and the exchange of stage 64.
template <int BASE>
__global__ void __launch_bounds__(kRowsThreads, kRowsCtas) quantize_rows_kernel(QuantArgs a, int64_t n_hi64, int64_t n_lo64) {
  extern __shared__ __align__(128) uint8_t rstage[];  // per warp 2 stages of 32 half-row slots
  __shared__ __align__(16) uint32_t smask_all[kRowsThreads / 32][64];
  const int lane = threadIdx.x & 31;
  // (the same in every lane: what follows from it stays in uniform registers)
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
  const int n_hi = (int)n_hi64, n_lo = (int)n_lo64;
  const uint32_t u_hi = (uint32_t)(n_hi + kTileSlots - 1) / kTileSlots;
  const uint32_t per_bh = u_hi + (uint32_t)(n_lo + kTileSlots - 1) / kTileSlots;
  const uint32_t total = (uint32_t)a.B * a.NL * a.H * per_bh;
  constexpr uint32_t kW = kRowsThreads / 32;
  const uint32_t first = (uint32_t)((uint64_t)total * blockIdx.x / gridDim.x);
  const uint32_t last = (uint32_t)((uint64_t)total * (blockIdx.x + 1) / gridDim.x);
  const uint32_t begin = first + warp;
  uint8_t* stages = rstage + warp * 2 * kWarpStageBytes;
  uint32_t* smask = smask_all[warp];
  const unsigned long long nz = opaque_neg_zero(smask);
  // the thresholds of both pools, a zero one as +0 (tq_fields): a copy per warp, which needs
  // no CTA barrier (they are inputs like the rows, read only after the wait)
  __shared__ float thr_all[BASE == SEMKV_BASE_TQ ? kRowsThreads / 32 : 1][2][8];
  float (*thr_sm)[8] = thr_all[BASE == SEMKV_BASE_TQ ? warp : 0];
  __syncwarp();
  pdl_wait();  // the slot maps, the rows and the tables come from earlier work on the stream
  pdl_trigger();
  auto advance = [&](RowsPos& p) {
    p.r += kW;
    while (p.r >= per_bh) {
      p.r -= per_bh;
      p.bhi++;
    }
  };
  // this lane's token of the tile at p (a lane past the pool's slots takes the last one)
  auto token = [&](const RowsPos& p) {
    const uint32_t b = p.bhi / (uint32_t)(a.NL * a.H);
    const bool hi = p.r < u_hi;
    const int s = (int)(hi ? p.r : p.r - u_hi) * kTileSlots + (lane >> 2);
    const int32_t* tokmap = hi ? a.hi_tok + (int64_t)b * a.hi_cap + a.hi_base
                               : a.lo_tok + (int64_t)b * a.lo_cap + a.lo_base;
    return tokmap[min(s, (hi ? n_hi : n_lo) - 1)];  // (tok_base comes off where it is used)
  };
  // row by row, so that an instruction reads 256 contiguous bytes of K and of V (slot i:
  // chunk c of 16 bytes of row 2 i + kind goes to half 2 row + (c >> 3))
  const int ch = lane & 15;
  const uint16_t* kv = (lane < 16 ? a.k : a.v) + 8 * ch;
  auto issue = [&](const RowsPos& p, int32_t tok, int st) {
    const uint16_t* src = kv + ((int64_t)p.bhi * a.Tsrc - a.tok_base) * kHeadDim;
    uint8_t* dst = stages + st * kWarpStageBytes + (2 * (lane >> 4) + (ch >> 3)) * kHalfStride + (ch & 7) * 16;
#pragma unroll
    for (int i = 0; i < kTileSlots; ++i)
      cp_async16(dst + 4 * i * kHalfStride,
                 src + (int64_t)__shfl_sync(0xffffffffu, tok, 4 * i) * kHeadDim);
    cp_async_commit();
  };
  if (begin >= last) return;
  const int trips = (int)((last - begin + kW - 1) / kW);
  RowsPos cur;
  cur.bhi = begin / per_bh;
  cur.r = begin - cur.bhi * per_bh;
  // the sign masks of (layer, head) lh
  auto signs_of = [&](uint32_t lh, char2 (&s2)[2]) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
      s2[i] = *reinterpret_cast<const char2*>(a.signs + (int64_t)lh * kHeadDim + 2 * (lane + 32 * i));
  };
  auto put_masks = [&](const char2 (&s2)[2]) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
      smask[lane + 32 * i] = (s2[i].x < 0 ? 0x8000u : 0u) | (s2[i].y < 0 ? 0x80000000u : 0u);
  };
  uint32_t masked = cur.bhi % (uint32_t)(a.NL * a.H);  // whose masks are in smask
  char2 s2[2];
  int32_t tok = token(cur);
  signs_of(masked, s2);
  float thr = 0.0f;
  if (BASE == SEMKV_BASE_TQ && (lane & 7) < ((lane & 8) ? a.L_lo : a.L_hi) - 1)
    thr = ((lane & 8) ? a.thr_lo : a.thr_hi)[lane & 7];
  issue(cur, tok, 0);
  RowsPos nxt = cur;
  if (trips > 1) {
    advance(nxt);
    tok = token(nxt);
  }
  put_masks(s2);
  if (BASE == SEMKV_BASE_TQ && lane < 16) thr_sm[lane >> 3][lane & 7] = __fadd_rn(thr, 0.0f);
  for (int i = 0; i < trips; ++i) {
    const int st = i & 1;
    const uint32_t lh = cur.bhi % (uint32_t)(a.NL * a.H);
    if (lh != masked) {
      masked = lh;
      signs_of(lh, s2);
      __syncwarp();
      put_masks(s2);
    }
    cp_async_wait<0>();
    __syncwarp();  // the tile has landed; the other stage's image has been stored
    RowsPos after = nxt;
    if (i + 1 < trips) {
      issue(nxt, tok, st ^ 1);
      if (i + 2 < trips) {
        advance(after);
        tok = token(after);
      }
    }
    uint8_t* stage = stages + st * kWarpStageBytes;
    const bool hi = cur.r < u_hi;
    const int L = hi ? a.L_hi : a.L_lo;
    const int s0 = (int)(hi ? cur.r : cur.r - u_hi) * kTileSlots;
    const int ns = min(kTileSlots, (hi ? n_hi : n_lo) - s0);
    uint8_t* rec = hi ? a.hi_pool + ((int64_t)cur.bhi * a.hi_cap + a.hi_base + s0) * record_bytes_rt(BASE, L)
                      : a.lo_pool + ((int64_t)cur.bhi * a.lo_cap + a.lo_base + s0) * record_bytes_rt(BASE, L);
    const float* thrs = thr_sm[hi ? 0 : 1];
    unsigned long long xp[32];
    uint32_t param;
    float invq, zq = 0.0f;
    bool live;
    rows_front<BASE>(L, stage, smask, nz, xp, param, invq, zq, live);
    switch (L) {
#define SEMKV_ROWS_CASE(LV) \
      case LV: rows_back<BASE, LV>(thrs, stage, rec, ns, nz, xp, param, invq, zq, live); break;
      SEMKV_ROWS_CASE(2) SEMKV_ROWS_CASE(3) SEMKV_ROWS_CASE(4) SEMKV_ROWS_CASE(5)
      SEMKV_ROWS_CASE(6) SEMKV_ROWS_CASE(7) SEMKV_ROWS_CASE(8)
#undef SEMKV_ROWS_CASE
      default: break;
    }
    cur = nxt;
    nxt = after;
  }
}
// ------------------------------------------------- fake quantization ---------
// Every row quantized at its token's precision and reconstructed to fp16 (the quality
// protocol of Sec. 4.1), in binary32 in this order:
//   affine: x^_d = fp16( z + s * c_d )
//   rotated affine: y = FWHT(z + s * c);  x^_d = fp16( (sign_d y_d) * fp32(1/sqrt 128) )
//   TQ:     y = FWHT(cb[c]) (the quantizer's butterflies);  x^_d = fp16( (sign_d y_d) * (n/128) )

// Affine base: a CTA of 128 threads per 64-token block, thread r on row r (K of token r/2
// when r is even, V when odd), rows staged through shared memory in and out
// (coalesced), each row kept as fp16 pairs (96 registers: 5 CTAs per SM).
__global__ void __launch_bounds__(128, 5) fake_affine_kernel(FakeArgs a) {
  __shared__ __align__(16) uint8_t stage[128 * kRowStride];
  const int tid = threadIdx.x;
  const int64_t bhs = (int64_t)a.B * a.NL * a.H;
  for (int64_t bhi = blockIdx.y; bhi < bhs; bhi += gridDim.y) {
    const int b = (int)(bhi / ((int64_t)a.H * a.NL));
    for (int t0 = blockIdx.x * kRowSlots; t0 < a.T; t0 += gridDim.x * kRowSlots) {
      const int nt = min(kRowSlots, a.T - t0);
      const int64_t row0 = bhi * a.T + t0;
      for (int c = tid; c < 128 * 16; c += 128) {
        const int r = c >> 4, ch = c & 15, i = r >> 1;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (i < nt) v = __ldg(reinterpret_cast<const uint4*>(((r & 1) ? a.v : a.k) + (row0 + i) * kHeadDim) + ch);
        *reinterpret_cast<uint4*>(stage + r * kRowStride + ch * 16) = v;
      }
      __syncthreads();
      const int i = tid >> 1;
      const bool hi = i < nt && (a.is_high == nullptr || a.is_high[(int64_t)b * a.T + t0 + i] != 0);
      const int L = (a.is_high == nullptr || hi) ? a.L_hi : a.L_lo;
      uint32_t ov[64];  // the row's fp16 outputs, in pairs
      {
        // x^_d = fp16(z + s c_d), the row kept as fp16 pairs (fewer registers, more CTAs)
        uint32_t hv[64];
#pragma unroll
        for (int ch = 0; ch < 16; ++ch) {
          const uint4 u = *reinterpret_cast<const uint4*>(stage + tid * kRowStride + ch * 16);
          hv[4 * ch] = u.x;
          hv[4 * ch + 1] = u.y;
          hv[4 * ch + 2] = u.z;
          hv[4 * ch + 3] = u.w;
        }
        // row minimum and maximum on fp16 pairs (exact)
        __half2 mn2 = *reinterpret_cast<const __half2*>(&hv[0]), mx2 = mn2;
#pragma unroll
        for (int j = 1; j < 64; ++j) {
          const __half2 x2 = *reinterpret_cast<const __half2*>(&hv[j]);
          mn2 = __hmin2(mn2, x2);
          mx2 = __hmax2(mx2, x2);
        }
        float mn = fminf(__low2float(mn2), __high2float(mn2));
        float mx = fmaxf(__low2float(mx2), __high2float(mx2));
        if (mn == 0.0f) mn = 0.0f;
        if (mx == 0.0f) mx = 0.0f;
        const uint16_t s16 = f16_param(__fdiv_rn(__fsub_rn(mx, mn), (float)(L - 1)));
        const float sv = f16_to_f32(s16), z = f16_to_f32(__half_as_ushort(__float2half_rn(mn)));
        const float inv = sv != 0.0f ? __fdiv_rn(1.0f, sv) : 0.0f;
        // c = rint(min((x - z) / s, L - 1)) as an integer-valued float (x >= z: z is the
        // row minimum; inv = 0 when s = 0, so every code is 0): adding and taking off
        // 1.5 * 2^23 rounds to nearest even, as the float-to-int conversion would
#pragma unroll
        for (int j = 0; j < 64; ++j) {
          float r[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float x = f16_to_f32((uint16_t)(hv[j] >> (16 * e)));
            const float y = fminf(__fmul_rn(__fsub_rn(x, z), inv), (float)(L - 1));
            const float c = __fsub_rn(__fadd_rn(y, 12582912.0f), 12582912.0f);
            r[e] = __fadd_rn(z, __fmul_rn(sv, c));
          }
          const __half2 h2 = __floats2half2_rn(r[0], r[1]);
          ov[j] = *reinterpret_cast<const uint32_t*>(&h2);
        }
      }
      __syncthreads();  // every row is read: the stage takes the outputs
#pragma unroll
      for (int ch = 0; ch < 16; ++ch)
        *reinterpret_cast<uint4*>(stage + tid * kRowStride + ch * 16) =
            make_uint4(ov[4 * ch], ov[4 * ch + 1], ov[4 * ch + 2], ov[4 * ch + 3]);
      __syncthreads();
      for (int c = tid; c < 128 * 16; c += 128) {
        const int r = c >> 4, ch = c & 15, ii = r >> 1;
        if (ii < nt)
          reinterpret_cast<uint4*>(((r & 1) ? a.v_out : a.k_out) + (row0 + ii) * kHeadDim)[ch] =
              *reinterpret_cast<const uint4*>(stage + r * kRowStride + ch * 16);
      }
      __syncthreads();
    }
  }
}

// Rotated affine and TQ: the rows quantizer's tiles (8 tokens, two lanes per row, each warp
// with its own two-stage pipeline) and its front half; then the values the codes stand for,
// the same butterflies back, and the fp16 rows through the stage, so that both ways move
// 512 contiguous bytes per instruction.

// The codebook entry of each of a pair's two values: c = #{k : u > thr_k} over the
// kLmax - 1 thresholds (the row's own L - 1 of them, then +inf), from the sign bits of
// thr_k - u as in tq_fields
template <int kLmax>
__device__ __forceinline__ unsigned long long tq_dequant2(unsigned long long u2,
                                                          const unsigned long long (&t2)[7],
                                                          const float* cb) {
  uint32_t cl = 0u, ch = 0u;
#pragma unroll
  for (int k = 0; k < kLmax - 1; ++k) {
    const unsigned long long d = f2_sub(t2[k], u2);
    cl += (uint32_t)d >> 31;
    ch += (uint32_t)(d >> 32) >> 31;
  }
  return f2_pack(cb[cl], cb[ch]);
}

// The values the row's codes stand for, in place of the rotated values in xp (pairs), and
// the reconstruction's final factor: fp32(1/sqrt 128), or n / 128
template <int BASE, int kLmax>
__device__ __forceinline__ float fake_values(int L, unsigned long long nz, const float* thr,
                                             const float* cb, bool active, uint32_t param,
                                             float invq, float zq, bool live,
                                             unsigned long long (&xp)[32]) {
  const unsigned long long inv2 = f2_pack(invq, invq);
  if constexpr (BASE == SEMKV_BASE_AFFINE_HAD) {
    const float sv = f16_to_f32((uint16_t)(param & 0xFFFFu)), top = (float)(L - 1);
    const unsigned long long z2 = f2_pack(zq, zq), s2 = f2_pack(sv, sv);
    const unsigned long long mg2 = f2_pack(12582912.0f, 12582912.0f);
#pragma unroll
    for (int j = 0; j < 32; ++j) xp[j] = f2_mul_only(f2_sub(xp[j], z2), inv2, nz);
    // (the clamp is needed only where the parameters were limited or subnormal: rows_back)
    const bool plain = zq > -65504.0f && sv >= 0x1p-14f && sv < 65504.0f;
    if (!__all_sync(0xffffffffu, plain || !active)) {
#pragma unroll
      for (int j = 0; j < 32; ++j)
        xp[j] = f2_pack(fminf(fmaxf(f2_lo(xp[j]), 0.0f), top), fminf(fmaxf(f2_hi(xp[j]), 0.0f), top));
    }
    // c = rint(...) as an integer-valued float (every code 0 when s = 0); z + s c: s c is
    // exact (an fp16 value times an integer below 8), so the fused multiply-add rounds as
    // the separate multiply and add
#pragma unroll
    for (int j = 0; j < 32; ++j) xp[j] = f2_fma(s2, f2_sub(f2_add(xp[j], mg2), mg2), z2);
    return kInvSqrtD;
  } else {
    unsigned long long t2[7];
#pragma unroll
    for (int k = 0; k < kLmax - 1; ++k) {
      // a zero-norm row compares against +inf (all codes 0)
      const float tk = live && k < L - 1 ? thr[k] : INFINITY;
      t2[k] = f2_pack(tk, tk);
    }
    // u = y * fl(1/n), rounded before the comparisons subtract it
#pragma unroll
    for (int j = 0; j < 32; ++j)
      xp[j] = tq_dequant2<kLmax>(f2_mul_only(xp[j], inv2, nz), t2, cb);
    return f16_to_f32((uint16_t)param) * 0.0078125f;
  }
}

// Warps over tiles of 8 tokens of one (sequence, layer, head), the CTA's range in turn.
// Bound by instruction issue: 4 layers x 16384 tokens of the rotated affine base 202 -> 128 us
// (4.2 TB/s), TQ 4/3 249 -> 167, against 64-token blocks with a CTA barrier each, clamps on
// every value and 16-byte stores a row apart.
template <int BASE>
__global__ void __launch_bounds__(kRowsThreads, kFakeCtas) fake_rows_kernel(FakeArgs a, int Lmax) {
  extern __shared__ __align__(128) uint8_t fstage[];  // per warp 2 stages of 32 half-row slots
  __shared__ __align__(16) uint32_t smask_all[kRowsThreads / 32][64];
  __shared__ float cbs[2][8], thr_sm[2][8];
  const int lane = threadIdx.x & 31, f = lane & 1;
  // (the same in every lane: what follows from it stays in uniform registers)
  const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0);
  constexpr uint32_t kW = kRowsThreads / 32;
  const uint32_t per_bh = (uint32_t)(a.T + kTileSlots - 1) / kTileSlots;
  const uint32_t total = (uint32_t)a.B * a.NL * a.H * per_bh;
  const uint32_t first = (uint32_t)((uint64_t)total * blockIdx.x / gridDim.x);
  const uint32_t last = (uint32_t)((uint64_t)total * (blockIdx.x + 1) / gridDim.x);
  const uint32_t begin = first + warp;
  uint8_t* stages = fstage + warp * 2 * kWarpStageBytes;
  uint32_t* smask = smask_all[warp];
  const unsigned long long nz = opaque_neg_zero(smask);
  if (BASE == SEMKV_BASE_TQ && threadIdx.x < 16) {
    const int which = threadIdx.x >> 3, k = threadIdx.x & 7;
    const int L = which ? a.L_lo : a.L_hi;
    cbs[which][k] = k < L ? (which ? a.cent_lo : a.cent_hi)[k] : 0.0f;
    // a zero threshold as +0 (tq_fields)
    thr_sm[which][k] = k < L - 1 ? __fadd_rn((which ? a.thr_lo : a.thr_hi)[k], 0.0f) : INFINITY;
  }
  __syncthreads();
  if (begin >= last) return;
  const int trips = (int)((last - begin + kW - 1) / kW);
  auto advance = [&](RowsPos& p) {
    p.r += kW;
    while (p.r >= per_bh) {
      p.r -= per_bh;
      p.bhi++;
    }
  };
  // a tile's 8 K rows and 8 V rows are 2 KB each: chunk c of 16 bytes of row 2 t + kind goes
  // to half 2 row + (c >> 3)
  const int ch = lane & 15;
  auto issue = [&](const RowsPos& p, int st) {
    const int t0 = (int)p.r * kTileSlots, n = a.T - t0;
    const int64_t row0 = (int64_t)p.bhi * a.T + t0;
    uint8_t* dst = stages + st * kWarpStageBytes + (ch >> 3) * kHalfStride + (ch & 7) * 16;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int t = 2 * (i & 3) + (lane >> 4), kind = i >> 2;
      if (t < n)
        cp_async16(dst + (2 * t + kind) * 2 * kHalfStride,
                   (kind ? a.v : a.k) + (row0 + t) * kHeadDim + 8 * ch);
    }
    cp_async_commit();
  };
  // whether this lane's token of the tile is a high one
  auto flag = [&](const RowsPos& p) -> uint32_t {
    if (a.is_high == nullptr) return 1u;
    const int64_t b = p.bhi / (uint32_t)(a.NL * a.H);
    return a.is_high[b * a.T + min((int)p.r * kTileSlots + (lane >> 2), a.T - 1)];
  };
  RowsPos cur;
  cur.bhi = begin / per_bh;
  cur.r = begin - cur.bhi * per_bh;
  issue(cur, 0);
  uint32_t hi_cur = flag(cur), hi_nxt = 0;
  uint32_t masked = 0xffffffffu;  // the (layer, head) whose masks are in smask
  for (int i = 0; i < trips; ++i) {
    const int st = i & 1;
    const uint32_t lh = cur.bhi % (uint32_t)(a.NL * a.H);
    if (lh != masked) {
      masked = lh;
      __syncwarp();
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const char2 s2 = *reinterpret_cast<const char2*>(a.signs + (int64_t)lh * kHeadDim + 2 * (lane + 32 * j));
        smask[lane + 32 * j] = (s2.x < 0 ? 0x8000u : 0u) | (s2.y < 0 ? 0x80000000u : 0u);
      }
    }
    cp_async_wait<0>();
    __syncwarp();  // the tile has landed; the other stage's rows have been stored
    RowsPos nxt = cur;
    if (i + 1 < trips) {
      advance(nxt);
      issue(nxt, st ^ 1);
      hi_nxt = flag(nxt);
    }
    uint8_t* stage = stages + st * kWarpStageBytes;
    const int t0 = (int)cur.r * kTileSlots, n = a.T - t0;
    const bool active = (lane >> 2) < n, hi = hi_cur != 0;
    const int L = hi ? a.L_hi : a.L_lo;
    unsigned long long xp[32];
    uint32_t param;
    float invq, zq = 0.0f, post = 0.0f;
    bool live;
    rows_front<BASE>(L, stage, smask, nz, xp, param, invq, zq, live);
    switch (BASE == SEMKV_BASE_TQ ? Lmax : 2) {
#define SEMKV_FAKE_CASE(LV) \
      case LV: post = fake_values<BASE, LV>(L, nz, thr_sm[hi ? 0 : 1], cbs[hi ? 0 : 1], active, param, invq, zq, live, xp); break;
      SEMKV_FAKE_CASE(2) SEMKV_FAKE_CASE(3) SEMKV_FAKE_CASE(4) SEMKV_FAKE_CASE(5)
      SEMKV_FAKE_CASE(6) SEMKV_FAKE_CASE(7) SEMKV_FAKE_CASE(8)
#undef SEMKV_FAKE_CASE
      default: break;
    }
    // ---- back: the butterflies, then sign_d (y_d * post) as fp16 into the lane's slot
    fwht_half(xp);
    fwht_stage64(xp, f);
    {
      const unsigned long long p2 = f2_pack(post, post);
      uint32_t out[32];
#pragma unroll
      for (int p = 0; p < 16; ++p) {
        const unsigned long long x = f2_mul(xp[2 * p], p2), y = f2_mul(xp[2 * p + 1], p2);
        const __half2 h0 = __floats2half2_rn(f2_lo(x), f2_lo(y));
        const __half2 h1 = __floats2half2_rn(f2_hi(x), f2_hi(y));
        out[p] = *reinterpret_cast<const uint32_t*>(&h0);
        out[16 + p] = *reinterpret_cast<const uint32_t*>(&h1);
      }
      const uint4* msk = reinterpret_cast<const uint4*>(smask + 32 * f);
      uint4* slot = reinterpret_cast<uint4*>(stage + lane * kHalfStride);
#pragma unroll
      for (int c = 0; c < 8; ++c) {
        const uint4 m = msk[c];
        slot[c] = make_uint4(out[4 * c] ^ m.x, out[4 * c + 1] ^ m.y, out[4 * c + 2] ^ m.z, out[4 * c + 3] ^ m.w);
      }
    }
    __syncwarp();
    {
      const int64_t row0 = (int64_t)cur.bhi * a.T + t0;
      const uint8_t* src = stage + (ch >> 3) * kHalfStride + (ch & 7) * 16;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int t = 2 * (j & 3) + (lane >> 4), kind = j >> 2;
        if (t < n)
          reinterpret_cast<uint4*>((kind ? a.v_out : a.k_out) + (row0 + t) * kHeadDim)[ch] =
              *reinterpret_cast<const uint4*>(src + (2 * t + kind) * 2 * kHalfStride);
      }
    }
    cur = nxt;
    hi_cur = hi_nxt;
  }
}

// ------------------------------------- dense-rotation TQ rows (tcgen05) --------
// Blocks of 64 slots of one pool of one (sequence, layer, KV head), as for the other
// bases: 128 rows (row r: K of slot r/2 when r is even, V when odd), one level count.
// Persistent CTAs of two groups of 4 warps (two CTAs per SM), each CTA over a range of
// blocks of one (sequence, layer, KV head) whose rotation M (128 x 128 fp16, the B
// operand, K-major: output dims x input dims) it stages once.  A group takes every other
// block of the range: thread r of the group brings row r with sixteen 16-byte cp.async
// copies into the group's A tile (K-major 8-row x 16-byte core matrices: byte
// kg * 2048 + r * 16 holds dims 8 kg .. 8 kg + 7), then one thread issues
// D = X M^T on tcgen05 (kind::f16, M = 128 rows, N = 128 output dims, K = 8 x 16) into
// the group's 128 columns of tensor memory, so TMEM lane r is row r and column c its
// output dim c.  While the MMAs run, thread r takes its row's fixed-tree norm from the
// tile; once they have completed it starts the copies of the group's next block and
// reads its row's w = M x a quarter (32 columns) at a time, the next quarter's load in
// flight while one is coded: u = w * fl(1/n), the codes
// from the thresholds, the quarter bit fields, and the row's bytes straight into its
// record.  The two groups' accumulators are distinct, so one group's MMAs overlap the
// other's epilogue.
constexpr int kDenseThreads = 256;
constexpr uint32_t kDenseM = 128 * 128 * 2;   // the rotation, bytes
constexpr uint32_t kDenseA = 128 * 128 * 2;   // one group's tile of 128 rows
constexpr uint32_t kDenseSmem = kDenseM + 2 * kDenseA + 1024;  // + alignment
// instruction descriptor: fp32 accumulate (bits 4-5 = 1), A and B fp16 (formats 0),
// both K-major, N >> 3 at bits 17-22, M >> 4 at bits 24-28
constexpr uint32_t kDenseIdesc = (1u << 4) | ((128u >> 3) << 17) | ((128u >> 4) << 24);

// shared-memory matrix descriptor without swizzle: start >> 4 (bits 0-13), leading
// (K-direction) core-matrix offset >> 4 (bits 16-29), stride (8-row group) offset >> 4
// (bits 32-45), descriptor version 1 (bits 46-47)
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}
// 32 columns of this warp's 32 TMEM lanes (lane i of the warp <- TMEM lane 32 (w % 4) + i):
// the load, and the wait that makes them readable.  The wait takes the registers as
// in-out operands, so no use of them can be scheduled before it.
__device__ __forceinline__ void tmem_ld32_start(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
        "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&v)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]),
                 "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]),
                 "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), "+r"(v[16]), "+r"(v[17]),
                 "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                 "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]),
                 "+r"(v[30]), "+r"(v[31])
               :
               : "memory");
}
__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
  return v;
}
// barrier of the 128 threads of group g (named barrier 1 + g), with an AND of p
__device__ __forceinline__ bool group_sync_and(int g, bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n"
      " barrier.cta.red.and.pred q, %2, 128, p;\n selp.u32 %0, 1, 0, q;\n}"
      : "=r"(r)
      : "r"((uint32_t)p), "r"(1 + g)
      : "memory");
  return r != 0;
}

// The field of one quarter from its 32 values u (thresholds as in tq_fields: t2[k] the
// pair (thr_k, thr_k)); pairs of neighbouring dims share each packed subtraction.
template <int L>
__device__ __forceinline__ void tq_quarter(const float (&u)[32], const unsigned long long (&t2)[7],
                                           uint32_t (&w)[3]) {
  using F = Fmt<L>;
  w[0] = w[1] = w[2] = 0u;
  if constexpr (F::G == 1 && F::LG == (1u << F::W)) {
    constexpr int W = F::W;
    uint32_t acc = 0u;
#pragma unroll
    for (int jp = 15; jp >= 0; --jp) {
      uint32_t dl[7], dh[7];
#pragma unroll
      for (int k = 0; k < L - 1; ++k) {
        const unsigned long long d = f2_sub(t2[k], f2_pack(u[2 * jp], u[2 * jp + 1]));
        dl[k] = (uint32_t)d;
        dh[k] = (uint32_t)(d >> 32);
      }
#pragma unroll
      for (int e = 1; e >= 0; --e) {  // dim 2jp + 1 first: most significant bit first
        const uint32_t* dd = e ? dh : dl;
        const int j = 2 * jp + e;
#pragma unroll
        for (int b = W - 1; b >= 0; --b) {
          uint32_t bit;
          if constexpr (L == 2) bit = dd[0];
          else if constexpr (L == 4) bit = b == 1 ? dd[1] : (dd[0] ^ dd[1] ^ dd[2]);
          else bit = b == 2 ? dd[3] : b == 1 ? (dd[1] ^ dd[3] ^ dd[5])
                                             : (dd[0] ^ dd[1] ^ dd[2] ^ dd[3] ^ dd[4] ^ dd[5] ^ dd[6]);
          acc = __funnelshift_l(bit, acc, 1);
          const int pbit = j * W + b;
          if ((pbit & 31) == 0) w[pbit >> 5] = acc;
        }
      }
    }
  } else {
    uint32_t t = 0u;
#pragma unroll
    for (int jp = 0; jp < 16; ++jp) {
      uint32_t c[2] = {0u, 0u};
#pragma unroll
      for (int k = 0; k < L - 1; ++k) {
        const unsigned long long d = f2_sub(t2[k], f2_pack(u[2 * jp], u[2 * jp + 1]));
        c[0] += (uint32_t)d >> 31;
        c[1] += (uint32_t)(d >> 32) >> 31;
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) field_push<L, 0u>(w, t, 2 * jp + e, c[e]);
    }
  }
}

// Row r of a block: codes from TMEM (taddr: this warp's lanes, the group's columns), the
// quarter fields, and the row's bytes into its record (rec: the record; kind 0 = K at
// byte 0, 1 = V at byte RB; its fp16 norm at byte 2 RB + 2 kind)
template <int L>
__device__ __forceinline__ void dense_row(uint32_t taddr, const float* thr, float inv, bool live,
                                          uint16_t n16, uint8_t* rec, int kind, bool store) {
  using F = Fmt<L>;
  constexpr int RB = F::RB;
  unsigned long long t2[7];
#pragma unroll
  for (int k = 0; k < L - 1; ++k) {
    const float tk = live ? __fadd_rn(__ldg(thr + k), 0.0f) : INFINITY;
    t2[k] = f2_pack(tk, tk);
  }
  uint32_t w[13];
#pragma unroll
  for (int k = 0; k < 13; ++k) w[k] = 0u;
  // quarter q + 1's columns load while quarter q is coded
  uint32_t vb[2][32];
  tmem_ld32_start(taddr, vb[0]);
  tmem_ld_wait(vb[0]);
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    if (q < 3) tmem_ld32_start(taddr + 32 * (q + 1), vb[(q + 1) & 1]);
    float u[32];
    // u = w * fl(1/n), rounded before the comparisons subtract it
#pragma unroll
    for (int j = 0; j < 32; ++j) u[j] = __fmul_rn(__uint_as_float(vb[q & 1][j]), inv);
    if (q < 3) tmem_ld_wait(vb[(q + 1) & 1]);
    uint32_t fw[3];
    tq_quarter<L>(u, t2, fw);
    or_field<13>(w, q * F::QB, fw);
  }
  if (!store) return;
  // the row's RB bytes: word-aligned for K; V starts 2 bytes into a word when RB = 2 mod 4
  if (kind == 0 || (RB & 3) == 0) {
    uint32_t* dst = reinterpret_cast<uint32_t*>(rec + kind * RB);
#pragma unroll
    for (int k = 0; k < RB / 4; ++k) dst[k] = w[k];
    if constexpr ((RB & 3) != 0)
      *reinterpret_cast<uint16_t*>(rec + kind * RB + 4 * (RB / 4)) = (uint16_t)w[RB / 4];
  } else {
    *reinterpret_cast<uint16_t*>(rec + RB) = (uint16_t)w[0];
    uint32_t* dst = reinterpret_cast<uint32_t*>(rec + RB + 2);
#pragma unroll
    for (int k = 0; k < (RB - 2) / 4; ++k) dst[k] = __funnelshift_r(w[k], w[k + 1], 16);
  }
  *reinterpret_cast<uint16_t*>(rec + 2 * RB + 2 * kind) = n16;
}

__global__ void __launch_bounds__(kDenseThreads, 2)
    quantize_tq_dense_kernel(QuantArgs a, int64_t n_hi, int64_t n_lo) {
  extern __shared__ uint8_t dsm_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(dsm_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* mb = base;                       // B: the rotation, core-matrix layout
  __shared__ __align__(8) uint64_t mma_bar[2];
  __shared__ uint32_t tmem_base;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int grp = warp >> 2, row = 32 * (warp & 3) + lane;
  uint8_t* xa = base + kDenseM + grp * kDenseA;  // A: this group's rows
  const int64_t bhl = blockIdx.y;
  const int h = (int)(bhl % a.H), l = (int)((bhl / a.H) % a.NL);
  const int b = (int)(bhl / ((int64_t)a.H * a.NL));
  const int nb_hi = (int)((n_hi + kRowSlots - 1) / kRowSlots);
  const int tiles = nb_hi + (int)((n_lo + kRowSlots - 1) / kRowSlots);
  const int per = (tiles + (int)gridDim.x - 1) / (int)gridDim.x;
  const int j0 = min(tiles, (int)blockIdx.x * per), j1 = min(tiles, j0 + per);

  if (tid == 0) {
    dbar_init(&mma_bar[0]);
    dbar_init(&mma_bar[1]);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(
                     dsmem_u32(&tmem_base))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the rotation: 16-byte chunk c = (row group, k group, row in group) at byte 16 c
  const uint4* msrc = reinterpret_cast<const uint4*>(a.rot + ((int64_t)l * a.H + h) * 128 * 128);
  for (int c = tid; c < 128 * 16; c += kDenseThreads) {
    const int rr = c & 7, kg = (c >> 3) & 15, r = (c >> 7) * 8 + rr;
    reinterpret_cast<uint4*>(mb)[c] = msrc[r * 16 + kg];
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tb = tmem_base;
  const uint32_t tcol = tb + (uint32_t)(grp * 128);           // this group's accumulator
  const uint32_t tlane = tcol + ((uint32_t)(32 * (warp & 3)) << 16);
  const int64_t bh = bhl;  // (sequence, layer, head) index of the pools and the rows

  // block j of the range: pool, first slot, slots
  auto block = [&](int j, bool& hi, int& s0, int& ns) {
    hi = j < nb_hi;
    s0 = (hi ? j : j - nb_hi) * kRowSlots;
    ns = (int)min((int64_t)kRowSlots, (hi ? n_hi : n_lo) - s0);
  };
  // this thread's row of block j into the group's tile
  auto load_row = [&](int j) {
    bool hi;
    int s0, ns;
    block(j, hi, s0, ns);
    if ((row >> 1) < ns) {
      const int64_t cap = hi ? a.hi_cap : a.lo_cap;
      const int32_t* tokmap = (hi ? a.hi_tok : a.lo_tok) + (int64_t)b * cap + (hi ? a.hi_base : a.lo_base);
      const int64_t tk = (int64_t)tokmap[s0 + (row >> 1)] - a.tok_base;
      const uint16_t* src = ((row & 1) ? a.v : a.k) + (bh * a.Tsrc + tk) * kHeadDim;
#pragma unroll
      for (int kg = 0; kg < 16; ++kg) cp_async16(xa + kg * 2048 + row * 16, src + 8 * kg);
    }
    cp_async_commit();
  };

  bool ok = true;
  int j = j0 + grp;
  if (j < j1) load_row(j);
  for (int it = 0; j < j1; j += 2, ++it) {
    bool hi;
    int s0, ns;
    block(j, hi, s0, ns);
    const bool mine = (row >> 1) < ns;
    cp_async_wait<0>();
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the rows, for the MMAs
    group_sync_and(grp, true);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (row == 0) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const uint64_t da = umma_desc(dsmem_u32(xa) + k * 4096, 2048, 128);
        const uint64_t db = umma_desc(dsmem_u32(mb) + k * 256, 128, 2048);
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}" ::"r"(tcol),
            "l"(da), "l"(db), "r"(kDenseIdesc), "r"((uint32_t)(k > 0))
            : "memory");
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              dsmem_u32(&mma_bar[grp]))
          : "memory");
    }
    // ---- while the MMAs run: the row's norm (fixed tree: 32 in-order partials of 4
    // squares, then the pairwise stages 16, 8, 4, 2, 1).  Partials g and g + 16 are
    // formed as a pair from chunks kg and kg + 8 (a square of an fp16 value is exact, so
    // a fused multiply-add rounds as the separate operations)
    uint16_t n16 = 0;
    float inv = 0.0f;
    {
      const uint32_t xs = dsmem_u32(xa);  // (shared-space loads: the tile is in shared memory)
      float pn[16];
#pragma unroll
      for (int kg = 0; kg < 8; ++kg) {
        const uint4 ua = ld_shared_v4(xs + kg * 2048 + row * 16);
        const uint4 ub = ld_shared_v4(xs + (kg + 8) * 2048 + row * 16);
        const uint32_t wa[4] = {ua.x, ua.y, ua.z, ua.w}, wb[4] = {ub.x, ub.y, ub.z, ub.w};
#pragma unroll
        for (int g2 = 0; g2 < 2; ++g2) {
          unsigned long long acc = 0ull;
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const uint32_t xw = wa[2 * g2 + (e >> 1)], yw = wb[2 * g2 + (e >> 1)];
            const int sh = 16 * (e & 1);
            const unsigned long long x2 = f2_pack(f16_to_f32((uint16_t)(xw >> sh)), f16_to_f32((uint16_t)(yw >> sh)));
            acc = e == 0 ? f2_mul(x2, x2) : f2_add(acc, f2_mul(x2, x2));
          }
          // partials 2kg + g2 and 2kg + g2 + 16, then their sum (stage 16)
          pn[2 * kg + g2] = __fadd_rn(f2_lo(acc), f2_hi(acc));
        }
      }
#pragma unroll
      for (int off = 8; off >= 1; off >>= 1)
#pragma unroll
        for (int g = 0; g < off; ++g) pn[g] = __fadd_rn(pn[g], pn[g + off]);
      n16 = f16_param(__fsqrt_rn(pn[0]));
      const float n = f16_to_f32(n16);
      inv = n != 0.0f ? __fdiv_rn(1.0f, n) : 0.0f;
    }
    ok = group_sync_and(grp, mbar_wait_bounded(&mma_bar[grp], (uint32_t)(it & 1)));
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    if (!ok) break;
    // the MMAs have read the tile and this thread its row: the next block's row
    if (j + 2 < j1) load_row(j + 2);
    // ---- codes and the record
    const int64_t cap = hi ? a.hi_cap : a.lo_cap;
    const int L = hi ? a.L_hi : a.L_lo;
    const int rec_bytes = 2 * row_bytes_rt(L) + 4;
    uint8_t* rec = (hi ? a.hi_pool : a.lo_pool) +
                   (bh * cap + (hi ? a.hi_base : a.lo_base) + s0 + (row >> 1)) * rec_bytes;
    const float* thr = hi ? a.thr_hi : a.thr_lo;
    const bool live = n16 != 0;
    switch (L) {
#define SEMKV_DENSE_CASE(LV) \
      case LV: dense_row<LV>(tlane, thr, inv, live, n16, rec, row & 1, mine); break;
      SEMKV_DENSE_CASE(2) SEMKV_DENSE_CASE(3) SEMKV_DENSE_CASE(4) SEMKV_DENSE_CASE(5)
      SEMKV_DENSE_CASE(6) SEMKV_DENSE_CASE(7) SEMKV_DENSE_CASE(8)
#undef SEMKV_DENSE_CASE
      default: break;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  }
  if (!ok && row == 0) raise_error(a.err, kDevWaitTimeout);
  cp_async_wait<0>();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tb) : "memory");
}

}  // namespace

cudaError_t launch_fake_quant(const FakeArgs& a, int num_sms, cudaStream_t stream) {
  const int64_t total = (int64_t)a.B * a.NL * a.H * a.T;
  if (total == 0) return cudaSuccess;
  const int64_t bhs = (int64_t)a.B * a.NL * a.H;
  const int64_t nblk = ((int64_t)a.T + kRowSlots - 1) / kRowSlots;
  if (a.base == SEMKV_BASE_AFFINE) {
    const dim3 grid((unsigned)(nblk < 65535 ? nblk : 65535), (unsigned)(bhs < 65535 ? bhs : 65535));
    fake_affine_kernel<<<grid, 128, 0, stream>>>(a);
    return cudaGetLastError();
  }
  static bool attr_set[kAttrDevices] = {};
  constexpr int kSmem = kRowsThreads / 32 * 2 * kWarpStageBytes;
  const cudaError_t e = once_per_device(attr_set, [] {
    cudaError_t r = cudaFuncSetAttribute(fake_rows_kernel<SEMKV_BASE_AFFINE_HAD>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(fake_rows_kernel<SEMKV_BASE_TQ>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, kSmem);
    return r;
  });
  if (e != cudaSuccess) return e;
  // tile indices are 32-bit (and a call of this size was refused by its 64-token blocks)
  const int64_t tiles = bhs * (((int64_t)a.T + kTileSlots - 1) / kTileSlots);
  if (bhs * nblk > INT32_MAX / 2 || tiles > UINT32_MAX / 2) return cudaErrorInvalidValue;
  constexpr int kRowWarps = kRowsThreads / 32;
  int64_t ctas = (int64_t)(num_sms > 0 ? num_sms : 1) * kFakeCtas;
  if (ctas > (tiles + kRowWarps - 1) / kRowWarps) ctas = (tiles + kRowWarps - 1) / kRowWarps;
  const int Lmax = a.L_hi > a.L_lo ? a.L_hi : a.L_lo;
  if (a.base == SEMKV_BASE_AFFINE_HAD)
    fake_rows_kernel<SEMKV_BASE_AFFINE_HAD><<<(unsigned)ctas, kRowsThreads, kSmem, stream>>>(a, Lmax);
  else
    fake_rows_kernel<SEMKV_BASE_TQ><<<(unsigned)ctas, kRowsThreads, kSmem, stream>>>(a, Lmax);
  return cudaGetLastError();
}

cudaError_t launch_quantize_pack(const QuantArgs& a, int64_t n_hi, int num_sms,
                                 cudaStream_t stream, bool maps_ready) {
  const int64_t total = (int64_t)a.B * a.NL * a.H * a.n;
  if (total == 0) return cudaSuccess;
  if (a.base == SEMKV_BASE_AFFINE) {
    if (!maps_ready) {
      const int64_t pairs = (int64_t)a.B * a.n;
      const cudaError_t e = launch_pdl(scatter_tok_kernel, dim3((unsigned)((pairs + 255) / 256)),
                                       dim3(256), 0, stream, a);
      if (e != cudaSuccess) return e;
    }
    // Grid x: bx_hi CTAs for the high pool of each (sequence, layer, head), the rest for the
    // low one, so that every warp has about the same number of units.  From a wave model:
    // with R resident CTAs (kAffineCtas per SM) the pass takes ceil(CTAs / R) waves of
    // (units per warp + 2), the 2 for a warp's start (its position, the first unit's token and
    // rows); the cheapest count up to 32 is taken.  (Sized by the larger pool alone and
    // without the start, a 32K prompt with 30% high two-level tokens got one unit per warp:
    // 51 us, 33 now.)  The head index runs over grid y (and loops past its limit of 65535).
    const int64_t bhs = (int64_t)a.B * a.NL * a.H;
    const int64_t rows = bhs < 65535 ? bhs : 65535;
    const int64_t resident = (int64_t)(num_sms > 0 ? num_sms : 1) * kAffineCtas;
    const int64_t u_hi = (n_hi + kAffineSlots - 1) / kAffineSlots;
    const int64_t u_lo = (a.n - n_hi + kAffineSlots - 1) / kAffineSlots;
    int64_t bx_hi = 0, bx_lo = 0, best = -1;
    for (int64_t pw = 32; pw >= 1; --pw) {
      const int64_t per = pw * kWarpsPerBlock;
      const int64_t xh = (u_hi + per - 1) / per, xl = (u_lo + per - 1) / per;
      const int64_t cost = (((xh + xl) * rows + resident - 1) / resident) * (pw + 2);
      if (best < 0 || cost < best) {
        best = cost;
        bx_hi = xh;
        bx_lo = xl;
      }
    }
    const dim3 grid((unsigned)(bx_hi + bx_lo), (unsigned)rows);
    const bool vec16 = ((reinterpret_cast<uintptr_t>(a.k) | reinterpret_cast<uintptr_t>(a.v)) & 15u) == 0;
    return launch_pdl(vec16 ? quantize_affine_kernel<true> : quantize_affine_kernel<false>, grid,
                      dim3(kWarpsPerBlock * 32), 0, stream, a, n_hi, a.n - n_hi, (int)bx_hi);
  }
  // TQ, rotated affine and dense-rotation TQ: slot -> token maps, then the rows by slot
  if (!maps_ready) {
    const int64_t pairs = (int64_t)a.B * a.n;
    const cudaError_t e = launch_pdl(scatter_tok_kernel, dim3((unsigned)((pairs + 255) / 256)),
                                     dim3(256), 0, stream, a);
    if (e != cudaSuccess) return e;
  }
  if (a.base == SEMKV_BASE_TQ_DENSE) {
    static bool attr_set[kAttrDevices] = {};
    const cudaError_t e = once_per_device(attr_set, [] {
      return cudaFuncSetAttribute(quantize_tq_dense_kernel,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kDenseSmem);
    });
    if (e != cudaSuccess) return e;
    const int64_t bhs = (int64_t)a.B * a.NL * a.H;
    if (bhs > 65535) return cudaErrorInvalidValue;
    const int64_t tiles = (n_hi + kRowSlots - 1) / kRowSlots + (a.n - n_hi + kRowSlots - 1) / kRowSlots;
    int64_t splits = (2 * (int64_t)num_sms + bhs - 1) / bhs;  // about two CTAs per SM
    // (each CTA's two groups take alternate blocks of its range)
    if (splits > (tiles + 1) / 2) splits = (tiles + 1) / 2;
    if (splits < 1) splits = 1;
    const dim3 grid((unsigned)splits, (unsigned)bhs);
    quantize_tq_dense_kernel<<<grid, kDenseThreads, kDenseSmem, stream>>>(a, n_hi, a.n - n_hi);
    return cudaGetLastError();
  }
  // kRowsCtas CTAs per SM, each a range of the tiles of both pools
  const int64_t bhs = (int64_t)a.B * a.NL * a.H;
  const int64_t tiles = bhs * ((n_hi + kTileSlots - 1) / kTileSlots +
                               (a.n - n_hi + kTileSlots - 1) / kTileSlots);
  int64_t ctas = (int64_t)(num_sms > 0 ? num_sms : 1) * kRowsCtas;
  constexpr int kRowWarps = kRowsThreads / 32;
  if (ctas > (tiles + kRowWarps - 1) / kRowWarps) ctas = (tiles + kRowWarps - 1) / kRowWarps;
  if (ctas < 1) return cudaSuccess;
  if (tiles > UINT32_MAX / 2) return cudaErrorInvalidValue;  // tile indices are 32-bit
  static bool rows_attr[kAttrDevices] = {};
  {
    const cudaError_t e = once_per_device(rows_attr, [] {
      cudaError_t r = cudaFuncSetAttribute(quantize_rows_kernel<SEMKV_BASE_AFFINE_HAD>,
                                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           kRowsThreads / 32 * 2 * kWarpStageBytes);
      if (r == cudaSuccess)
        r = cudaFuncSetAttribute(quantize_rows_kernel<SEMKV_BASE_TQ>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, kRowsThreads / 32 * 2 * kWarpStageBytes);
      return r;
    });
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(a.base == SEMKV_BASE_AFFINE_HAD ? quantize_rows_kernel<SEMKV_BASE_AFFINE_HAD>
                                                    : quantize_rows_kernel<SEMKV_BASE_TQ>,
                    dim3((unsigned)ctas), dim3(kRowsThreads), kRowsThreads / 32 * 2 * kWarpStageBytes, stream, a,
                    n_hi, a.n - n_hi);
}

}  // namespace semkv
