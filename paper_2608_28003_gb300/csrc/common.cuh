// Shared device/host helpers of libw8a8 (sm_103a).
#pragma once

#include <utility>

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>
#include <stdint.h>
#include <stddef.h>

#include "../../include/w8a8.h"

namespace w8a8 {

// ------------------------------------------------------------------------- host status
void set_error(const char* fmt, ...);
const char* get_error();

#define W8A8_CHECK_ARG(cond, code, ...)   \
  do {                                    \
    if (!(cond)) {                        \
      ::w8a8::set_error(__VA_ARGS__);     \
      return code;                        \
    }                                     \
  } while (0)

#define W8A8_CUDA(call)                                                                        \
  do {                                                                                         \
    cudaError_t e_ = (call);                                                                   \
    if (e_ != cudaSuccess) {                                                                   \
      ::w8a8::set_error("CUDA error %s at %s:%d", cudaGetErrorString(e_), __FILE__, __LINE__); \
      return W8A8_ERR_CUDA;                                                                    \
    }                                                                                          \
  } while (0)

#define W8A8_LAUNCH_CHECK() W8A8_CUDA(cudaGetLastError())

// Programmatic dependent launch.  Kernels are launched with programmatic stream serialization: the
// next kernel in the stream may start while this one runs, so that it can set up and stream its
// weights early.  Every such kernel calls pdl_wait() before its first read of data an earlier kernel
// wrote and before its first global write; pdl_wait() returns once the preceding grid has completed
// and its writes are visible (at once when the launch allowed no overlap).  Because every kernel
// waits before it can finish, completion is ordered along the whole stream.
//
// What a kernel may read ahead of its wait.  The arguments of a call, weights and scales included, may
// be the result of any work before it on the stream, and kernels let their dependents start at once, so
// a call's first launch reads nothing ahead: it waits, and only then triggers its own dependents (its
// `settled` argument is false).  The call's later launches (settled) cannot start before every CTA of
// the first one has passed its wait, when all work before the call is complete: they trigger at once and
// read whatever the call itself does not write ahead of their wait.  The decoder's calls begin with a
// launch that allows no overlap (set_int), so all of their others are settled.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
// Let the next kernel in the stream begin launching (its CTAs start as resources free up).
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }

template <typename... KArgs, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

#define W8A8_TRY(expr)            \
  do {                            \
    w8a8_status s_ = (expr);      \
    if (s_ != W8A8_OK) return s_; \
  } while (0)

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline cudaStream_t as_stream(void* s) { return reinterpret_cast<cudaStream_t>(s); }
inline size_t round_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

w8a8_status check_device();  // current device must be sm_103

// ---------------------------------------------------------------------- exact conversions
__device__ __forceinline__ float bf16_bits_to_f32(uint32_t bits16) { return __uint_as_float(bits16 << 16); }
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }

__device__ __forceinline__ uint16_t f32_to_bf16_bits(float x) {
  __nv_bfloat16 b = __float2bfloat16_rn(x);
  return *reinterpret_cast<uint16_t*>(&b);
}

// int8 code (as int) -> fp16 bit pattern; exact for |q| <= 2048.
__device__ __forceinline__ uint16_t int_to_f16_bits(int q) {
  __half h = __int2half_rn(q);
  return *reinterpret_cast<uint16_t*>(&h);
}

// Four signed bytes of `w` (byte b0 lowest) -> two f16x2 words {f16(b0), f16(b1)} and
// {f16(b2), f16(b3)}, exact for codes in [-128, 127].  Flipping the sign bit of each byte gives
// u = b + 128 in [0, 255]; the half 0x6400 | u is 1024 + u exactly, so subtracting 1152 leaves b.
__device__ __forceinline__ void i8x4_to_f16x2x2(uint32_t w, uint32_t& lo, uint32_t& hi) {
  const uint32_t u = w ^ 0x80808080u;
  const uint32_t plo = __byte_perm(u, 0x64646464u, 0x4140u);
  const uint32_t phi = __byte_perm(u, 0x64646464u, 0x4342u);
  const __half2 bias = __halves2half2(__ushort_as_half(0x6480u), __ushort_as_half(0x6480u));  // 1152
  __half2 a = __hsub2(*reinterpret_cast<const __half2*>(&plo), bias);
  __half2 b = __hsub2(*reinterpret_cast<const __half2*>(&phi), bias);
  lo = *reinterpret_cast<uint32_t*>(&a);
  hi = *reinterpret_cast<uint32_t*>(&b);
}

// Two fp32 values -> two e4m3 codes (lo in the low byte): round to nearest even, saturating at
// +-448 (the hardware conversion with .satfinite).
__device__ __forceinline__ uint32_t e4m3x2_of(float lo, float hi) {
  return (uint32_t)__nv_cvt_float2_to_fp8x2(make_float2(lo, hi), __NV_SATFINITE, __NV_E4M3);
}
// Two e4m3 codes (low byte first) -> their values as an fp16 pair, low half first (exact: every
// e4m3 value is an fp16 value).
__device__ __forceinline__ uint32_t e4m3x2_to_f16x2(uint32_t codes16) {
  const __half2_raw h = __nv_cvt_fp8x2_to_halfraw2((__nv_fp8x2_storage_t)(codes16 & 0xFFFFu), __NV_E4M3);
  return (uint32_t)h.x | ((uint32_t)h.y << 16);
}

// ------------------------------------------------------------------------- legacy MMA
// D[16x8] += A[16x16] * B[16x8], fp32 accumulate.
__device__ __forceinline__ void mma_f16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                              uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_bf16_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                               uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// ----------------------------------------------------------------- streaming global loads
__device__ __forceinline__ uint4 ldg_stream(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}
__device__ __forceinline__ uint4 ldg_keep(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "l"(p));
  return v;
}

// ------------------------------------------------------------- mbarrier and bulk copies
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait for the phase with the given parity to complete, for at most `budget` SM cycles.
// Returns false on timeout (the caller records an error and stops waiting).
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, long long budget) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity))
    if (clock64() - t0 > budget) return false;
  return true;
}
// The same for a whole warp: the result, and so the control flow that depends on it, is uniform.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, long long budget) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const long long t0 = clock64();
  while (!__all_sync(0xffffffffu, mbar_try_wait(bar, parity)))
    if (__any_sync(0xffffffffu, clock64() - t0 > budget)) return false;
  return true;
}
// One lane of a converged warp, the same one every time.
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(r));
  return r != 0;
}
// Start fetching a tensor map (a kernel parameter) so the first copy does not wait for it.
__device__ __forceinline__ void prefetch_tmap(const void* tmap) {
  asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(tmap)) : "memory");
}
// 2-D tiled TMA load of one box (coordinates: c0 = innermost element index, c1 = row) into shared
// memory; completion is counted on `bar` in bytes (out-of-bounds elements are zero-filled and counted).
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const void* tmap, int c0, int c1, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}
// An L2 policy that marks the lines it brings in as the first to evict: decode weights are read
// once per step (far more bytes than L2 holds), and so should not push the KV cache, the
// activations and the small per-step tables out of L2.
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;\n" : "=l"(p));
  return p;
}
// tma_load_2d with an L2 cache policy.
__device__ __forceinline__ void tma_load_2d_policy(uint32_t dst, const void* tmap, int c0, int c1, uint32_t bar,
                                                   uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, "
      "%3}], [%4], %5;\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(tmap)), "r"(c0), "r"(c1), "r"(bar), "l"(policy)
      : "memory");
}
// 1-D bulk copy global -> shared (async proxy); completion is counted on `bar` in bytes.
// dst and src 16-byte aligned, bytes a multiple of 16.
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void named_bar_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(nthreads) : "memory");
}
// Named barrier `id` of nthreads threads that also returns whether every one of them passed ok.
__device__ __forceinline__ bool named_bar_all(int id, int nthreads, bool ok) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.u32 p, %1, 0;\n bar.red.and.pred p, %2, %3, p;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)ok), "r"(id), "r"(nthreads)
      : "memory");
  return r != 0;
}
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

// Device-side error bits (reserved workspace word at kErrWordOffset): set by a bounded wait
// that gave up; read and cleared by w8a8_workspace_check.
enum DevErr : unsigned int { DEVERR_CONSUMER_WAIT = 1u, DEVERR_PRODUCER_WAIT = 2u, DEVERR_DRAIN_WAIT = 4u };
constexpr size_t kErrWordOffset = 36864;
constexpr long long kWaitBudgetCycles = 4000000000LL;  // ~2 s at 2 GHz

// ------------------------------------------------------------------------ packed fp32
// Two fp32 values in one 64-bit register: each half of a packed operation is one IEEE operation,
// rounded to nearest even.  A packed multiply feeding a packed add is contracted into one fused
// operation whatever the rounding modifier says, so f2_mul adds a -0 that the compiler cannot know
// (f2_neg_zero, for kernels whose gridDim.z is 1: the tcgen05 GEMM and the decode GEMV; not the attention
// kernels, whose z is the batch); a b + (-0) is the rounded product, signs included.
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 f2_pack(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;\n" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 f2_both(uint32_t bits) { return ((f32x2)bits << 32) | bits; }
__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ f32x2 f2_neg_zero() { return f2_both(0x7fffffffu + gridDim.z); }
__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b, f32x2 neg_zero) { return f2_fma(a, b, neg_zero); }

// ------------------------------------------------------------------------ INT8 codes
// Codes rint(fl(x_hat r)) of two values (Eq. xint8) as an fp16 pair: the fp32 sum of the product and
// 1.5 2^23 rounds it to the nearest integer, ties to even, and its low bits (`shifted`) are the code.
// With r = fl(127 / max |x_hat|) a finite product rounds into [-127, 127] and needs no clamp; `bad`
// becomes NaN when a product is NaN or infinite (NaN input, or r infinite for a row of tiny
// values), and the caller then redoes the row by integer conversion, which maps NaN to 0 and clamps.
constexpr uint32_t kCodeMagic = 0x4b400000u;  // 1.5 2^23
__device__ __forceinline__ uint32_t code_pair(f32x2 xh, f32x2 r2, f32x2 nz, f32x2& bad, f32x2& shifted) {
  const f32x2 p = f2_mul(xh, r2, nz);
  bad = f2_fma(p, 0ull, bad);
  shifted = f2_add(p, f2_both(kCodeMagic));
  float a, b;
  uint32_t h;
  f2_unpack(f2_add(shifted, f2_both(kCodeMagic | 0x80000000u)), a, b);
  asm("cvt.rn.f16x2.f32 %0, %1, %2;\n" : "=r"(h) : "f"(b), "f"(a));
  return h;
}
// The codes of four such pairs as bytes.
__device__ __forceinline__ uint2 code_bytes(const f32x2 (&s)[4]) {
  uint32_t w[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t a = __byte_perm((uint32_t)s[2 * h], (uint32_t)(s[2 * h] >> 32), 0x0040u);
    const uint32_t b = __byte_perm((uint32_t)s[2 * h + 1], (uint32_t)(s[2 * h + 1] >> 32), 0x0040u);
    w[h] = __byte_perm(a, b, 0x5410u);
  }
  return make_uint2(w[0], w[1]);
}
// Two integer codes as an fp16 pair.
__device__ __forceinline__ uint32_t f16_codes(int lo, int hi) {
  return (uint32_t)int_to_f16_bits(lo) | ((uint32_t)int_to_f16_bits(hi) << 16);
}

// --------------------------------------------------------------------- GeGLU fp32 recipe
// gelu_tanh(g) = g / (1 + 2^w), w = -2 log2(e) * sqrt(2/pi) * (g + 0.044715 g^3), each step one
// IEEE fp32 operation rounded to nearest-even, in the order below (no contraction into FMA).
// 2^w = 2^n * p(f), n = rint(w), f = w - n in [-1/2, 1/2], p = degree-7 Taylor polynomial of
// e^{f ln 2} (coefficients (ln 2)^k / k! rounded to fp32), Horner's rule.
__device__ __forceinline__ float exp2_recipe(float w) {
  const float n = rintf(w);
  const float f = __fsub_rn(w, n);
  float p = __uint_as_float(0x377fe5feu);  // (ln2)^7/7!
  p = __fadd_rn(__fmul_rn(p, f), __uint_as_float(0x39218489u));  // (ln2)^6/6!
  p = __fadd_rn(__fmul_rn(p, f), __uint_as_float(0x3aaec3ffu));  // (ln2)^5/5!
  p = __fadd_rn(__fmul_rn(p, f), __uint_as_float(0x3c1d955bu));  // (ln2)^4/4!
  p = __fadd_rn(__fmul_rn(p, f), __uint_as_float(0x3d635847u));  // (ln2)^3/3!
  p = __fadd_rn(__fmul_rn(p, f), __uint_as_float(0x3e75fdf0u));  // (ln2)^2/2!
  p = __fadd_rn(__fmul_rn(p, f), __uint_as_float(0x3f317218u));  // ln2
  p = __fadd_rn(__fmul_rn(p, f), 1.0f);
  const int ni = __float2int_rn(n);                      // |n| <= 126
  const float scale = __int_as_float((ni + 127) << 23);  // 2^n, a normal number
  return __fmul_rn(p, scale);
}

__device__ __forceinline__ float gelu_tanh_recipe(float g) {
  const float g2 = __fmul_rn(g, g);
  const float g3 = __fmul_rn(g2, g);
  const float t = __fadd_rn(g, __fmul_rn(__uint_as_float(0x3d372713u), g3));  // 0.044715
  const float z = __fmul_rn(__uint_as_float(0x3f4c422au), t);                  // sqrt(2/pi)
  float w = __fmul_rn(__uint_as_float(0xc038aa3bu), z);                        // -2 log2(e)
  w = fminf(fmaxf(w, -126.0f), 126.0f);
  const float e = exp2_recipe(w);
  return __fdiv_rn(g, __fadd_rn(1.0f, e));
}

__device__ __forceinline__ float geglu_recipe(float g, float u) { return __fmul_rn(gelu_tanh_recipe(g), u); }

// Whether geglu_pair takes this gate: 2^-60 <= |g| <= 2^60 or +0 (an INT32 sum of 0); NaN, infinities
// and -0 are left to geglu_recipe.
__device__ __forceinline__ bool geglu_in_range(float g) {
  const uint32_t b = __float_as_uint(g);
  return (b & 0x7fffffffu) - 0x21800000u <= 0x5d800000u - 0x21800000u || b == 0u;
}

// geglu_recipe of two (gate, up) pairs, bit for bit, for gates in range: packed operations and no
// branch.  The recipe's division compiles to a routine with a branch to a slow path for extreme
// operands (1 + 2^w reaches 2^126), so neighbouring elements could not be interleaved and the GeGLU
// epilogue, not the MMAs, bounded the GEMM: 2048 x 1152 -> 13824 W8A8 69 us (50 us without GeGLU),
// now 52; bf16 52.9 -> 45.8.
// What makes the steps below the recipe's:
//  * rint(w) is the fp32 sum w + 1.5 2^23 less 1.5 2^23 (|w| < 2^22, ties to even), whose low
//    mantissa bits are the integer;
//  * w is clamped at -60 instead of -126: 1 + 2^w rounds to 1 either way;
//  * everything from 2^w on is scaled by 2^-64 (exact: no step leaves the normal range), which keeps
//    the reciprocal of 1 + 2^w normal;
//  * the quotient is refined by Markstein's method (Computation of elementary functions on the IBM RISC
//    System/6000, 1990): a reciprocal within one ulp, corrected once by its exact residual, then the
//    quotient corrected by its own residual.  From any such reciprocal that rounds correctly for every divisor
//    but the significands 0xfffffd and 0xffffff (checked on the host over all divisors and the dividends
//    whose quotients lie nearest a rounding boundary).  With those, which 1 + 2^w reaches (g = 2^-24), it rests on
//    this GPU's reciprocal: compared with the recipe on all 2.0e9 gates in range (test_gpu_geglu_pair.py), no bit
//    differs.  Leaving the divisors near the top of a binade to the recipe instead cost 3 us of the 93 us
//    FFN block at 2048 tokens.
__device__ __forceinline__ void geglu_pair(float g0, float g1, float u0, float u1, f32x2 nz, float& h0, float& h1) {
  const f32x2 magic = f2_both(0x4b400000u), minus1 = f2_both(0xbf800000u), tiny = f2_both(0x1f800000u);  // 2^-64
  const f32x2 g = f2_pack(g0, g1);
  const f32x2 g3 = f2_mul(f2_mul(g, g, nz), g, nz);
  const f32x2 t = f2_add(g, f2_mul(f2_both(0x3d372713u), g3, nz));
  const f32x2 w2 = f2_mul(f2_both(0xc038aa3bu), f2_mul(f2_both(0x3f4c422au), t, nz), nz);
  float wa, wb;
  f2_unpack(w2, wa, wb);
  wa = fminf(fmaxf(wa, -60.0f), 126.0f);
  wb = fminf(fmaxf(wb, -60.0f), 126.0f);
  const f32x2 w = f2_pack(wa, wb);
  const f32x2 shifted = f2_add(w, magic);
  const f32x2 f = f2_add(w, f2_fma(shifted, minus1, magic));  // w - rint(w)
  f32x2 p = f2_both(0x377fe5feu);
  p = f2_add(f2_mul(p, f, nz), f2_both(0x39218489u));
  p = f2_add(f2_mul(p, f, nz), f2_both(0x3aaec3ffu));
  p = f2_add(f2_mul(p, f, nz), f2_both(0x3c1d955bu));
  p = f2_add(f2_mul(p, f, nz), f2_both(0x3d635847u));
  p = f2_add(f2_mul(p, f, nz), f2_both(0x3e75fdf0u));
  p = f2_add(f2_mul(p, f, nz), f2_both(0x3f317218u));
  p = f2_add(f2_mul(p, f, nz), f2_both(0x3f800000u));
  float sa, sb;
  f2_unpack(shifted, sa, sb);
  const f32x2 scale = f2_pack(__uint_as_float((__float_as_uint(sa) << 23) + (63u << 23)),
                              __uint_as_float((__float_as_uint(sb) << 23) + (63u << 23)));  // 2^(n - 64)
  const f32x2 d = f2_add(tiny, f2_mul(p, scale, nz)), nd = f2_mul(d, minus1, nz);
  float da, db, ya, yb;
  f2_unpack(d, da, db);
  asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(ya) : "f"(da));
  asm("rcp.approx.ftz.f32 %0, %1;\n" : "=f"(yb) : "f"(db));
  f32x2 y = f2_pack(ya, yb);
  y = f2_fma(y, f2_fma(nd, y, f2_both(0x3f800000u)), y);
  f32x2 q = f2_mul(g, y, nz);
  q = f2_fma(f2_fma(nd, q, g), y, q);
  f2_unpack(f2_mul(f2_mul(q, tiny, nz), f2_pack(u0, u1), nz), h0, h1);
}

// ------------------------------------------------------------------------- reductions
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Orderable key for a float (NaN-free): larger float -> larger key.
__device__ __forceinline__ uint32_t float_order_key(float v) {
  const uint32_t b = __float_as_uint(v + 0.0f);  // -0 -> +0
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// The value behind a key's upper half (the inverse of float_order_key); NaN for the empty key.
__device__ __forceinline__ float key_value(unsigned long long key) {
  const uint32_t k = (uint32_t)(key >> 32);
  return __uint_as_float((k & 0x80000000u) ? k ^ 0x80000000u : ~k);
}
// max that is NaN when an operand is
__device__ __forceinline__ float max_nan(float a, float b) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;\n" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

}  // namespace w8a8
