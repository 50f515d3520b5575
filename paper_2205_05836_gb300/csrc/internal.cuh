// Internal helpers shared by the CUDA translation units of libcutqc.
// Nothing here is part of the public C ABI (see include/cutqc.h).
#pragma once

#include <cuda_runtime.h>
#include <cuda_fp16.h>
#include <stdint.h>
#include <stddef.h>

#include "../../include/cutqc.h"

namespace cutqc {

// ---------------------------------------------------------------- host side

// Records a message for cutqc_last_error() (thread-local) and returns code.
int set_error(int code, const char* fmt, ...);
// Maps a CUDA runtime error to CUTQC_ECUDA with its text.
int cuda_error(cudaError_t e, const char* where);

#define CUTQC_CUDA_TRY(expr)                                          \
  do {                                                                \
    cudaError_t _e = (expr);                                          \
    if (_e != cudaSuccess) return ::cutqc::cuda_error(_e, #expr);     \
  } while (0)

// Kernels enqueued (or captured into a graph) by the library, process-wide:
// every launch site is followed by one CUTQC_LAUNCH_CHECK, which counts it;
// a check that covers several launches adds the others with count_launches.
void count_launches(int n);

#define CUTQC_LAUNCH_CHECK(where)                                     \
  do {                                                                \
    ::cutqc::count_launches(1);                                       \
    cudaError_t _e = cudaGetLastError();                              \
    if (_e != cudaSuccess) return ::cutqc::cuda_error(_e, where);     \
  } while (0)

// Device-side status word: kernels that wait on a barrier give up after a
// bounded time and record why here; the host reads it with
// cutqc_device_status().
int* device_status_ptr();

// Number of SMs of the current device (cached per device).
int sm_count();

// Launch of a kernel whose CTAs may start while the kernel before it on the
// stream is still running its last ones (programmatic dependent launch): it
// must call grid_dependency_wait() before it touches anything that kernel
// writes (or reads, if it overwrites it).
template <class... P, class... A>
inline cudaError_t launch_dependent(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                    A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ---------------------------------------------------------------- device side

__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

__device__ __forceinline__ void record_status(int* status, int code) {
  if (status) atomicCAS(status, 0, code);
}

// IEEE 754 binary64 -> binary32, round to nearest, ties to even, on the
// integer pipes.  GB300's FP64 pipe converts only a few values per SM per
// clock, which is what bounded the FP64 attribution loads; this follows the
// two formats' definitions instead.  Binary64 fields: sign, 11-bit exponent
// e (bias 1023), 52-bit fraction; binary32: 8-bit exponent (bias 127), 23-bit
// fraction, subnormals in units of 2^-149.  NaN stays a (quiet) NaN.
// The rare cases: binary32 subnormals and underflow, overflow, infinities,
// NaN (e in 1..896 or 1151..2047).
__device__ __forceinline__ float f64_to_f32_rare(unsigned hi, unsigned lo) {
  const unsigned sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7ffu);
  const unsigned fh = hi & 0xfffffu;                        // fraction bits 51..32
  if (e == 0x7ff) return __uint_as_float(sign | ((fh | lo) ? 0x7fc00000u : 0x7f800000u));
  if (e >= 1151) return __uint_as_float(sign | 0x7f800000u);  // |d| >= 2^128
  // binary32 subnormal or zero: d = sig * 2^(e - 1075) with sig = 2^52 +
  // fraction, i.e. sig * 2^(e - 926) units of 2^-149
  const int s = 926 - e;                                     // >= 30 here
  if (e == 0 || s >= 54) return __uint_as_float(sign);
  const unsigned long long sig = (1ull << 52) | ((unsigned long long)fh << 32) | lo;
  unsigned long long q = sig >> s;
  const unsigned long long rem = sig & ((1ull << s) - 1), half = 1ull << (s - 1);
  q += (rem > half || (rem == half && (q & 1ull))) ? 1ull : 0ull;
  return __uint_as_float(sign | (unsigned)q);
}

// The common case in a handful of instructions: a binary32 normal result
// (biased exponent e - 896 in 1..254: rebias the exponent, keep fraction bits
// 51..29, round on bits 28..0, the low bit of r deciding a tie; a carry out
// of the fraction bumps the exponent, to infinity above the largest float),
// or zero for e = 0 (zero or a binary64 subnormal).  The rare cases run only
// in warps that hold one, behind a vote, so that the common path keeps its
// registers and needs no branch per value.
__device__ __forceinline__ float f64_to_f32_rn(double d) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(d);
  const unsigned hi = (unsigned)(u >> 32), lo = (unsigned)u;
  const unsigned mag = hi & 0x7fffffffu;
  const unsigned e = mag >> 20;
  unsigned r = ((mag - (896u << 20)) << 3) | (lo >> 29);
  r += ((lo & 0x1fffffffu) + (r & 1u)) > 0x10000000u ? 1u : 0u;
  r = e == 0 ? 0u : r;
  float f = __uint_as_float((hi & 0x80000000u) | r);
  const bool rare = e != 0 && e - 897u >= 254u;
  if (__any_sync(__activemask(), rare)) {
    if (rare) f = f64_to_f32_rare(hi, lo);
  }
  return f;
}

// Two fused multiply-adds per lane and instruction (each half rounded as
// fmaf rounds).  On GB300 scalar FFMA reaches 60 TFLOP/s and the packed form
// 76 (register-only loops), with half the issue slots.
__device__ __forceinline__ unsigned long long ffma2(unsigned long long a, unsigned long long b,
                                                    unsigned long long c) {
  unsigned long long d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ unsigned long long pair2(float a) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(a));
  return d;
}
__device__ __forceinline__ unsigned long long pack2(uint32_t a, uint32_t b) {
  unsigned long long d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "r"(a), "r"(b));
  return d;
}
__device__ __forceinline__ unsigned long long fadd2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ unsigned long long fmul2(unsigned long long a, unsigned long long b) {
  unsigned long long d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float2 unpack2(unsigned long long v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}

// A float32 sum that carries its rounding errors beside it (Knuth's two-sum:
// each step's error is exact), for totals that go on in float64.  A float64
// add per group of outputs is exact too, but GB300's FP64 pipe takes a few
// lanes per clock.  Terms up to the float32 range over their number.
struct Sum2 {
  float s = 0.f, e = 0.f;
  __device__ __forceinline__ void add(float v) {
    const float t = __fadd_rn(s, v), b = __fsub_rn(t, s);
    e = __fadd_rn(e, __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(v, b)));
    s = t;
  }
  __device__ __forceinline__ void add(const Sum2& o) {
    add(o.s);
    e = __fadd_rn(e, o.e);
  }
  // (after an infinity or a NaN the errors mean nothing)
  __device__ __forceinline__ double value() const { return isfinite(s) ? (double)s + (double)e : (double)s; }
};
// Two of them in the halves of packed registers.
struct Sum2x2 {
  unsigned long long s = 0ull, e = 0ull;
  static __device__ __forceinline__ unsigned long long sub(unsigned long long a, unsigned long long b) {
    return fadd2(a, b ^ 0x8000000080000000ull);
  }
  __device__ __forceinline__ void add(unsigned long long v) {
    const unsigned long long t = fadd2(s, v), b = sub(t, s);
    e = fadd2(e, fadd2(sub(s, sub(t, b)), sub(v, b)));
    s = t;
  }
  __device__ __forceinline__ double value() const {
    const float2 a = unpack2(s), b = unpack2(e);
    return (isfinite(a.x) ? (double)a.x + (double)b.x : (double)a.x) +
           (isfinite(a.y) ? (double)a.y + (double)b.y : (double)a.y);
  }
};

// Software bit deposit: scatter the low bits of v to the set bits of mask.
__host__ __device__ __forceinline__ uint64_t pdep64(uint64_t v, uint64_t mask) {
  uint64_t r = 0;
  while (mask) {
    uint64_t low = mask & (~mask + 1);
    if (v & 1) r |= low;
    v >>= 1;
    mask &= mask - 1;
  }
  return r;
}

// A bit deposit whose mask is known on the host.  Masks below 2^32 (every
// output of DD, and most of FD) take the five shift-and-select steps of the
// parallel expand (Warren, Hacker's Delight, section 7-5), a dozen dependent
// instructions; the loop above takes some thirty cycles per mask bit, which
// was most of a small task's time in the persistent DD kernel.
struct Deposit {
  uint64_t mask;
  uint32_t mv[5];     // bits that step i moves up by 2^i
  int fast;           // mask < 2^32
  uint64_t bit[2];    // places of bits 0 and 1
  // the place of a value plus the value deposited at d
  __device__ __forceinline__ uint64_t next(uint64_t at, uint64_t d) const { return ((at | ~mask) + d) & mask; }
  __device__ __forceinline__ uint64_t operator()(uint64_t v) const {
    if (!fast) return pdep64(v, mask);
    uint32_t x = (uint32_t)v;
#pragma unroll
    for (int i = 4; i >= 0; --i) {
      const uint32_t m = mv[i];
      x = (x & ~m) | ((x << (1 << i)) & m);
    }
    return x & (uint32_t)mask;
  }
};
inline Deposit make_deposit(uint64_t mask) {
  Deposit d{};
  d.mask = mask;
  d.bit[0] = pdep64(1, mask);
  d.bit[1] = pdep64(2, mask);
  d.fast = (mask >> 32) == 0;
  uint32_t m = (uint32_t)mask, mk = ~m << 1;     // mk: zeros to the right of each bit, counted
  for (int i = 0; i < 5 && d.fast; ++i) {
    uint32_t mp = mk ^ (mk << 1);
    mp ^= mp << 2;
    mp ^= mp << 4;
    mp ^= mp << 8;
    mp ^= mp << 16;
    const uint32_t mv = mp & m;                  // bits an odd number of 2^i places up
    m = (m ^ mv) | (mv >> (1 << i));
    mk &= ~mp;
    d.mv[i] = mv;
  }
  return d;
}

// Software bit extract: gather the bits of v at the set bits of mask.
__host__ __device__ __forceinline__ uint64_t pext64(uint64_t v, uint64_t mask) {
  uint64_t r = 0;
  int k = 0;
  while (mask) {
    uint64_t low = mask & (~mask + 1);
    if (v & low) r |= (uint64_t)1 << k;
    ++k;
    mask &= mask - 1;
  }
  return r;
}

// A contraction step's operand view and result layout (see contract.cu).
struct OperandView {
  const float* src;      // [2^o][4^k] fp32 tensor (rows x, columns c)
  int o;                 // output bits of the source tensor
  int k;                 // cut digits of the source tensor (columns 4^k)
  uint64_t open_dmask;   // bit mask (2 bits per digit) of the open digits in c
  uint64_t shared_dmask; // bit mask of the shared (contracted) digits in c
  int n_open;            // number of open digits
  int n_shared;          // number of shared digits
  int64_t rows() const { return ((int64_t)1 << o) << (2 * n_open); }
  int64_t kdim() const { return (int64_t)1 << (2 * n_shared); }
};

}  // namespace cutqc
