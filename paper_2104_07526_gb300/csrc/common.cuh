// Device helpers shared by the render kernels.
//
// Projection (Sec. 3.1, Listing "basic"): clip = M (x, y, z, 1)^T with M
// row-major; each clip row is summed left to right, every product and sum a
// separately rounded float32 operation (__fmul_rn / __fadd_rn never fuse into
// an FMA), the division is IEEE (__fdiv_rn).  The point is culled unless
// w > 0 and finite, and unless 0 <= s < size on both axes with
// s = (clip / w * 0.5 + 0.5) * size.  pixel = floor(sx) + floor(sy) * width.
//
// Two forms here compute the same results with fewer instructions:
// - ndc * 0.5 + 0.5 is one fused multiply-add.  ndc * 0.5 is exact unless
//   |ndc| < 2^-125, and then both forms round to 0.5.
// - The tests are integer compares of bit patterns.  w lies in (0, inf)
//   exactly when bits(w) - 1 < 0x7F7FFFFF: -0, negatives and NaNs fail.  For
//   s, 0 <= s < size exactly when bits(s) < bits(size): s is never -0, and
//   negatives and NaNs have larger patterns.
// The projection has no branch: every slot of a chunk is projected, and
// culled slots drop out at the one visibility test.  The compiler can then
// interleave the divisions of a lane's slots.
//
// project_slots computes the same results for a lane's slots, two at a time:
// Blackwell's paired float32 instructions (each half rounded on its own, as
// the scalar instruction rounds it) for the matrix rows and the screen
// transform, and one reciprocal per slot shared by both screen divisions,
// with Markstein's correction making each quotient the IEEE one.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace pcr {

constexpr uint32_t kFullMask = 0xFFFFFFFFu;
constexpr uint32_t kNoPixel = 0xFFFFFFFFu;  // viewport is at most 16384^2 < 2^32
constexpr unsigned long long kEmptyKey = 0xFFFFFFFFFFFFFFFFull;
constexpr uint32_t kInfBits = 0x7F800000u;

// Rows 0, 1 and 3 of the matrix plus the viewport, passed by value so every
// thread reads them from the constant bank.
struct ViewParams {
  float r0[4];
  float r1[4];
  float r3[4];
  float fw, fh;
  uint32_t width;
  uint32_t height;
};

__device__ __forceinline__ float row_dot(const float r[4], float x, float y, float z) {
  return __fadd_rn(__fadd_rn(__fadd_rn(__fmul_rn(r[0], x), __fmul_rn(r[1], y)), __fmul_rn(r[2], z)), r[3]);
}

__device__ __forceinline__ float to_screen(float c, float w, float size) {
  return __fmul_rn(__fmaf_rn(__fdiv_rn(c, w), 0.5f, 0.5f), size);
}

// Returns true and the pixel/depth when the point is visible.
__device__ __forceinline__ bool project(const ViewParams& v, float x, float y, float z, uint32_t& pixel,
                                        float& w) {
  w = row_dot(v.r3, x, y, z);
  const bool w_ok = __float_as_uint(w) - 1u < 0x7F7FFFFFu;
  const float cx = row_dot(v.r0, x, y, z);
  const float cy = row_dot(v.r1, x, y, z);
  const float sx = to_screen(cx, w, v.fw);
  const float sy = to_screen(cy, w, v.fh);
  if (!(w_ok && __float_as_uint(sx) < __float_as_uint(v.fw) && __float_as_uint(sy) < __float_as_uint(v.fh)))
    return false;
  // 0 <= s < size here, so converting with round-toward-minus-infinity is floor
  pixel = __float2uint_rd(sx) + __float2uint_rd(sy) * v.width;
  return true;
}

// ---------------------------------------------------------------------------
// Two slots at once.
// ---------------------------------------------------------------------------

// Two floats in one 64-bit register pair: slot a in the low half, slot b in
// the high half.  mul/fma .rn.f32x2 round each half on its own, exactly as
// the scalar .rn instruction would (no flush to zero).
using f32x2 = unsigned long long;

__device__ __forceinline__ f32x2 f2_pack(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void f2_unpack(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 f2_bcast(float x) { return f2_pack(x, x); }
__device__ __forceinline__ f32x2 f2_mul(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 f2_fma(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

__device__ __forceinline__ f32x2 f2_add(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// -0 in both halves, from a value (a viewport size, positive) that the
// assembler cannot know.
__device__ __forceinline__ f32x2 f2_opaque_neg_zero(float positive) {
  return f2_bcast(__uint_as_float((__float_as_uint(positive) & 0x80000000u) ^ 0x80000000u));
}

// One matrix row for two slots, every product and sum rounded on its own.
// A product is written as a fused multiply-add of -0, which rounds as the
// product does (and keeps its sign when it is zero): ptxas fuses a plain
// paired product into a following paired add despite the .rn modifier, which
// would change roundings, but it has no operation for the sum of a fused
// multiply-add and another value.  `nz` must not be a constant it can see.
// Six instructions a row for two slots; nine with scalar sums.
__device__ __forceinline__ f32x2 row_dot2(const float r[4], f32x2 x, f32x2 y, f32x2 z, f32x2 nz) {
  const f32x2 a = f2_fma(f2_bcast(r[0]), x, nz);
  const f32x2 b = f2_fma(f2_bcast(r[1]), y, nz);
  const f32x2 c = f2_fma(f2_bcast(r[2]), z, nz);
  return f2_add(f2_add(f2_add(a, b), c), f2_bcast(r[3]));
}

// Hardware reciprocal estimate (within 1 ulp of 1/w).
__device__ __forceinline__ float rcp_estimate(float w) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(w));
  return r;
}

// w for which the reciprocal path below is exact: [2^-40, 2^40).  Every
// quantity it forms is then a normal number or an exact zero, or the point
// is culled either way (below).
constexpr float kRcpWindowBottom = 0x1p-40f, kRcpWindowTop = 0x1p40f;

__device__ __forceinline__ bool in_rcp_window(float w) {
  return w >= kRcpWindowBottom && w < kRcpWindowTop;
}

// RN(1/w) for both halves: one Newton step with fused operations on the
// estimate y0, y1 = y0 + y0 (1 - w y0).  nw holds -w.
__device__ __forceinline__ f32x2 reciprocal2(f32x2 nw, float wa, float wb) {
  const f32x2 y0 = f2_pack(rcp_estimate(wa), rcp_estimate(wb));
  return f2_fma(y0, f2_fma(nw, y0, f2_bcast(1.0f)), y0);
}

// c / w rounded to nearest even, given y = RN(1/w) (Markstein, IBM J. Res.
// Dev. 34(1), 1990): q0 = RN(c y) lies within one ulp of c / w, so the
// remainder r = c - q0 w is exact in one fused operation, and RN(q0 + r y)
// is the correctly rounded quotient.  That holds while nothing overflows or
// underflows: for w in the window and |c / w| >= 2^-30 every term is normal
// or an exact zero.  Smaller quotients come out below 2^-27 in magnitude, and
// every such quotient gives ndc * 0.5 + 0.5 = 0.5 exactly, as the exact one
// does.  Where c y overflows (|c / w| near 2^128) the result is infinite or
// NaN, and the point is culled, as with the exact quotient (|c / w| > 2).
__device__ __forceinline__ f32x2 quotient2(f32x2 c, f32x2 nw, f32x2 y) {
  const f32x2 q0 = f2_mul(c, y);
  return f2_fma(f2_fma(q0, nw, c), y, q0);
}

// A positive w outside the window, zero or infinity among two slots.  Where
// this is false, w is valid exactly when it is positive: a NaN gives false
// here and is culled by that test.
__device__ __forceinline__ bool leaves_window(float most, float least_magnitude) {
  return most >= kRcpWindowTop || least_magnitude < kRcpWindowBottom;
}

// Screen coordinates of two slots from their clip coordinates and w, with the
// one reciprocal each.
__device__ __forceinline__ void screen_pair(const ViewParams& v, f32x2 cx, f32x2 cy, const float (&w)[2],
                                            float (&sx)[2], float (&sy)[2]) {
  const f32x2 nw = f2_mul(f2_pack(w[0], w[1]), f2_bcast(-1.0f));
  const f32x2 rw = reciprocal2(nw, w[0], w[1]);
  const f32x2 half = f2_bcast(0.5f);
  f2_unpack(f2_mul(f2_fma(quotient2(cx, nw, rw), half, half), f2_bcast(v.fw)), sx[0], sx[1]);
  f2_unpack(f2_mul(f2_fma(quotient2(cy, nw, rw), half, half), f2_bcast(v.fh)), sy[0], sy[1]);
}

// project() for U slots (even U): the same results, bit for bit.  The matrix
// rows are summed in the same order with the same roundings; the screen
// transform is the same fused multiply-add and product; each quotient equals
// the IEEE one (quotient2).  A slot whose w leaves the window takes the IEEE
// divisions, with its pair, or with ONE_TEST (which forms every w first) with
// all slots of the lane.  ONE_TEST saves instructions where the records die
// with the projection: the 800M-point key frame takes 1.852 ms with it and
// 1.869 without, HQS1R (whose records' colours live on) 0.615 and 0.593 ms at
// 100M points, the 8 x 8 batch 21.98 and 21.70 ms.  (With scalar sums and a
// test per slot they took 1.888, 0.609 and 22.21 ms.)  pix[u] is meaningful
// only when vis[u].
template <int U, bool ONE_TEST = false>
__device__ __forceinline__ void project_slots(const ViewParams& v, const uint4 (&r)[U], uint32_t (&pix)[U],
                                              float (&w)[U], bool (&vis)[U]) {
  static_assert(U % 2 == 0, "slots project in pairs");
  const f32x2 nz = f2_opaque_neg_zero(v.fw);
  const uint32_t bw = __float_as_uint(v.fw), bh = __float_as_uint(v.fh);
  auto x = [&](int u) { return f2_pack(__uint_as_float(r[u].x), __uint_as_float(r[u + 1].x)); };
  auto y = [&](int u) { return f2_pack(__uint_as_float(r[u].y), __uint_as_float(r[u + 1].y)); };
  auto z = [&](int u) { return f2_pack(__uint_as_float(r[u].z), __uint_as_float(r[u + 1].z)); };
  if constexpr (ONE_TEST) {
    float most = 0.0f, least = kRcpWindowTop;
#pragma unroll
    for (int u = 0; u < U; u += 2) {
      f2_unpack(row_dot2(v.r3, x(u), y(u), z(u), nz), w[u], w[u + 1]);
      most = fmaxf(fmaxf(most, w[u]), w[u + 1]);
      least = fminf(fminf(least, fabsf(w[u])), fabsf(w[u + 1]));
    }
    if (__builtin_expect(leaves_window(most, least), 0)) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        pix[u] = 0;
        vis[u] = project(v, __uint_as_float(r[u].x), __uint_as_float(r[u].y), __uint_as_float(r[u].z), pix[u], w[u]);
      }
      return;
    }
  }
#pragma unroll
  for (int u = 0; u < U; u += 2) {
    if constexpr (!ONE_TEST) f2_unpack(row_dot2(v.r3, x(u), y(u), z(u), nz), w[u], w[u + 1]);
    const f32x2 cx = row_dot2(v.r0, x(u), y(u), z(u), nz);
    const f32x2 cy = row_dot2(v.r1, x(u), y(u), z(u), nz);
    float sx[2], sy[2];
    screen_pair(v, cx, cy, {w[u], w[u + 1]}, sx, sy);
    if constexpr (!ONE_TEST) {
      if (__builtin_expect(leaves_window(fmaxf(w[u], w[u + 1]), fminf(fabsf(w[u]), fabsf(w[u + 1]))), 0)) {
        float ex[2], ey[2];
        f2_unpack(cx, ex[0], ex[1]);
        f2_unpack(cy, ey[0], ey[1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          sx[k] = w[u + k] < __uint_as_float(kInfBits) ? to_screen(ex[k], w[u + k], v.fw) : -1.0f;  // infinity: culled
          sy[k] = to_screen(ey[k], w[u + k], v.fh);
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      vis[u + k] = w[u + k] > 0.0f && __float_as_uint(sx[k]) < bw && __float_as_uint(sy[k]) < bh;
      pix[u + k] = __float2uint_rd(sx[k]) + __float2uint_rd(sy[k]) * v.width;
    }
  }
}

// 16-byte point load that streams past L1 and marks the line first for
// eviction in L2, so the point stream does not push the framebuffer out.
// The point buffer is read-only while a kernel runs, so the load is a pure
// function of its address and the compiler may schedule it freely.
__device__ __forceinline__ uint4 load_point_stream(const uint4* p, uint64_t policy) {
  uint4 r;
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0,%1,%2,%3}, [%4], %5;"
      : "=r"(r.x), "=r"(r.y), "=r"(r.z), "=r"(r.w)
      : "l"(p), "l"(policy));
  return r;
}

// Two neighbouring 16-byte records (32-byte aligned) in one 32-byte load,
// with the same caching as load_point_stream.
__device__ __forceinline__ void load_pair_stream(const uint4* p, uint64_t policy, uint4& a, uint4& b) {
  asm("ld.global.nc.L1::no_allocate.L2::cache_hint.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8], %9;"
      : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
      : "l"(p), "l"(policy));
}

__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// Unsynchronised read of a framebuffer word for the early depth test
// (Sec. 3.2).  A relaxed load is not a data race against the atomics; a
// stale value can only be larger than the current one (values only
// decrease), which costs an extra atomic and never a wrong pixel.  These
// reads and the atomics below are volatile (kept in program order among
// themselves) but carry no memory clobber: nothing in a render kernel reads
// the framebuffer through ordinary loads.
__device__ __forceinline__ unsigned long long load_relaxed_u64(const unsigned long long* p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}

__device__ __forceinline__ uint32_t load_relaxed_u32(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
  return v;
}

// Fire-and-forget atomic minimum / add (the result is never read), with an
// L2 evict-last hint so the framebuffer stays resident.
__device__ __forceinline__ void red_min_u64(unsigned long long* p, unsigned long long v, uint64_t policy) {
  asm volatile("red.relaxed.gpu.global.min.u64.L2::cache_hint [%0], %1, %2;" ::"l"(p), "l"(v), "l"(policy));
}

__device__ __forceinline__ void red_min_u32(uint32_t* p, uint32_t v, uint64_t policy) {
  asm volatile("red.relaxed.gpu.global.min.u32.L2::cache_hint [%0], %1, %2;" ::"l"(p), "r"(v), "l"(policy));
}

__device__ __forceinline__ void red_add_u64(unsigned long long* p, unsigned long long v, uint64_t policy) {
  asm volatile("red.relaxed.gpu.global.add.u64.L2::cache_hint [%0], %1, %2;" ::"l"(p), "l"(v), "l"(policy));
}

// Atomic add that returns the previous value (needed by the single-atomic
// high-quality pass to detect a full primary word).
__device__ __forceinline__ unsigned long long atom_add_u64(unsigned long long* p, unsigned long long v,
                                                           uint64_t policy) {
  unsigned long long old;
  asm volatile("atom.relaxed.gpu.global.add.u64.L2::cache_hint %0, [%1], %2, %3;"
               : "=l"(old)
               : "l"(p), "l"(v), "l"(policy));
  return old;
}

__device__ __forceinline__ unsigned long long atom_exch_u64(unsigned long long* p, unsigned long long v) {
  unsigned long long old;
  asm volatile("atom.relaxed.gpu.global.exch.b64 %0, [%1], %2;" : "=l"(old) : "l"(p), "l"(v));
  return old;
}

__device__ __forceinline__ uint32_t lane_id() { return threadIdx.x & 31u; }

// Start of every kernel (see launch_kernel): returns once the previous kernel
// of the stream, and so everything before it, has finished and its writes are
// visible; no kernel but
// k_clear_sums touches global memory before.  The branch, never taken,
// keeps the compiler from moving loads it takes for constant (of const
// __restrict__ parameters) above the wait: past it they would be speculative.
__device__ __forceinline__ void after_previous() {
  uint32_t never;
  asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, 0;" : "=r"(never)::"memory");
  if (never != 0u) {
    asm volatile("exit;");
    __builtin_unreachable();
  }
}

// Lets the next kernel's blocks start once every block of this one has called
// it: only for a next kernel that touches nothing of this one's before its own
// after_previous().
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

}  // namespace pcr
