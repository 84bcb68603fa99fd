// Prefill quantisers of the inner-grouped cache: the middle tokens of every unit into the ROW store (groups of G
// channels inside a token, Section "InnerQ" for keys) and the BLOCK store (per-channel groups of G tokens, values).
//
// Both are built around one work item: 32 values of one group held in the registers of one thread (a group of
// 64 or 128 values is 2 or 4 such threads, which exchange their minima / maxima and error sums).  The thread
// makes the passes the method needs over its registers: min / max, then (hybrid mode only) the L1 errors of both
// candidates, then the codes of the chosen mode.  All value arithmetic is the same sequence of single, correctly
// rounded fp32 operations as in group_params / asym_code / sym_code, so stored bits do not depend on the kernel:
// rounding to an integer is done by adding 1.5 * 2^23 (round-to-nearest-even at unit granularity, identical to
// rintf for |t| < 2^22), which leaves the code in the low mantissa bits.  |t| before the clamp is at most a few times 2^b
// plus the rounding error of the zero-point in units of the scale: keys are divided by the root of their largest value, so
// their zero-point is below 2^8 and off by 2^-4 at most, and the smallest fp16 scale is 2^-24, hence |t| < 2^21.
//
// What bounds them: instruction issue (both read and write far below the HBM rate).  Values are kept as PAIRS and most
// adds / multiplies are packed fp32x2 instructions, whose two halves are rounded exactly as the scalar ones.  A packed (or
// half-precision pair) instruction occupies its pipe and the issue for two cycles, as two scalar ones do; it saves
// instruction fetches and registers, not time.
#include <algorithm>
#include <atomic>
#include <type_traits>

#include "innerq_device.cuh"
#include "innerq_div_const.h"
#include "innerq_kernels.h"

namespace iq {

namespace {

constexpr float kMagic = 12582912.0f;       // 1.5 * 2^23
constexpr int kSeg = 32;                    // values per thread and group
constexpr int kCopies = 8;                  // 16-byte copies in flight per thread
constexpr int kRowsCtasPerSm = 4;           // of 128 threads and 128 registers (5 or 6 with fewer registers: +-1 %)

// ---- two fp32 values in a 64-bit register pair
using F2 = unsigned long long;
__device__ __forceinline__ F2 f2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 unf2(F2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// Product rounded by itself, as a * b + (-0).  A mul.rn.f32x2 (or an fma with a literal -0) is contracted by the
// assembler with a following packed add, although its scalar form never is, and that moves codes at rounding ties; so
// the -0 comes from a kernel argument, whose value the assembler does not know.
struct Mul2 {
  F2 neg_zero;
  __device__ __forceinline__ explicit Mul2(float nz) : neg_zero(f2(nz, nz)) {}
  __device__ __forceinline__ F2 operator()(F2 a, F2 b) const { return fma2(a, b, neg_zero); }
};

// group_params (innerq_device.cuh) with its divisions by constants and reciprocals in their cheaper correctly rounded
// forms: the same bits.
template <int BITS> __device__ __forceinline__ GroupParams seg_params(float mn, float mx, int sym_variant) {
  GroupParams p;
  constexpr int L = (1 << BITS) - 1, half = 1 << (BITS - 1);
  p.L = (float)L;
  p.half = (float)half;
  p.sa_bits = f2h_bits(div_const<L>(__fsub_rn(mx, mn)));
  p.z_bits = f2h_bits(mn);
  p.s_a = h2f_bits(p.sa_bits);
  p.z_a = h2f_bits(p.z_bits);
  p.inv_a = p.s_a == 0.f ? 0.f : __frcp_rn(p.s_a);
  const float am = fmaxf(fabsf(mn), fabsf(mx));
  if (sym_variant == 0) {
    p.ss_bits = f2h_bits(div_const<half - 1>(am));
    p.q_lo = -(float)(half - 1);
  } else {
    p.ss_bits = f2h_bits(div_const<L>(am));
    p.q_lo = -(float)half;
  }
  p.q_hi = (float)(half - 1);
  p.s_s = h2f_bits(p.ss_bits);
  p.inv_s = p.s_s == 0.f ? 0.f : __frcp_rn(p.s_s);
  return p;
}

// Clamp bounds of both candidates in the magic domain, and whether any value of the group can need them.
struct Bounds {
  float off_s, lo_s, hi_s, hi_a;            // symmetric: magic + 2^(b-1) and its bounds; asymmetric: [magic, hi_a]
  bool no_clip;
  __device__ __forceinline__ Bounds(Mul2 mul2, const GroupParams& p, float mn, float mx)
      : off_s(kMagic + p.half), lo_s(off_s + p.q_lo), hi_s(off_s + p.q_hi), hi_a(kMagic + p.L) {
    // Both coders are non-decreasing in x (each step is a correctly rounded monotone operation and the reciprocal
    // scales are >= 0), so if the group's minimum and maximum land inside the code range, every value does.
    const F2 ends = f2(mn, mx);
    const float2 a = unf2(add2(mul2(add2(ends, f2(-p.z_a, -p.z_a)), f2(p.inv_a, p.inv_a)), f2(kMagic, kMagic)));
    const float2 s = unf2(add2(mul2(ends, f2(p.inv_s, p.inv_s)), f2(off_s, off_s)));
    no_clip = a.x >= kMagic && a.y <= hi_a && s.x >= lo_s && s.y <= hi_s;
  }
};

// The coders for a pair of values whose parameters may differ (two channels) or not (two values of one group).
// Asymmetric: ((x - z) * inv) + magic; symmetric: (x * inv) + (magic + 2^(b-1)): the low mantissa bits are the stored
// code.  CLAMP = false leaves out the clamp to the code range, for groups where no_clip holds.
struct PairCoder {
  Mul2 mul2;
  F2 nz_a, inv_a, ns_a, inv_s, off_s, noff_s, ns_s;
  float2 hi_a, lo_s, hi_s;
  __device__ __forceinline__ PairCoder(Mul2 mul, const GroupParams& p, const Bounds& b, const GroupParams& q, const Bounds& d)
      : mul2(mul), nz_a(f2(-p.z_a, -q.z_a)), inv_a(f2(p.inv_a, q.inv_a)), ns_a(f2(-p.s_a, -q.s_a)), inv_s(f2(p.inv_s, q.inv_s)),
        off_s(f2(b.off_s, d.off_s)), noff_s(f2(-b.off_s, -d.off_s)), ns_s(f2(-p.s_s, -q.s_s)),
        hi_a(make_float2(b.hi_a, d.hi_a)), lo_s(make_float2(b.lo_s, d.lo_s)), hi_s(make_float2(b.hi_s, d.hi_s)) {}
  static __device__ __forceinline__ F2 clamp2(F2 t, float2 lo, float2 hi) {
    const float2 v = unf2(t);
    return f2(fminf(fmaxf(v.x, lo.x), hi.x), fminf(fmaxf(v.y, lo.y), hi.y));
  }
  // L1 reconstruction errors (signed) of both candidates: used only to pick the mode of a hybrid group
  template <bool CLAMP> __device__ __forceinline__ float2 err_asym(F2 x) const {
    const F2 d = add2(x, nz_a);
    F2 t = add2(mul2(d, inv_a), f2(kMagic, kMagic));
    if (CLAMP) t = clamp2(t, make_float2(kMagic, kMagic), hi_a);
    return unf2(fma2(ns_a, add2(t, f2(-kMagic, -kMagic)), d));
  }
  template <bool CLAMP> __device__ __forceinline__ float2 err_sym(F2 x) const {
    F2 t = add2(mul2(x, inv_s), off_s);
    if (CLAMP) t = clamp2(t, lo_s, hi_s);
    return unf2(fma2(ns_s, add2(t, noff_s), x));
  }
};

// The coder of the chosen mode as one formula, clamp(((x - z) * inv) + off): symmetric is z = 0 (x - 0 is exact).
struct ChosenPair {
  Mul2 mul2;
  F2 nz, inv, off;
  float2 lo, hi;
  __device__ __forceinline__ ChosenPair(Mul2 mul, const GroupParams& p, const Bounds& b, bool asym_p, const GroupParams& q,
                                        const Bounds& d, bool asym_q)
      : mul2(mul), nz(f2(asym_p ? -p.z_a : 0.f, asym_q ? -q.z_a : 0.f)), inv(f2(asym_p ? p.inv_a : p.inv_s, asym_q ? q.inv_a : q.inv_s)),
        off(f2(asym_p ? kMagic : b.off_s, asym_q ? kMagic : d.off_s)),
        lo(make_float2(asym_p ? kMagic : b.lo_s, asym_q ? kMagic : d.lo_s)),
        hi(make_float2(asym_p ? b.hi_a : b.hi_s, asym_q ? d.hi_a : d.hi_s)) {}
  // bits of (1.5 * 2^23 + code) of both values: the low byte is the code
  template <bool CLAMP> __device__ __forceinline__ uint2 code_bits(F2 x) const {
    F2 t = add2(mul2(add2(x, nz), inv), off);
    if (CLAMP) t = PairCoder::clamp2(t, lo, hi);
    const float2 v = unf2(t);
    return make_uint2(__float_as_uint(v.x), __float_as_uint(v.y));
  }
};

// Both candidates' L1 errors with fewer operations than PairCoder's, for the groups whose mode they settle beyond doubt
// (quick_mode); the others get the sums above.  A segment's sums of one channel; packed and half-precision instructions
// issue over two cycles, so what counts is operations: 11 per value above, 12.4 cycles measured.  32 units x 16384 tokens,
// both tensors: 150 us before, 132 with 2 bits; 4 bits 151 and 138; groups that nothing but the sums above decides (equal
// errors everywhere) cost 10 % more.
//   2 bits: the distance to the nearest of four equidistant levels is | ||x - c| - s| - s/2 | with c in their middle, to
//           the nearest of -s, 0, s it is s/2 - ||x| - s/2|: 6 operations, 6.7 cycles; a scalar addition takes the
//           absolute value of its operand for free.
//   3, 4 bits: y = x / s + const is rounded at 2^-16 by a fused multiply-add whose result lies in [128, 256): the low 16
//           bits are the distance to the nearest code as a signed fraction.  Its absolute value (the smaller of it and its
//           complement, one unit off where it is negative) is summed by dp2a: 7.4 cycles.  Needs codes within their
//           range (no_clip), scales that are not zero and a zero-point of at most 64 scales.
template <int BITS> struct QuickErr {
  F2 nc, inv_a, off_a, inv_s;               // pairs for the two operands of add()
  float2 s_a, h_a, h_s;
  float2 a = make_float2(0.f, 0.f), t = make_float2(0.f, 0.f);
  uint32_t ua0 = 0, ua1 = 0, us0 = 0, us1 = 0;
  static constexpr float kFrac = 192.f;     // 1.5 * 2^7
  __device__ __forceinline__ QuickErr(const GroupParams& p, const GroupParams& q)
      : nc(f2(-fmaf(1.5f, p.s_a, p.z_a), -fmaf(1.5f, q.s_a, q.z_a))), inv_a(f2(p.inv_a, q.inv_a)),
        off_a(f2(fmaf(-p.z_a, p.inv_a, kFrac), fmaf(-q.z_a, q.inv_a, kFrac))), inv_s(f2(p.inv_s, q.inv_s)),
        s_a(make_float2(p.s_a, q.s_a)), h_a(make_float2(0.5f * p.s_a, 0.5f * q.s_a)), h_s(make_float2(0.5f * p.s_s, 0.5f * q.s_s)) {}
  // values lo and hi of one group: distances to their nearest codes, in the two halves of a word
  static __device__ __forceinline__ uint32_t frac_abs(float lo, float hi) {
    const uint32_t f = __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x5410);
    return __vminu2(f, ~f);
  }
  static __device__ __forceinline__ void acc2(uint32_t& acc, uint32_t f) {
    asm("dp2a.lo.u32.u32 %0, %1, %2, %0;" : "+r"(acc) : "r"(f), "r"(0x0101));
  }
  // x, y: two pairs, the first halves of both belong to one group and the second halves to another (or to the same one)
  __device__ __forceinline__ void add(F2 x, F2 y) {
    if constexpr (BITS == 2) {
      one(x);
      one(y);
    } else {
      const F2 k = f2(kFrac, kFrac);
      const float2 ax = unf2(fma2(x, inv_a, off_a)), ay = unf2(fma2(y, inv_a, off_a));
      const float2 sx = unf2(fma2(x, inv_s, k)), sy = unf2(fma2(y, inv_s, k));
      acc2(ua0, frac_abs(ax.x, ay.x));
      acc2(ua1, frac_abs(ax.y, ay.y));
      acc2(us0, frac_abs(sx.x, sy.x));
      acc2(us1, frac_abs(sx.y, sy.y));
    }
  }
  __device__ __forceinline__ void one(F2 x) {
    const float2 v = unf2(x), d = unf2(add2(x, nc));
    a.x += fabsf(fabsf(fabsf(d.x) - s_a.x) - h_a.x);
    a.y += fabsf(fabsf(fabsf(d.y) - s_a.y) - h_a.y);
    t.x += fabsf(fabsf(v.x) - h_s.x);
    t.y += fabsf(fabsf(v.y) - h_s.y);
  }
  // (asymmetric - symmetric) error sum of the n values that went into the first / second halves
  __device__ __forceinline__ float2 difference(float n) const {
    if constexpr (BITS == 2) return make_float2(a.x - fmaf(n, h_s.x, -t.x), a.y - fmaf(n, h_s.y, -t.y));
    const float u = 0x1p-16f;
    return make_float2(u * (s_a.x * (float)ua0 - 2.f * h_s.x * (float)us0), u * (s_a.y * (float)ua1 - 2.f * h_s.y * (float)us1));
  }
};

// How far a group's difference of the quick sums and that of PairCoder's can be apart; infinite where the quick sums mean
// nothing (infinite or NaN also where a value is infinite: no comparison with it settles anything).  A NaN shows in neither
// scale nor bound, and 3- and 4-bit sums count it as 0: groups with one get PairCoder's sums, whose NaN makes them symmetric
// as in the append (see `nan`: the maximum that propagates NaN costs what the other one does, the branch 1 to 1.5 % of a
// prefill; parameters that the rare path below makes anew instead cost 4 %).  2-bit sums show a NaN themselves.  m = largest
// |x| of the group.
// 2 bits: a value's rounding errors are below 2^-20 m in each form, those of adding up 32 of them in two chains below
// 2^-20 m a value; a value beyond the outer symmetric level (whose fp16 scale may be rounded down) counts with the wrong
// sign.  3, 4 bits: in units of 2^-16 scales a value is off by 1 (complement), 1/2 (constant), 1/2 (rounding) and 1/8
// (reciprocal scales, the other form's own roundings).
template <int BITS>
__device__ __forceinline__ float quick_bound(const GroupParams& p, const Bounds& b, float mn, float mx, int G) {
  const float m = fmaxf(fabsf(mn), fabsf(mx)), n = (float)G;
  if constexpr (BITS == 2)
    return n * (m * 0x1p-18f + 2.f * fmaxf(0.f, m - p.s_s));
  else
    return b.no_clip && p.s_a > 0.f && p.s_s > 0.f && fabsf(p.z_a) * p.inv_a < 60.f ? n * 3.f * 0x1p-16f * (p.s_a + p.s_s) : INFINITY;
}
// 1: asymmetric, 0: symmetric, -1: the quick sums do not tell
__device__ __forceinline__ int quick_mode(float difference, float bound) {
  return difference > bound ? 0 : difference < -bound ? 1 : -1;
}

__device__ __forceinline__ float min3(float a, float b, float c) {
  float r;
  asm("min.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// the same; with 3 and 4 bits a NaN among the three is the result
template <int BITS> __device__ __forceinline__ float max3_nan(float a, float b, float c) {
  if constexpr (BITS == 2) return max3(a, b, c);
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// low bytes of four code words as the four bytes of one word
__device__ __forceinline__ uint32_t bytes4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  return __byte_perm(__byte_perm(a, b, 0x0040), __byte_perm(c, d, 0x0040), 0x5410);
}

// 3-bit codes in byte order (see row_pos_i8_3 / block_pos_i8_3): four codes in the bytes of w become the 2-bit plane's
// bytes (bit position 0) and the 1-bit plane's bytes (bit 0); `odd` (the bit position of the segment is odd) picks the
// split of a code between the planes.
__device__ __forceinline__ void split_planes(uint32_t w, int odd, uint32_t& lo, uint32_t& hi) {
  lo = (w >> odd) & 0x03030303u;
  hi = (w >> (odd ? 0 : 2)) & 0x01010101u;
}

// Reduce-scatter by OR over the four lanes 4q .. 4q+3 of 2 * NJ words v[NH * j + h], j = 0..3 (h = 0..NH-1): lane
// `pos` of the four ends up with the complete words of j = pos.
template <int NH> __device__ __forceinline__ void quad_reduce_scatter(const uint32_t (&v)[4 * NH], int pos, uint32_t (&out)[NH]) {
  uint32_t m[2 * NH];                          // step 1: keep the j of my parity (j = 2 i + (pos & 1))
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int h = 0; h < NH; ++h) {
      const uint32_t keep = (pos & 1) ? v[NH * (2 * i + 1) + h] : v[NH * (2 * i) + h];
      const uint32_t give = (pos & 1) ? v[NH * (2 * i) + h] : v[NH * (2 * i + 1) + h];
      m[NH * i + h] = keep | __shfl_xor_sync(0xffffffffu, give, 1);
    }
#pragma unroll
  for (int h = 0; h < NH; ++h) {               // step 2: keep i = pos >> 1
    const uint32_t keep = (pos & 2) ? m[NH + h] : m[h];
    const uint32_t give = (pos & 2) ? m[h] : m[NH + h];
    out[h] = keep | __shfl_xor_sync(0xffffffffu, give, 2);
  }
}

// How prefill_first_kernel divides the keys for their maxima: slices of 128 rows (per_unit of them), `ctas` CTAs with a
// contiguous share each, which leave one row of 128 partial maxima per unit they meet, in that unit's `stride` rows.
struct MaxShares {
  int per_unit, ctas, stride;
  __host__ __device__ int total(int U) const { return U * per_unit; }
  // (products of a slice and a CTA stay below 2^32: a slice is 32 KB of keys)
  __host__ __device__ int begin(int U, int cta) const { return (int)((uint32_t)total(U) * (uint32_t)cta / (uint32_t)ctas); }
  __host__ __device__ int cta_of(int U, int slice) const {      // whose share holds the slice
    return (int)(((uint32_t)(slice + 1) * (uint32_t)ctas + (uint32_t)total(U) - 1u) / (uint32_t)total(U)) - 1;
  }
};
// Key norm of one channel from the partial maxima: sqrt(max |K|), 0 -> 1 (Section "Per-channel Normalization of K").
__device__ __forceinline__ float key_norm(const float* __restrict__ absmax, const MaxShares& ms, int U, int u, int c) {
  const float* p = absmax + (size_t)u * ms.stride * kD + c;
  const int n_part = ms.cta_of(U, (u + 1) * ms.per_unit - 1) - ms.cta_of(U, u * ms.per_unit) + 1;
  float m = 0.f;
#pragma unroll 8
  for (int i = 0; i < n_part; ++i) m = fmaxf(m, __ldcg(p + (size_t)i * kD));
  const float n = __fsqrt_rn(m);
  return n == 0.f ? 1.0f : n;
}

// Chunk record ci (32 tokens) of a unit: chunk_rec_ptr with the group size's shift instead of divisions (a group has
// 1 << sh chunks; the inner-grouped record starts with its chunks).
__device__ __forceinline__ unsigned char* chunk_ptr(const Rec& rec, const Store& S, int ci, int sh) {
  return group_ptr(rec, ci >> sh) + (ci & ((1 << sh) - 1)) * S.chunk_stride;
}

// ------------------------------------------------------------------ ROW store
// A warp quantises 8 consecutive tokens per iteration: lane = 4 * (token in the batch) + segment, segment =
// channels 32*seg .. 32*seg+31, which is one bit position (2, 3 bits: p = seg; 4 bits: nibble seg % 2 of row half
// seg / 2) of the bytes of the packed row.  The four lanes of a token exchange their words so that each stores a
// contiguous run of complete ones; the 8 packed rows and their metadata entries are contiguous in the chunk record.
// (Through shared memory with an atomic OR per word instead: 22 more shared-memory operations per 32 values.)
// CTA x of the grid takes the x-th part of all units' batches (a contiguous run, so every CTA ends at the same time
// whatever the number of units), unit by unit.
// NORM: the unit's key norm comes from `absmax`, the partial maxima that prefill_first_kernel wrote; every
// unit's norm is stored once.  The launch may start before that kernel has ended (griddepcontrol.wait).
template <int BITS, bool NORM>
__global__ void __launch_bounds__(128, kRowsCtasPerSm)
quantize_rows_prefill_kernel(const __grid_constant__ Layout L, const __half* __restrict__ X, int N, int n_q,
                             unsigned char* __restrict__ cache, const float* __restrict__ absmax, const MaxShares ms, float neg_zero) {
  const Mul2 mul2(neg_zero);
  const Store& S = L.k;
  constexpr int RW = 4 * BITS;                // 32-bit words per packed row
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int seg = lane & 3, tk = lane >> 2;
  const int gl = L.G >> 5, sh = gl >> 1;      // lanes per group: 1, 2 or 4, and its logarithm
  // reciprocal key norms: segment rows padded to 36 words, so that the four lanes of a token read different banks
  __shared__ __align__(16) float inv_s[NORM ? 4 * 36 : 4];
  // What follows may start: a kernel of this cache waits before it touches anything (innerq_quantize_prefill has reset N_safe
  // and reads_settled; a paged decode looks at its page table before that, which no kernel writes), one of another cache that
  // does not touches nothing that a prefill writes, and the triggers and waits in between keep the kernels of that cache in
  // their order.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  if constexpr (NORM) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    float* norm = reinterpret_cast<float*>(cache + L.norm_off);
    for (int u = blockIdx.x; u < L.U; u += gridDim.x) norm[(size_t)u * kD + threadIdx.x] = key_norm(absmax, ms, L.U, u, threadIdx.x);
  }
  const int n_batches = (n_q + 7) >> 3;
  const long long total = (long long)L.U * n_batches;
  long long at = total * blockIdx.x / gridDim.x;
  const long long end = total * (blockIdx.x + 1) / gridDim.x;
  while (at < end) {
    const int u = (int)(at / n_batches);
    int bi = (int)(at - (long long)u * n_batches) + warp;
    const int b_end = (int)(end - (long long)u * n_batches < n_batches ? end - (long long)u * n_batches : n_batches);
    at = (long long)(u + 1) * n_batches;
    if constexpr (NORM) {
      __syncthreads();                          // the previous unit's norms are no longer read
      inv_s[(threadIdx.x >> 5) * 36 + (threadIdx.x & 31)] = __fdiv_rn(1.0f, key_norm(absmax, ms, L.U, u, threadIdx.x));
      __syncthreads();
    }
    const Rec rec = unit_rec(L, cache, u);
    const __half* Xu = X + ((size_t)u * N + L.w_sink) * kD + kSeg * seg;
    uint4 raw[4];
    if (bi < b_end) {
      const uint4* src = reinterpret_cast<const uint4*>(Xu + (size_t)min(bi * 8 + tk, n_q - 1) * kD);
#pragma unroll
      for (int k = 0; k < 4; ++k) raw[k] = __ldg(src + k);
    }
    for (; bi < b_end; bi += 4) {
      const int i0 = bi * 8;
      F2 x[kSeg / 2];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const __half2* h = reinterpret_cast<const __half2*>(&raw[k]);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float2 v = __half22float2(h[i]);
          x[4 * k + i] = f2(v.x, v.y);
        }
      }
      if (bi + 4 < b_end) {                     // next batch's rows are requested before this one is worked on
        const uint4* src = reinterpret_cast<const uint4*>(Xu + (size_t)min((bi + 4) * 8 + tk, n_q - 1) * kD);
#pragma unroll
        for (int k = 0; k < 4; ++k) raw[k] = __ldg(src + k);
      }
      if constexpr (NORM) {
#pragma unroll
        for (int e = 0; e < kSeg / 4; ++e) {
          const float4 v = *reinterpret_cast<const float4*>(inv_s + seg * 36 + 4 * e);
          x[2 * e] = mul2(x[2 * e], f2(v.x, v.y));
          x[2 * e + 1] = mul2(x[2 * e + 1], f2(v.z, v.w));
        }
      }
      float mn, mx;                             // three-input min / max: two values per instruction
      {
        const float2 v = unf2(x[0]);
        mn = fminf(v.x, v.y); mx = max3_nan<BITS>(v.x, v.x, v.y);
#pragma unroll
        for (int e = 1; e < kSeg / 2; ++e) {
          const float2 w = unf2(x[e]);
          mn = min3(mn, w.x, w.y); mx = max3_nan<BITS>(mx, w.x, w.y);
        }
      }
      const bool nan = BITS > 2 && mx != mx;
      if (nan) {                                // the largest number
#pragma unroll
        for (int e = 0; e < kSeg / 2; ++e) {
          const float2 w = unf2(x[e]);
          mx = max3(mx, w.x, w.y);
        }
      }
      for (int o = 1; o < gl; o <<= 1) {
        mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      }
      const GroupParams p = seg_params<BITS>(mn, mx, L.sym_variant);
      const Bounds bd(mul2, p, mn, mx);               // the same for all lanes of a group
      bool asym = S.mode == 1;
      if (S.mode == 2) {
        int quick = -1;
        if (L.sym_variant == 0) {               // (the literal formula clips the tails of every group)
          QuickErr<BITS> qe(p, p);
#pragma unroll
          for (int e = 0; e < kSeg / 2; e += 2) qe.add(x[e], x[e + 1]);
          const float2 d2 = qe.difference((float)(kSeg / 2));
          float d = d2.x + d2.y;
          for (int o = 1; o < gl; o <<= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
          quick = quick_mode(d, quick_bound<BITS>(p, bd, mn, mx, L.G));      // the same in all lanes of a group
        }
        asym = quick > 0;
        if (__any_sync(0xffffffffu, quick < 0 || nan)) {
          const PairCoder pc(mul2, p, bd, p, bd);
          float2 ea = make_float2(0.f, 0.f), es = make_float2(0.f, 0.f);
          auto sums = [&](auto clamp) {
#pragma unroll
            for (int e = 0; e < kSeg / 2; ++e) {
              const float2 a = pc.template err_asym<decltype(clamp)::value>(x[e]), s = pc.template err_sym<decltype(clamp)::value>(x[e]);
              ea.x += fabsf(a.x); ea.y += fabsf(a.y);
              es.x += fabsf(s.x); es.y += fabsf(s.y);
            }
          };
          if (bd.no_clip) sums(std::false_type{});
          else sums(std::true_type{});
          float a = ea.x + ea.y, s = es.x + es.y;
          for (int o = 1; o < gl; o <<= 1) {
            a += __shfl_xor_sync(0xffffffffu, a, o);
            s += __shfl_xor_sync(0xffffffffu, s, o);
          }
          asym = a < s;
        }
      }
      uint32_t w8[8];                           // [2 * j + h]: bytes 16 h + 4 j .. + 3 of the segment's bit position
      {
        const ChosenPair cc(mul2, p, bd, asym, p, bd, asym);
        auto codes = [&](auto clamp) {
#pragma unroll
          for (int lw = 0; lw < 8; ++lw) {
            const uint2 a = cc.template code_bits<decltype(clamp)::value>(x[2 * lw]), b = cc.template code_bits<decltype(clamp)::value>(x[2 * lw + 1]);
            w8[2 * (lw & 3) + (lw >> 2)] = bytes4(a.x, a.y, b.x, b.y);
          }
        };
        if (bd.no_clip) codes(std::false_type{});
        else codes(std::true_type{});
      }
      __syncwarp();
      const int i = i0 + tk;
      unsigned char* chunk = chunk_ptr(rec, S, i0 / kChunk, sh);
      const int in_chunk = (i0 % kChunk) + tk;
      uint32_t* row = reinterpret_cast<uint32_t*>(chunk + S.code_in_rec) + in_chunk * RW;
      if constexpr (BITS == 4) {
        // segments 2q, 2q + 1 are the nibbles of the same 8 words: each of the two lanes keeps the words of two j
        const int half = seg >> 1, odd = seg & 1;
        uint32_t o4[4];
#pragma unroll
        for (int k = 0; k < 8; ++k) w8[k] <<= 4 * odd;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t keep = odd ? w8[4 + k] : w8[k], give = odd ? w8[k] : w8[4 + k];
          o4[k] = keep | __shfl_xor_sync(0xffffffffu, give, 1);
        }
        if (i < n_q) {
          *reinterpret_cast<uint2*>(row + 4 * (2 * odd) + 2 * half) = make_uint2(o4[0], o4[1]);
          *reinterpret_cast<uint2*>(row + 4 * (2 * odd + 1) + 2 * half) = make_uint2(o4[2], o4[3]);
        }
      } else {
        uint32_t o2[2];
        if constexpr (BITS == 3) {
          const int b0 = hi_bit_i8(seg, 0), b1 = hi_bit_i8(seg, 1);
          uint32_t h4[4], o1[1];
#pragma unroll
          for (int jj = 0; jj < 4; ++jj) {
            uint32_t lo0, hi0, lo1, hi1;
            split_planes(w8[2 * jj], seg & 1, lo0, hi0);
            split_planes(w8[2 * jj + 1], seg & 1, lo1, hi1);
            w8[2 * jj] = lo0; w8[2 * jj + 1] = lo1;
            h4[jj] = (hi0 << b0) | (hi1 << b1);
          }
          quad_reduce_scatter<1>(h4, seg, o1);
          if (i < n_q) row[8 + seg] = o1[0];
        }
#pragma unroll
        for (int k = 0; k < 8; ++k) w8[k] <<= 2 * seg;
        quad_reduce_scatter<2>(w8, seg, o2);
        if (i < n_q) *reinterpret_cast<uint2*>(row + 2 * seg) = make_uint2(o2[0], o2[1]);
      }
      if (i < n_q && (lane & (gl - 1)) == 0)
        store_meta(chunk + S.meta_in_rec, (in_chunk << (2 - sh)) + (seg >> sh), S.meta_bytes, group_meta(p, asym));
    }
  }
}

// ------------------------------------------------------------------ BLOCK store
// 64 * (G / 32) threads quantise one group of G tokens x 128 channels, a CTA of 256 threads 4 / (G / 32) groups at a
// time: thread (channel pair cp, chunk k) owns tokens 32k .. 32k+31 of channels 2cp and 2cp+1, read straight from global
// memory (one 32-bit load per token: a warp reads 128 contiguous bytes of each token row).  A pair of values is the two
// channels of one token.  The two channels are the two row halves of one MMA fragment row pair, and the pairs that
// share words of the packed chunk are adjacent lanes, which exchange them and store 16 contiguous bytes each (3-bit:
// the 1-bit plane's words are shared with the other channel half, a warp away).
// CTA `part` of `n_parts` takes a contiguous run of all units' groups, and between reading a step's values and working on
// them a slice of the keys for their maxima (KeyMax).
// A warp's 32 tokens x 64 channels come through its own 4 KB of shared memory, requested (cp.async) as soon as the values
// before them are in registers: read straight from global memory the loads of a group were waited for with nothing else to
// do, two thirds of the cycles without an instruction.
constexpr int kStage = 8 * 4096 / 16;                   // uint4: a step's values, or a slice of keys, of 8 warps
constexpr int kStats = 4 * 128 + 4 * 32;                // statistics of 4 chunks, 1-bit plane words of 4 chunks
constexpr int kFirstSmem = (2 * kStage + kStats) * 16;  // bytes of prefill_first_kernel: values, keys, statistics

// Maxima of |K| per channel over a CTA's share of the keys, a slice of 128 rows at a time: 16 lanes of 8 channels each, 16
// rows per warp, through 4 KB of shared memory that nobody but the lane which requested a piece reads.
struct KeyMax {
  const __half* K;
  float* out;
  MaxShares ms;
  int N, U, cta, at, end;
  uint4* stage;
  __half2 m[4];
  __device__ __forceinline__ KeyMax(const __half* K_, float* out_, const MaxShares& s, int N_, int U_, int cta_, uint4* stage_)
      : K(K_), out(out_), ms(s), N(N_), U(U_), cta(cta_), stage(stage_) {
    at = end = 0;
    if (cta >= 0 && cta < ms.ctas) { at = ms.begin(U, cta); end = ms.begin(U, cta + 1); }
    clear();
    if (at < end) request();
  }
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 4; ++i) m[i] = __float2half2_rn(0.f);
  }
  __device__ __forceinline__ void request() const {
    const int u = at / ms.per_unit, r0 = (at - u * ms.per_unit) * 128 + (threadIdx.x >> 5) * 16 + ((threadIdx.x >> 4) & 1);
    const __half* src = K + (size_t)u * N * kD + (threadIdx.x & 15) * 8;
    const uint32_t to = (uint32_t)__cvta_generic_to_shared(stage + (threadIdx.x >> 5) * 256 + (threadIdx.x & 31));
#pragma unroll
    for (int i = 0; i < 8; ++i)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(to + i * 512), "l"(src + (size_t)min(r0 + 2 * i, N - 1) * kD) : "memory");
  }
  // the slice that has arrived (cp.async.wait_all); requests the next one
  __device__ __forceinline__ void take() {
    if (at >= end) return;
    const uint4* mine = stage + (threadIdx.x >> 5) * 256 + (threadIdx.x & 31);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const uint4 v = mine[i * 32];
      const __half2* h = reinterpret_cast<const __half2*>(&v);
#pragma unroll
      for (int k = 0; k < 4; ++k) m[k] = __hmax2(m[k], __habs2(h[k]));
    }
    const int u = at / ms.per_unit;
    ++at;
    if (at >= end || at == (u + 1) * ms.per_unit) flush(u);
    if (at < end) request();
  }
  __device__ __forceinline__ void flush(int u) {        // the unit's maxima of this CTA: one row
    float* red = reinterpret_cast<float*>(stage);       // [16][kD]
    const int cg = threadIdx.x & 15, rg = threadIdx.x >> 4;
    __syncthreads();                                    // everyone has taken the last slice
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      red[rg * kD + cg * 8 + 2 * i] = __low2float(m[i]);
      red[rg * kD + cg * 8 + 2 * i + 1] = __high2float(m[i]);
    }
    __syncthreads();
    if (threadIdx.x < kD) {
      float v = 0.f;
#pragma unroll
      for (int i = 0; i < 16; ++i) v = fmaxf(v, red[i * kD + threadIdx.x]);
      out[((size_t)u * ms.stride + cta - ms.cta_of(U, u * ms.per_unit)) * kD + threadIdx.x] = v;
    }
    __syncthreads();
    clear();
  }
};

template <int BITS>
__device__ __forceinline__ void quantize_blocks(const Layout& L, const __half* __restrict__ X, int N, int n_q,
                                                unsigned char* __restrict__ cache, int part, int n_parts, uint4* smem_q,
                                                KeyMax& keys, Mul2 mul2) {
  const Store& S = L.v;
  const int G = L.G, CH = G >> 5, sh = CH >> 1, per_cta = 4 >> sh, n_groups = n_q / G;
  const int tid = threadIdx.x, cp = tid & 63, k4 = tid >> 6, k = k4 & (CH - 1), c0 = 2 * cp;
  uint4* stats = smem_q + 2 * kStage;
  float4* red_m = reinterpret_cast<float4*>(stats);                              // [4][64]: min, max of both channels
  float4* red_e = red_m + 4 * 64;                                                // [4][64]: error sums of both channels
  uint4* red_h = stats + 4 * 128;                                                // [4][32]: 1-bit plane words
  const int lane = tid & 31;
  unsigned char* mine = reinterpret_cast<unsigned char*>(smem_q) + (tid >> 5) * 4096;      // this warp's [32 tokens][64 channels]
  const uint32_t mine_u32 = (uint32_t)__cvta_generic_to_shared(mine);
  const bool wide = (reinterpret_cast<size_t>(X) & 15) == 0;
  const int m = 4 * (c0 >> 6) + ((c0 >> 1) & 3), gid = (c0 >> 3) & 7;             // fragment coordinates of the pair
  // Barriers of the warps that exchange something, instead of the whole CTA's: the CH warps with the same channels of a
  // group (the statistics), the two warps of a chunk (the 1-bit plane).
  const int my_group = 1 + ((k4 >> sh) << 1) + ((tid >> 5) & 1);
  auto group_sync = [&]() { asm volatile("barrier.sync %0, %1;" ::"r"(my_group), "r"(32 * CH) : "memory"); };
  auto group_or = [&](bool p) {
    int any;
    asm volatile("{.reg .pred p, q; setp.ne.s32 p, %1, 0; barrier.red.or.pred q, %2, %3, p; selp.s32 %0, 1, 0, q;}"
                 : "=r"(any) : "r"((int)p), "r"(my_group), "r"(32 * CH) : "memory");
    return any != 0;
  };
  [[maybe_unused]] auto pair_sync = [&]() { asm volatile("barrier.sync %0, 64;" ::"r"(9 + k4) : "memory"); };
  const int items = L.U * n_groups, steps = (items + per_cta - 1) / per_cta;      // a group is 8 KB at least: 31 bits hold them
  int s_begin = 0, s_end = 0;
  if (part >= 0 && part < n_parts) {
    s_begin = (int)((long long)steps * part / n_parts);
    s_end = (int)((long long)steps * (part + 1) / n_parts);
  }
  int u = 0, j = 0;                                         // unit and group of this thread's item of the step
  bool valid = false;
  auto locate = [&](int step) {
    int item = step * per_cta + (k4 >> sh);
    valid = item < items;                                   // the last step may have fewer groups than the CTA takes
    if (!valid) item = items - 1;
    u = item / n_groups;
    j = item - u * n_groups;
  };
  auto request = [&]() {                                    // the warp's values of (u, j), into its shared memory
    const __half* src = X + ((size_t)u * N + L.w_sink + (size_t)j * G + kSeg * k) * kD + 64 * ((tid >> 5) & 1);
    if (wide) {
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int p = i * 32 + lane;                        // 16-byte piece: token p / 8, channels 8 (p % 8) ..
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(mine_u32 + p * 16), "l"(src + (p >> 3) * kD + (p & 7) * 8) : "memory");
      }
    } else {
#pragma unroll 4
      for (int i = 0; i < kSeg; ++i)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(mine_u32 + (i * 32 + lane) * 4), "l"(src + i * kD + 2 * lane) : "memory");
    }
  };
  if (s_begin < s_end) {
    locate(s_begin);
    request();
  }
  for (int step = s_begin; step < s_end; ++step) {
    const int u_now = u, j_now = j;
    const bool valid_now = valid;
    F2 x[kSeg];
    {
      uint32_t raw[kSeg];
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncwarp();
#pragma unroll
      for (int t = 0; t < kSeg; ++t) raw[t] = *reinterpret_cast<const uint32_t*>(mine + t * 128 + lane * 4);
      __syncwarp();                                         // all lanes have theirs: the next values may come
      if (step + 1 < s_end) {
        locate(step + 1);
        request();
      }
      keys.take();
#pragma unroll
      for (int t = 0; t < kSeg; ++t) {
        const float2 v = __half22float2(*reinterpret_cast<const __half2*>(&raw[t]));
        x[t] = f2(v.x, v.y);
      }
    }
    float2 mn = unf2(x[0]), mx = mn;
    {
      const float2 v = unf2(x[1]);
      mn.x = fminf(mn.x, v.x); mn.y = fminf(mn.y, v.y);
      mx.x = max3_nan<BITS>(mx.x, mx.x, v.x); mx.y = max3_nan<BITS>(mx.y, mx.y, v.y);
    }
#pragma unroll
    for (int t = 2; t < kSeg; t += 2) {
      const float2 v = unf2(x[t]), w = unf2(x[t + 1]);
      mn.x = min3(mn.x, v.x, w.x); mn.y = min3(mn.y, v.y, w.y);
      mx.x = max3_nan<BITS>(mx.x, v.x, w.x); mx.y = max3_nan<BITS>(mx.y, v.y, w.y);
    }
    const bool nan = BITS > 2 && (mx.x != mx.x || mx.y != mx.y);
    if (nan) {                                               // the largest numbers
#pragma unroll
      for (int t = 0; t < kSeg; ++t) {
        const float2 v = unf2(x[t]);
        mx.x = fmaxf(mx.x, v.x); mx.y = fmaxf(mx.y, v.y);
      }
    }
    if (CH > 1) {
      group_sync();                                          // the previous group's words are no longer read
      red_m[k4 * 64 + cp] = make_float4(mn.x, mx.x, mn.y, mx.y);
      group_sync();
      for (int kk = 0; kk < CH; ++kk) {
        const float4 o = red_m[(k4 - k + kk) * 64 + cp];
        mn.x = fminf(mn.x, o.x); mx.x = fmaxf(mx.x, o.y);
        mn.y = fminf(mn.y, o.z); mx.y = fmaxf(mx.y, o.w);
      }
    }
    const GroupParams p0 = seg_params<BITS>(mn.x, mx.x, L.sym_variant), p1 = seg_params<BITS>(mn.y, mx.y, L.sym_variant);
    const Bounds b0(mul2, p0, mn.x, mx.x), b1(mul2, p1, mn.y, mx.y);
    const bool no_clip = b0.no_clip && b1.no_clip;
    bool asym0 = S.mode == 1, asym1 = asym0;
    if (S.mode == 2) {
      bool close = true;
      if (L.sym_variant == 0) {
        QuickErr<BITS> qe(p0, p1);
#pragma unroll
        for (int t = 0; t < kSeg; t += 2) qe.add(x[t], x[t + 1]);
        float2 d = qe.difference((float)kSeg);
        if (CH > 1) {
          float2* red_d = reinterpret_cast<float2*>(red_e);         // the first half of the thread's own entry
          red_d[2 * (k4 * 64 + cp)] = d;
          group_sync();
          d = make_float2(0.f, 0.f);
          for (int kk = 0; kk < CH; ++kk) {
            const float2 o = red_d[2 * ((k4 - k + kk) * 64 + cp)];
            d.x += o.x; d.y += o.y;
          }
        }
        const int quick0 = quick_mode(d.x, quick_bound<BITS>(p0, b0, mn.x, mx.x, G));
        const int quick1 = quick_mode(d.y, quick_bound<BITS>(p1, b1, mn.y, mx.y, G));
        asym0 = quick0 > 0;
        asym1 = quick1 > 0;
        close = quick0 < 0 || quick1 < 0 || nan;
      }
      if (CH > 1 ? group_or(close) : (bool)__any_sync(0xffffffffu, close)) {
        const PairCoder pc(mul2, p0, b0, p1, b1);
        float2 a0 = make_float2(0.f, 0.f), a1 = a0, s0 = a0, s1 = a0;      // even / odd tokens
        auto sums = [&](auto clamp) {
          constexpr bool C = decltype(clamp)::value;
#pragma unroll
          for (int t = 0; t < kSeg; t += 2) {
            const float2 ae = pc.template err_asym<C>(x[t]), ao = pc.template err_asym<C>(x[t + 1]);
            a0.x += fabsf(ae.x); a0.y += fabsf(ae.y); a1.x += fabsf(ao.x); a1.y += fabsf(ao.y);
            const float2 se = pc.template err_sym<C>(x[t]), so = pc.template err_sym<C>(x[t + 1]);
            s0.x += fabsf(se.x); s0.y += fabsf(se.y); s1.x += fabsf(so.x); s1.y += fabsf(so.y);
          }
        };
        if (no_clip) sums(std::false_type{});
        else sums(std::true_type{});
        float4 e = make_float4(a0.x + a1.x, s0.x + s1.x, a0.y + a1.y, s0.y + s1.y);
        if (CH > 1) {
          red_e[k4 * 64 + cp] = e;
          group_sync();
          e = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int kk = 0; kk < CH; ++kk) {
            const float4 o = red_e[(k4 - k + kk) * 64 + cp];
            e.x += o.x; e.y += o.y; e.z += o.z; e.w += o.w;
          }
        }
        asym0 = e.x < e.y;
        asym1 = e.z < e.w;
      }
    }
    // codes of token t sit in byte t / 8 of word [2 * (t % 4) + (t % 8) / 4] (see block_pos_i8), at bit position 0 here
    uint32_t w[2][8];
    {
      const ChosenPair cc(mul2, p0, b0, asym0, p1, b1, asym1);
      auto codes = [&](auto clamp) {
        constexpr bool C = decltype(clamp)::value;
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const uint2 a = cc.template code_bits<C>(x[t]), b = cc.template code_bits<C>(x[t + 8]),
                      c = cc.template code_bits<C>(x[t + 16]), d = cc.template code_bits<C>(x[t + 24]);
          w[0][2 * (t & 3) + (t >> 2)] = bytes4(a.x, b.x, c.x, d.x);
          w[1][2 * (t & 3) + (t >> 2)] = bytes4(a.y, b.y, c.y, d.y);
        }
      };
      if (no_clip) codes(std::false_type{});
      else codes(std::true_type{});
    }
    const Rec rec = unit_rec(L, cache, u_now);
    unsigned char* group = group_ptr(rec, j_now);
    uint32_t* chunk = reinterpret_cast<uint32_t*>(group + k * S.chunk_stride + S.code_in_rec);
    if constexpr (BITS == 4) {
      // The two channel pairs cp = 2q, 2q + 1 (adjacent lanes) fill the two nibbles of the same 16 words: after one
      // exchange lane `pos` holds the complete words of j = 2 pos, 2 pos + 1 (16 contiguous bytes each).
      const int pos = cp & 1, W = m >> 1;
#pragma unroll
      for (int i = 0; i < 8; ++i) { w[0][i] <<= 4 * pos; w[1][i] <<= 4 * pos; }
#pragma unroll
      for (int jj = 0; jj < 2; ++jj) {
        uint32_t f4[4];
#pragma unroll
        for (int rh = 0; rh < 2; ++rh)
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            const uint32_t keep = pos ? w[rh][2 * (2 + jj) + half] : w[rh][2 * jj + half];
            const uint32_t give = pos ? w[rh][2 * jj + half] : w[rh][2 * (2 + jj) + half];
            f4[2 * half + rh] = keep | __shfl_xor_sync(0xffffffffu, give, 1);
          }
        if (valid_now) *reinterpret_cast<uint4*>(chunk + W * 128 + (4 * gid + 2 * pos + jj) * 4) = make_uint4(f4[0], f4[1], f4[2], f4[3]);
      }
    } else {
      // The four channel pairs cp = 4q .. 4q+3 (adjacent lanes) fill the four bit positions of the same 16 words:
      // after two exchange steps lane `pos` holds the complete words of j = pos (two halves, two row halves), which
      // are 16 contiguous bytes of the chunk.
      const int pos = cp & 3, W = c0 >> 6;
      uint32_t lo[16], out[4];                              // [4 * j + 2 * half + rh]: the word order in the chunk
      [[maybe_unused]] uint32_t hi[16];
      const int sh_hi = hi_bit_i8(pos, W);
#pragma unroll
      for (int rh = 0; rh < 2; ++rh)
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          uint32_t l = w[rh][i];
          if constexpr (BITS == 3) {
            uint32_t h;
            split_planes(w[rh][i], pos & 1, l, h);
            hi[2 * i + rh] = h << sh_hi;
          }
          lo[2 * i + rh] = l << (2 * pos);
        }
      quad_reduce_scatter<4>(lo, pos, out);
      if (valid_now) *reinterpret_cast<uint4*>(chunk + W * 128 + (4 * gid + pos) * 4) = make_uint4(out[0], out[1], out[2], out[3]);
      if constexpr (BITS == 3) {
        // 1-bit plane: the words of lane group gid hold the bits of both halves W of the channels, which two warps
        // of this chunk's 64 threads computed: the second hands its words to the first through shared memory
        uint4* hx = red_h + k4 * 32 + (cp & 31);
        quad_reduce_scatter<4>(hi, pos, out);
        const uint4 mine = make_uint4(out[0], out[1], out[2], out[3]);
        pair_sync();                                        // the words before these have been read
        if (W == 1) *hx = mine;
        pair_sync();
        if (W == 0 && valid_now) {
          const uint4 o = *hx;
          *reinterpret_cast<uint4*>(chunk + 256 + (4 * gid + pos) * 4) =
              make_uint4(mine.x | o.x, mine.y | o.y, mine.z | o.z, mine.w | o.w);
        }
      }
    }
    if (k == 0 && valid_now) {
      store_meta(group + S.meta_in_rec, block_meta_index(c0), S.meta_bytes, group_meta(p0, asym0));
      store_meta(group + S.meta_in_rec, block_meta_index(c0 + 1), S.meta_bytes, group_meta(p1, asym1));
    }
  }
  while (keys.at < keys.end) {
    asm volatile("cp.async.wait_all;" ::: "memory");
    keys.take();
  }
}

// ------------------------------------------------------------------ windows, counts
// The fp16 windows of both tensors and the counts that the decode kernel compares with its own N (see append_publish), and
// the norms (1) unless the key quantiser computes them.  CTA `part` of `n_parts`, 256 threads.  Bound by memory latency in
// this kernel's two CTAs per SM: kCopies 16-byte pieces are in flight per thread, and stepping from piece to piece takes no
// division.  (One piece at a time with its division: 600 units x 1000 tokens, all in the windows, 260 us; now 136.)
__device__ __forceinline__ void copy_windows(const Layout& L, const Counts& cn, const __half* __restrict__ K,
                                             const __half* __restrict__ V, unsigned char* __restrict__ cache, bool set_norm,
                                             int part, int n_parts) {
  const int N = cn.N, i0 = part * 256 + threadIdx.x, n = n_parts * 256;
  uint32_t* counts = reinterpret_cast<uint32_t*>(cache + L.appended_off);
  for (int i = i0; i < L.U; i += n) counts[i] = (uint32_t)N;
  if (set_norm) {
    float* norm = reinterpret_cast<float*>(cache + L.norm_off);
    for (int i = i0; i < L.U * kD; i += n) norm[i] = 1.0f;
  }
#pragma unroll 1
  for (int s = 0; s < 2; ++s) {
    const Store& S = s ? L.v : L.k;
    const __half* X = s ? V : K;
    const int n_q = s ? cn.n_qv : cn.n_qk, per_unit = (N - n_q) * 16;      // 16-byte pieces of the tokens kept in fp16
    if (per_unit == 0) continue;
    // piece r of unit u; a thread's next one is n pieces further on
    const int step_u = n / per_unit, step_r = n - step_u * per_unit, ring0 = n_q % S.ring_cap;
    int u = i0 / per_unit, r = i0 - u * per_unit;
    while (u < L.U) {
      uint4 x[kCopies];
      uint4* to[kCopies];
#pragma unroll
      for (int k = 0; k < kCopies; ++k) {
        to[k] = nullptr;
        if (u < L.U) {
          const int w = r >> 4;                                            // the w-th token kept in fp16
          const bool sink = w < cn.n_sink;
          x[k] = __ldg(reinterpret_cast<const uint4*>(X + ((size_t)u * N + (sink ? w : w + n_q)) * kD) + (r & 15));
          int slot = w;
          if (!sink) {                                                     // the recent tokens fit the ring: it wraps once
            slot = ring0 + w - cn.n_sink;
            if (slot >= S.ring_cap) slot -= S.ring_cap;
          }
          unsigned char* base = cache + (sink ? S.sink_off + (size_t)u * S.sink_stride : S.ring_off + (size_t)u * S.ring_stride);
          to[k] = reinterpret_cast<uint4*>(base) + (size_t)slot * 16 + (r & 15);
          u += step_u;
          r += step_r;
          if (r >= per_unit) { r -= per_unit; ++u; }
        }
      }
#pragma unroll
      for (int k = 0; k < kCopies; ++k)
        if (to[k]) *to[k] = x[k];
    }
  }
}

// First of the two launches of an inner-grouped prefill: everything that does not need the key norms.  CTAs [k0, k0 + ms.ctas)
// take the key maxima, CTAs [v0, v0 + n_val) the value groups, CTAs [w0, w0 + n_win) the windows.  A prompt that fills the
// GPU gives all CTAs of one wave a share of all three: the maxima's keys arrive while the value groups are worked on, every
// load but a CTA's first is requested a step ahead (32 units x 16384 tokens, 2 bits, G = 128: 78 us as CTAs of several
// roles, four waves of them).  A short one spreads the roles over CTAs of their own; it is bound by its launches, not by its
// kernels: ten of them (clear, maxima, norms, two quantisers, four window copies, counts) took 38.9 us for 512 tokens of 8
// heads (3 bits, symmetric; calls through the binding, one after the other), the two take 10.2 us.
template <int VBITS>
__global__ void __launch_bounds__(256, 2)
prefill_first_kernel(const __grid_constant__ Layout L, const Counts cn, const __half* __restrict__ K,
                     const __half* __restrict__ V, unsigned char* __restrict__ cache, float* __restrict__ absmax,
                     const MaxShares ms, int k0, int v0, int n_val, int w0, int n_win, float neg_zero) {
  extern __shared__ uint4 first_smem[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  // a programmatic dependent of whatever comes before it, for its launch to overlap that kernel's end; keys and values may be
  // that kernel's results, and the cache and workspace what it reads
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int b = blockIdx.x;
  KeyMax keys(K, absmax, ms, cn.N, L.U, b - k0, first_smem + kStage);
  if (b >= w0 && b < w0 + n_win) copy_windows(L, cn, K, V, cache, ms.ctas == 0, b - w0, n_win);
  quantize_blocks<VBITS>(L, V, cn.N, cn.n_qv, cache, b - v0, n_val, first_smem, keys, Mul2(neg_zero));
}

// The same for a cache that has nothing else to do here: empty, unquantised (everything goes to the sink array) or
// outer-grouped (its quantisers are launches of their own).  Grid (share, unit, tensor), a kernel of few registers: full
// occupancy hides the latency (32 units x 65536 tokens, unquantised: 316 us, 6.8 TB/s; as a role of the kernel above 354).
__global__ void __launch_bounds__(256) prefill_windows_kernel(const __grid_constant__ Layout L, const Counts cn,
                                                              const __half* __restrict__ K, const __half* __restrict__ V,
                                                              unsigned char* __restrict__ cache) {
  const int u = blockIdx.y, N = cn.N;
  const Store& S = blockIdx.z ? L.v : L.k;
  const int n_q = blockIdx.z ? cn.n_qv : cn.n_qk;
  if (blockIdx.x == 0 && blockIdx.z == 0) {
    if (threadIdx.x < kD) reinterpret_cast<float*>(cache + L.norm_off)[(size_t)u * kD + threadIdx.x] = 1.0f;
    if (threadIdx.x == kD) reinterpret_cast<uint32_t*>(cache + L.appended_off)[u] = (uint32_t)N;
  }
  const uint4* X = reinterpret_cast<const uint4*>((blockIdx.z ? V : K) + (size_t)u * N * kD);
  uint4* sink = reinterpret_cast<uint4*>(cache + S.sink_off + (size_t)u * S.sink_stride);
  uint4* ring = reinterpret_cast<uint4*>(cache + S.ring_off + (size_t)u * S.ring_stride);
  const int n_sink = S.kind == kNone ? N : cn.n_sink, per_unit = (N - n_q) * 16;
  for (int i = blockIdx.x * 256 + threadIdx.x; i < per_unit; i += gridDim.x * 256) {
    const int w = i >> 4, piece = i & 15;
    if (w < n_sink) sink[i] = __ldg(X + i);
    else ring[(size_t)((w + n_q - n_sink) % S.ring_cap) * 16 + piece] = __ldg(X + (size_t)(w + n_q) * 16 + piece);
  }
}

int clamp_int(long long n, int lo, int hi) { return (int)(n < lo ? lo : (n > hi ? hi : n)); }

int window_ctas(const Layout& L, const Counts& cn) {      // about four 16-byte pieces per thread, eight CTAs per SM at most
  const long long pieces = (long long)L.U * 16 * (2ll * cn.N - cn.n_qk - cn.n_qv) + L.U * kD;
  return clamp_int((pieces + 1023) / 1024, 1, 148 * 8);
}

template <int KBITS>
int launch_rows(const Layout& L, const Counts& cn, const __half* K, unsigned char* cache, const float* absmax,
                const MaxShares& ms, cudaStream_t st) {
  // one wave of CTAs, each with at least one batch of 8 rows per warp; with norms at least one CTA (it stores them)
  const long long batches = (long long)L.U * ((cn.n_qk + 7) / 8);
  if (batches == 0 && !absmax) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(clamp_int((batches + 3) / 4, absmax ? (L.U < 148 ? L.U : 148) : 1, 148 * kRowsCtasPerSm));
  cfg.blockDim = dim3(128); cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // see prefill_first_kernel
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = absmax ? 1 : 0;
  const cudaError_t e =
      absmax ? cudaLaunchKernelEx(&cfg, quantize_rows_prefill_kernel<KBITS, true>, L, K, cn.N, cn.n_qk, cache, absmax, ms, -0.f)
             : cudaLaunchKernelEx(&cfg, quantize_rows_prefill_kernel<KBITS, false>, L, K, cn.N, cn.n_qk, cache, absmax, ms, -0.f);
  return e == cudaSuccess ? 1 : -1;
}

}  // namespace

int launch_prefill_windows(const Layout& L, const Counts& cn, unsigned char* cache, const __half* K, const __half* V,
                           cudaStream_t st) {
  const int n_fp16 = cn.N - std::min(cn.n_qk, cn.n_qv);
  prefill_windows_kernel<<<dim3(clamp_int((n_fp16 + 15) / 16, 1, 1024), L.U, 2), 256, 0, st>>>(L, cn, K, V, cache);
  return cudaGetLastError() == cudaSuccess ? 1 : -1;
}

int launch_prefill_inner(const Layout& L, const Counts& cn, unsigned char* cache, unsigned char* ws, const __half* K,
                         const __half* V, cudaStream_t st) {
  float* absmax = L.k_normalize ? reinterpret_cast<float*>(ws + L.ws_partial_off) : nullptr;
  // key maxima: their results go where the decode keeps its split partials, max_splits rows of more than 128 floats per unit
  static_assert(kPartialStride >= kD, "a row of partial maxima fits a split partial");
  const int wave = 2 * 148;
  MaxShares ms = {(cn.N + 127) / 128, 0, 0};
  // a unit meets at most ceil(ctas / U) + 1 CTAs
  if (absmax) ms.ctas = clamp_int(std::min<long long>((long long)L.U * ms.per_unit, (long long)L.U * (L.max_splits - 1)), 1, wave);
  ms.stride = (ms.ctas + L.U - 1) / L.U + 1;
  const long long steps = cn.n_qv > 0 ? ((long long)L.U * (cn.n_qv / L.G) * (L.G / kChunk) + 3) / 4 : 0;
  int k0 = 0, v0 = 0, n_val = clamp_int(steps, 0, wave), w0 = 0, n_win = window_ctas(L, cn), grid;
  if (ms.ctas + n_val <= 2 * wave && std::max(ms.ctas, n_val) < wave) {
    // Roles apart: 32 units x 768 tokens, 4 bits, G = 128 (192 + 128 + 198 CTAs), 17.4 us, together 20.3; x 1001 tokens (256 +
    // 192 + 187) 16.8 and 19.1; 56 x 576 (280 + 168 + 222) 18.8 and 20.8.  With a full wave of keys it is the slower form: 48 x
    // 900 tokens, 2 bits, G = 32 (296 + 288): 21.4 and 20.7.  Where the three need more than a wave, the value groups, which
    // take longest, start first and the windows fill the end: 24 x 900, 4 bits, G = 128 (192 + 144 + 102): keys first 14.1 us,
    // values first 13.1.
    if (ms.ctas + n_val + n_win > wave) k0 = n_val;
    else v0 = ms.ctas;
    w0 = ms.ctas + n_val;
    grid = w0 + n_win;
  } else {
    if (n_win > wave) w0 = std::max(ms.ctas, n_val);      // long windows: CTAs of their own
    else n_win = std::max(ms.ctas, n_val);
    grid = std::max(std::max(ms.ctas, n_val), w0 + n_win);
  }
  auto go = [&](auto kernel, std::atomic<unsigned long long>& configured) {
    if (!opt_in_dynamic_smem(kernel, kFirstSmem, configured)) return false;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid); cfg.blockDim = dim3(256); cfg.dynamicSmemBytes = kFirstSmem; cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr; cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kernel, L, cn, K, V, cache, absmax, ms, k0, v0, n_val, w0, n_win, -0.f) == cudaSuccess;
  };
  static std::atomic<unsigned long long> configured[3];
  if (!(L.v.bits == 2   ? go(prefill_first_kernel<2>, configured[0])
        : L.v.bits == 3 ? go(prefill_first_kernel<3>, configured[1])
                        : go(prefill_first_kernel<4>, configured[2]))) return -1;
  if (cudaGetLastError() != cudaSuccess) return -1;
  const int rows = L.k.bits == 2   ? launch_rows<2>(L, cn, K, cache, absmax, ms, st)
                   : L.k.bits == 3 ? launch_rows<3>(L, cn, K, cache, absmax, ms, st)
                                   : launch_rows<4>(L, cn, K, cache, absmax, ms, st);
  return rows < 0 ? -1 : 1 + rows;
}

}  // namespace iq
