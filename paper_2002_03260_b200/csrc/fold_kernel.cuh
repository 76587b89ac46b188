// One uniform axis of the KDFT formulation whose matrix is applied in folded form (paper Eq. 12 with Eq. 14's kernel).
//
// The N x N matrix of a uniform grid repeats itself: with N = R*m, j = i + s*m and k = R*kappa + q,
//     X[R*kappa + q] = sum_i exp(+-2*pi*i * i*kappa/m) * u_q[i],
//     u_q[i] = exp(+-2*pi*i * i*q/N) * sum_s exp(+-2*pi*i * s*q/R) * x[i + s*m],
// so the R residue classes of the output share ONE m x m matrix (m <= 64).  u is R-point sums, additions mostly, that a
// thread forms in registers on the CUDA cores; the product is one real GEMM with K = N = 2m whose table (both fp16
// pieces, at most 64 KB) stays in shared memory.  Tensor work falls by N/m = R against the product with the full
// matrix, and neither the table nor a line is read twice.
//
// Pieces: x = hi + 2^-11 * lo', W likewise, hi and lo' in fp16 (11-bit significands); hi x [W_hi | W_lo'] is one MMA of
// twice the width, lo' x W_hi is added to its upper half, and the store forms hi*hi + 2^-11 * cross in fp32.  Because
// the lo pieces carry their own 2^11 they stay normal numbers: an element is held to 2^-23 of itself down to 2^-25 of the
// largest one and to about 2^-46 of that one below; the R-point sums and the phases round in fp32 on top.  The chains on the
// large accumulator are 2m/16 <= 8 MMAs long.  Scales are exact powers of two (table 1024 * W, data from the largest input
// magnitude; TF32 pieces: see FoldRange).
//
// Roofline: HBM, 16 B per point.  Per tile of 128 lanes (128/R lines x R classes) and m = 64: 24 MMAs = 1536 clk of the
// tensor pipe and about 2600 clk of shared-memory traffic against 5700 clk of an SM's share of the HBM stream.
//
// Measured (per transform, the reduction over the input included; overlapped launches): 512^3 4.7 -> 1.48-1.6 ms, 1024^3 75
// -> 13.1 ms, 64^3 38 -> 19.1 us against the full matrix; a contiguous 1024-point pass moves 5.8 TB/s, a strided one 4.2-4.6
// TB/s.  Relative error against 64-bit results 2e-7 to 5e-7 per 3D transform (full matrix: 1.5e-6 to 2.6e-6).
//
// Organisation (one persistent CTA per SM, 640 threads):
//   warp 0       table load; one thread issues tcgen05.mma (both operands from shared memory)
//   warps 4-7    epilogue: tensor memory -> registers -> global
//   warps 8-19   global -> registers -> R-point sums, phase, split -> shared memory; L2 prefetch two tiles ahead
// Two operand buffers and two accumulators, so the three run on different tiles.  No TMA on the data: the loads are
// coalesced as they are (16 or more neighbouring columns, or consecutive points of a line) and need no alignment beyond
// a complex number's 8 bytes (contiguous lines of even m: 16 bytes, which every plan asks of its arrays).
#pragma once
#include <type_traits>
#include "kdft_f16_kernel.cuh"
#include "split_f16.cuh"

namespace dft3d {

struct FoldParams {
  const float2* in;
  float2* out;
  const uint8_t* w_image;   // table as it lies in shared memory: [panel of 128 bytes][hi rows, lo rows][128 B], swizzled
  const float4* tw;         // [R][mp/2] phases exp(+-2*pi*i*i*q/N) of i, i+1: (re, re', im, im'), zero beyond m
  int n, m, mp;             // N, m, m rounded up to whole groups
  int np;                   // MMA N of one piece: 2m rounded up to 16
  int ks;                   // MMA steps along the contraction: 32 bytes, K = 16 halves or 8 TF32 words
  int panels;               // panels of 128 bytes
  unsigned w_bytes;
  unsigned groups;          // groups of B consecutive i per line
  unsigned groups_magic;    // ceil(2^24 / groups)
  unsigned lines;
  unsigned C, off;          // STRIDED, natural order: line l starts at (l / C) * pitch + off + l % C, its points are `step` apart
  size_t pitch, step;
  int prefetch;             // L2 prefetch of later units
  int twin;                 // TF32 pieces: two accumulators
  int in_blocked, out_blocked;   // columns per block, 0 = natural order: layouts of the intermediate between axes 0 and 1, see fold_place
  unsigned n0, n1, n2;      // the cube or the slice of its last axis (blocked layouts only)
  unsigned units;           // groups of fold_lines lines
  unsigned tasks;           // warp-sized shares of a unit's loads and sums
  unsigned block_tasks;     // TF32 pieces: the tasks that hold the groups of a line, block_tasks consecutive ones for up to 32 lines
  int split_warps;          // warps that take the tasks
  float out_mul;
  const unsigned int* amax_in;
  unsigned int* amax_out;
  unsigned int* status;
  WaitControl wc;
};

struct FoldShared {
  uint64_t a_full[2], a_empty[2], d_full[2], d_empty[2], w_full;
  uint32_t tmem_base;
  volatile int abort_flag;
  long long wait_limit;
};

// TF32 pieces need no scale unless a line lies near an end of the float range: with its largest component in [2^-96, 2^116) no
// piece that matters is subnormal and no sum overflows.  Every task notes which of its lines have a component in that range and
// which have one beyond; the epilogue passes over a unit that has a line with too large ones, or with too small ones only, and
// the CTA takes these units once more when it is through with the others: then the tasks of a line wait for each other's
// exponents and scale it to about 1.  (512-point axes 0 / 1 / 2 of 512^3: every line scaled that way 591 / 485 / 456 us, because
// all warps wait for the slowest load of a unit; this way 479 / 444 / 416; no notes and no scale 496 / 444 / 401.)
constexpr uint32_t kFoldLow = 127 - 96, kFoldHigh = 127 + 115;     // exponent fields
constexpr unsigned kFoldTops = 8;        // units whose notes are kept: a warp that enters unit u has left u - 2 or a later one, whose
                                         // buffer was free, so the product of u - 4 had been issued, the sums of u - 6 read
constexpr unsigned kFoldMarks = 1 << 16; // units that a CTA can pass over; with more all take the second form
struct FoldRange {
  uint64_t top_full[kFoldTops][4];       // second form, per block of 32 lines: the exponents are complete
  uint64_t split_done, first_done;       // every unit has been split once; has been stored or marked
  // Words of a unit carry its position in the order of work plus one, so that an older one never counts.
  uint32_t top[kFoldTops * 128];          // << 8 | 0: the line has a component in the range; second form: largest exponent field
  uint32_t far[kFoldTops * 128];          // << 1 | 1: the line has a component above the range, | 0: one below (and not zero)
  volatile uint32_t any_far[kFoldTops];
  volatile uint32_t marks[kFoldMarks / 32];
  volatile uint32_t marked;
  volatile uint32_t far_seen;            // 0: nothing to take once more, no role waits for the others at its end
};

constexpr int kFoldThreads = 640;
constexpr int kFoldSplitWarps = 12;
// consecutive i that a thread takes at a time
__host__ __device__ constexpr int fold_group(int R) { return R >= 10 ? 2 : 4; }
// A unit is the lines whose R-point sums are formed together, 32 warps' worth at most: one tile of 128 lanes (128/R lines
// x R classes), or, on the strided axes with R = 16, two tiles of 16 lines x 8 classes, so that every row of the data is
// read and written in pieces of at least a 128-byte line.  (With one tile of 8 lines the halves of the lines were fetched
// from DRAM twice: 1.8 instead of 1.07 GB at 128 x 1024 x 1024, 652 us.)
__host__ __device__ constexpr int fold_tiles(bool strided, int R) { return strided && R >= 10 ? 2 : 1; }
// lines per unit: the largest power of two that 128 lanes hold (R = 3, 5, 6 and 10 leave some lanes idle)
__host__ __device__ constexpr int fold_lines(bool strided, int R) {
  int l = 1;
  while (2 * l * (R / fold_tiles(strided, R)) <= 128) l *= 2;
  return l;
}
constexpr int kFoldPanelBytes = 128 * 128;      // 128 lanes x 128 bytes
__host__ __device__ constexpr size_t fold_smem_bytes(unsigned w_bytes, int panels, int tw_entries, bool t32) {
  return size_t(w_bytes) + size_t(4) * panels * kFoldPanelBytes + size_t(tw_entries) * 12 + sizeof(FoldShared) +
         (t32 ? sizeof(FoldRange) : 0) + 1024;
}

// ---- Two complex numbers at a time: re and im hold the real and the imaginary parts of two neighbouring points, so that
// every operation is one packed instruction and a product with i costs no register moves.
struct C2 {
  uint64_t re, im;
};
__device__ __forceinline__ uint64_t dup2(float a) { return pack2(a, a); }
__device__ __forceinline__ C2 c2_add(C2 a, C2 b) { return {add2(a.re, b.re), add2(a.im, b.im)}; }
__device__ __forceinline__ C2 c2_sub(C2 a, C2 b) { return {sub2(a.re, b.re), sub2(a.im, b.im)}; }
// a +- s*i*f with s = +1 or -1 (sp = (s, s), sn = (-s, -s))
__device__ __forceinline__ C2 c2_add_i(C2 a, C2 f, uint64_t sp, uint64_t sn) {
  return {fma2(f.im, sn, a.re), fma2(f.re, sp, a.im)};
}
// x * (c + i*d), d2n = -d
__device__ __forceinline__ C2 c2_mul(C2 x, uint64_t c, uint64_t d, uint64_t dn) {
  return {fma2(x.im, dn, mul2(x.re, c)), fma2(x.re, d, mul2(x.im, c))};
}
__device__ __forceinline__ void dft4(C2& x0, C2& x1, C2& x2, C2& x3, uint64_t sp, uint64_t sn) {
  const C2 a = c2_add(x0, x2), b = c2_sub(x0, x2), c = c2_add(x1, x3), d = c2_sub(x1, x3);
  x0 = c2_add(a, c);
  x2 = c2_sub(a, c);
  x1 = c2_add_i(b, d, sp, sn);
  x3 = c2_add_i(b, d, sn, sp);
}
__device__ __forceinline__ void dft3(C2& x0, C2& x1, C2& x2, uint64_t sp, uint64_t sn) {
  const uint64_t half = dup2(-0.5f), h = dup2(0.86602540378443864676f);
  const C2 t = c2_add(x1, x2), d = c2_sub(x1, x2), b = {mul2(d.re, h), mul2(d.im, h)};
  const C2 a = {fma2(t.re, half, x0.re), fma2(t.im, half, x0.im)};
  x0 = c2_add(x0, t);
  x1 = c2_add_i(a, b, sp, sn);
  x2 = c2_add_i(a, b, sn, sp);
}
__device__ __forceinline__ void dft5(C2& x0, C2& x1, C2& x2, C2& x3, C2& x4, uint64_t sp, uint64_t sn) {
  const uint64_t c1 = dup2(0.30901699437494742410f), c2 = dup2(-0.80901699437494742410f);
  const uint64_t s1 = dup2(0.95105651629515357212f), s2 = dup2(0.58778525229247312917f), s1n = dup2(-0.95105651629515357212f);
  const C2 t1 = c2_add(x1, x4), t2 = c2_add(x2, x3), t3 = c2_sub(x1, x4), t4 = c2_sub(x2, x3);
  const C2 a1 = {fma2(t2.re, c2, fma2(t1.re, c1, x0.re)), fma2(t2.im, c2, fma2(t1.im, c1, x0.im))};
  const C2 a2 = {fma2(t2.re, c1, fma2(t1.re, c2, x0.re)), fma2(t2.im, c1, fma2(t1.im, c2, x0.im))};
  const C2 b1 = {fma2(t4.re, s2, mul2(t3.re, s1)), fma2(t4.im, s2, mul2(t3.im, s1))};
  const C2 b2 = {fma2(t4.re, s1n, mul2(t3.re, s2)), fma2(t4.im, s1n, mul2(t3.im, s2))};
  x0 = c2_add(x0, c2_add(t1, t2));
  x1 = c2_add_i(a1, b1, sp, sn);
  x4 = c2_add_i(a1, b1, sn, sp);
  x2 = c2_add_i(a2, b2, sp, sn);
  x3 = c2_add_i(a2, b2, sn, sp);
}
__device__ __forceinline__ void c2_swap(C2& a, C2& b) { const C2 t = a; a = b; b = t; }

// x[s] -> sum_s exp(sign*2*pi*i*s*q/R) x[s], natural order
template <int R>
__device__ __forceinline__ void dft_r(C2 (&x)[R], float s) {
  constexpr float kC1 = 0.92387953251128675613f, kS1 = 0.38268343236508977173f, kH = 0.70710678118654752440f;
  const uint64_t sp = dup2(s), sn = dup2(-s);
  if constexpr (R == 2) {
    const C2 a = x[0];
    x[0] = c2_add(a, x[1]);
    x[1] = c2_sub(a, x[1]);
  } else if constexpr (R == 3) {
    dft3(x[0], x[1], x[2], sp, sn);
  } else if constexpr (R == 5) {
    dft5(x[0], x[1], x[2], x[3], x[4], sp, sn);
  } else if constexpr (R == 6 || R == 10) {     // even and odd points, then the odd half turned by exp(s*2*pi*i*q/R)
    constexpr int K = R / 2;
    constexpr float kCos[5] = {1.0f, R == 6 ? 0.5f : 0.80901699437494742410f, R == 6 ? -0.5f : 0.30901699437494742410f,
                               -0.30901699437494742410f, -0.80901699437494742410f};
    constexpr float kSin[5] = {0.0f, R == 6 ? 0.86602540378443864676f : 0.58778525229247312917f,
                               R == 6 ? 0.86602540378443864676f : 0.95105651629515357212f, 0.95105651629515357212f,
                               0.58778525229247312917f};
    C2 e[K], o[K];
#pragma unroll
    for (int q = 0; q < K; ++q) { e[q] = x[2 * q]; o[q] = x[2 * q + 1]; }
    if constexpr (K == 3) {
      dft3(e[0], e[1], e[2], sp, sn);
      dft3(o[0], o[1], o[2], sp, sn);
    } else {
      dft5(e[0], e[1], e[2], e[3], e[K - 1], sp, sn);
      dft5(o[0], o[1], o[2], o[3], o[K - 1], sp, sn);
    }
#pragma unroll
    for (int q = 0; q < K; ++q) {
      const C2 t = q == 0 ? o[0] : c2_mul(o[q], dup2(kCos[q]), dup2(s * kSin[q]), dup2(-s * kSin[q]));
      x[q] = c2_add(e[q], t);
      x[q + K] = c2_sub(e[q], t);
    }
  } else if constexpr (R == 4) {
    dft4(x[0], x[1], x[2], x[3], sp, sn);
  } else if constexpr (R == 8) {
    dft4(x[0], x[2], x[4], x[6], sp, sn);
    dft4(x[1], x[3], x[5], x[7], sp, sn);
    const uint64_t h = dup2(kH), hs = dup2(s * kH), hn = dup2(-s * kH);
    const C2 e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6];
    const C2 o0 = x[1], o1 = c2_mul(x[3], h, hs, hn), o2 = x[5], o3 = c2_mul(x[7], dup2(-kH), hs, hn);
    x[0] = c2_add(e0, o0);
    x[4] = c2_sub(e0, o0);
    x[1] = c2_add(e1, o1);
    x[5] = c2_sub(e1, o1);
    x[2] = c2_add_i(e2, o2, sp, sn);
    x[6] = c2_add_i(e2, o2, sn, sp);
    x[3] = c2_add(e3, o3);
    x[7] = c2_sub(e3, o3);
  } else if constexpr (R == 16) {
#pragma unroll
    for (int a = 0; a < 4; ++a) dft4(x[a], x[a + 4], x[a + 8], x[a + 12], sp, sn);
    // x[a + 4*q0] *= w^(a*q0), w = exp(s*2*pi*i/16)
    const uint64_t c1 = dup2(kC1), s1 = dup2(kS1), h = dup2(kH), hm = dup2(-kH);
    const uint64_t c1s = dup2(s * kC1), c1n = dup2(-s * kC1), s1s = dup2(s * kS1), s1n = dup2(-s * kS1);
    const uint64_t hs = dup2(s * kH), hn = dup2(-s * kH);
    x[5] = c2_mul(x[5], c1, s1s, s1n);
    x[6] = c2_mul(x[6], h, hs, hn);
    x[7] = c2_mul(x[7], s1, c1s, c1n);
    x[9] = c2_mul(x[9], h, hs, hn);
    x[10] = {mul2(x[10].im, sn), mul2(x[10].re, sp)};
    x[11] = c2_mul(x[11], hm, hs, hn);
    x[13] = c2_mul(x[13], s1, c1s, c1n);
    x[14] = c2_mul(x[14], hm, hs, hn);
    x[15] = c2_mul(x[15], dup2(-kC1), s1n, s1s);
#pragma unroll
    for (int q0 = 0; q0 < 4; ++q0) dft4(x[4 * q0], x[4 * q0 + 1], x[4 * q0 + 2], x[4 * q0 + 3], sp, sn);
    // entry q0 + 4*q1 now sits at 4*q0 + q1: transpose the 4 x 4 (register renaming)
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = a + 1; b < 4; ++b) c2_swap(x[4 * a + b], x[4 * b + a]);
  }
}

// two complex numbers -> fp16 pairs: hi, and the remainder times 2^11
__device__ __forceinline__ void split_half2_scaled(C2 x, uint32_t& hi0, uint32_t& hi1, uint32_t& lo0, uint32_t& lo1) {
  float r0, r1, i0, i1;
  unpack2(x.re, r0, r1);
  unpack2(x.im, i0, i1);
  const __half2 h0 = __floats2half2_rn(r0, i0), h1 = __floats2half2_rn(r1, i1);
  const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
  const uint64_t up = dup2(2048.0f);
  unpack2(mul2(sub2(x.re, pack2(f0.x, f1.x)), up), r0, r1);
  unpack2(mul2(sub2(x.im, pack2(f0.y, f1.y)), up), i0, i1);
  const __half2 l0 = __floats2half2_rn(r0, i0), l1 = __floats2half2_rn(r1, i1);
  hi0 = *reinterpret_cast<const uint32_t*>(&h0);
  hi1 = *reinterpret_cast<const uint32_t*>(&h1);
  lo0 = *reinterpret_cast<const uint32_t*>(&l0);
  lo1 = *reinterpret_cast<const uint32_t*>(&l1);
}

__device__ __forceinline__ float max_abs3(float a, float b, float c) {
  float r;
  asm("max.abs.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// Exponent fields as FoldRange holds them.  A line with an infinity (255) has no finite result at any scale.
__device__ __forceinline__ uint32_t fold_field(float top) { return top > 0.0f ? max(__float_as_uint(top) >> 23, 1u) : 0; }
__device__ __forceinline__ bool fold_outside(uint32_t f) { return f != 0 && f != 255 && (f < kFoldLow || f > kFoldHigh); }
__device__ __forceinline__ int fold_shift(uint32_t f) { return f == 0 || f == 255 ? 0 : max(127 - int(f), -100); }
__device__ __forceinline__ float pow2f(int e) { return __uint_as_float(uint32_t(127 + e) << 23); }
// the first marked unit from `from` on, or `units`
__device__ __forceinline__ unsigned fold_next(const FoldRange& rg, bool all, unsigned from, unsigned units) {
  if (all || from >= units) return min(from, units);
  unsigned w = from >> 5;
  uint32_t b = rg.marks[w] & (0xffffffffu << (from & 31));
  while (b == 0) {
    if (++w * 32 >= units) return units;
    b = rg.marks[w];
  }
  return w * 32 + __ffs(b) - 1;
}

// Two complex numbers -> TF32 pieces (re, im, re', im'): hi is the raw word (the tensor core ignores the low 13 bits of the
// mantissa), lo the remainder rounded to TF32.
__device__ __forceinline__ void split_tf32(C2 x, uint32_t (&hi)[4], uint32_t (&lo)[4]) {
  float v[4];
  unpack2(x.re, v[0], v[2]);
  unpack2(x.im, v[1], v[3]);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    hi[i] = __float_as_uint(v[i]);
    lo[i] = (__float_as_uint(v[i] - __uint_as_float(hi[i] & 0xffffe000u)) + 0x1000u) & 0xffffe000u;
  }
}

// Loads of the data (ordinary ones: a pass may run in place, and may start while its predecessor still writes), and explicit
// shared-memory accesses.  The 8-byte form takes whole lines per warp; of the 16-byte form a
// warp's lanes may be 32 bytes apart, and the second load finds the other halves of the sectors in L1 (512-point lines:
// 582 us with, 620 us without).
__device__ __forceinline__ void ld_stream8(const float2* p, float& a, float& b) {
  asm volatile("ld.global.L1::no_allocate.v2.f32 {%0, %1}, [%2];" : "=f"(a), "=f"(b) : "l"(p));
}
__device__ __forceinline__ void ld_stream16(const float2* p, float& a, float& b, float& c, float& d) {
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(a), "=f"(b), "=f"(c), "=f"(d) : "l"(p));
}
__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }
__device__ __forceinline__ void lds_2x64(uint32_t addr, uint64_t& a, uint64_t& b) {
  asm volatile("ld.shared.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "r"(addr));
}
__device__ __forceinline__ void lds_64(uint32_t addr, uint64_t& a) {
  asm volatile("ld.shared.b64 %0, [%1];" : "=l"(a) : "r"(addr));
}
__device__ __forceinline__ void sts_64(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void sts_128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// Where line l starts and how far apart its points are, in complex numbers.  Natural order: [batch][j][C].  Blocked order,
// between the passes over axis 0 and axis 1 of one transform: [n2 / 16][i1][k0][16 columns] (eight where one of the two axes has no folded form), in which the axis-0 pass
// writes contiguous blocks (its rows are n1*n2 points apart in natural order, and writing such rows piecewise is slow)
// and the axis-1 pass reads whole 128-byte lines.
struct LinePlace {
  size_t base, step;
};
__device__ __forceinline__ LinePlace fold_place(const FoldParams& p, unsigned l, bool in_blocked, bool out_blocked) {
  if (in_blocked) {            // axis 1: l = k0 * n2 + i2
    const unsigned b = l / p.C, c = l - b * p.C, w = unsigned(p.in_blocked), t = w == 16 ? c >> 4 : c / w;
    return {(size_t(t) * p.n1 * p.n0 + b) * w + (c - t * w), size_t(p.n0) * w};
  }
  if (out_blocked) {           // axis 0: l = i1 * n2 + i2
    const unsigned i1 = l / p.n2, i2 = l - i1 * p.n2, w = unsigned(p.out_blocked), t = w == 16 ? i2 >> 4 : i2 / w;
    return {(size_t(t) * p.n1 + i1) * p.n0 * w + (i2 - t * w), w};
  }
  const unsigned b = l / p.C, c = l - b * p.C;
  return {size_t(b) * p.pitch + p.off + c, p.step};
}

#define FOLD_WAIT(bar, parity, code)                                                   \
  if (!bounded_wait((bar), (parity), &sh.abort_flag, sh.wait_limit)) {                 \
    sh.abort_flag = 1;                                                                 \
    atomicCAS(p.status, 0u, (unsigned)(code));                                         \
    goto role_done;                                                                    \
  }
#define FOLD_WAIT_WARP_ELSE(bar, parity, code, leave)                                                     \
  if (!__all_sync(0xffffffffu, bounded_wait((bar), (parity), &sh.abort_flag, sh.wait_limit) ? 1 : 0)) {   \
    sh.abort_flag = 1;                                                                                    \
    atomicCAS(p.status, 0u, (unsigned)(code));                                                            \
    leave;                                                                                                \
  }
#define FOLD_WAIT_WARP(bar, parity, code) FOLD_WAIT_WARP_ELSE(bar, parity, code, goto role_done)

// T32: TF32 pieces instead of fp16 ones (twice the bytes per operand, so m <= 32; scales as FoldRange says)
template <int MODE, int R, bool T32>
__global__ void __launch_bounds__(kFoldThreads, 1) fold_axis_kernel(const FoldParams p, const float sign) {
  constexpr int H = fold_tiles(MODE == KDFT_STRIDED, R);   // tiles per unit
  constexpr int Q = R / H;          // residue classes per tile
  constexpr int L = fold_lines(MODE == KDFT_STRIDED, R);   // lines per unit (and per tile)
  // How many units ahead the L2 prefetch runs, 64 or 128 KB per unit (512 x 1024 x 1024, microseconds per pass without the
  // reduction: strided R = 16 2147 / 1820 / 2040 / 2170 for no prefetch, 1, 2 and 3 units; contiguous R = 8 2270 / 1870 / 1720 /
  // 1860).
  constexpr unsigned kAhead = H == 2 ? 1 : 2;
  constexpr int B = fold_group(R);  // consecutive i a thread takes at a time
  constexpr int kLog2R = R <= 4 ? 2 : (R <= 8 ? 3 : 4);    // at least log2(R)
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = ptx::align_1024(smem_raw);
  uint8_t* smem_w = smem;
  uint8_t* smem_a = smem + p.w_bytes;                    // [buffer][hi, lo'][panel][128 rows][128 B]
  const uint32_t piece_bytes = uint32_t(p.panels) * kFoldPanelBytes;
  // phases times the input scale, for pairs of neighbouring i: (re, re', im, im') and, behind them, (-im, -im')
  const uint32_t t_entries = uint32_t(R * p.mp) / 2;
  float4* smem_t = reinterpret_cast<float4*>(smem_a + 4 * size_t(piece_bytes));
  float2* smem_tn = reinterpret_cast<float2*>(smem_t + t_entries);
  FoldShared& sh = *reinterpret_cast<FoldShared*>(smem_tn + t_entries);
  FoldRange& rg = *reinterpret_cast<FoldRange*>(&sh + 1);                   // TF32 pieces only
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // this CTA's units: blockIdx.x, blockIdx.x + gridDim.x, ...
  const unsigned my_units = blockIdx.x < p.units ? (p.units - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  // Positions in the order of work: first the units one by one, then (TF32 pieces) those that the epilogue marked.
  const bool all = T32 && my_units > kFoldMarks;
  const unsigned first = all ? 0 : my_units;

  ptx::griddep_launch();
  if (tid == 0) {
    for (int i = 0; i < 2; ++i) {
      ptx::mbar_init(&sh.a_full[i], p.tasks);
      ptx::mbar_init(&sh.a_empty[i], 1);
      ptx::mbar_init(&sh.d_full[i], 1);
      ptx::mbar_init(&sh.d_empty[i], 4);
    }
    if (T32) {
      ptx::mbar_init(&rg.split_done, unsigned(p.split_warps));
      ptx::mbar_init(&rg.first_done, 4);
      rg.marked = 0;
      rg.far_seen = all;
    }
    ptx::mbar_init(&sh.w_full, 1);
    sh.abort_flag = 0;
    sh.wait_limit = p.wc.limit_clocks > 0 ? p.wc.limit_clocks : kDefaultWaitClocks;
    ptx::fence_mbar_init();
    if (!p.wc.silent_producer) {
      ptx::mbar_arrive_expect_tx(&sh.w_full, p.w_bytes);
      ptx::bulk_load(smem_w, p.w_image, p.w_bytes, &sh.w_full);
    }
  }
  if (warp == 1) {
    ptx::tmem_alloc(&sh.tmem_base, 512);
    ptx::tmem_relinquish();
  }
  ptx::griddep_wait();
  // The largest |component| of the input, at most 2^(e+1), is scaled so that the R-point sums (modulus at most R*sqrt(2)
  // times that) stay below 2^15.5.  The scale rides on the phases; data near the top of the float range are brought down
  // first so that the sums cannot overflow.
  float in_scale = 1.0f, out_mul2 = 1.0f, pre = 1.0f;
  if (T32) {
    if (tid < 4 * kFoldTops) ptx::mbar_init(&rg.top_full[0][0] + tid, p.block_tasks);
    if (tid < kFoldTops) rg.any_far[tid] = 0;
    for (uint32_t i = tid; i < kFoldTops * L; i += kFoldThreads) rg.top[i] = rg.far[i] = 0;
    if (!all)
      for (uint32_t i = tid; i < (my_units + 31) / 32; i += kFoldThreads) rg.marks[i] = 0;
  } else {
    const float a = __uint_as_float(*p.amax_in);
    if (a > 0.0f) {                      // never an infinity: the reduction and the epilogues leave those out
      constexpr int kTop = 14 - kLog2R;
      const int e = max(ilogbf(a), -113);
      const int down = e > 100 ? 16 : 0;
      pre = down ? 0x1p-16f : 1.0f;
      in_scale = ldexpf(1.0f, kTop - e + down);
      out_mul2 = ldexpf(1.0f, e - kTop);
    }
  }
  for (uint32_t i = tid; i < t_entries; i += kFoldThreads) {
    const float4 t = __ldg(p.tw + i);
    smem_t[i] = make_float4(t.x * in_scale, t.y * in_scale, t.z * in_scale, t.w * in_scale);
    smem_tn[i] = make_float2(-t.z * in_scale, -t.w * in_scale);
  }
  if (2 * p.mp < (T32 ? 8 : 16) * p.ks) {   // columns of the contraction that no group writes
    uint4* z = reinterpret_cast<uint4*>(smem_a);
    for (uint32_t i = tid; i < 4 * piece_bytes / 16; i += kFoldThreads) z[i] = make_uint4(0, 0, 0, 0);
    ptx::fence_proxy_async_smem();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = sh.tmem_base;

  // TF32 steps contract 8 instead of 16: twice as many additions that truncate.  Even and odd steps take accumulators of
  // their own (np <= 64 there), which the epilogue adds in round-to-nearest fp32.
  // Only where fp16 pieces are what the axis would have otherwise: it costs up to 9 % (100 x 66 x 250: 36.8 -> 40.1 us).
  const bool twin = T32 && p.twin && p.ks >= 2;

  if (warp < 4) {
    ptx::setmaxnreg_dec<32>();
    if (warp == 0 && lane == 0) {
      // ------------------------------------------------------------ MMA issuer
      const uint32_t idesc = T32 ? ptx::make_idesc_tf32(128, p.np) : ptx::make_idesc_f16(128, p.np);
      const uint32_t idesc_wide = T32 ? ptx::make_idesc_tf32(128, 2 * p.np) : ptx::make_idesc_f16(128, 2 * p.np);
      const uint64_t w0 = ptx::make_kmajor_sw128_desc(ptx::smem_u32(smem_w));
      const uint64_t a0 = ptx::make_kmajor_sw128_desc(ptx::smem_u32(smem_a));
      const uint32_t w_panel = uint32_t(2 * p.np * 128) >> 4;     // in descriptor address units
      FOLD_WAIT(&sh.w_full, 0, 0x701);
      unsigned tiles = first * H;
      for (unsigned k = 0;; ++k) {
        if (k == tiles) {
          if (!T32 || tiles != first * H) break;
          if (!rg.far_seen) break;
          FOLD_WAIT(&rg.first_done, 0, 0x707);
          tiles += (all ? my_units : rg.marked) * H;
          if (k == tiles) break;
        }
        const uint32_t buf = k & 1, ph = (k >> 1) & 1;
        FOLD_WAIT(&sh.d_empty[buf], ph ^ 1, 0x703);
        FOLD_WAIT(&sh.a_full[buf], ph, 0x702);
        ptx::tc_fence_after();
        const uint32_t d = tmem + buf * 256;
        const uint64_t ah = a0 + uint64_t(buf * 2 * piece_bytes >> 4), al = ah + uint64_t(piece_bytes >> 4);
        for (int s = 0; s < p.ks; ++s) {
          const uint32_t a_off = uint32_t(s >> 2) * (kFoldPanelBytes >> 4) + (s & 3) * 2;
          const uint64_t wd = w0 + uint32_t(s >> 2) * w_panel + (s & 3) * 2;
          if (T32) {
            const uint32_t dt = d + (twin && (s & 1) ? 128 : 0);
            ptx::mma_tf32_ss(dt, ah + a_off, wd, idesc_wide, s > (twin ? 1 : 0));
            ptx::mma_tf32_ss(dt + p.np, al + a_off, wd, idesc, 1);
          } else {
            ptx::mma_f16_ss(d, ah + a_off, wd, idesc_wide, s != 0);
            ptx::mma_f16_ss(d + p.np, al + a_off, wd, idesc, 1);
          }
        }
        ptx::tc_commit(&sh.a_empty[buf]);
        ptx::tc_commit(&sh.d_full[buf]);
      }
    }
  } else if (warp < 8) {
    // -------------------------------------------------------------- epilogue
    ptx::setmaxnreg_inc<112>();
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_addr = tmem + (uint32_t((warp & 3) * 32) << 16);
    const int q = MODE == KDFT_CONTIG ? row % Q : row / L;
    const unsigned line = MODE == KDFT_CONTIG ? row / Q : row % L;
    const uint64_t down11 = dup2(T32 ? 1.0f : 0x1p-11f);
    // one factor where it is a normal number, else the two one after the other
    const float both = p.out_mul * out_mul2;
    const bool one_step = both > 1e-30f && both < 1e30f;
    const uint64_t mul_a = dup2(one_step ? both : p.out_mul), mul_b = dup2(out_mul2);
    float amax = 0.0f;
    // tile k in the order of work, of unit `unit`; false: a wait gave up
    auto drain = [&](auto again, unsigned k, unsigned unit) -> bool {
      constexpr bool kSecond = decltype(again)::value;
      const uint32_t buf = k & 1, ph = (k >> 1) & 1;
      const unsigned l = (blockIdx.x + unit * gridDim.x) * L + line;
      const bool live = l < p.lines && (MODE == KDFT_CONTIG ? line < unsigned(L) : q < Q);   // not an idle lane
      float2* dst;
      size_t step;
      if (MODE == KDFT_CONTIG) {
        dst = p.out + size_t(l) * p.n + q;
        step = R;
      } else {
        const LinePlace at = fold_place(p, l, false, p.out_blocked);
        dst = p.out + at.base + (q + (k % H) * Q) * at.step;
        step = at.step * R;
      }
      FOLD_WAIT_WARP_ELSE(&sh.d_full[buf], ph, 0x704, return false);
      ptx::tc_fence_after();
      int shift = 0;
      bool pass_over = false;
      if (T32) {
        const unsigned slot = k / H % kFoldTops, tag = k / H + 1;
        const volatile uint32_t *top = rg.top + slot * L, *far = rg.far + slot * L;
        if (kSecond) {
          if (live) shift = fold_shift(top[line] & 0xff);
        } else if (rg.any_far[slot] == tag) {
          for (int i = lane; i < L; i += 32) pass_over |= far[i] >> 1 == tag && ((far[i] & 1) || top[i] >> 8 != tag);
          pass_over = __any_sync(0xffffffffu, pass_over);
          if (pass_over && k % H == H - 1 && warp == 4 && lane == 0) {
            rg.marks[unit >> 5] = rg.marks[unit >> 5] | 1u << (unit & 31);
            rg.marked = rg.marked + 1;
          }
        }
      }
      for (int c0 = 0; c0 < 2 * p.m; c0 += 32) {
        uint32_t hh[32], xx[32];
        ptx::tmem_ld_32x32(lane_addr + buf * 256 + c0, hh);
        ptx::tmem_ld_32x32(lane_addr + buf * 256 + p.np + c0, xx);
        ptx::tc_wait_ld();
        if (twin) {
          uint32_t more[32];
          ptx::tmem_ld_32x32(lane_addr + buf * 256 + 128 + c0, more);
          ptx::tc_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) hh[i] = __float_as_uint(__uint_as_float(hh[i]) + __uint_as_float(more[i]));
          ptx::tmem_ld_32x32(lane_addr + buf * 256 + 128 + p.np + c0, more);
          ptx::tc_wait_ld();
#pragma unroll
          for (int i = 0; i < 32; ++i) xx[i] = __float_as_uint(__uint_as_float(xx[i]) + __uint_as_float(more[i]));
        }
        if (c0 + 32 >= 2 * p.m) {     // the accumulator has been read: the next tile may overwrite it
          ptx::tc_fence_before();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&sh.d_empty[buf]);
        }
        uint64_t v[16];
#pragma unroll
        for (int i = 0; i < 16; ++i)
          v[i] = mul2(fma2(pack2_bits(xx[2 * i], xx[2 * i + 1]), down11, pack2_bits(hh[2 * i], hh[2 * i + 1])), mul_a);
        if (T32 ? kSecond && shift != 0 : !one_step) {
          const uint64_t f = T32 ? dup2(pow2f(-shift)) : mul_b;
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = mul2(v[i], f);
        }
        const int count = live && !pass_over ? p.m - c0 / 2 : 0;       // outputs of this line among the sixteen
        float top = 0.0f;
        if (!kSecond && count >= 16) {
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            float re, im;
            unpack2(v[i], re, im);
            *dst = make_float2(re, im);
            dst += step;
            top = fmaxf(top, fmaxf(fabsf(re), fabsf(im)));
          }
        } else {
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (i < count) {
              float re, im;
              unpack2(v[i], re, im);
              *dst = make_float2(re, im);
              dst += step;
              top = fmaxf(top, fmaxf(fabsf(re), fabsf(im)));
            }
        }
        amax = fmaxf(amax, finite_magnitude(top));       // a line with an infinity has no say in the next pass's scale
      }
      return true;
    };
    unsigned k = 0;
    for (; k < first * H; ++k)
      if (!drain(std::false_type(), k, k / H)) goto role_done;
    if (T32 && __builtin_expect(rg.far_seen != 0, 0)) {
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&rg.first_done);
      FOLD_WAIT_WARP(&rg.first_done, 0, 0x707);
      for (unsigned unit = fold_next(rg, all, 0, my_units); unit < my_units; unit = fold_next(rg, all, unit + 1, my_units))
        for (int h = 0; h < H; ++h, ++k)
          if (!drain(std::true_type(), k, unit)) goto role_done;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    if (!T32 && lane == 0 && amax > 0.0f) atomicMax(p.amax_out, __float_as_uint(amax));
  } else {
    // -------------------------------------------------------------- load, R-point sums, phase, split
    ptx::setmaxnreg_inc<112>();
    if (p.wc.silent_producer || warp - 8 >= p.split_warps) goto role_done;
    const bool wide = (p.m & 1) == 0;                              // 16-byte loads on the contiguous axis
    const uint32_t a_base = ptx::smem_u32(smem_a), t_base = ptx::smem_u32(smem_t), tn_base = ptx::smem_u32(smem_tn);
    // The tasks of all units go round the warps.  The host picks the number of warps such that no warp is so far ahead of
    // the buffers that the parity of a_empty could mean an older phase: consecutive units of a warp are neighbours, or
    // at most two apart where a unit uses one of the two buffers.
    // Task j of unit `unit`, the k-th in the order of work; false: a wait gave up.  (Two copies of the code: one that also waits for the
    // lines' exponents took 63 instead of 56 us on 256-point axes 0 of 256^3.)
    auto split = [&](auto again, unsigned k, unsigned j, unsigned unit) -> bool {
      constexpr bool kSecond = decltype(again)::value;
      const uint32_t buf = H == 2 ? 0 : k & 1, ph = (H == 2 ? k : k >> 1) & 1;
      unsigned line, grp;
      if (MODE == KDFT_CONTIG) {
        const unsigned id = j * 32 + lane;
        line = unsigned((uint64_t(id) * p.groups_magic) >> 24);
        grp = id - line * p.groups;
      } else {
        // sixteen lines: eight of them and two groups per half warp, so that its 8-byte operand stores meet every bank once
        // more than 32 lines: block by block
        line = L == 16 ? (lane & 7) | ((lane >> 4) << 3) : lane;
        grp = L == 16 ? j * 2 + ((lane >> 3) & 1) : j;
        if (L > 32) {
          const unsigned block = unsigned((uint64_t(j) * p.groups_magic) >> 24);
          line += block * 32;
          grp -= block * p.groups;
        }
      }
      const bool mine = line < unsigned(L) && grp < p.groups;
      C2 x[B / 2][R];
      {
        const unsigned l = (blockIdx.x + unit * gridDim.x) * L + line;
        const float2* src;
        size_t C = 1;                                              // distance of neighbouring points of a line
        if (MODE == KDFT_CONTIG) {
          src = p.in + size_t(l) * p.n + grp * B;
        } else {
          const LinePlace at = fold_place(p, l, p.in_blocked, false);
          C = at.step;
          src = p.in + at.base + size_t(grp * B) * C;
        }
        const size_t sstep = size_t(p.m) * C;
        const bool live = mine && l < p.lines;
        if (!kSecond && live && (grp + 1) * B <= unsigned(p.m)) {
          if (MODE == KDFT_CONTIG && wide) {
#pragma unroll
            for (int s = 0; s < R; ++s, src += sstep)
#pragma unroll
              for (int b = 0; b < B / 2; ++b) {
                float v0, v1, v2, v3;
                ld_stream16(src + 2 * b, v0, v1, v2, v3);
                x[b][s] = {pack2(v0, v2), pack2(v1, v3)};
              }
          } else {
#pragma unroll
            for (int b = 0; b < B / 2; ++b) {
              const float2* at = src + (2 * b) * C;
#pragma unroll
              for (int s = 0; s < R; ++s, at += sstep) {
                float v0, v1, v2, v3;
                ld_stream8(at, v0, v1);
                ld_stream8(at + C, v2, v3);
                x[b][s] = {pack2(v0, v2), pack2(v1, v3)};
              }
            }
          }
        } else {
#pragma unroll
          for (int b = 0; b < B / 2; ++b)
#pragma unroll
            for (int s = 0; s < R; ++s) {
              float v0 = 0.0f, v1 = 0.0f, v2 = 0.0f, v3 = 0.0f;
              if (live && grp * B + 2 * b < unsigned(p.m)) ld_stream8(src + s * sstep + (2 * b) * C, v0, v1);
              if (live && grp * B + 2 * b + 1 < unsigned(p.m)) ld_stream8(src + s * sstep + (2 * b + 1) * C, v2, v3);
              x[b][s] = {pack2(v0, v2), pack2(v1, v3)};
            }
        }
      }
      // bring a later unit of this CTA into L2 meanwhile
      if (p.prefetch && !kSecond && unit + kAhead < my_units) {
        const unsigned l0 = (blockIdx.x + (unit + kAhead) * gridDim.x) * L;
        if (l0 < p.lines) {
          if (MODE == KDFT_CONTIG) {
            const char* base = reinterpret_cast<const char*>(p.in + size_t(l0) * p.n);
            const unsigned bytes = min(unsigned(L), p.lines - l0) * unsigned(p.n) * 8;
            for (unsigned o = (j * 32 + lane) * 128; o < bytes; o += p.tasks * 4096) prefetch_l2(base + o);
          } else {
            constexpr unsigned kLpr = L * 8 > 128 ? L * 8 / 128 : 1;  // 128-byte lines per row
            for (unsigned o = j * 32 + lane; o < unsigned(p.n) * kLpr; o += p.tasks * 32) {
              const unsigned seg = (o % kLpr) * 16;
              if (l0 + seg < p.lines) {
                const LinePlace at = fold_place(p, l0 + seg, p.in_blocked, false);
                prefetch_l2(p.in + at.base + (o / kLpr) * at.step);
              }
            }
          }
        }
      }
      float factor = pre;
      if (T32) {                                                   // this task's share of its lines' exponents
        float top = 0.0f;
#pragma unroll
        for (int b = 0; b < B / 2; ++b)
#pragma unroll
          for (int s = 0; s < R; ++s) {
            float v0, v1, v2, v3;
            unpack2(x[b][s].re, v0, v2);
            unpack2(x[b][s].im, v1, v3);
            top = max_abs3(max_abs3(top, v0, v1), v2, v3);
          }
        const unsigned slot = k % kFoldTops, tag = k + 1;
        const uint32_t field = fold_field(top);
        const uint32_t at = slot * L + (mine ? line : 0);
        uint32_t* word = &rg.top[at];
        if (!kSecond) {
          if (mine && field != 0) {
            if (!fold_outside(field)) {
              *const_cast<volatile uint32_t*>(word) = tag << 8;
            } else {
              atomicMax(&rg.far[at], tag << 1 | (field > kFoldHigh));
              rg.any_far[slot] = tag;
              rg.far_seen = 1;
            }
          }
        } else {
          if (mine) atomicMax(word, tag << 8 | field);
          const unsigned i = k - first, block = L > 32 ? unsigned((uint64_t(j) * p.groups_magic) >> 24) : 0;
          uint64_t* bar = &rg.top_full[i % kFoldTops][block];
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(bar);
          FOLD_WAIT_WARP_ELSE(bar, (i / kFoldTops) & 1, 0x706, return false);
          factor = pow2f(mine ? fold_shift(*const_cast<volatile uint32_t*>(word) & 0xff) : 0);
        }
      }
      if (T32 ? kSecond : factor != 1.0f) {
#pragma unroll
        for (int b = 0; b < B / 2; ++b)
#pragma unroll
          for (int s = 0; s < R; ++s) x[b][s] = {mul2(x[b][s].re, dup2(factor)), mul2(x[b][s].im, dup2(factor))};
      }
      {
        const uint32_t col = grp * (B * (T32 ? 8 : 4));            // bytes along the contraction
        const uint32_t chunk = (col >> 4) & 7, low = col & 15;
        const uint32_t at0 = a_base + buf * 2 * piece_bytes + (col >> 7) * kFoldPanelBytes + low +
                             (MODE == KDFT_CONTIG ? line * Q * 128 : line * 128);
        const uint32_t t_at = t_base + grp * (B * 8), tn_at = tn_base + grp * (B * 4);
        uint32_t hi[B], lo[B];
        if (B == 4) {
#pragma unroll
          for (int b = 0; b < B / 2; ++b) dft_r<R>(x[b], sign);
        } else {
          dft_r<R>(x[0], sign);
        }
#pragma unroll
        for (int h = 0; h < H; ++h) {
          FOLD_WAIT_WARP_ELSE(&sh.a_empty[buf + h], ph ^ 1, 0x705, return false);
          if (mine) {
#pragma unroll
            for (int q = h * Q; q < (h + 1) * Q; ++q) {
              // row (operand lane): line * R + q or q * L + line; the swizzle XORs the 16-byte chunk with row & 7
              const uint32_t sw = MODE == KDFT_CONTIG ? (line * Q + q) & 7 : line & 7;
              const uint32_t row_at = at0 + h * 2 * piece_bytes + (q - h * Q) * (MODE == KDFT_CONTIG ? 128 : L * 128);
              const uint32_t at = row_at + ((chunk ^ sw) << 4);
#pragma unroll
              for (int b = 0; b < B / 2; ++b) {
                uint64_t c, d, dn;
                C2 u = x[b][0];
                if (!T32 || q != 0) lds_2x64(t_at + (uint32_t(q) * p.mp / 2 + b) * 16, c, d);
                if (q == 0) {                  // the phases are 1, times the scale that the fp16 pieces need
                  if (!T32) u = {mul2(u.re, c), mul2(u.im, c)};
                } else {
                  lds_64(tn_at + (uint32_t(q) * p.mp / 2 + b) * 8, dn);
                  u = c2_mul(x[b][q], c, d, dn);
                }
                if constexpr (T32) {           // two points fill a chunk of 16 bytes
                  uint32_t th[4], tl[4];
                  split_tf32(u, th, tl);
                  const uint32_t to = row_at + (((chunk + b) ^ sw) << 4);
                  sts_128(to, th[0], th[1], th[2], th[3]);
                  sts_128(to + piece_bytes, tl[0], tl[1], tl[2], tl[3]);
                } else {
                  split_half2_scaled(u, hi[2 * b], hi[2 * b + 1], lo[2 * b], lo[2 * b + 1]);
                }
              }
              if constexpr (T32) {
              } else if constexpr (B == 4) {
                sts_128(at, hi[0], hi[1], hi[2], hi[3]);
                sts_128(at + piece_bytes, lo[0], lo[1], lo[2], lo[3]);
              } else {
                sts_64(at, hi[0], hi[1]);
                sts_64(at + piece_bytes, lo[0], lo[1]);
              }
            }
          }
          ptx::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive(&sh.a_full[buf + h]);
        }
      }
      return true;
    };
    unsigned k = 0, j = unsigned(warp - 8);
    for (; j >= p.tasks; ++k) j -= p.tasks;
    while (k < first) {
      if (!split(std::false_type(), k, j, k)) goto role_done;
      for (j += unsigned(p.split_warps); j >= p.tasks; ++k) j -= p.tasks;
    }
    if constexpr (T32) {
      // far_seen is final when every warp has split its share
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(&rg.split_done);
      FOLD_WAIT_WARP(&rg.split_done, 0, 0x708);
      if (__builtin_expect(rg.far_seen != 0, 0)) {
        FOLD_WAIT_WARP(&rg.first_done, 0, 0x707);
        unsigned unit = fold_next(rg, all, 0, my_units);
        for (unsigned i = first; i < k; ++i) unit = fold_next(rg, all, unit + 1, my_units);
        while (unit < my_units) {
          if (!split(std::true_type(), k, j, unit)) goto role_done;
          for (j += unsigned(p.split_warps); j >= p.tasks; ++k) {
            j -= p.tasks;
            unit = fold_next(rg, all, unit + 1, my_units);
          }
        }
      }
    }
  }

role_done:
  if (warp == 0 && lane == 0 && sh.abort_flag) {
    // give the table load that was already issued a bounded chance to land before the CTA goes away
    const long long t0 = clock64();
    while (clock64() - t0 < 2000000LL) { }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (warp == 1) ptx::tmem_dealloc(tmem, 512);
}

#undef FOLD_WAIT
#undef FOLD_WAIT_WARP
#undef FOLD_WAIT_WARP_ELSE

}  // namespace dft3d
