// fio_fx.cuh -- FP64- and FP32-accurate stage products on the tensor cores (sm_103a) in fixed
// point: every operand is cut into 8-bit digits, the digits are multiplied as FP16 integers by
// tcgen05.mma, and the products are summed exactly.
//
// Why.  The stage products are dense contractions, and the CUDA cores bound them: GB300 has 2 FP64
// multiply-adds per clock and SM (1.2 TFLOP/s) and 128 FP32 ones (78 TFLOP/s), against about 3600
// FP16 ones with FP32 accumulation on the tensor cores.  The method is error-free splitting (Ozaki,
// Ogita, Oishi and Rump, "Error-free transformations of matrix multiplication by using fast
// routines of matrix multiplication", 2012) in its fixed-point form:
//   the rows and columns of the (complex, interleaved) factor are scaled by powers of two, Er and Ec, to
//   entries below 1 with one above 1/2 in every row (k_fx_exps); the column scales go into the
//   gathered vector, whose entries are cut below 2^ej > max |x_c| 2^Ec; each real
//   becomes an integer (f = 62 in FP64, 30 in FP32), v_a = a 2^(f-Er-Ec), v_x = x 2^(f+Ec-ej), written
//   in balanced base 256, v = sum_i d_i 256^(S-1-i), -128 <= d_i <= 127, S = 8 resp. 4 digits;
//   sum_k v_a v_x = sum_o 256^(2S-2-o) sum_{i+l=o} (D_i^a D_l^x): every digit product is an
//   integer of at most 2^14, exact in FP16 x FP16 -> FP32, and sums of all products of one order o
//   over at most 128 (FP64) or 256 (FP32) real columns stay within 2^24: the FP32 accumulators
//   hold them exactly whatever the order of summation.  Orders 0..S-1 are kept; what is dropped is
//   about 2^-59 resp. 2^-27 of the product, below the rounding of an FMA chain of the operands'
//   own type (FP64 chain 2^-51, FP32 2^-23 over 500 columns).
//   Those are errors of the largest scaled product of a block; an FMA chain's are of a row's own sum of
//   products.  The column scales keep the two together: a real operator's HIF blocks have columns that
//   differ by 2^6, and vectors that differ the other way.  Example 3 n = 128, G-dot in FP64 (relative
//   error, CPU restatement): FMA chain 1.4e-15; rows scaled alone 1.6e-15, with columns 2.6e-16; right-hand
//   sides that span 40 binary orders, n = 64: 1.1e-15, 1.5e-15, 3.6e-16; K-dot 1.6e-15, 1.2e-16, 1.2e-16.
//   The accumulators are drained every 128 / 256 columns into 96- resp. 64-bit integers, so a
//   whole output is summed without any rounding and rounded once, to nearest, at the end.
// Columns that hold infinities, NaN, or exponents near the end of the range are computed in plain
// arithmetic instead (fx::plain): the same values as the CUDA-core kernels.
//
// Layouts.  Cutting a real into digits costs 14 integer instructions and 1.5 per digit, at 64 per
// clock and SM: done in the stage kernel it bound it (2400 clocks per 16 KB of factor, against 760
// for its HBM stream).  So the factor is cut once, at upload, into a copy of the same size in bytes
// (k_fx_pack), and the vector once per stage (k_fx_gather, which also takes the columns' scales:
// a column's maximum is needed before its first digit).  In both, the 4 bytes of digit i of two
// complex columns (re, im, re, im) are one word, and two byte permutes with the constant 0x64
// make it two pairs of FP16 numbers 1024 + byte, from which 1152 is taken off exactly.
// A unit's data (128-row tile of a block) is contiguous, in chunks of 128 bytes per row:
//   [K step of 8 complex columns][pair of digits][half of the K step][row] x 16 bytes
//   (2 digits x 4 complex columns); the vector's likewise with right-hand sides for rows.
//
// k_stage_fx: persistent, one CTA per SM, 28 warps, over units (block, 128-row tile, tile of BT
// right-hand sides), largest first; the right-hand-side tiles of a unit go to neighbouring CTAs so
// that the factor is read from HBM once and then from L2.
//   copy warp       factor and vector chunks by bulk copies into a ring of raw slots;
//   16 slicer warps in four groups, group g for the K steps g mod 4: chunk -> S digit tiles of the
//                   factor, the K-major 128-byte-swizzled operand of the MMA (a tile's 128-byte rows
//                   are four slots of one K = 16 step each: group g writes slot g), and of the vector
//                   with the complex sign pattern (fio_tc.cuh), digit l in rows l 2BT .. (l+1) 2BT - 1;
//   MMA warp        per K step one MMA per digit i of the factor: A_i against the concatenated
//                   digits B_0 .. B_{S-1-i}, whose products land in the accumulator columns of
//                   order i + l (N up to 256: one read of A_i serves all of them);
//   8 drain warps   accumulators (two buffers) -> integers, and the scaled rows to their outputs.
// A slicer step is a chain of waits, shared-memory round trips and a proxy fence; four groups hide
// it from one another.  Registers are moved to the drain warps (setmaxnreg), which keep a row's sums.
//
// Measured (one GB300, the shapes of the 2D transform at n = 256, 548 M entries, K-dot; before: the
// best CUDA-core kernel): FP64 b = 1 / 8 / 16 / 32: 5.53 / 32.9 / 65.6 / 129 ms before, 2.02 / 2.25 /
// 3.07 / 5.97 now; FP32 b = 16 / 32: 2.26 / 3.45 before, 1.53 / 1.94 now.  On 64 blocks of 512 x 512, FP64 b = 16, a K step
// takes 0.65 us (1340 clocks); it moves 147 KB through shared memory (copies in 18, read 18, digits
// written 40, operands read 71), 1150 clocks at 128 bytes a clock: L1 and shared memory are 73% busy on the busiest
// SM, the tensor cores 46%, HBM 43% (its stream needs 760 clocks).
// All waits are bounded as in fio_tc.cuh.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "fio_internal.h"
#include "fio_kernels.cuh"
#include "fio_tc.cuh"

namespace fio {

struct FxArgs {
  const FxUnit* units;
  int nunits;
  int nrt;            // right-hand-side tiles
  const uint8_t* A;   // digit copy of the factor (k_fx_pack)
  const uint8_t* X;   // digit copy of the gathered vector (k_fx_gather)
  const int* ej;      // scale exponent of every (block, right-hand side), block stride b
  const short* rexp;  // scale exponent Er of every (block, row of the product), block stride lrow
  const int2* list;   // per block and column of the product: the index gathered there (-1: none), its scale
  int llist;          // exponent Ec; block stride, a multiple of 16 not below lcol
  const int* rowidx;  // output index lists (forward: out, adjoint: in), block stride lrow
  const int* colidx;  // gather index lists, block stride lcol
  int lrow, lcol;
  int maxcols;        // columns of the widest block, whole chunks
  const int2* dims;   // per block (valid rows, valid columns) of the forward block
  const int2* xofs;   // per block: columns before it in X (FP64, FP32 chunking)
  long long xcols;    // columns of one right-hand-side tile of X
  int nblk;
  int R, C;           // packed block shape
  const void* M;      // the factor itself (columns that need plain arithmetic)
  const void* x;
  long long xrs, xcs;
  void* y;
  long long yrs, ycs;
  int b;
  int nraw;           // raw ring slots (2 .. kMaxRaw)
  long long steps;    // K steps of all units (host side)
  int* timeout;       // set when a bounded wait gave up
};

namespace fx {

constexpr int kDrainWarps = 8, kSlots = 4;  // slots: K steps (16 reals) in a digit tile's 128-byte rows
constexpr int kGroupWarps = 4;              // slicer warps per slot
constexpr int kThreads = 32 * (kDrainWarps + kSlots * kGroupWarps + 4);  // 896: 72 registers a thread
// registers per role; over the 7 warpgroups: 2 x 128 + 4 x 48 + 56 = 7 x 72
constexpr int kDrainRegs = 128, kSliceRegs = 48, kCtrlRegs = 56;
static_assert(2 * kDrainRegs + 4 * kSliceRegs + kCtrlRegs <= 7 * 72, "more registers than the launch has: would wait forever");
// Raw slots at most.  A chunk's arrival barrier is the chunk's number mod 8, whatever the slots: the
// chunks that a slicer group takes from one barrier are 8 apart, each consumed before the next is
// issued, so that no group waits for a phase two ahead (which a parity wait would let pass).
constexpr int kMaxRaw = 8;
// Chunks that the copy warp asks L2 for ahead of the ring: shared memory holds three to five slots
// beside the digit tiles, 55 KB in flight an SM, and under load HBM answers after 1.5 us or more.
// (2D n = 256 FP64 b = 16: 3.23 ms without, 3.06 with; where several CTAs share a unit's factor they
// already run ahead of one another, and 1D b = 64 lost 0.4%.)
constexpr int kAhead = 6;
constexpr uint32_t kBufCols = 256;
constexpr int kPlain = 1 << 20;  // scale exponent that marks a column for plain()

template <typename R> struct Cfg;
template <> struct Cfg<double> {
  using V = double2;
  using F = uint2;  // fixed-point value, each byte a digit + 128
  static constexpr int S = 8, KPC = 1, G = 8;  // digits, K steps per raw chunk, K steps per drain
};
template <> struct Cfg<float> {
  using V = float2;
  using F = uint32_t;
  static constexpr int S = 4, KPC = 2, G = 16;
};
// a raw slot: a chunk of the factor (128 rows x 128 bytes) and of the vector (BT x 128 bytes)
template <int BT> constexpr int raw_bytes() { return 16384 + BT * 128; }
template <typename R, int BT> constexpr int smem_fixed() { return 1024 + Cfg<R>::S * (16384 + 2 * BT * 128); }

// 4 accumulator columns of 32 lanes (no wait)
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, float (&r)[4]) {
  uint32_t a, b, c, d;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(a), "=r"(b), "=r"(c), "=r"(d)
               : "r"(taddr));
  r[0] = __uint_as_float(a);
  r[1] = __uint_as_float(b);
  r[2] = __uint_as_float(c);
  r[3] = __uint_as_float(d);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
template <int N> __device__ __forceinline__ void regs_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N)); }
template <int N> __device__ __forceinline__ void regs_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N)); }
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ uint64_t evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}
// contiguous copy of a multiple of 16 bytes into shared memory
__device__ __forceinline__ void bulk(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(tc::su32(bar))
               : "memory");
}
__device__ __forceinline__ void bulk(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(tc::su32(bar)), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* src, uint32_t bytes, uint64_t policy) {
  asm volatile("cp.async.bulk.prefetch.L2.global.L2::cache_hint [%0], %1, %2;" ::"l"(src), "r"(bytes), "l"(policy) : "memory");
}
__device__ __forceinline__ void expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc::su32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((e + 127) << 23); }  // -126 <= e <= 127

// fixed-point value of a under the scale 2^E, as digits + 128 (zeros and subnormals have no implicit bit: with
// it a zero would count as 2^-1023, up to 2^-41 of a column whose largest entry is near 2^-982)
__device__ __forceinline__ uint2 fix(double a, int E) {
  const uint32_t hi = (uint32_t)__double2hiint(a), lo = (uint32_t)__double2loint(a);
  const uint32_t be = (hi >> 20) & 0x7ffu;
  const int sh = min(max(1023 + E - (int)max(be, 1u), 0), 63);
  unsigned long long v = ((((unsigned long long)((hi & 0xfffffu) | (be ? 0x100000u : 0u))) << 32) | lo) << 10;
  v >>= sh;
  const long long s = (long long)((int)hi >> 31);
  v = (v ^ (unsigned long long)s) - (unsigned long long)s + 0x8080808080808080ull;
  return make_uint2((uint32_t)v, (uint32_t)(v >> 32));
}
__device__ __forceinline__ uint32_t fix(float a, int E) {
  const int s = 30 - E, h = s >> 1;  // -119 .. 176
  return (uint32_t)__float2int_rn(a * pow2f(h) * pow2f(s - h)) + 0x80808080u;
}
template <typename F> __device__ __forceinline__ F fix_zero();
template <> __device__ __forceinline__ uint2 fix_zero<uint2>() { return make_uint2(0x80808080u, 0x80808080u); }
template <> __device__ __forceinline__ uint32_t fix_zero<uint32_t>() { return 0x80808080u; }

// bytes B of two complex values: (re0, im0, re1, im1)
template <int B>
__device__ __forceinline__ uint32_t gather_byte(uint32_t re0, uint32_t im0, uint32_t re1, uint32_t im1) {
  return __byte_perm(__byte_perm(re0, im0, B | ((4 + B) << 4)), __byte_perm(re1, im1, B | ((4 + B) << 4)), 0x5410);
}
template <int I>  // digit I, 0 the most significant
__device__ __forceinline__ uint32_t digit_word(uint2 re0, uint2 im0, uint2 re1, uint2 im1) {
  constexpr int B = 7 - I;
  return B >= 4 ? gather_byte<(B & 3)>(re0.y, im0.y, re1.y, im1.y) : gather_byte<(B & 3)>(re0.x, im0.x, re1.x, im1.x);
}
template <int I>
__device__ __forceinline__ uint32_t digit_word(uint32_t re0, uint32_t im0, uint32_t re1, uint32_t im1) {
  return gather_byte<3 - I>(re0, im0, re1, im1);
}
// digits 2P, 2P + 1 of four complex columns, as stored
template <int P, typename F>
__device__ __forceinline__ uint4 digit_pair(const F (&re)[4], const F (&im)[4]) {
  return make_uint4(digit_word<2 * P>(re[0], im[0], re[1], im[1]), digit_word<2 * P>(re[2], im[2], re[3], im[3]),
                    digit_word<2 * P + 1>(re[0], im[0], re[1], im[1]), digit_word<2 * P + 1>(re[2], im[2], re[3], im[3]));
}
// two of a word's bytes (digits + 128) as FP16 integers: HI = 0 the first two, 1 the last two
template <int HI>
__device__ __forceinline__ uint32_t half2_of(uint32_t w) {
  uint32_t d;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(d) : "r"(__byte_perm(w, 0x64646464u, HI ? 0x4342 : 0x4140)), "r"(0x64806480u));
  return d;
}
__device__ __forceinline__ void st128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

// one output of a block by the CUDA-core kernels' sum (columns whose entries the fixed point cannot
// hold).  X: the column's entries, which k_fx_gather left as they are in the place of the digits
template <typename V, bool ADJ>
__device__ __noinline__ V plain(const V* M, int ldm, const int* cidx, int ncols, int r, const uint8_t* X, int wt, int j) {
  constexpr int S = Cfg<typename std::conditional<sizeof(V) == 16, double, float>::type>::S, PER = 16 / (int)sizeof(V);
  V acc = czero<V>();
  for (int c = 0; c < ncols; ++c) {
    const V* item = reinterpret_cast<const V*>(X + ((size_t)((c >> 3) * S + (c & 7) / PER) * wt + j) * 16);
    const V v = cidx[c] >= 0 ? item[c % PER] : czero<V>();
    acc = ADJ ? cmacc(acc, M[(size_t)c * ldm + r], v) : cmac(acc, M[(size_t)r * ldm + c], v);
  }
  return acc;
}

// biased exponent of the larger part (subnormals: 1), -1 for zero
__device__ __forceinline__ int biased(double2 v) {
  const uint32_t x = (uint32_t)__double2hiint(v.x) & 0x7fffffffu, y = (uint32_t)__double2hiint(v.y) & 0x7fffffffu;
  const uint32_t any = x | y | (uint32_t)__double2loint(v.x) | (uint32_t)__double2loint(v.y);
  return any ? (int)max(max(x, y) >> 20, 1u) : -1;
}
__device__ __forceinline__ int biased(float2 v) {
  const uint32_t m = max(__float_as_uint(v.x) & 0x7fffffffu, __float_as_uint(v.y) & 0x7fffffffu);
  return m ? (int)max(m >> 23, 1u) : -1;
}

// An entry's exponent under its column scale, as a key > 0 that grows with it (0: zero); infinities and NaN above all
constexpr int kKeyBias = 64, kKeyBad = 1 << 14;
template <typename V>
__device__ __forceinline__ int scale_key(V v, int ce) {
  const int be = biased(v);
  return be < 0 ? 0 : be == (sizeof(V) == 16 ? 2047 : 255) ? kKeyBad : be + ce + kKeyBias;
}
// scale exponent of a gathered vector from its largest key (0 for a zero vector)
template <typename R>
__device__ __forceinline__ int col_exp(int key) {
  constexpr bool W = std::is_same<R, double>::value;
  if (key == 0) return 0;
  const int be = key - kKeyBias;
  if (be < 40 || be > (W ? 2047 - 40 : 255 - 40)) return kPlain;
  return be - (W ? 1022 : 126);
}

// 96-bit sum of FP64's drains: hi 2^32 + lo
struct Acc96 {
  long long hi;
  uint32_t lo;
};
// v 2^s, rounded to nearest, in 32-bit integer steps (the FP64 pipe's two lanes a clock would take
// four times as long for the conversion of a tile as its sums take to form)
__device__ __forceinline__ double to_double(Acc96 v, int s) {
  uint32_t w2 = (uint32_t)((unsigned long long)v.hi >> 32), w1 = (uint32_t)v.hi, w0 = v.lo;
  const uint32_t sg = (uint32_t)((int)w2 >> 31);
  // magnitude: negated where the sign is set
  asm("{\n\txor.b32 %0, %0, %3;\n\txor.b32 %1, %1, %3;\n\txor.b32 %2, %2, %3;\n\t"
      "sub.cc.u32 %0, %0, %3;\n\tsubc.cc.u32 %1, %1, %3;\n\tsubc.u32 %2, %2, %3;\n\t}"
      : "+r"(w0), "+r"(w1), "+r"(w2)
      : "r"(sg));
  int e = s + 95;  // exponent of w2's first bit
  if (w2 == 0) {
    w2 = w1;
    w1 = w0;
    w0 = 0;
    e -= 32;
  }
  if (w2 == 0) {
    w2 = w1;
    w1 = 0;
    e -= 32;
  }
  const int lz = __clz((int)w2);
  const uint32_t h = __funnelshift_l(w1, w2, lz), l = __funnelshift_l(w0, w1, lz);
  e -= lz;
  // 53 of the 64 bits, to nearest (a carry out of a mantissa of ones goes into the exponent)
  uint32_t mh = h >> 11, ml = __funnelshift_r(l, h, 11);
  const uint32_t up = (l >> 10) & 1u;
  asm("add.cc.u32 %0, %0, %2;\n\taddc.u32 %1, %1, 0;" : "+r"(ml), "+r"(mh) : "r"(up));
  const int be = e + 1022;  // the leading bit adds the last 1
  if (h == 0) return 0.0;
  if (be < 0 || be > 2044) {
    const double m = ldexp((double)(((unsigned long long)mh << 32) | ml), e - 52);
    return sg ? -m : m;
  }
  return __hiloint2double((int)((mh + ((uint32_t)be << 20)) | (sg & 0x80000000u)), (int)ml);
}
// the upper 41 bits and the lower 23 converted apart: at most 2^-24 off before the last rounding
// (the 64-bit conversion instruction is many times slower)
__device__ __forceinline__ float to_float(long long v, int s) {
  const float lo = __int_as_float(0x4b000000 | (int)(v & 0x7fffff)) - 8388608.0f;
  const int h = s >> 1;
  return fmaf((float)(int)(v >> 23), 8388608.0f, lo) * pow2f(h) * pow2f(s - h);
}

template <int I> using Int = std::integral_constant<int, I>;

}  // namespace fx

// The gathered vector of every block as digits (layout above), and its columns' scale exponents.
// A CTA per (block, right-hand-side tile), a thread for every CS-th group of four columns of one
// right-hand side.  Bound by the latency of its two dependent loads, list and vector: the entries of
// up to HOLD groups stay in registers between the maximum and the cut (stages of at most 4 CS HOLD columns a
// block; no more than a stage needs, for the registers), those of longer blocks are loaded twice (HOLD 0).
template <typename R, bool ADJ, int BT, int HOLD>
__global__ void __launch_bounds__(256) k_fx_gather(const FxArgs a, uint8_t* X, int* ej) {
  using namespace fx;
  using C = Cfg<R>;
  using V = typename C::V;
  using F = typename C::F;
  constexpr bool W = std::is_same<R, double>::value;
  constexpr int CS = 256 / BT;
  __shared__ int s_key[BT];
  const int blk = blockIdx.x, rt = blockIdx.y;
  const int j0 = rt * BT, wt = min(BT, a.b - j0);
  const int2 d = a.dims[blk];
  const int ncols = ADJ ? d.x : d.y;
  const int nk = C::KPC * ((ncols + 8 * C::KPC - 1) / (8 * C::KPC)), nq = 2 * nk;
  const int4* list = reinterpret_cast<const int4*>(a.list + (size_t)blk * a.llist);  // two columns each
  const V* x = (const V*)a.x;
  const int tid = threadIdx.x;
  pdl_go();
  if (tid < BT) s_key[tid] = 0;
  // lanes along the right-hand sides (BT a power of two; those beyond wt idle)
  const int j = tid % BT, c0 = tid / BT;
  const bool on = j < wt;
  struct Four {
    V v[4];
    int ce[4];
  };
  auto get = [&](Four& f, const int4& p, const int4& q) {
    const int idx[4] = {p.x, p.z, q.x, q.z};
    f.ce[0] = p.y;
    f.ce[1] = p.w;
    f.ce[2] = q.y;
    f.ce[3] = q.w;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      f.v[i] = on && idx[i] >= 0 ? x[(long long)idx[i] * a.xrs + (long long)(j0 + j) * a.xcs] : czero<V>();
  };
  auto key = [&](const Four& f, int m) {
#pragma unroll
    for (int i = 0; i < 4; ++i) m = max(m, scale_key(f.v[i], f.ce[i]));
    return m;
  };
  constexpr bool hold = HOLD > 0;
  Four held[HOLD + 1];
  int4 lp[HOLD + 1], lq[HOLD + 1];
  const int4 none = make_int4(-1, 0, -1, 0);
  if constexpr (hold) {
#pragma unroll
    for (int k = 0; k < HOLD; ++k) {
      const int q = c0 + k * CS;
      lp[k] = q < nq ? list[2 * q] : none;
      lq[k] = q < nq ? list[2 * q + 1] : none;
    }
  }
  __syncthreads();
  pdl_wait();
  int m = 0;
  if constexpr (hold) {
#pragma unroll
    for (int k = 0; k < HOLD; ++k) get(held[k], lp[k], lq[k]);
#pragma unroll
    for (int k = 0; k < HOLD; ++k) m = key(held[k], m);
  } else {
#pragma unroll 1
    for (int q = c0; q < nq; q += CS) {
      Four f;
      get(f, list[2 * q], list[2 * q + 1]);
      m = key(f, m);
    }
  }
  if (on) atomicMax(&s_key[j], m);
  __syncthreads();
  if (!on) return;
  const int e = col_exp<R>(s_key[j]);
  if (c0 == 0) ej[(size_t)blk * a.b + j0 + j] = e;
  const int2 xo = a.xofs[blk];
  uint4* out = reinterpret_cast<uint4*>(X + ((long long)rt * BT * a.xcols + (long long)(W ? xo.x : xo.y) * wt) * sizeof(V));
  auto put = [&](int q, const Four& f) {  // half q & 1 of K step q / 2
    uint4* o = out + ((size_t)(q >> 1) * C::S + (q & 1)) * wt + j;
    if (e == kPlain) {  // for fx::plain, entry by entry; the products of these bytes are not used
      constexpr int PER = 16 / (int)sizeof(V);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        V* item = reinterpret_cast<V*>(out + ((size_t)(q >> 1) * C::S + (4 * (q & 1) + i) / PER) * wt + j);
        item[i % PER] = f.v[i];
      }
      return;
    }
    F re[4], im[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      re[i] = fix(f.v[i].x, e - f.ce[i]);
      im[i] = fix(f.v[i].y, e - f.ce[i]);
    }
    o[0] = digit_pair<0>(re, im);
    o[2 * wt] = digit_pair<1>(re, im);
    if constexpr (W) {
      o[4 * wt] = digit_pair<2>(re, im);
      o[6 * wt] = digit_pair<3>(re, im);
    }
  };
  if constexpr (hold) {
#pragma unroll
    for (int k = 0; k < HOLD; ++k)
      if (c0 + k * CS < nq) put(c0 + k * CS, held[k]);
  } else {
#pragma unroll 1
    for (int q = c0; q < nq; q += CS) {
      Four f;
      get(f, list[2 * q], list[2 * q + 1]);
      put(q, f);
    }
  }
}

template <typename R, bool ADJ, int BT>
__global__ void __launch_bounds__(fx::kThreads, 1) k_stage_fx(const FxArgs a) {
  using namespace tc;
  using namespace fx;
  using C = fx::Cfg<R>;
  using V = typename C::V;
  constexpr bool W = std::is_same<R, double>::value;
  constexpr int S = C::S, KPC = C::KPC, G = C::G;
  constexpr int NS = 2 * BT;                // accumulator columns of one order
  constexpr int KC = 8 * KPC;               // complex columns per raw chunk
  constexpr uint32_t RAW = raw_bytes<BT>();
  static_assert(S * NS <= (int)kBufCols, "an accumulator buffer holds every order");
  constexpr uint32_t BBYTES = NS * 128;     // one digit of the vector operand
  __shared__ uint32_t s_tmem;
  __shared__ __align__(8) uint64_t raw_full[kMaxRaw], raw_empty[kMaxRaw];
  __shared__ __align__(8) uint64_t dig_full[kSlots], dig_empty[kSlots];
  __shared__ __align__(8) uint64_t acc_full[2], acc_empty[2], s_done;
  extern __shared__ __align__(16) uint8_t smem_dyn[];
  const uint32_t base = (su32(smem_dyn) + 1023u) & ~1023u;
  uint8_t* gbase = smem_dyn + (base - su32(smem_dyn));
  constexpr uint32_t OFF_B = S * 16384u, OFF_RAW = OFF_B + S * BBYTES;

  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const int total = a.nunits * a.nrt;
  const uint32_t nraw = (uint32_t)a.nraw;
  // every role reads the unit after its current one ahead of time (a unit may be two K steps long)
  auto unit = [&](int u) { return a.units[min(u, total - 1) / a.nrt]; };

  if (warp == 0) tmem_alloc(&s_tmem, 512);
  if (tid == 0) {
    for (int q = 0; q < kMaxRaw; ++q) {
      mbar_init(&raw_full[q], 1);
      mbar_init(&raw_empty[q], KPC * kGroupWarps);
    }
    for (int q = 0; q < kSlots; ++q) {
      mbar_init(&dig_full[q], kGroupWarps);
      mbar_init(&dig_empty[q], 1);
    }
    for (int q = 0; q < 2; ++q) {
      mbar_init(&acc_full[q], 1);
      mbar_init(&acc_empty[q], kDrainWarps);
    }
    mbar_init(&s_done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
  pdl_go();  // only now: a kernel started behind this one may hold tensor memory while it waits for it
  bool ok = true;

  if (warp < kDrainWarps) {
    regs_inc<kDrainRegs>();
    // ---- accumulators -> integers -> rows -----------------------------------------------------
    const int quad = warp & 3, half = warp >> 2;
    uint32_t g = 0;  // drains so far
    int oidx, er, ejl;  // output row, its scale; lane l keeps the scale of the warp's l-th right-hand side
    auto row_of = [&](const FxUnit& e, int u) {
      const int row = e.r0 + quad * 32 + lane, jl = (u % a.nrt) * BT + half * (BT / 2) + lane;
      const bool live = row < e.nrows;
      oidx = live ? a.rowidx[(size_t)e.blk * a.lrow + row] : -1;
      er = live ? (int)a.rexp[(size_t)e.blk * a.lrow + row] : 0;
      ejl = lane < BT / 2 && jl < a.b ? a.ej[(size_t)e.blk * a.b + jl] : 0;
    };
    FxUnit nx = unit(blockIdx.x);
    pdl_wait();
    row_of(nx, blockIdx.x);
    for (int u = blockIdx.x; u < total && ok; u += gridDim.x) {
      const FxUnit e = nx;
      nx = unit(u + gridDim.x);
      const int j0 = (u % a.nrt) * BT;
      const int nk = KPC * ((e.ncols + KC - 1) / KC);
      using Acc = typename std::conditional<W, Acc96, long long>::type;
      Acc acc[BT];
#pragma unroll
      for (int c = 0; c < BT; ++c) acc[c] = Acc{};
      for (int k = 0; k < nk; k += G, ++g) {
        const uint32_t buf = g & 1;
        if (!__all_sync(0xffffffffu, mbar_wait(&acc_full[buf], (g >> 1) & 1) ? 1 : 0)) {
          ok = false;
          break;
        }
        fence_after();
        if (e.r0 + quad * 32 < e.nrows) {
          const uint32_t t0 = tmem + ((uint32_t)(quad * 32) << 16) + buf * kBufCols + (uint32_t)(half * BT);
#pragma unroll
          for (int c = 0; c < BT; c += 4) {
            float v[S][4];
#pragma unroll
            for (int o = 0; o < S; ++o) tmem_ld4(t0 + (uint32_t)(o * NS + c), v[o]);
            tmem_ld_wait();
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const long long h = (long long)__float2int_rn(v[0][q]) * 16777216 + (long long)__float2int_rn(v[1][q]) * 65536 +
                                  ((long long)__float2int_rn(v[2][q]) * 256 + __float2int_rn(v[3][q]));
              if constexpr (W) {
                const long long l = (long long)__float2int_rn(v[4][q]) * 16777216 + (long long)__float2int_rn(v[5][q]) * 65536 +
                                    ((long long)__float2int_rn(v[6][q]) * 256 + __float2int_rn(v[7][q]));
                const unsigned long long t = (unsigned long long)acc[c + q].lo + (uint32_t)l;
                acc[c + q].lo = (uint32_t)t;
                acc[c + q].hi += h + (l >> 32) + (long long)(t >> 32);
              } else {
                acc[c + q] += h;
              }
            }
          }
        }
        fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[buf]);
      }
      if (!ok) break;
      const int oidx_u = oidx, er_u = er, ejl_u = ejl;
      if (u + (int)gridDim.x < total) row_of(nx, u + gridDim.x);  // the next unit's, during this one's stores
      if (e.r0 + quad * 32 < e.nrows) {
        V* yr = (V*)a.y + (long long)(oidx_u < 0 ? 0 : oidx_u) * a.yrs;
        // FP32 pairs of right-hand sides as one 16-byte store where the rows allow it
        const bool pairs = !W && a.ycs == 1 && (a.yrs & 1) == 0 && ((uintptr_t)a.y & 15) == 0;
#pragma unroll
        for (int c = 0; c < BT; c += 4) {
          const int e0 = er_u + __shfl_sync(0xffffffffu, ejl_u, c / 2), e1 = er_u + __shfl_sync(0xffffffffu, ejl_u, c / 2 + 1);
          const int j = j0 + half * (BT / 2) + c / 2;
          const bool on0 = oidx_u >= 0 && j < a.b, on1 = oidx_u >= 0 && j + 1 < a.b;
          if constexpr (W) {
            if (on0) yr[(long long)j * a.ycs] = make_double2(to_double(acc[c], e0 - 68), to_double(acc[c + 1], e0 - 68));
            if (on1) yr[(long long)(j + 1) * a.ycs] = make_double2(to_double(acc[c + 2], e1 - 68), to_double(acc[c + 3], e1 - 68));
          } else {
            const float4 v = make_float4(to_float(acc[c], e0 - 36), to_float(acc[c + 1], e0 - 36), to_float(acc[c + 2], e1 - 36),
                                         to_float(acc[c + 3], e1 - 36));
            if (pairs && on1) {
              *reinterpret_cast<float4*>(yr + j) = v;
            } else {
              if (on0) yr[(long long)j * a.ycs] = make_float2(v.x, v.y);
              if (on1) yr[(long long)(j + 1) * a.ycs] = make_float2(v.z, v.w);
            }
          }
        }
      }
      // columns for plain arithmetic (what was stored above is replaced)
      if (__any_sync(0xffffffffu, ejl_u == kPlain)) {
        const int rt = u % a.nrt, wt = min(BT, a.b - rt * BT);
        const uint8_t* X = a.X + ((long long)rt * BT * a.xcols + (long long)(W ? e.x64 : e.x32) * wt) * sizeof(V);
        for (int q = 0; q < BT / 2; ++q) {
          if (__shfl_sync(0xffffffffu, ejl_u, q) == kPlain && oidx_u >= 0) {
            const int jt = half * (BT / 2) + q;
            ((V*)a.y)[(long long)oidx_u * a.yrs + (long long)(j0 + jt) * a.ycs] =
                plain<V, ADJ>((const V*)a.M + (size_t)e.blk * a.R * a.C, a.C, a.colidx + (size_t)e.blk * a.lcol, e.ncols,
                              e.r0 + quad * 32 + lane, X, wt, jt);
          }
        }
      }
    }
  } else if (warp < kDrainWarps + kSlots * kGroupWarps) {
    regs_dec<kSliceRegs>();
    // ---- chunk -> digit tiles -----------------------------------------------------------------
    const int slot = (warp - kDrainWarps) / kGroupWarps;
    const int r = tid & 127;      // row of the tile, and item of the vector
    uint32_t ks = 0;              // K steps before the unit
    uint32_t s = slot / KPC, par = 1;  // the group's raw slot; phase of its digit slot
    const uint32_t d0 = base + (uint32_t)(r * 128);
    FxUnit nx = unit(blockIdx.x);
    for (int u = blockIdx.x; u < total && ok; u += gridDim.x) {
      const FxUnit e = nx;
      nx = unit(u + gridDim.x);
      const int wt = min(BT, a.b - (u % a.nrt) * BT);
      const int nk = KPC * ((e.ncols + KC - 1) / KC);
      const int rp = min(128, (e.nrows - e.r0 + 31) & ~31);  // stored rows of the tile
      const bool live = r < rp;                              // uniform in the warp
      // the group's K steps of the unit: those with (ks + k) mod 4 == slot
      for (int k = (int)((slot - ks) & (kSlots - 1)); k < nk; k += kSlots) {
        while (s >= nraw) s -= nraw;
        // the group's last chunk on this barrier was 8 back, so its phase is at most one ahead
        const uint32_t c = (ks + (uint32_t)k) / KPC;  // chunk
        ok = __all_sync(0xffffffffu, mbar_wait(&raw_full[c % kMaxRaw], (c / kMaxRaw) & 1) && mbar_wait(&dig_empty[slot], par) ? 1 : 0) != 0;
        if (!ok) break;
        const uint8_t* raw = gbase + OFF_RAW + s * RAW;
        const int kk = KPC == 1 ? 0 : (int)((ks + (uint32_t)k) & 1);  // K step of the chunk
        if (live) {
          const uint8_t* rr = raw + (kk * S * rp + r) * 16;
#pragma unroll
          for (int h = 0; h < 2; ++h) {  // half of the K step: the row's 16-byte column 2 slot + h, swizzled
            const uint32_t d = d0 + (uint32_t)(((2 * slot + h) ^ (r & 7)) << 4);
            uint4 w[S / 2];
#pragma unroll
            for (int p = 0; p < S / 2; ++p) w[p] = *reinterpret_cast<const uint4*>(rr + (2 * p + h) * rp * 16);
#pragma unroll
            for (int p = 0; p < S / 2; ++p) {
              st128(d + 2 * p * 16384u, half2_of<0>(w[p].x), half2_of<1>(w[p].x), half2_of<0>(w[p].y), half2_of<1>(w[p].y));
              st128(d + (2 * p + 1) * 16384u, half2_of<0>(w[p].z), half2_of<1>(w[p].z), half2_of<0>(w[p].w), half2_of<1>(w[p].w));
            }
          }
        }
        // the vector: items (digit pair and half, right-hand side) of 16 bytes
        const int j = r % BT, q = r / BT;
        if (q < S && j < wt) {
          const uint4 w = *reinterpret_cast<const uint4*>(raw + 16384 + ((kk * S + q) * wt + j) * 16);
          const int col = 2 * slot + (q & 1);
          const uint32_t d = base + OFF_B + (uint32_t)(q >> 1) * 2 * BBYTES;
          const uint32_t e0 = d + swz(2 * j, col), e1 = d + swz(2 * j + 1, col);
          // forward rows (re, -im), (im, re); adjoint (re, im), (im, -re)
          auto put = [&](uint32_t ofs, uint32_t w0, uint32_t w1) {
            const uint32_t t0 = half2_of<0>(w0), t1 = half2_of<1>(w0), t2 = half2_of<0>(w1), t3 = half2_of<1>(w1);
            constexpr uint32_t N0 = ADJ ? 0u : 0x80000000u, N1 = ADJ ? 0x80000000u : 0u;
            st128(e0 + ofs, t0 ^ N0, t1 ^ N0, t2 ^ N0, t3 ^ N0);
            st128(e1 + ofs, __byte_perm(t0, t0, 0x1032) ^ N1, __byte_perm(t1, t1, 0x1032) ^ N1,
                  __byte_perm(t2, t2, 0x1032) ^ N1, __byte_perm(t3, t3, 0x1032) ^ N1);
          };
          put(0u, w.x, w.y);
          put(BBYTES, w.z, w.w);
        }
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&raw_empty[s]);
          mbar_arrive(&dig_full[slot]);
        }
        s += kSlots / KPC;
        par ^= 1;
      }
      ks += (uint32_t)nk;
    }
  } else {
   regs_dec<kCtrlRegs>();
   if (warp == kDrainWarps + kSlots * kGroupWarps) {
    // ---- copies -------------------------------------------------------------------------------
    if (lane == 0) {
      const uint64_t pol = evict_first();
      uint32_t ic = 0, s = 0, ph = 1;
      FxUnit nx = unit(blockIdx.x);
      // the chunk to ask L2 for next: unit pu, pk chunks left of it
      int pu = blockIdx.x, pk = 0;
      uint32_t pbytes = 0;
      const uint8_t* pA = nullptr;
      auto ask = [&]() {
        if (pk == 0) {
          if (pu >= total) return;
          const FxUnit f = unit(pu);
          pu += gridDim.x;
          pk = (f.ncols + KC - 1) / KC;
          pbytes = (uint32_t)min(128, (f.nrows - f.r0 + 31) & ~31) * 128u;
          pA = a.A + (size_t)(uint32_t)(W ? f.a64 : f.a32) * 128;
        }
        prefetch_l2(pA, pbytes, pol);
        pA += pbytes;
        --pk;
      };
      if (a.nrt == 1)
        for (int q = 0; q < kAhead; ++q) ask();
      for (int u = blockIdx.x; u < total && ok; u += gridDim.x) {
        const FxUnit e = nx;
        nx = unit(u + gridDim.x);
        const int rt = u % a.nrt, wt = min(BT, a.b - rt * BT);
        const int nch = (e.ncols + KC - 1) / KC;
        const uint32_t abytes = (uint32_t)min(128, (e.nrows - e.r0 + 31) & ~31) * 128u, xbytes = (uint32_t)wt * 128u;
        const uint8_t* A = a.A + (size_t)(uint32_t)(W ? e.a64 : e.a32) * 128;
        const uint8_t* X = a.X + ((long long)rt * BT * a.xcols + (long long)(W ? e.x64 : e.x32) * wt) * sizeof(V);
        for (int k = 0; k < nch; ++k, ++ic) {
          if (ic >= nraw && !mbar_wait(&raw_empty[s], ph)) {
            ok = false;
            break;
          }
          if (a.nrt == 1) ask();
          const uint32_t dst = base + OFF_RAW + s * RAW;
          uint64_t* full = &raw_full[ic % kMaxRaw];
          expect(full, abytes + xbytes);
          if (a.nrt == 1) bulk(dst, A, abytes, full, pol);
          else bulk(dst, A, abytes, full);
          if (ic == 0) pdl_wait();  // the factor's first chunk does not wait for the vector
          bulk(dst + 16384, X, xbytes, full);
          A += abytes;
          X += xbytes;
          if (++s == nraw) {
            s = 0;
            ph ^= 1;
          }
        }
      }
      // every copy issued has landed before the CTA may leave (after a timeout as well)
      for (uint32_t i = ic > nraw ? ic - nraw : 0; i < ic; ++i)
        if (!mbar_wait(&raw_full[i % kMaxRaw], (i / kMaxRaw) & 1)) ok = false;
    }
    __syncwarp();
   } else if (warp == kDrainWarps + kSlots * kGroupWarps + 1) {
    // ---- MMAs (warp-uniform, so that descriptors stay in uniform registers) --------------------
    const bool lead = elect_one();
    uint32_t ks = 0, g = 0;
    int nx = unit(blockIdx.x).ncols;
    for (int u = blockIdx.x; u < total && ok; u += gridDim.x) {
      const int ncols = __shfl_sync(0xffffffffu, nx, 0);
      nx = unit(u + gridDim.x).ncols;
      const int nk = KPC * ((ncols + KC - 1) / KC);
      for (int k = 0; k < nk; ++k, ++ks) {
        const uint32_t buf = g & 1;
        const bool first = k % G == 0;
        const uint32_t slot = ks % kSlots;
        bool got = true;
        if (first && g >= 2) got = mbar_wait(&acc_empty[buf], ((g >> 1) - 1) & 1);
        got = got && mbar_wait(&dig_full[slot], (ks / kSlots) & 1);
        ok = __all_sync(0xffffffffu, got ? 1 : 0) != 0;
        if (!ok) break;
        fence_after();
        const uint64_t dA = sdesc(base + 32u * slot), dB = sdesc(base + OFF_B + 32u * slot);
        const uint32_t d = tmem + buf * kBufCols;
        if (lead) {
#pragma unroll
          for (int i = 0; i < S; ++i)
            mma<true>(d + i * NS, dA + i * (16384u >> 4), dB, idesc(0u, 128, (S - i) * NS), (first && i == 0) ? 0u : 1u);
          mma_commit(&dig_empty[slot]);
          if (k % G == G - 1 || k == nk - 1) mma_commit(&acc_full[buf]);
        }
        __syncwarp();
        if (k % G == G - 1 || k == nk - 1) ++g;
      }
    }
    // every MMA issued is finished before the tiles and tensor memory are released
    if (lead) mma_commit(&s_done);
    __syncwarp();
    if (!mbar_wait(&s_done, 0)) ok = false;
   }
  }

  if (!ok) atomicExch(a.timeout, 1);
  fence_before();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// ---- upload --------------------------------------------------------------------------------------
// Scale exponents of a stage per direction: ef, er (forward: columns C a block, rows R), af, ar (adjoint:
// columns R a block, rows C).  A column's is half way between its largest entry and its largest entry under
// the rows' own scales, both below the block's (for a Hermitian positive definite block the square root of
// the diagonal: in either extreme alone one of a real operator's HIF stages loses bits, see above); a row's is
// its largest entry under the columns' scales.  A largest entry or a scale outside 2^-60 .. 2^60, an
// infinity or NaN marks the stage in bad[0] (its factor then keeps the CUDA-core kernels).
__global__ void k_fx_exps(const double2* M, const int* in, const int* out, const int2* dims, int R, int C, short* ef,
                          short* er, short* af, short* ar, int* bad) {
  const int blk = blockIdx.x;
  const double2* Mb = M + (size_t)blk * R * C;
  const int2 d = dims[blk];
  const int* bi = in + (size_t)blk * C;
  const int* bo = out + (size_t)blk * R;
  ef += (size_t)blk * C;
  er += (size_t)blk * R;
  af += (size_t)blk * R;
  ar += (size_t)blk * C;
  constexpr int kNone = -32768;  // no entry but zeros
  __shared__ int s_top[4];       // largest of er, ef, af, ar after the first two passes
  if (threadIdx.x < 4) s_top[threadIdx.x] = kNone;
  __syncthreads();
  auto expo = [&](int r, int c) {
    const int be = bo[r] >= 0 && bi[c] >= 0 ? fx::biased(Mb[(size_t)r * C + c]) : -1;
    return be < 0 ? kNone : be - 1022;
  };
  // rowto[r], colto[c]: the largest of a row and of a column, under colby resp. rowby (or as they are)
  auto maxima = [&](const short* colby, short* rowto, const short* rowby, short* colto, int* top) {
    auto put = [&](short* dst, int m, int* t) {
      if (m != kNone && (m < (top && colby ? -120 : -60) || m > 60)) atomicExch(bad, 1);
      if (t) atomicMax(t, m);
      *dst = (short)(m == kNone ? kNone : min(max(m, -120), 60));
    };
    for (int r = threadIdx.x >> 5; r < d.x; r += blockDim.x >> 5) {  // a warp each
      int m = kNone;
      for (int c = threadIdx.x & 31; c < d.y; c += 32) {
        const int e = expo(r, c);
        if (e != kNone) m = max(m, colby ? e - colby[c] : e);
      }
      for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
      if ((threadIdx.x & 31) == 0) put(rowto + r, m, top ? top : nullptr);
    }
    for (int c = threadIdx.x; c < d.y; c += blockDim.x) {  // a thread each
      int m = kNone;
      for (int r = 0; r < d.x; ++r) {
        const int e = expo(r, c);
        if (e != kNone) m = max(m, rowby ? e - rowby[r] : e);
      }
      put(colto + c, m, top ? top + 1 : nullptr);
    }
    __syncthreads();
  };
  maxima(nullptr, er, nullptr, ef, s_top);
  maxima(ef, af, er, ar, s_top + 2);
  auto half = [&](short* own, short other, int t0, int t1) {
    const int m = *own == kNone ? 0 : (*own - t0 + other - t1) >> 1;
    if (m < -60) atomicExch(bad, 1);
    *own = (short)max(m, -60);
  };
  for (int r = threadIdx.x; r < d.x; r += blockDim.x) half(af + r, er[r], s_top[2], s_top[0]);
  for (int c = threadIdx.x; c < d.y; c += blockDim.x) half(ef + c, ar[c], s_top[1], s_top[3]);
  __syncthreads();
  maxima(ef, er, af, ar, nullptr);
  for (int r = threadIdx.x; r < d.x; r += blockDim.x)
    if (er[r] == kNone) er[r] = 0;
  for (int c = threadIdx.x; c < d.y; c += blockDim.x)
    if (ar[c] == kNone) ar[c] = 0;
}

// Gather list of a stage for one direction (FxArgs::list): a CTA a block
static __global__ void k_fx_list(const int* colidx, const short* cexp, const int2* dims, bool adj, int lcol, int llist, int2* list) {
  const int blk = blockIdx.x, ncols = adj ? dims[blk].x : dims[blk].y;
  for (int c = threadIdx.x; c < llist; c += blockDim.x)
    list[(size_t)blk * llist + c] = c < ncols ? make_int2(colidx[(size_t)blk * lcol + c], cexp[(size_t)blk * lcol + c]) : make_int2(-1, 0);
}

// Digit copy of a factor for one direction: a CTA per unit, a thread per (row, half K step).
// Rows and columns outside the block, or that are not read or written, are zero.
template <typename R, bool ADJ>
__global__ void __launch_bounds__(256) k_fx_pack(const FxUnit* units, const typename fx::Cfg<R>::V* M, const int* rowidx,
                                                 const int* colidx, const short* rexp, const short* cexp, int Rr, int Cc,
                                                 uint8_t* A) {
  using namespace fx;
  using C = Cfg<R>;
  using V = typename C::V;
  using F = typename C::F;
  constexpr bool W = std::is_same<R, double>::value;
  const FxUnit e = units[blockIdx.x];
  const int lrow = ADJ ? Cc : Rr, lcol = ADJ ? Rr : Cc;
  const int rp = min(128, (e.nrows - e.r0 + 31) & ~31);
  const int nh = 2 * C::KPC * ((e.ncols + 8 * C::KPC - 1) / (8 * C::KPC));  // half K steps
  const V* Mb = M + (size_t)e.blk * Rr * Cc;
  uint4* out = reinterpret_cast<uint4*>(A + (size_t)(uint32_t)(W ? e.a64 : e.a32) * 128);
  for (int t = threadIdx.x; t < rp * nh; t += 256) {
    const int q = t / rp, rl = t - q * rp, r = e.r0 + rl;
    const bool row = r < e.nrows && rowidx[(size_t)e.blk * lrow + r] >= 0;
    const int E = r < e.nrows ? (int)rexp[(size_t)e.blk * lrow + r] : 0;
    F re[4], im[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int c = 4 * q + i;
      re[i] = im[i] = fix_zero<F>();
      if (row && c < e.ncols && colidx[(size_t)e.blk * lcol + c] >= 0) {
        const V v = ADJ ? Mb[(size_t)c * Cc + r] : Mb[(size_t)r * Cc + c];
        const int Ec = cexp[(size_t)e.blk * lcol + c];
        re[i] = fix(v.x, E + Ec);
        im[i] = fix(v.y, E + Ec);
      }
    }
    uint4* o = out + ((size_t)(q >> 1) * C::S + (q & 1)) * rp + rl;
    o[0] = digit_pair<0>(re, im);
    o[2 * rp] = digit_pair<1>(re, im);
    if constexpr (W) {
      o[4 * rp] = digit_pair<2>(re, im);
      o[6 * rp] = digit_pair<3>(re, im);
    }
  }
}

}  // namespace fio
