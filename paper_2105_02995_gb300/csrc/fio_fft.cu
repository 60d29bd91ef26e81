// fio_fft.cu -- the DFT F of the paper's problem statement (section 1) and its inverse, on the
// device: u = K F f, so the full solve is f = F^{-1} (K^{-1} u), and F is the step after the
// approximate inverse.
//
//   F      f-hat(xi) = n^{-d} sum_x exp(-2 pi i x.xi) f(x)       (section 1, the DFT of f)
//   F^{-1} f(x)      =         sum_xi exp(+2 pi i x.xi) f-hat(xi)
// on the grids x = k/n, xi = j - n/2 per dimension (2D index i1 + n*i2).  With xi = j - n/2,
// exp(-+2 pi i x.xi) = (-1)^(k_1+..+k_d) exp(-+2 pi i k.j/n): F is the standard DFT of the
// sign-modulated input scaled by n^{-d}, F^{-1} the sign-modulated standard inverse DFT.
//
// Kernel: k_fft_pass, a batch of power-of-two transforms of length L <= 2048, 2048 / L transforms per
// CTA of 256 threads (one right-hand side per grid row).  Element e of transform t is read at
// t*xt + e*xe and written at t*yt + e*ye of the right-hand side's vector, so one kernel serves the
// contiguous and the strided axes; the threads walk whichever index is contiguous in memory.
// Stockham's autosort form with eight values per thread in registers: one stage of radix 2 or 4
// when log2 L is not a multiple of three, then stages of radix 8; the first stage reads and the last
// one writes global memory, between them the values go through shared memory (L = 256: two
// exchanges; a radix-2 form in shared memory needs a barrier and a round trip for each of its eight
// stages, and took 74 us for the two passes of 32 transforms of 256 x 256 in FP32 against 29 us: now bound
// by the latency of its loads and exchanges, at 2.3 TB/s through L2).
// Twiddles exp(2 pi i k / 2048) come from a table made at upload.
// Optional per-element factors: the (-1)^k sign modulation on the input (F) or on the output
// (F^{-1}), the four-step twiddle exp(s 2 pi i t e / N) on the output, and a scale.
// Plans: 2D n x n = transforms along i1, then along i2; 1D N <= 2048 = one pass; 1D N > 2048 =
// four-step (N = N1 N2, N1 <= N2): length-N2 transforms over j2 with the twiddle, then length-N1
// transforms over j1 written to k2 + N2 k1.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "fio.h"
#include "fio_internal.h"

namespace {

constexpr int kFftElems = 2048;  // complex elements per CTA
constexpr int kFftThreads = 256;

struct FftPass {
  const void* x;
  void* y;
  long long ldx, ldy;  // per right-hand side
  int L, logL;         // transform length and log2
  int T;               // transforms per right-hand side
  long long xt, xe;    // input offset of element e of transform t: t*xt + e*xe
  long long yt, ye;    // output offset
  const void* tw;      // exp(2 pi i k / 2048), k < 2048, in the vectors' precision
  int twN;             // > 0: multiply output (t, e) by exp(sign 2 pi i (t e mod twN) / twN)
  int mod_in, mod_out; // (-1)^(grid coordinate sum) of the input / output linear index
  int n, logn, d;      // grid (for the modulation)
  double scale;        // output scale
};

template <typename R> struct Cplx;
template <> struct Cplx<float> {
  using T = float2;
  static __device__ __forceinline__ T make(float a, float b) { return make_float2(a, b); }
  static __device__ __forceinline__ void sincospi_(float a, float* s, float* c) { sincospif(a, s, c); }
};
template <> struct Cplx<double> {
  using T = double2;
  static __device__ __forceinline__ T make(double a, double b) { return make_double2(a, b); }
  static __device__ __forceinline__ void sincospi_(double a, double* s, double* c) { sincospi(a, s, c); }
};

// (offsets within one right-hand side's vector fit an int: N <= 2^22)
__device__ __forceinline__ bool odd_coord_sum(int k, const FftPass& p) {
  return ((p.d == 1 ? k : k ^ (k >> p.logn)) & 1) != 0;
}

template <typename V> __device__ __forceinline__ V cadd(V a, V b) { a.x += b.x; a.y += b.y; return a; }
template <typename V> __device__ __forceinline__ V csub(V a, V b) { a.x -= b.x; a.y -= b.y; return a; }
template <typename V> __device__ __forceinline__ V cmul(V a, V b) {
  V r;
  r.x = a.x * b.x - a.y * b.y;
  r.y = a.x * b.y + a.y * b.x;
  return r;
}
// a times exp(SIGN pi i / 2)
template <int SIGN, typename V> __device__ __forceinline__ V times_i(V a) {
  V r;
  r.x = SIGN > 0 ? -a.y : a.y;
  r.y = SIGN > 0 ? a.x : -a.x;
  return r;
}
template <int SIGN, typename V> __device__ __forceinline__ void dft2(V& a, V& b) {
  const V t = b;
  b = csub(a, t);
  a = cadd(a, t);
}
// in place, results in natural order
template <int SIGN, typename V> __device__ __forceinline__ void dft4(V& a, V& b, V& c, V& d) {
  const V s0 = cadd(a, c), s1 = csub(a, c), s2 = cadd(b, d), s3 = times_i<SIGN>(csub(b, d));
  a = cadd(s0, s2);
  b = cadd(s1, s3);
  c = csub(s0, s2);
  d = csub(s1, s3);
}
template <int SIGN, typename V> __device__ __forceinline__ void dft8(V (&v)[8]) {
  V e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6], o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
  dft4<SIGN>(e0, e1, e2, e3);
  dft4<SIGN>(o0, o1, o2, o3);
  // o1 exp(SIGN pi i / 4), o2 exp(SIGN pi i / 2), o3 exp(SIGN 3 pi i / 4)
  using S = decltype(o1.x);
  const S h = (S)0.70710678118654752440;
  const V q1 = times_i<SIGN>(o1), q3 = times_i<SIGN>(o3);
  V w1 = cadd(o1, q1), w3 = csub(q3, o3);
  w1.x *= h;
  w1.y *= h;
  w3.x *= h;
  w3.y *= h;
  const V w2 = times_i<SIGN>(o2);
  v[0] = cadd(e0, o0);
  v[4] = csub(e0, o0);
  v[1] = cadd(e1, w1);
  v[5] = csub(e1, w1);
  v[2] = cadd(e2, w2);
  v[6] = csub(e2, w2);
  v[3] = cadd(e3, w3);
  v[7] = csub(e3, w3);
}

// where element e of transform tl lies in shared memory: strides of 8 elements, and neighbouring
// transforms of the strided axes, are spread over the banks
constexpr int kFftPad = 2;
constexpr int kFftShared = kFftElems + kFftElems / 16 + kFftPad * (kFftElems / 16);
__device__ __forceinline__ int place(int tl, int e, int L) {
  return tl * (L + (L >> 4) + (L >= 16 ? kFftPad : 0)) + e + (e >> 4);
}

// The stage of radix RX after stages of product Ns, for this thread's 8 / RX butterflies: butterfly
// (transform tl, index j < L / RX) takes elements j + r L / RX, turned by exp(2 pi i r (j mod Ns) / (Ns RX)),
// and leaves element (j / Ns) Ns RX + j mod Ns + r Ns.
template <typename R, int SIGN, int RX>
__device__ __forceinline__ void fft_stage(const FftPass& p, typename Cplx<R>::T* s, const typename Cplx<R>::T* x,
                                          typename Cplx<R>::T* y, int t0, int Ns, bool e_fast, bool oe_fast) {
  using C = Cplx<R>;
  using V = typename C::T;
  constexpr int NB = 8 / RX, LOGRX = RX == 8 ? 3 : RX == 4 ? 2 : 1;
  const int L = p.L, logLR = p.logL - LOGRX, logTT = 11 - p.logL, logNs = __ffs(Ns) - 1;  // all powers of two
  const bool first = Ns == 1, last = Ns * RX == L;
  const V* tw = reinterpret_cast<const V*>(p.tw);
  const int xt = (int)p.xt, xe = (int)p.xe, yt = (int)p.yt, ye = (int)p.ye;
  V v[NB][RX];
  int tl[NB], j[NB];
  // which of (transform, index) runs along the threads: as global memory wants it at the two ends
  const bool fast = last ? oe_fast : e_fast;
#pragma unroll
  for (int k = 0; k < NB; ++k) {
    const int i = threadIdx.x + kFftThreads * k;
    tl[k] = fast ? i >> logLR : i & ((1 << logTT) - 1);
    j[k] = fast ? i & ((1 << logLR) - 1) : i >> logTT;
    if (first) {
      const int at = (t0 + tl[k]) * xt + j[k] * xe, step = xe << logLR;
      const bool on = t0 + tl[k] < p.T;
#pragma unroll
      for (int r = 0; r < RX; ++r) v[k][r] = on ? x[at + r * step] : C::make(0, 0);
      if (p.mod_in) {
#pragma unroll
        for (int r = 0; r < RX; ++r)
          if (odd_coord_sum(at + r * step, p)) v[k][r] = C::make(-v[k][r].x, -v[k][r].y);
      }
    } else {
#pragma unroll
      for (int r = 0; r < RX; ++r) v[k][r] = s[place(tl[k], j[k] + (r << logLR), L)];
    }
    if (!first) {
      const int q = (j[k] & (Ns - 1)) << (11 - logNs - LOGRX);
#pragma unroll
      for (int r = 1; r < RX; ++r) {
        V w = tw[r * q];
        if (SIGN < 0) w.y = -w.y;
        v[k][r] = cmul(v[k][r], w);
      }
    }
    if constexpr (RX == 2) dft2<SIGN>(v[k][0], v[k][1]);
    if constexpr (RX == 4) dft4<SIGN>(v[k][0], v[k][1], v[k][2], v[k][3]);
    if constexpr (RX == 8) dft8<SIGN>(v[k]);
  }
  if (!first) __syncthreads();  // every value is read before any is replaced
#pragma unroll
  for (int k = 0; k < NB; ++k) {
    const int e0 = ((j[k] >> logNs) << (logNs + LOGRX)) + (j[k] & (Ns - 1));
    if (!last) {
#pragma unroll
      for (int r = 0; r < RX; ++r) s[place(tl[k], e0 + (r << logNs), L)] = v[k][r];
      continue;
    }
    const int t = t0 + tl[k];
    if (t >= p.T) continue;
    const int at = t * yt + e0 * ye, step = ye << logNs;
#pragma unroll
    for (int r = 0; r < RX; ++r) {
      V u = v[k][r];
      if (p.twN > 0) {
        const int q = (t * (e0 + (r << logNs))) & (p.twN - 1);  // t e < N <= 2^22
        R sn, cs;
        C::sincospi_((R)(2 * q) / (R)p.twN, &sn, &cs);
        u = cmul(u, C::make(cs, SIGN > 0 ? sn : -sn));
      }
      R sc = (R)p.scale;
      if (p.mod_out && odd_coord_sum(at + r * step, p)) sc = -sc;
      y[at + r * step] = C::make(sc * u.x, sc * u.y);
    }
  }
  if (!last) __syncthreads();
}

template <typename R, int SIGN>
__global__ void __launch_bounds__(kFftThreads) k_fft_pass(FftPass p) {
  using V = typename Cplx<R>::T;
  __shared__ V s[kFftShared];
  fio::pdl_go();
  fio::pdl_wait();
  const int t0 = blockIdx.x * (kFftElems / p.L);
  const V* x = reinterpret_cast<const V*>(p.x) + (long long)blockIdx.y * p.ldx;
  V* y = reinterpret_cast<V*>(p.y) + (long long)blockIdx.y * p.ldy;
  const bool e_fast = p.xe == 1 || p.xt != 1, oe_fast = p.ye == 1 || p.yt != 1;
  int Ns = 1;
  const int rem = p.logL % 3;
  if (rem == 1) {
    fft_stage<R, SIGN, 2>(p, s, x, y, t0, Ns, e_fast, oe_fast);
    Ns = 2;
  } else if (rem == 2) {
    fft_stage<R, SIGN, 4>(p, s, x, y, t0, Ns, e_fast, oe_fast);
    Ns = 4;
  }
  for (; Ns < p.L; Ns *= 8) fft_stage<R, SIGN, 8>(p, s, x, y, t0, Ns, e_fast, oe_fast);
}

// exp(2 pi i k / 2048) in both precisions, the FP32 one rounded from FP64
__global__ void k_fft_twiddles(double2* t64, float2* t32) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= kFftElems) return;
  double sn, cs;
  sincospi(2.0 * k / kFftElems, &sn, &cs);
  t64[k] = make_double2(cs, sn);
  t32[k] = make_float2((float)cs, (float)sn);
}

int ilog2(long long v) {
  int l = 0;
  while ((1LL << l) < v) ++l;
  return l;
}

template <typename R>
int run_pass(const FftPass& p, bool inverse, int b, cudaStream_t s) {
  const int TT = kFftElems / p.L;
  dim3 grid((unsigned)((p.T + TT - 1) / TT), (unsigned)b);
  if (inverse) pdl_launch(true, k_fft_pass<R, 1>, grid, kFftThreads, 0, s, p);
  else pdl_launch(true, k_fft_pass<R, -1>, grid, kFftThreads, 0, s, p);
  return FIO_OK;
}

// y = F x (inverse = false) or F^{-1} x (inverse = true); tmp: N x b scratch (ld N)
template <typename R>
int apply_dft(fio_op op, bool inverse, const void* x, void* y, long long ld, int b, void* tmp, cudaStream_t s) {
  const int n = (int)op->n, d = op->d;
  const long long N = op->N;
  FftPass p{};
  p.tw = sizeof(R) == 8 ? op->fft_tw : (const void*)((const double2*)op->fft_tw + kFftElems);
  p.n = n;
  p.logn = ilog2(n);
  p.d = d;
  const double scale_last = inverse ? 1.0 : 1.0 / (double)N;
  int rc;
  if (d == 2 || N > kFftElems) {
    // two passes: (2D) along i1 then along i2; (1D four-step) over j2 with twiddle, then over j1
    const int L1 = d == 2 ? n : (int)(1LL << (ilog2(N) / 2)), L2 = (int)(N / L1);
    FftPass a = p, c = p;
    a.x = x;
    a.y = tmp;
    a.ldx = ld;
    a.ldy = N;
    a.mod_in = inverse ? 0 : 1;
    a.scale = 1.0;
    c.x = tmp;
    c.y = y;
    c.ldx = N;
    c.ldy = ld;
    c.mod_out = inverse ? 1 : 0;
    c.scale = scale_last;
    if (d == 2) {
      a.L = n, a.T = n, a.xt = n, a.xe = 1, a.yt = n, a.ye = 1;   // along i1 for each i2
      c.L = n, c.T = n, c.xt = 1, c.xe = n, c.yt = 1, c.ye = n;   // along i2 for each i1
    } else {
      a.L = L2, a.T = L1, a.xt = 1, a.xe = L1, a.yt = 1, a.ye = L1, a.twN = (int)N;  // j1 + L1 j2 -> j1 + L1 k2
      c.L = L1, c.T = L2, c.xt = L1, c.xe = 1, c.yt = 1, c.ye = L2;                  // -> k2 + L2 k1
    }
    a.logL = ilog2(a.L);
    c.logL = ilog2(c.L);
    if ((rc = run_pass<R>(a, inverse, b, s))) return rc;
    if ((rc = run_pass<R>(c, inverse, b, s))) return rc;
  } else {
    p.x = x;
    p.y = y;
    p.ldx = ld;
    p.ldy = ld;
    p.L = (int)N;
    p.logL = ilog2(N);
    p.T = 1;
    p.xt = p.yt = 0;
    p.xe = p.ye = 1;
    p.mod_in = inverse ? 0 : 1;
    p.mod_out = inverse ? 1 : 0;
    p.scale = scale_last;
    if ((rc = run_pass<R>(p, inverse, b, s))) return rc;
  }
  return cudaGetLastError() == cudaSuccess ? FIO_OK : FIO_ECUDA;
}

int dft_entry(fio_op op, bool inverse, const void* x, void* y, int64_t ld, int b, int dtype, int precision,
              void* stream) {
  if (!op || b < 0 || b > 65535 || ld < (op ? op->N : 0)) return FIO_EINVAL;  // b: grid rows
  if (!((dtype == FIO_C128 && precision == FIO_P64) || (dtype == FIO_C64 && precision == FIO_P32)))
    return FIO_EINVAL;
  if (b > 0 && (!x || !y || x == y)) return FIO_EINVAL;
  const long long n = op->n;
  if (n < 2 || (n & (n - 1)) != 0 || op->N > (long long)kFftElems * kFftElems) return FIO_ENOTSUP;
  const size_t es = dtype == FIO_C128 ? 16 : 8;
  const size_t span = ((size_t)ld * (b > 0 ? b - 1 : 0) + op->N) * es;
  const uint8_t *xb = (const uint8_t*)x, *yb = (const uint8_t*)y;
  if (b > 0 && xb < yb + span && yb < xb + span) return FIO_EINVAL;  // overlap
  if (b == 0) return FIO_OK;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaGetLastError() != cudaSuccess) return FIO_ECUDA;
  void* bufs[5];
  int rc = fio_scratch(op, b, es, s, bufs);
  if (rc) return rc;
  return dtype == FIO_C128 ? apply_dft<double>(op, inverse, x, y, ld, b, bufs[4], s)
                           : apply_dft<float>(op, inverse, x, y, ld, b, bufs[4], s);
}

}  // namespace

int fft_build(fio_op op, cudaStream_t s) {
  const size_t bytes = kFftElems * (sizeof(double2) + sizeof(float2));
  if (cudaMalloc(&op->fft_tw, bytes) != cudaSuccess) {
    cudaGetLastError();
    op->fft_tw = nullptr;
    return FIO_ENOMEM;
  }
  op->fft_bytes = bytes;
  k_fft_twiddles<<<kFftElems / 256, 256, 0, s>>>((double2*)op->fft_tw, (float2*)((double2*)op->fft_tw + kFftElems));
  return FIO_OK;
}

extern "C" int fio_apply_F(fio_op op, const void* f, void* fhat, int64_t ld, int b, int dtype, int precision,
                           void* stream) {
  return dft_entry(op, false, f, fhat, ld, b, dtype, precision, stream);
}

extern "C" int fio_apply_Finv(fio_op op, const void* fhat, void* f, int64_t ld, int b, int dtype, int precision,
                              void* stream) {
  return dft_entry(op, true, fhat, f, ld, b, dtype, precision, stream);
}
