// fio_fx.cu -- host side of the fixed-point tensor-core stage kernel (fio_fx.cuh): which stages it
// takes, their digit copies and work units at upload, and its launches.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>
#include <vector>

#include "fio.h"
#include "fio_fx.cuh"
#include "fio_internal.h"

using namespace fio;

namespace {

// Stages the kernel may take.  In FP64: all of an operator above kSmallOp unknowns; in smaller ones,
// above kTinyOp, those with at least kMinUnits 128-row tiles or blocks of at most one 64-row tile (a
// CUDA-core FP64 tile of a 28-row block takes 22 us at b = 8 and 55 at b = 32 whatever the number of
// blocks; this kernel 8 to 12): the rest keeps the CUDA-core sums, which every tile shape reproduces bit
// for bit.  In FP32: with kMinUnits tiles, blocks of more than kSmallDim rows or columns.
constexpr int64_t kSmallOp = 4096, kTinyOp = 1024;
constexpr int kMinUnits = 96;
constexpr int kSmallDim = 32;

inline size_t al256(size_t v) { return (v + 255) & ~(size_t)255; }
inline int list_stride(int lcol) { return (lcol + 15) & ~15; }  // whole FP32 chunks, 16-byte aligned

template <typename R, bool ADJ>
void pack(const Stage& st, const FxUnit* units, uint8_t* A, cudaStream_t s) {
  using V = typename fx::Cfg<R>::V;
  const V* M = (const V*)(std::is_same<R, double>::value ? (const void*)st.M64 : (const void*)st.M32);
  k_fx_pack<R, ADJ><<<st.n_fx_units[ADJ], 256, 0, s>>>(units, M, ADJ ? st.in : st.out, ADJ ? st.out : st.in, st.fx_exp[ADJ], st.fx_cexp[ADJ],
                                                       (int)st.R, (int)st.C, A);
}

// dynamic shared memory opt-in, once per device and kernel
bool opt_in(const void* f, int bytes) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, int> granted;
  std::lock_guard<std::mutex> lock(mu);
  int& cap = granted[std::make_pair(dev, f)];
  if (bytes <= cap) return true;
  if (cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cap = bytes;
  return true;
}

int sm_count() {
  thread_local int last = -1, n = 1;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  if (dev != last && (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)) n = 1;
  last = dev;
  return n;
}

template <typename R, bool ADJ, int BT>
bool launch(FxArgs a, uint8_t* X, int* ej, cudaStream_t s) {
  a.nrt = (a.b + BT - 1) / BT;
  constexpr int fixed = fx::smem_fixed<R, BT>(), raw = fx::raw_bytes<BT>();
  a.nraw = std::min(fx::kMaxRaw, (227 * 1024 - 512 - fixed) / raw);  // 512: the static barriers
  const int need = fixed + a.nraw * raw;
  const long long total = (long long)a.nunits * a.nrt;
  if (total > 0x7fffffffLL || a.nrt > 65535) return false;
  if (!opt_in((const void*)k_stage_fx<R, ADJ, BT>, need)) return false;
  // the gather is started early behind short stages only: behind a long one its CTAs crowd the
  // multiprocessors that finish first (2D n = 256 FP64 b = 1, 440 K steps an SM: 2.04 ms without, 2.10 with;
  // 1D N = 16384 b = 5, 15 K steps: 414 us without, 360 with)
  const bool early = (long long)a.steps * a.nrt <= 300LL * sm_count();
  const int groups = (a.maxcols + 4 * (256 / BT) - 1) / (4 * (256 / BT));
  // (four groups kept take 126 registers: where the CTAs are more than two a multiprocessor, the loop of 54
  // is no slower; 2D n = 256 FP64 b = 1, K-dot 2031 us with four, 2023 without)
  auto gather = groups <= 1   ? k_fx_gather<R, ADJ, BT, 1>
                : groups <= 2 ? k_fx_gather<R, ADJ, BT, 2>
                : groups <= 4 && (long long)a.nblk * a.nrt <= 2LL * sm_count() ? k_fx_gather<R, ADJ, BT, 4>
                              : k_fx_gather<R, ADJ, BT, 0>;
  pdl_launch(early, gather, dim3((unsigned)a.nblk, (unsigned)a.nrt), 256, 0, s, a, X, ej);
  pdl_launch(true, k_stage_fx<R, ADJ, BT>, (unsigned)std::min<long long>(total, sm_count()), fx::kThreads, need, s, a);
  return true;
}

template <typename R, bool ADJ>
bool launch_b(const FxArgs& a, uint8_t* X, int* ej, cudaStream_t s) {
  if (a.b <= 8) return launch<R, ADJ, 8>(a, X, ej, s);
  if constexpr (std::is_same<R, float>::value)
    if (a.b > 16) return launch<R, ADJ, 32>(a, X, ej, s);
  return launch<R, ADJ, 16>(a, X, ej, s);
}

}  // namespace

int fx_build(fio_op op, const std::vector<int2>& meta, const std::vector<size_t>& mdims, cudaStream_t s) {
  // (the FP32 copies serve the corrections asked for in split TF32, and variant 50 when it is pinned)
  bool want[2] = {(op->mask & FIO_MASK_P64) != 0, op->arena32 && op->arena_tc};
  if (!want[0] && !want[1]) return FIO_OK;
  struct Plan {
    int stage;
    bool want[2];
    size_t units[2], exps, xofs[2], list[2], digits[2][2];  // offsets: entries, entries, entries, entries, bytes
  };
  std::vector<Plan> plans;
  std::vector<FxUnit> units;
  std::vector<int2> xofs;
  size_t nexp = 0, nlist = 0, dbytes[2] = {0, 0};
  for (size_t si = 0; si < op->st.size(); ++si) {
    Stage& st = op->st[si];
    int2 n = make_int2(0, 0);
    bool ok = st.nblk > 0;
    for (uint32_t b = 0; ok && b < st.nblk; ++b) {
      const int2 d = meta[mdims[si] + b];
      ok = d.x > 0 && d.y > 0;
      st.nnz = (b ? st.nnz : 0) + (long long)d.x * d.y;
      n.x += (d.x + 127) / 128;
      n.y += (d.y + 127) / 128;
    }
    const bool few = std::min(n.x, n.y) < kMinUnits;
    Plan p;
    p.stage = (int)si;
    const bool narrow = std::max(st.maxcols[0], st.maxcols[1]) <= 64;
    p.want[0] = ok && want[0] && (op->N > kSmallOp || !few || (op->N > kTinyOp && narrow));
    p.want[1] = ok && want[1] && !few && std::max(st.maxcols[0], st.maxcols[1]) > kSmallDim;
    if (!p.want[0] && !p.want[1]) continue;
    p.exps = nexp;
    nexp += 2 * (size_t)st.nblk * (st.R + st.C);
    for (int dir = 0; dir < 2; ++dir) {
      p.list[dir] = nlist;
      nlist += (size_t)st.nblk * list_stride(dir ? st.R : st.C);
    }
    long long cols[2] = {0, 0};
    size_t bytes[2][2];
    const size_t u0 = units.size(), x0 = xofs.size();
    for (int dir = 0; dir < 2; ++dir) {
      p.units[dir] = units.size();
      p.xofs[dir] = xofs.size();
      long long xo[2] = {0, 0};
      for (uint32_t b = 0; b < st.nblk; ++b) {
        const int2 d = meta[mdims[si] + b];
        const int rows = dir ? d.y : d.x, c = dir ? d.x : d.y;
        for (int r0 = 0; r0 < rows; r0 += 128) units.push_back(FxUnit{(int)b, r0, rows, c, 0, 0, (int)xo[0], (int)xo[1]});
        xofs.push_back(make_int2((int)xo[0], (int)xo[1]));
        xo[0] += (c + 7) / 8 * 8;
        xo[1] += (c + 15) / 16 * 16;
      }
      for (int t = 0; t < 2; ++t) cols[t] = std::max(cols[t], xo[t]);
      st.fx_cols[dir] = make_int2((int)xo[0], (int)xo[1]);
      std::stable_sort(units.begin() + p.units[dir], units.end(), [](const FxUnit& x, const FxUnit& y) { return x.ncols > y.ncols; });
      long long at[2] = {0, 0};  // 128-byte rows of the digit copies
      for (size_t k = p.units[dir]; k < units.size(); ++k) {
        FxUnit& u = units[k];
        const int rp = std::min(128, (u.nrows - u.r0 + 31) & ~31);
        u.a64 = (int)at[0];
        u.a32 = (int)at[1];
        at[0] += (long long)rp * ((u.ncols + 7) / 8);
        at[1] += (long long)rp * ((u.ncols + 15) / 16);
      }
      ok = ok && std::max(at[0], at[1]) < 0x7fffffffLL && std::max(xo[0], xo[1]) < 0x7fffffffLL;
      for (int t = 0; t < 2; ++t) bytes[t][dir] = (size_t)at[t] * 128;
      st.n_fx_units[dir] = (int)(units.size() - p.units[dir]);
      st.fx_steps[dir] = 0;
      for (size_t k = p.units[dir]; k < units.size(); ++k) st.fx_steps[dir] += (units[k].ncols + 7) / 8;
    }
    if (!ok) {
      units.resize(u0);
      xofs.resize(x0);
      continue;
    }
    for (int t = 0; t < 2; ++t)
      for (int dir = 0; p.want[t] && dir < 2; ++dir) {
        p.digits[t][dir] = dbytes[t];
        dbytes[t] += al256(bytes[t][dir]);
      }
    for (int t = 0; t < 2; ++t)
      if (p.want[t]) op->fx_max_cols[t] = std::max(op->fx_max_cols[t], cols[t]);
    op->fx_max_blk = std::max(op->fx_max_blk, (long long)st.nblk);
    plans.push_back(p);
  }
  if (plans.empty()) return FIO_OK;
  const size_t oe = al256(units.size() * sizeof(FxUnit)), ox = oe + al256(nexp * sizeof(short)),
               ol = ox + al256(xofs.size() * sizeof(int2)), ob = ol + al256(nlist * sizeof(int2)),
               od = ob + al256(plans.size() * sizeof(int));
  // The copies take at most half of the free memory, so that scratch, solver vectors and other operators
  // find the room they had without them: both types', or FP64's alone, or none (the CUDA-core kernels serve).
  size_t room = 0, all = 0;
  if (cudaMemGetInfo(&room, &all) != cudaSuccess) room = 0;
  cudaGetLastError();
  for (const bool both : {true, false}) {
    const size_t bytes = od + dbytes[0] + (both ? dbytes[1] : 0);
    if (op->fx || bytes == od || bytes > room / 2) continue;
    if (cudaMalloc(&op->fx, bytes) != cudaSuccess) {
      cudaGetLastError();
      op->fx = nullptr;
      continue;
    }
    op->fx_bytes = bytes;
    want[1] = want[1] && both;
  }
  if (!op->fx) want[0] = want[1] = false;
  for (int t = 0; t < 2; ++t)
    if (!want[t]) op->fx_max_cols[t] = 0;
  if (!op->fx) return FIO_OK;
  for (Plan& p : plans) p.want[1] = p.want[1] && want[1];
  uint8_t *p0 = (uint8_t*)op->fx, *pd[2] = {p0 + od, p0 + od + dbytes[0]};
  int* bad = (int*)(p0 + ob);
  if (cudaMemcpyAsync(p0, units.data(), units.size() * sizeof(FxUnit), cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(p0 + ox, xofs.data(), xofs.size() * sizeof(int2), cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemsetAsync(p0 + oe, 0, ox - oe, s) != cudaSuccess || cudaMemsetAsync(bad, 0, od - ob, s) != cudaSuccess)
    return FIO_ECUDA;
  for (size_t k = 0; k < plans.size(); ++k) {
    const Plan& p = plans[k];
    Stage& st = op->st[p.stage];
    short* ef = (short*)(p0 + oe) + p.exps;
    short *er = ef + (size_t)st.nblk * st.C, *af = er + (size_t)st.nblk * st.R, *ar = af + (size_t)st.nblk * st.R;
    st.fx_cexp[0] = ef;
    st.fx_exp[0] = er;
    st.fx_cexp[1] = af;
    st.fx_exp[1] = ar;
    k_fx_exps<<<st.nblk, 512, 0, s>>>(st.M64, st.in, st.out, st.dims, (int)st.R, (int)st.C, ef, er, af, ar, bad + k);
    for (int dir = 0; dir < 2; ++dir) {
      const int lcol = (int)(dir ? st.R : st.C);
      int2* list = (int2*)(p0 + ol) + p.list[dir];
      k_fx_list<<<st.nblk, 128, 0, s>>>(dir ? st.out : st.in, st.fx_cexp[dir], st.dims, dir == 1, lcol, list_stride(lcol), list);
      st.fx_list[dir] = list;
      st.fx_units[dir] = (const FxUnit*)p0 + p.units[dir];
      st.fx_xofs[dir] = (const int2*)(p0 + ox) + p.xofs[dir];
      for (int t = 0; t < 2; ++t) st.fxA[t][dir] = p.want[t] ? pd[t] + p.digits[t][dir] : nullptr;
    }
    if (p.want[0]) {
      pack<double, false>(st, st.fx_units[0], pd[0] + p.digits[0][0], s);
      pack<double, true>(st, st.fx_units[1], pd[0] + p.digits[0][1], s);
    }
    if (p.want[1]) {
      pack<float, false>(st, st.fx_units[0], pd[1] + p.digits[1][0], s);
      pack<float, true>(st, st.fx_units[1], pd[1] + p.digits[1][1], s);
    }
  }
  std::vector<int> hbad(plans.size(), 1);
  if (cudaMemcpyAsync(hbad.data(), bad, plans.size() * sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return FIO_ECUDA;
  for (size_t k = 0; k < plans.size(); ++k)
    for (int t = 0; t < 2; ++t) op->st[plans[k].stage].fx_ok[t] = plans[k].want[t] && !hbad[k];
  return FIO_OK;
}

size_t fx_scratch_bytes(fio_op op, int b, size_t elem) {
  const int t = elem == sizeof(double2) ? 0 : 1;
  if (!op->fx || op->fx_max_cols[t] == 0) return 0;
  return al256((size_t)op->fx_max_cols[t] * (size_t)b * elem) + al256((size_t)op->fx_max_blk * (size_t)b * sizeof(int));
}

// The built-in choice.  FP64 from b = 5 on: the CUDA-core kernels need 2 to 20 times as long on every
// stage.  FP64 at b <= 4 and FP32 by estimated time, in microseconds.
//   this kernel   9 for its two launches, and the busiest SM's K steps at their measured time, or
//                 1.4 a unit (the drain of a short one)
//   FP64, b <= 4  k_stage_vec: 7, and b times the entries a CTA slot streams, at 2.2 ns (wide blocks) to
//                 4 ns (narrow ones) forward and 1.25 to 1.9 adjoint.  Measured on both sides of the line,
//                 b = 1: 141 blocks of 58 x 58 forward 28 against 16, adjoint 15 against 16; 4096 blocks
//                 of 16 x 16 adjoint 30 against 63; 72 blocks of 228 x 228 67 against 27
//   FP32          31 TFLOP/s up to 16 right-hand sides, 42 above.  Measured at b = 32: blocks of 415 x 250
//                 0.60 ms against 0.34, of 58 x 58 0.030 against 0.035.  FP32 also needs two tiles for
//                 every SM: below, the smaller CUDA-core tiles fill the chip better.
bool fx_takes(const Stage& st, bool adj, bool wide, int b) {
  if (!st.fx_ok[wide ? 0 : 1]) return false;
  if (wide && b > 4) return true;
  const int sms = sm_count(), bt = wide ? (b <= 8 ? 8 : 16) : (b <= 8 ? 8 : b <= 16 ? 16 : 32);
  const long long nrt = (b + bt - 1) / bt, units = st.n_fx_units[adj] * nrt;
  const double step = wide ? (bt == 8 ? 0.55 : 0.80) : (bt == 8 ? 0.33 : bt == 16 ? 0.37 : 0.45);
  const double a_unit = std::max(1.4, step * (double)st.fx_steps[adj] / st.n_fx_units[adj]);
  const double fx = 9.0 + a_unit * (double)((units + sms - 1) / sms);
  if (wide) {
    const bool broad = std::max(st.maxcols[0], st.maxcols[1]) >= 128;
    const double ns = adj ? (broad ? 1.25 : 1.9) : (broad ? 2.2 : 4.0);
    const int tiles = std::min(sms, std::max(1, adj ? st.ntiles_adj : st.ntiles_fwd));
    return fx < 7.0 + 1e-3 * b * ns * (double)st.nnz / tiles;
  }
  const int bp = b <= 16 ? 16 : (b + 31) / 32 * 32;
  return b > 8 && units >= 2LL * sms && fx < 8e-6 * (double)st.nnz * bp / (b <= 16 ? 31.0 : 42.0);
}

bool fx_all_wide(fio_op op) {
  if (op->fx_max_cols[0] == 0) return false;
  for (const Stage& st : op->st)
    if (st.nblk && !st.fx_ok[0]) return false;
  return op->fx != nullptr;
}

bool fx_launch(const Stage& st, bool adj, bool wide, const void* x, long long xrs, long long xcs, void* y, long long yrs,
               long long ycs, int b, void* scratch, size_t scratch_bytes, int* timeout, cudaStream_t s) {
  const int dir = adj ? 1 : 0;
  const size_t elem = wide ? sizeof(double2) : sizeof(float2);
  const long long cols = wide ? st.fx_cols[dir].x : st.fx_cols[dir].y;
  const size_t xb = al256((size_t)cols * (size_t)b * elem);
  if (!scratch || xb + (size_t)st.nblk * (size_t)b * sizeof(int) > scratch_bytes) return false;
  FxArgs a;
  a.units = st.fx_units[dir];
  a.nunits = st.n_fx_units[dir];
  a.nrt = 1;
  a.A = st.fxA[wide ? 0 : 1][dir];
  a.X = (const uint8_t*)scratch;
  a.ej = (const int*)((uint8_t*)scratch + xb);
  a.rexp = st.fx_exp[dir];
  a.rowidx = adj ? st.in : st.out;
  a.colidx = adj ? st.out : st.in;
  a.lrow = adj ? (int)st.C : (int)st.R;
  a.lcol = adj ? (int)st.R : (int)st.C;
  a.list = st.fx_list[dir];
  a.llist = list_stride(a.lcol);
  a.maxcols = (st.maxcols[dir] + 15) & ~15;
  a.dims = st.dims;
  a.xofs = st.fx_xofs[dir];
  a.xcols = cols;
  a.nblk = (int)st.nblk;
  a.R = (int)st.R;
  a.C = (int)st.C;
  a.M = wide ? (const void*)st.M64 : (const void*)st.M32;
  a.x = x;
  a.xrs = xrs;
  a.xcs = xcs;
  a.y = y;
  a.yrs = yrs;
  a.ycs = ycs;
  a.b = b;
  a.nraw = 0;
  a.steps = st.fx_steps[dir];
  a.timeout = timeout;
  uint8_t* X = (uint8_t*)scratch;
  int* ej = (int*)(X + xb);
  if (wide) return adj ? launch_b<double, true>(a, X, ej, s) : launch_b<double, false>(a, X, ej, s);
  return adj ? launch_b<float, true>(a, X, ej, s) : launch_b<float, false>(a, X, ej, s);
}
