// fio_capi.cu -- the C ABI of include/fio.h: upload of the packed factors, the applies of
// K-dot (paper section 2), K-dot* , G-dot (section 4) and G-dot K-dot* (section 5), and the
// operator bookkeeping.  The iterative solvers live in fio_solve.cu.
#include <cuda_runtime.h>
#include <cudaTypedefs.h>
#include <stdint.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <type_traits>
#include <new>
#include <vector>

#include "fio.h"
#include "fio_internal.h"
#include "fio_kernels.cuh"
#include "fio_tc.cuh"
#include "fio_tma.cuh"

using namespace fio;

namespace {

constexpr size_t kHeader = 256;
constexpr int kTileRows = 64;  // output rows per CTA of every k_stage_mm / k_stage_mm_pipe shape
constexpr size_t kStageBytes = 64;

template <typename T>
T rd(const uint8_t* p, size_t off) {
  T v;
  memcpy(&v, p + off, sizeof(T));
  return v;
}

uint64_t checksum(const uint8_t* p, size_t start, size_t end) {
  uint64_t s = 0;
  const size_t nw = (end - start) / 8;
  for (size_t k = 0; k < nw; ++k) {
    uint64_t w;
    memcpy(&w, p + start + 8 * k, 8);
    s += w * (2 * (uint64_t)k + 1);
  }
  return s;
}

// every valid index of `idx` in [0, len) and each value of [0, len) exactly once
bool is_permutation(const int32_t* idx, size_t n, int64_t len) {
  std::vector<uint8_t> seen((size_t)len, 0);
  int64_t cnt = 0;
  for (size_t k = 0; k < n; ++k) {
    const int32_t v = idx[k];
    if (v < 0) continue;
    if (v >= len || seen[v]) return false;
    seen[v] = 1;
    ++cnt;
  }
  return cnt == len;
}

// cuTensorMapEncodeTiled from the driver (looked up once; no link-time dependency on libcuda)
PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    cudaGetLastError();
  });
  return fn;
}

// 2D tensor map over a stage's factor copy for the TMA kernel: rows = nblk * rows_per_blk, each of
// 2 * ld elements (FP32 or BF16), boxes of 32 rows x 128 bytes (four make one 128-row operand
// tile), 128-byte swizzle (the K-major operand layout of tcgen05.mma).  False when the copy's base or row stride is not 16-byte
// aligned (the stage then keeps the other kernels).
bool encode_tmap(CUtensorMap* map, const void* base, bool bf16, long long rows, int ld) {
  PFN_cuTensorMapEncodeTiled_v12000 fn = encode_fn();
  if (!fn || !base || rows <= 0 || ld <= 0) return false;
  const int esz = bf16 ? 2 : 4;
  const cuuint64_t dims[2] = {(cuuint64_t)(2 * ld), (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)(2 * ld) * esz};
  const cuuint32_t box[2] = {(cuuint32_t)(128 / esz), (cuuint32_t)tma::kBoxRows};
  const cuuint32_t estr[2] = {1u, 1u};
  if (((uintptr_t)base & 15) || (strides[0] & 15) || rows > 0x7fffffffLL) return false;
  return fn(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<void*>(base),
            dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// work units of the TMA kernel for one stage: per direction and per unit size G in {1, 2, 4}
// row tiles, every block's 128-row tiles in groups of at most G, sorted by work (tiles x valid
// columns) with the largest first, so that the persistent CTAs' round-robin walk ends evenly
int build_units(fio_op op, const std::vector<int2>& meta, const std::vector<size_t>& mdims) {
  static const int kG[3] = {1, 2, 4};
  std::vector<int4> all;
  std::vector<size_t> off;
  for (size_t si = 0; si < op->st.size(); ++si) {
    const Stage& st = op->st[si];
    for (int dir = 0; dir < 2; ++dir)
      for (int g = 0; g < 3; ++g) {
        std::vector<std::pair<long long, int4>> u;
        for (uint32_t b = 0; b < st.nblk; ++b) {
          const int2 d = meta[mdims[si] + b];
          const int rows = dir ? d.y : d.x, cols = dir ? d.x : d.y;
          const int nt = (rows + kTcRows - 1) / kTcRows;
          for (int t0 = 0; t0 < nt; t0 += kG[g]) {
            const int k = std::min(kG[g], nt - t0);
            u.push_back(std::make_pair((long long)k * cols, make_int4((int)b, t0, k, 0)));
          }
        }
        std::stable_sort(u.begin(), u.end(), [](const std::pair<long long, int4>& x, const std::pair<long long, int4>& y) {
          return x.first > y.first;
        });
        off.push_back(all.size());
        for (auto& e : u) all.push_back(e.second);
      }
  }
  off.push_back(all.size());
  if (all.empty()) return FIO_OK;
  if (cudaMalloc(&op->units, all.size() * sizeof(int4)) != cudaSuccess) {
    cudaGetLastError();
    return FIO_ENOMEM;
  }
  op->units_bytes = all.size() * sizeof(int4);
  if (cudaMemcpy(op->units, all.data(), op->units_bytes, cudaMemcpyHostToDevice) != cudaSuccess) return FIO_ECUDA;
  size_t k = 0;
  for (auto& st : op->st)
    for (int dir = 0; dir < 2; ++dir)
      for (int g = 0; g < 3; ++g, ++k) {
        st.units[dir][g] = (const int4*)op->units + off[k];
        st.nunits[dir][g] = (int)(off[k + 1] - off[k]);
      }
  return FIO_OK;
}

}  // namespace

// ---------------------------------------------------------------------------------------------
// upload
// ---------------------------------------------------------------------------------------------
extern "C" int fio_upload_factors(const void* packed, size_t nbytes, unsigned mask, void* stream,
                                  fio_op* out) {
  if (!packed || !out) return FIO_EINVAL;
  *out = nullptr;
  if (mask == 0) mask = FIO_MASK_P64 | FIO_MASK_P32 | FIO_MASK_TC | FIO_MASK_DF;
  const uint8_t* p = (const uint8_t*)packed;
  if (nbytes < kHeader || memcmp(p, "FIOPACK1", 8) != 0) return FIO_EBADFACTORS;
  const uint32_t version = rd<uint32_t>(p, 8), d = rd<uint32_t>(p, 12);
  const int64_t n = rd<int64_t>(p, 16), N = rd<int64_t>(p, 24);
  const uint32_t n_bf = rd<uint32_t>(p, 32), n_hif = rd<uint32_t>(p, 36), n_root = rd<uint32_t>(p, 40);
  const uint64_t tab = rd<uint64_t>(p, 64), data = rd<uint64_t>(p, 72), total = rd<uint64_t>(p, 80),
                 csum = rd<uint64_t>(p, 88);
  if (version != 1 || (d != 1 && d != 2) || n <= 0 || N <= 0 || N > (int64_t)1 << 31) return FIO_EBADFACTORS;
  if ((d == 1 && N != n) || (d == 2 && N != n * n)) return FIO_EBADFACTORS;
  if (total != nbytes || data > total || (total - data) % 8 || n_root > 1 || n_bf == 0) return FIO_EBADFACTORS;
  const uint64_t nst = (uint64_t)n_bf + n_hif + n_root;
  if (tab < kHeader || tab + nst * kStageBytes > data) return FIO_EBADFACTORS;
  if (checksum(p, data, total) != csum) return FIO_EBADFACTORS;

  fio_op_s* op = new (std::nothrow) fio_op_s();
  if (!op) return FIO_ENOMEM;
  op->d = (int)d;
  op->n = n;
  op->N = N;
  op->n_bf = (int)n_bf;
  op->n_hif = (int)n_hif;
  op->n_root = (int)n_root;
  op->mask = mask;
  op->max_len = N;
  size_t m_elems = 0;
  int64_t prev_out = N;
  for (uint64_t s = 0; s < nst; ++s) {
    const size_t e = tab + s * kStageBytes;
    Stage st{};
    st.kind = rd<uint32_t>(p, e);
    st.nblk = rd<uint32_t>(p, e + 4);
    st.R = rd<uint32_t>(p, e + 8);
    st.C = rd<uint32_t>(p, e + 12);
    st.in_len = rd<int64_t>(p, e + 16);
    st.out_len = rd<int64_t>(p, e + 24);
    st.offM = rd<uint64_t>(p, e + 32);
    st.offIn = rd<uint64_t>(p, e + 40);
    st.offOut = rd<uint64_t>(p, e + 48);
    st.level = rd<uint32_t>(p, e + 56);
    st.role = rd<uint32_t>(p, e + 60);
    const uint64_t mb = (uint64_t)st.nblk * st.R * st.C * 16, ib = (uint64_t)st.nblk * st.C * 4,
                   ob = (uint64_t)st.nblk * st.R * 4;
    const bool bf = s < n_bf;
    bool ok = st.kind <= 1 && st.offM % 16 == 0 && st.offIn % 4 == 0 && st.offOut % 4 == 0 &&
              st.offM >= data && st.offIn >= data && st.offOut >= data && st.offM + mb <= total &&
              st.offIn + ib <= total && st.offOut + ob <= total && st.in_len > 0 && st.out_len > 0 &&
              st.in_len < ((int64_t)1 << 31) && st.out_len < ((int64_t)1 << 31) &&
              (st.nblk == 0 || (st.R > 0 && st.C > 0));
    if (ok && bf) {
      ok = st.kind == 0 && st.in_len == prev_out &&
           is_permutation((const int32_t*)(p + st.offIn), (size_t)st.nblk * st.C, st.in_len) &&
           is_permutation((const int32_t*)(p + st.offOut), (size_t)st.nblk * st.R, st.out_len);
      prev_out = st.out_len;
      if (st.out_len > op->max_len) op->max_len = st.out_len;
      if (s + 1 == n_bf && st.out_len != N) ok = false;
    } else if (ok) {
      // INPLACE: square blocks, identical in/out lists, disjoint index sets inside [0, N)
      ok = st.kind == 1 && st.R == st.C && st.in_len == N && st.out_len == N &&
           memcmp(p + st.offIn, p + st.offOut, ib) == 0;
      if (ok) {
        std::vector<uint8_t> seen((size_t)N, 0);
        const int32_t* ii = (const int32_t*)(p + st.offIn);
        for (size_t k = 0; ok && k < (size_t)st.nblk * st.C; ++k) {
          const int32_t v = ii[k];
          if (v < 0) continue;
          if (v >= N || seen[v]) ok = false;
          else seen[v] = 1;
        }
      }
    }
    if (!ok) {
      delete op;
      return FIO_EBADFACTORS;
    }
    st.launch_rows = 0;
    m_elems += (size_t)st.nblk * st.R * st.C;
    op->st.push_back(st);
  }

  // per block: extent of the valid rows / columns; CTA tile lists (64-row tiles) per direction
  std::vector<int2> meta;
  std::vector<size_t> mdims(nst), mfwd(nst), madj(nst), m128f(nst), m128a(nst);
  for (uint64_t si = 0; si < nst; ++si) {
    fio::Stage& st = op->st[si];
    const int32_t* ii = (const int32_t*)(p + st.offIn);
    const int32_t* oo = (const int32_t*)(p + st.offOut);
    mdims[si] = meta.size();
    for (uint32_t b = 0; b < st.nblk; ++b) {
      int rb = 0, cb = 0;
      for (uint32_t r = 0; r < st.R; ++r)
        if (oo[(size_t)b * st.R + r] >= 0) rb = (int)r + 1;
      for (uint32_t c = 0; c < st.C; ++c)
        if (ii[(size_t)b * st.C + c] >= 0) cb = (int)c + 1;
      meta.push_back(make_int2(rb, cb));
      st.maxcols[0] = std::max(st.maxcols[0], cb);
      st.maxcols[1] = std::max(st.maxcols[1], rb);
    }
    mfwd[si] = meta.size();
    for (uint32_t b = 0; b < st.nblk; ++b)
      for (int t = 0; t * kTileRows < meta[mdims[si] + b].x; ++t) meta.push_back(make_int2((int)b, t));
    st.ntiles_fwd = (int)(meta.size() - mfwd[si]);
    madj[si] = meta.size();
    for (uint32_t b = 0; b < st.nblk; ++b)
      for (int t = 0; t * kTileRows < meta[mdims[si] + b].y; ++t) meta.push_back(make_int2((int)b, t));
    st.ntiles_adj = (int)(meta.size() - madj[si]);
    m128f[si] = meta.size();
    for (uint32_t b = 0; b < st.nblk; ++b)
      for (int t = 0; t * kTcRows < meta[mdims[si] + b].x; ++t) meta.push_back(make_int2((int)b, t));
    st.n128_fwd = (int)(meta.size() - m128f[si]);
    m128a[si] = meta.size();
    for (uint32_t b = 0; b < st.nblk; ++b)
      for (int t = 0; t * kTcRows < meta[mdims[si] + b].y; ++t) meta.push_back(make_int2((int)b, t));
    st.n128_adj = (int)(meta.size() - m128a[si]);
  }

  cudaStream_t s = (cudaStream_t)stream;
  if (!meta.empty()) {
    if (cudaMalloc(&op->meta, meta.size() * sizeof(int2)) != cudaSuccess) {
      cudaGetLastError();
      delete op;
      return FIO_ENOMEM;
    }
    op->meta_bytes = meta.size() * sizeof(int2);
    if (cudaMemcpy(op->meta, meta.data(), op->meta_bytes, cudaMemcpyHostToDevice) != cudaSuccess) {
      fio_release(op);
      return FIO_ECUDA;
    }
    for (uint64_t si = 0; si < nst; ++si) {
      op->st[si].dims = (const int2*)op->meta + mdims[si];
      op->st[si].tiles_fwd = (const int2*)op->meta + mfwd[si];
      op->st[si].tiles_adj = (const int2*)op->meta + madj[si];
      op->st[si].t128_fwd = (const int2*)op->meta + m128f[si];
      op->st[si].t128_adj = (const int2*)op->meta + m128a[si];
    }
  }
  if (cudaMalloc(&op->arena, nbytes) != cudaSuccess) {
    cudaGetLastError();
    delete op;
    return FIO_ENOMEM;
  }
  op->arena_bytes = nbytes;
  if (cudaMemcpyAsync(op->arena, packed, nbytes, cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess) {
    fio_release(op);
    return FIO_ECUDA;
  }
  if (mask & FIO_MASK_P32) {
    if (cudaMalloc(&op->arena32, (m_elems + nst) * sizeof(float2) + 256) != cudaSuccess) {
      cudaGetLastError();
      fio_release(op);
      return FIO_ENOMEM;
    }
    op->arena32_bytes = (m_elems + nst) * sizeof(float2) + 256;
  }
  if (mask & FIO_MASK_DF) {
    if (cudaMalloc(&op->arena_df, (m_elems + nst) * sizeof(dfc) + 256) != cudaSuccess) {
      cudaGetLastError();
      fio_release(op);
      return FIO_ENOMEM;
    }
    op->arena_df_bytes = (m_elems + nst) * sizeof(dfc) + 256;
  }
  size_t off32 = 0;
  for (auto& st : op->st) {
    const size_t ne = (size_t)st.nblk * st.R * st.C;
    st.M64 = (const double2*)((const uint8_t*)op->arena + st.offM);
    st.in = (const int*)((const uint8_t*)op->arena + st.offIn);
    st.out = (const int*)((const uint8_t*)op->arena + st.offOut);
    if (op->arena32) {
      float2* dst = (float2*)op->arena32 + off32;
      st.M32 = dst;
      if (ne) {
        k_cast_c128_c64<<<(unsigned)((ne + 255) / 256), 256, 0, s>>>(st.M64, dst, ne);
      }
    }
    if (op->arena_df) {
      dfc* dst = (dfc*)op->arena_df + off32;
      st.Mdf = dst;
      if (ne) k_split_df<<<(unsigned)((ne + 255) / 256), 256, 0, s>>>(st.M64, dst, ne);
    }
    off32 += ne + (ne & 1);  // every stage's complex64 blocks start 16-byte aligned
  }
  if ((mask & FIO_MASK_TC) && op->arena32) {
    auto al = [](size_t x) { return (x + 255) & ~(size_t)255; };
    size_t tot = 0;
    for (auto& st : op->st) {
      const size_t ne = (size_t)st.nblk * st.R * st.C;
      const int ldbf = (int)((st.C + 3) & ~3u), ldbft = (int)((st.R + 3) & ~3u);
      tot += al(ne * sizeof(float2)) + al((size_t)st.nblk * st.R * ldbf * 4) + al((size_t)st.nblk * st.C * ldbft * 4);
    }
    if (cudaMalloc(&op->arena_tc, tot + 256) != cudaSuccess) {
      cudaGetLastError();
      fio_release(op);
      return FIO_ENOMEM;
    }
    op->arena_tc_bytes = tot + 256;
    uint8_t* q = (uint8_t*)op->arena_tc;
    for (auto& st : op->st) {
      const size_t ne = (size_t)st.nblk * st.R * st.C;
      st.ldbf = (int)((st.C + 3) & ~3u);
      st.ldbft = (int)((st.R + 3) & ~3u);
      float2* t32 = (float2*)q;
      q += al(ne * sizeof(float2));
      __nv_bfloat162* bf = (__nv_bfloat162*)q;
      q += al((size_t)st.nblk * st.R * st.ldbf * 4);
      __nv_bfloat162* bft = (__nv_bfloat162*)q;
      q += al((size_t)st.nblk * st.C * st.ldbft * 4);
      st.M32t = t32;
      st.Mbf = bf;
      st.Mbft = bft;
      if (!ne) continue;
      const unsigned g = (unsigned)((ne + 255) / 256);
      k_transpose_blocks<<<g, 256, 0, s>>>(st.M32, t32, (int)st.nblk, (int)st.R, (int)st.C);
      const size_t n1 = (size_t)st.nblk * st.R * st.ldbf, n2 = (size_t)st.nblk * st.C * st.ldbft;
      k_to_bf16<<<(unsigned)((n1 + 255) / 256), 256, 0, s>>>(st.M32, bf, (int)st.nblk, (int)st.R, (int)st.C, st.ldbf);
      k_to_bf16<<<(unsigned)((n2 + 255) / 256), 256, 0, s>>>(t32, bft, (int)st.nblk, (int)st.C, (int)st.R, st.ldbft);
    }
    // the TMA kernel's tensor maps (forward / adjoint x FP32 / BF16) and work units
    for (auto& st : op->st) {
      const long long nb = st.nblk;
      st.tma_ok[0][0] = encode_tmap(&st.tmap[0][0], st.M32, false, nb * st.R, (int)st.C);
      st.tma_ok[1][0] = encode_tmap(&st.tmap[1][0], st.M32t, false, nb * st.C, (int)st.R);
      st.tma_ok[0][1] = encode_tmap(&st.tmap[0][1], st.Mbf, true, nb * st.R, st.ldbf);
      st.tma_ok[1][1] = encode_tmap(&st.tmap[1][1], st.Mbft, true, nb * st.C, st.ldbft);
    }
    const int urc = build_units(op, meta, mdims);
    if (urc != FIO_OK) {
      fio_release(op);
      return urc;
    }
  }
  int fxrc = fft_build(op, s);
  if (fxrc == FIO_OK) fxrc = fx_build(op, meta, mdims, s);
  if (fxrc != FIO_OK) {
    fio_release(op);
    return fxrc;
  }
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(s) != cudaSuccess) {
    fio_release(op);
    return FIO_ECUDA;
  }
  *out = op;
  return FIO_OK;
}

extern "C" int fio_release(fio_op op) {
  if (!op) return FIO_OK;
  cudaDeviceSynchronize();
  if (op->arena) cudaFree(op->arena);
  if (op->arena32) cudaFree(op->arena32);
  if (op->arena_df) cudaFree(op->arena_df);
  if (op->meta) cudaFree(op->meta);
  if (op->units) cudaFree(op->units);
  if (op->fx) cudaFree(op->fx);
  if (op->fft_tw) cudaFree(op->fft_tw);
  if (op->arena_tc) cudaFree(op->arena_tc);
  if (op->scratch) cudaFree(op->scratch);
  if (op->fx_scratch) cudaFree(op->fx_scratch);
  if (op->flag_host) cudaFreeHost(op->flag_host);
  fio_solver_free(op);
  cudaGetLastError();
  delete op;
  return FIO_OK;
}

extern "C" int fio_query(fio_op op, int* d, int64_t* n, int64_t* N, size_t* device_bytes) {
  if (!op) return FIO_EINVAL;
  if (d) *d = op->d;
  if (n) *n = op->n;
  if (N) *N = op->N;
  if (device_bytes)
    *device_bytes = op->arena_bytes + op->arena32_bytes + op->arena_tc_bytes + op->arena_df_bytes + op->meta_bytes +
                    op->units_bytes + op->fx_bytes + op->fft_bytes + op->scratch_bytes +
                    op->fx_scratch_bytes + op->solver_bytes;
  return FIO_OK;
}

extern "C" const char* fio_strerror(int status) {
  switch (status) {
    case FIO_OK: return "ok";
    case FIO_EINVAL: return "invalid argument";
    case FIO_ENOMEM: return "out of device memory";
    case FIO_EBADFACTORS: return "packed factor buffer is damaged or inconsistent";
    case FIO_ENOCONV: return "iterative solve did not reach the tolerance";
    case FIO_ETIMEOUT: return "bounded device wait timed out";
    case FIO_ECUDA: return "CUDA runtime error";
    case FIO_ENOTSUP: return "operator lacks the factors this call needs";
    default: return "unknown status";
  }
}

// ---------------------------------------------------------------------------------------------
// scratch pool: 5 work arrays of max(max_len, N) x b complex elements each
// ---------------------------------------------------------------------------------------------
int fio_scratch(fio_op op, int b, size_t elem, cudaStream_t s, void** bufs, void** fxbuf, size_t* fxbytes) {
  const size_t per = (size_t)op->max_len * (size_t)(elem == 8 ? (b + 1) & ~1 : b) * elem;  // row_stride
  const size_t per_al = (per + 255) & ~(size_t)255;
  // FIO_OK, FIO_ENOMEM (the buffer is gone) or FIO_ECUDA
  auto grow = [&](void** buf, size_t* bytes, size_t need) {
    if (need <= *bytes) return FIO_OK;
    if (*buf) {
      if (cudaStreamSynchronize(s) != cudaSuccess) return FIO_ECUDA;
      cudaFree(*buf);
      *buf = nullptr;
      *bytes = 0;
    }
    if (cudaMalloc(buf, need) != cudaSuccess) {
      cudaGetLastError();
      *buf = nullptr;
      return FIO_ENOMEM;
    }
    *bytes = need;
    return FIO_OK;
  };
  int rc = grow(&op->scratch, &op->scratch_bytes, 5 * per_al);
  if (rc == FIO_ENOMEM && op->fx_scratch) {  // what the fixed-point kernel holds may be what is missing
    cudaFree(op->fx_scratch);
    op->fx_scratch = nullptr;
    op->fx_scratch_bytes = 0;
    rc = grow(&op->scratch, &op->scratch_bytes, 5 * per_al);
  }
  if (rc) return rc;
  for (int k = 0; k < 5; ++k) bufs[k] = (uint8_t*)op->scratch + k * per_al;
  // no room for the fixed-point kernel's: this call runs on the CUDA cores (so does a captured call whose
  // sizing call had none: nothing may be allocated now)
  const size_t fxneed = fxbuf ? fx_scratch_bytes(op, b, elem) : 0;
  auto captured = [&] {
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    const bool yes = cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone;
    if (yes) cudaGetLastError();
    return yes;
  };
  rc = fxneed && (fxneed <= op->fx_scratch_bytes || !captured()) ? grow(&op->fx_scratch, &op->fx_scratch_bytes, fxneed) : FIO_ENOMEM;
  if (rc == FIO_ECUDA) return rc;
  if (fxbuf) *fxbuf = rc == FIO_OK ? op->fx_scratch : nullptr;
  if (fxbytes) *fxbytes = rc == FIO_OK ? fxneed : 0;
  return FIO_OK;
}

// ---------------------------------------------------------------------------------------------
// stage launches
// ---------------------------------------------------------------------------------------------
namespace {

// optional per-stage event marks (fio_apply_profiled); null in the ordinary applies
struct Marks {
  cudaEvent_t* ev;
  int cap, n;
  void mark(cudaStream_t s) {
    if (ev && n < cap) cudaEventRecord(ev[n++], s);
  }
};
thread_local Marks* g_marks = nullptr;
inline void mark(cudaStream_t s) {
  if (g_marks) g_marks->mark(s);
}

// Row stride of the work vectors: in complex64 rounded up to even from b = 5 on, so that every row is
// 16-byte aligned and the pipelined kernels serve odd counts too (they may read, never write, the odd
// column; b = 13 at N = 4096: 0.36 ms a direct solve unpadded, 0.24 padded)
template <typename V>
inline int row_stride(int b) { return sizeof(V) == 8 && b >= 5 ? (b + 1) & ~1 : b; }

template <typename V> const V* stage_M(const Stage& st);
template <> const double2* stage_M<double2>(const Stage& st) { return st.M64; }
template <> const float2* stage_M<float2>(const Stage& st) { return st.M32; }
template <> const dfc* stage_M<dfc>(const Stage& st) { return st.Mdf; }

template <typename V> struct ChunkK;
template <> struct ChunkK<double2> { static constexpr int v = 16; };
template <> struct ChunkK<float2> { static constexpr int v = 32; };
template <> struct ChunkK<dfc> { static constexpr int v = 16; };

int num_sms();

// Stage launches whose CTAs are light enough to be started early (pdl_launch), by the complex
// multiply-adds of a CTA's tile and the grid.  Early CTAs, of more than one launch ahead, take the places
// that are free when they come, and later run two on one multiprocessor while others idle: a loss of up
// to a tile's time against a gain of 2 us a launch.  The limits follow the type's rate (FP64 2 lanes an SM and
// clock, FP32 128) and how much of the chip the grid covers.  Measured, speed of a K-dot or inverse against
// plain launches, with the limits of the columns:
//   a grid of at most an eighth of the SMs never shares one: any tile up to 110000 (1D N = 256, FP64
//     b = 8 1.19, FP32 b = 16 1.67)
//   at most half of the SMs      110000         smaller
//     FP32  1D N = 1024 b = 8    1.71           1.36 (30000)
//     double-float               0.93           1.03 (30000)   Example 3 n = 32, b = 16
//     FP64  40 tiles 64 x 230    0.46           1.05 (8000)    PCG, b = 5
//   more                         110000         smaller
//     FP32  1D N = 16384 b = 16  0.94           1.03 (80000)   K-dot*; inverse 1.38 and 1.49
//           1D N = 4096 b = 16   0.92           1.22 (80000, 1.10 at 34000)
//           2D n = 128 b = 6     0.74           1.08 (80000)   K-dot*; inverse 0.92 and 1.11
//           1D N = 65536 b = 16  1.41           1.29 (80000)   inverse; 7 times as many CTAs as SMs: from
//           four on the waves even themselves out
//     FP64  1D N = 4096 b = 1    0.65           1.18 (2500, 0.65 at 8000)   K-dot*
constexpr long long kLightMacs = 110000;
template <bool ADJ, typename V>
bool light(const StageArgs<V>& a, int rows, int rhs, const dim3& grid) {
  const long long ctas = (long long)grid.x * grid.y * grid.z, sms = num_sms();
  const bool many = 2 * ctas > sms;
  const long long limit = 8 * ctas <= sms                    ? kLightMacs
                          : sizeof(V) == sizeof(float2)      ? (many && ctas <= 4 * sms ? 80000 : kLightMacs)
                          : std::is_same<V, dfc>::value      ? (many ? 30000 : 50000)
                                                             : (many ? 2500 : 12000);
  return (long long)rows * (ADJ ? a.R : a.C) * std::min(rhs, a.b) <= limit * a.ksplit;
}

template <typename V, bool ADJ, int TX, int TB, int TR>
void launch_mm(StageArgs<V> a, cudaStream_t s) {
  constexpr int RT = (256 / TX) * TR, BT = TX * TB;
  static_assert(RT == kTileRows, "tile lists are built for 64-row tiles");
  const int nrows = ADJ ? a.C : a.R;
  a.ntiles = (nrows + RT - 1) / RT;
  const long long ncta = a.tiles ? a.ntiles_list : (long long)a.nblk * a.ntiles;
  if (ncta == 0) return;
  dim3 grid((unsigned)ncta, (unsigned)((a.b + BT - 1) / BT));
  pdl_launch(light<ADJ>(a, RT, BT, grid), k_stage_mm<V, ADJ, TX, TB, TR, ChunkK<V>::v>, grid, 256, 0, s, a);
}

// Dynamic shared memory above 48 KB is opted into per kernel and per device: remember, per (device,
// kernel), the largest amount granted so far.  False when the attribute call fails (the launch
// then fails and the call reports FIO_ECUDA, or the caller picks another variant).
bool smem_opt_in(const void* func, int need) {
  if (need <= 48 * 1024) return true;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, int> granted;
  std::lock_guard<std::mutex> lock(mu);
  int& cap = granted[std::make_pair(dev, func)];
  if (need <= cap) return true;
  if (cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, need) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  cap = need;
  return true;
}

template <typename V, bool ADJ, int TX, int TB, int TR>
void launch_pipe(StageArgs<V> a, cudaStream_t s) {
  constexpr int CK = ChunkK<V>::v;
  using S = PipeShape<V, ADJ, TX, TB, TR, CK>;
  smem_opt_in((const void*)k_stage_mm_pipe<V, ADJ, TX, TB, TR, CK>, S::SMEM);
  static_assert(S::RT == kTileRows, "tile lists are built for 64-row tiles");
  const int nrows = ADJ ? a.C : a.R;
  a.ntiles = (nrows + S::RT - 1) / S::RT;
  const long long ncta = a.tiles ? a.ntiles_list : (long long)a.nblk * a.ntiles;
  if (ncta == 0) return;
  dim3 grid((unsigned)ncta, (unsigned)((a.b + S::BT - 1) / S::BT));
  pdl_launch(light<ADJ>(a, S::RT, S::BT, grid), k_stage_mm_pipe<V, ADJ, TX, TB, TR, CK>, grid, 256, S::SMEM, s, a);
}
// the same tiles with three real products per complex product (FP64 and double-float only)
template <typename V, bool ADJ, int TX, int TB, int TR>
bool launch_pipe3(StageArgs<V> a, cudaStream_t s) {
  if constexpr (std::is_same<V, double2>::value || std::is_same<V, dfc>::value) {
    constexpr int CK = ChunkK<V>::v;
    using S = PipeShape<V, ADJ, TX, TB, TR, CK>;
    constexpr int smem = S::smem(true);
    if (!smem_opt_in((const void*)k_stage_mm_pipe<V, ADJ, TX, TB, TR, CK, true>, smem)) return false;
    const int nrows = ADJ ? a.C : a.R;
    a.ntiles = (nrows + S::RT - 1) / S::RT;
    const long long ncta = a.tiles ? a.ntiles_list : (long long)a.nblk * a.ntiles;
    if (ncta == 0) return true;
    dim3 grid((unsigned)ncta, (unsigned)((a.b + S::BT - 1) / S::BT));
    pdl_launch(light<ADJ>(a, S::RT, S::BT, grid), k_stage_mm_pipe<V, ADJ, TX, TB, TR, CK, true>, grid, 256, smem, s, a);
    return true;
  } else {
    return false;
  }
}

// complex64 tiles with contiguous per-thread rows and right-hand sides (k_stage_mm_vt); 64- or
// 128-row tiles (the latter from the stage's list of 128-row tiles)
template <bool ADJ, int TX, int TB, int TR, int NT, int CK = 32, int MINB = (NT == 128 && TX == 8 ? 4 : 1)>
bool launch_vt(StageArgs<float2> a, cudaStream_t s) {
  using S = VtShape<ADJ, TX, TB, TR, NT, CK>;
  static_assert(S::RT == kTileRows || S::RT == 2 * kTileRows, "tile lists hold 64- and 128-row tiles");
  if (S::RT != kTileRows) {
    if (!a.tiles128) return false;
    a.tiles = a.tiles128;
    a.ntiles_list = a.ntiles128;
  }
  if (!smem_opt_in((const void*)k_stage_mm_vt<ADJ, TX, TB, TR, NT, CK, MINB>, S::SMEM)) return false;
  const int nrows = ADJ ? a.C : a.R;
  a.ntiles = (nrows + S::RT - 1) / S::RT;
  const long long ncta = a.tiles ? a.ntiles_list : (long long)a.nblk * a.ntiles;
  if (ncta == 0) return true;
  dim3 grid((unsigned)ncta, (unsigned)((a.b + S::BT - 1) / S::BT), (unsigned)a.ksplit);
  pdl_launch(light<ADJ>(a, S::RT, S::BT, grid), k_stage_mm_vt<ADJ, TX, TB, TR, NT, CK, MINB>, grid, NT, S::SMEM, s, a);
  return true;
}
template <typename V, bool ADJ, int TX, int TB, int TR, int NT, int CK = 32,
          int MINB = (NT == 128 && TX == 8 ? 4 : 1)>
bool launch_vt_if(const StageArgs<V>& a, cudaStream_t s) {
  if constexpr (std::is_same<V, float2>::value) {
    return launch_vt<ADJ, TX, TB, TR, NT, CK, MINB>(a, s);
  } else {
    return false;
  }
}

// small blocks (k_stage_small, FP64 and FP32): a warp per block, 32 right-hand sides per CTA row
template <typename V>
bool small_ok(const StageArgs<V>& a) {
  return (std::is_same<V, float2>::value || std::is_same<V, double2>::value) && a.R <= kSmallMaxDim &&
         a.C <= kSmallMaxDim && a.R > 0 && a.C > 0;
}
template <typename V, bool ADJ>
bool launch_small(const StageArgs<V>& a, cudaStream_t s) {
  if constexpr (std::is_same<V, float2>::value || std::is_same<V, double2>::value) {
    if (!small_ok(a)) return false;
    const int smem = kSmallWarps * (a.R * a.C + 32 * (ADJ ? a.R : a.C)) * (int)sizeof(V);
    if (!smem_opt_in((const void*)k_stage_small<V, ADJ>, smem)) return false;
    if (a.nblk == 0) return true;
    dim3 grid((unsigned)((a.nblk + kSmallWarps - 1) / kSmallWarps), (unsigned)((a.b + 31) / 32));
    pdl_launch(true, k_stage_small<V, ADJ>, grid, 32 * kSmallWarps, smem, s, a);
    return true;
  } else {
    return false;
  }
}

// the pipelined kernel needs row-major x with 16-byte aligned rows of M and of x
template <typename V>
bool pipe_ok(const StageArgs<V>& a) {
  const int vpc = 16 / (int)sizeof(V);
  return a.xcs == 1 && a.xrs >= a.b && a.xrs % vpc == 0 && a.C % vpc == 0 &&
         ((uintptr_t)a.M & 15) == 0 && ((uintptr_t)a.x & 15) == 0;
}

// few right-hand sides: k_stage_vec when the tile's gathered input fits in shared memory (false:
// the caller falls back to the tiled kernel)
template <typename V, bool ADJ, int B>
bool launch_vec_b(StageArgs<V> a, cudaStream_t s) {
  const long long slots = (long long)(ADJ ? std::max<int>(a.R, 256) : a.C) * B;
  const long long need = slots * (long long)sizeof(V);
  if (need > 200 * 1024) return false;
  if (!smem_opt_in((const void*)k_stage_vec<V, ADJ, B>, (int)need)) return false;
  const int nrows = ADJ ? a.C : a.R;
  a.ntiles = (nrows + kTileRows - 1) / kTileRows;
  const long long ncta = a.tiles ? a.ntiles_list : (long long)a.nblk * a.ntiles;
  if (ncta == 0) return true;
  pdl_launch(light<ADJ>(a, kTileRows, B, dim3((unsigned)ncta)), k_stage_vec<V, ADJ, B>, (unsigned)ncta, 256, (size_t)need, s, a);
  return true;
}
template <typename V, bool ADJ>
bool launch_vec(const StageArgs<V>& a, cudaStream_t s) {
  switch (a.b) {
    case 1: return launch_vec_b<V, ADJ, 1>(a, s);
    case 2: return launch_vec_b<V, ADJ, 2>(a, s);
    case 3: return launch_vec_b<V, ADJ, 3>(a, s);
    case 4: return launch_vec_b<V, ADJ, 4>(a, s);
    default: return false;
  }
}

// ---- kernel variants (the autotuner's candidates) -----------------------------------------
// 1..7: tile shapes <TX, TB, TR> of the tiled kernel (256 threads, 64-row tiles, TX x TB
// right-hand sides per CTA): 1 <8,1,2>, 2 <16,1,4>, 3 <16,2,4>, 4 <8,2,2>, 5 <8,4,2>,
// 6 <32,1,8>, 7 <16,4,4>; 8: k_stage_vec (b <= 4); complex64 only, contiguous per-thread tiles
// (k_stage_mm_vt): 9 <16,2,8> with 128 threads, 10 <16,2,4> with 256 threads, 11 <8,4,8> with 128
// threads on 128-row tiles (32 accumulators per thread, 16-column chunks), 12 the same with the
// in-place stages split over their columns (partial sums reduced in a fixed order); 13
// k_stage_small (a warp per block, FP64 and FP32, padded blocks up to 32 x 32); 14, 15, 16 the
// FP64 and double-float tiles of 3, 6, 2 with three real products per complex product
// (k_stage_mm_pipe's G3) on the butterfly stages (the in-place stages, where the HIF's
// conditioning amplifies rounding, keep four products); 17 the tile of 9 with 16-column chunks
// (half the shared memory: up to five CTAs per SM instead of two); 18 the tile of 11 without its
// register cap (three CTAs per SM).  Shapes 2..7, 9..12, 14..17
// need the pipelined kernel's layout (row-major, 16-byte aligned rows); shape 1 falls back to the
// plain tiled kernel.
// the TMA-fed persistent tensor-core kernel (k_stage_tma): 30 units of as many row tiles as tensor
// memory holds and the deepest A ring; 31 the same with in-place stages split over K; 32 units
// sized for about eight per SM; 33 an A ring of at most six slots (split TF32: a six-slot tail
// ring instead of three)
constexpr int kTmaVariant = 30;
constexpr int kTmaSplitVariant = 31;
constexpr int kTmaBalancedVariant = 32;
constexpr int kTmaShallowVariant = 33;
inline bool is_tma_variant(int v) { return v >= kTmaVariant && v <= kTmaShallowVariant; }
// with a tensor-core precision: this stage launch on the FP32 CUDA cores instead (at least as
// accurate; the small blocks of the lowest HIF levels run faster there)
constexpr int kFp32CoresVariant = 40;
inline int rhs_bucket(int b) { return b <= 4 ? 0 : (b <= 8 ? 1 : (b <= 16 ? 2 : (b <= 32 ? 3 : 4))); }
// candidates per bucket, the built-in choice first
constexpr int kSmallVariant = 13;
constexpr int kVtChunk16Variant = 17;
constexpr int kVtUncappedVariant = 18;
constexpr int kMaxCudaCoreVariant = 18;
inline bool is_fp32_tile_variant(int v) { return (v >= 9 && v <= 12) || v == kVtChunk16Variant || v == kVtUncappedVariant; }
inline bool is_3m_variant(int v) { return v >= 14 && v <= 16; }
// the four-product variant a three-product one stands for on the in-place stages
inline int four_product_of(int v) { return v == 14 ? 3 : v == 15 ? 6 : v == 16 ? 2 : v; }
constexpr int kNCand = 13;
constexpr int kCand[5][kNCand] = {{8, 1}, {1, 2, 13, 16}, {2, 4, 3, 13, 14, 16},
                                  {3, 5, 6, 9, 10, 11, 12, 13, 14, 15, 17, 18},
                                  {3, 5, 6, 7, 9, 10, 11, 12, 13, 14, 15, 17, 18}};

// launch with variant `var`; false when it does not apply to this launch
template <typename V, bool ADJ>
bool launch_variant(const StageArgs<V>& a, cudaStream_t s, int var) {
  const bool pipe = pipe_ok(a);
  switch (var) {
    case 1:
      if (pipe) launch_pipe<V, ADJ, 8, 1, 2>(a, s);
      else launch_mm<V, ADJ, 8, 1, 2>(a, s);
      return true;
    case 2: if (!pipe) return false; launch_pipe<V, ADJ, 16, 1, 4>(a, s); return true;
    case 3: if (!pipe) return false; launch_pipe<V, ADJ, 16, 2, 4>(a, s); return true;
    case 4: if (!pipe) return false; launch_pipe<V, ADJ, 8, 2, 2>(a, s); return true;
    case 5: if (!pipe) return false; launch_pipe<V, ADJ, 8, 4, 2>(a, s); return true;
    case 6: if (!pipe) return false; launch_pipe<V, ADJ, 32, 1, 8>(a, s); return true;
    case 7: if (!pipe) return false; launch_pipe<V, ADJ, 16, 4, 4>(a, s); return true;
    case 8: return a.b <= kVecMaxRhs && launch_vec<V, ADJ>(a, s);
    case 9: return pipe && launch_vt_if<V, ADJ, 16, 2, 8, 128>(a, s);
    case 10: return pipe && launch_vt_if<V, ADJ, 16, 2, 4, 256>(a, s);
    case 11:
    case 12: return pipe && launch_vt_if<V, ADJ, 8, 4, 8, 128, 16>(a, s);
    case kSmallVariant: return launch_small<V, ADJ>(a, s);
    case 14: return pipe && launch_pipe3<V, ADJ, 16, 2, 4>(a, s);
    case 15: return pipe && launch_pipe3<V, ADJ, 32, 1, 8>(a, s);
    case 16: return pipe && launch_pipe3<V, ADJ, 16, 1, 4>(a, s);
    case kVtChunk16Variant: return pipe && launch_vt_if<V, ADJ, 16, 2, 8, 128, 16>(a, s);
    case kVtUncappedVariant: return pipe && launch_vt_if<V, ADJ, 8, 4, 8, 128, 16, 1>(a, s);
    default: return false;
  }
}

// whether CUDA-core variant `var` runs this launch as itself (else launch_variant declines it)
template <typename V>
bool variant_applies(const StageArgs<V>& a, int var) {
  const bool pipe = pipe_ok(a);
  if (var == 1) return true;
  if (var >= 2 && var <= 7) return pipe;
  if (var == 8) return a.b <= kVecMaxRhs;
  if (is_fp32_tile_variant(var))
    return pipe && std::is_same<V, float2>::value && ((var != 11 && var != 12 && var != kVtUncappedVariant) || a.tiles128);
  if (var == kSmallVariant) return small_ok(a);
  if (is_3m_variant(var)) return pipe && !std::is_same<V, float2>::value;
  return false;
}

// var: the tuned variant of this launch (0 = none): else the built-in choice by b
template <typename V, bool ADJ>
void launch_stage_dir(const StageArgs<V>& a, cudaStream_t s, int var) {
  if (var > 0 && launch_variant<V, ADJ>(a, s, var)) return;
  // many blocks of at most 16 x 16: a warp each (a 64-row tile leaves three quarters of its rows
  // idle); the same sums.  FP32 at b = 32: 4096 blocks 56 us in tiles, 18 so; 1024 blocks 20 and 12; 256
  // blocks 12 and 10; 28 x 28 blocks, up to 512 of them, 8 to 10 us in tiles, 14 to 18 so
  if (a.b >= 5 && a.xcs == 1 && a.R <= 16 && a.C <= 16 && a.nblk >= 1024 && launch_small<V, ADJ>(a, s)) return;
  if (a.b >= 5 && pipe_ok(a)) {
    // complex64 from 17 right-hand sides on: contiguous thread tiles (variant 9; 252 x 252 blocks,
    // b = 32: 0.109 ms a K-dot of 4 stages against 0.119), the same sums
    if (a.b > 16 && launch_vt_if<V, ADJ, 16, 2, 8, 128>(a, s)) return;
    if (a.b <= 8) launch_pipe<V, ADJ, 8, 1, 2>(a, s);
    else if (a.b <= 16) launch_pipe<V, ADJ, 16, 1, 4>(a, s);
    else launch_pipe<V, ADJ, 16, 2, 4>(a, s);
    return;
  }
  if (a.b <= kVecMaxRhs && launch_vec<V, ADJ>(a, s)) return;
  if (a.b <= 8) {  // also b <= 4 on blocks too wide for k_stage_vec's shared-memory gather
    launch_mm<V, ADJ, 8, 1, 2>(a, s);
  } else if (a.b <= 16) {
    launch_mm<V, ADJ, 16, 1, 4>(a, s);
  } else {
    launch_mm<V, ADJ, 16, 2, 4>(a, s);
  }
}

// stage arithmetic of the float2 path: 0 FP32 CUDA cores, or a k_stage_tc operand mode on the
// tensor cores (kTcTF32, kTcBF16, kTcX3 = split TF32); set for the duration of one public call
// (TcMode), read by launch_stage
thread_local int g_tc_mode = 0;
struct TcMode {
  int prev;
  explicit TcMode(int m) : prev(g_tc_mode) { g_tc_mode = m; }
  ~TcMode() { g_tc_mode = prev; }
};
inline int tc_mode_of(int prec) {
  return prec == FIO_PTF32 ? kTcTF32 : (prec == FIO_PBF16 ? kTcBF16 : (prec == FIO_PTF32X3 ? kTcX3 : 0));
}

template <bool ADJ, int MODE>
void launch_tc_dir(const TcArgs& a, int ncta, cudaStream_t s) {
  const int need = tc_smem_bytes(MODE, a.nmax, a.ncmax);
  smem_opt_in((const void*)k_stage_tc<ADJ, MODE>, need);
  dim3 grid((unsigned)ncta, (unsigned)((a.b + kTcMaxRhs - 1) / kTcMaxRhs));
  pdl_launch((long long)kTcRows * a.ncmax * a.b <= kLightMacs, k_stage_tc<ADJ, MODE>, grid, 128, need, s, a);
}

// the ring variant with S stages; false when its shared memory does not fit
template <bool ADJ, int MODE, int S>
bool launch_tc_ring(const TcArgs& a, int ncta, cudaStream_t s) {
  const int need = tc_ring_smem_bytes(MODE, a.nmax, a.ncmax, S);
  if (need > 227 * 1024) return false;
  if (!smem_opt_in((const void*)k_stage_tc_ring<ADJ, MODE, S>, need)) return false;
  dim3 grid((unsigned)ncta, (unsigned)((a.b + kTcMaxRhs - 1) / kTcMaxRhs));
  pdl_launch(false, k_stage_tc_ring<ADJ, MODE, S>, grid, 192, need, s, a);
  return true;
}

// tensor-core variants: 0 the single-buffer kernel, 20 + (S - 2) the ring kernel with S stages
template <bool ADJ, int MODE>
bool launch_tc_var(const TcArgs& a, int ncta, cudaStream_t s, int var) {
  switch (var) {
    case 0: launch_tc_dir<ADJ, MODE>(a, ncta, s); return true;
    case 20: return launch_tc_ring<ADJ, MODE, 2>(a, ncta, s);
    case 21: return launch_tc_ring<ADJ, MODE, 3>(a, ncta, s);
    case 22: return launch_tc_ring<ADJ, MODE, 4>(a, ncta, s);
    default: return false;
  }
}

// multiprocessor count of the current device (cached per thread for the last device: every stage launch asks)
int num_sms() {
  thread_local int last = -1, n = 1;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 1;
  }
  if (dev == last) return n;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
    cudaGetLastError();
    n = 1;
  }
  last = dev;
  return n;
}

// the TMA-fed persistent kernel (variant 30); false when it does not apply to this launch:
// x must be the row-major work layout with 16-byte aligned rows (b even), and the stage's tensor
// map must exist
bool launch_tma(const Stage& st, bool adj, const float2* x, long long xrs, long long xcs, float2* y, long long yrs,
                long long ycs, int b, cudaStream_t s, int var = kTmaVariant, int ksplit = 1, float2* part = nullptr,
                int gsel = -1) {
  const bool bf = g_tc_mode == kTcBF16;
  const int dir = adj ? 1 : 0;
  if (!st.tma_ok[dir][bf ? 1 : 0] || xcs != 1 || (xrs & 1) || (b & 1) || ((uintptr_t)x & 15) || b < 8) return false;
  TmaArgs a;
  a.rowidx = adj ? st.in : st.out;
  a.colidx = adj ? st.out : st.in;
  a.lrow = adj ? (int)st.C : (int)st.R;
  a.lcol = adj ? (int)st.R : (int)st.C;
  a.rows_per_blk = adj ? (int)st.C : (int)st.R;
  a.dims = st.dims;
  a.b = b;
  a.nmax = 2 * ((std::min(b, kTcMaxRhs) + 7) & ~7);
  // units of 4, 2 or 1 row tiles: G x nmax accumulator columns fit one of the two buffers
  a.nrhs_tiles = (b + kTcMaxRhs - 1) / kTcMaxRhs;
  // units of up to 4, 2 or 1 row tiles (G x nmax accumulator columns fit one of the two tensor
  // memory buffers): the largest G that still gives every SM about eight units, so that the
  // persistent CTAs' walk ends evenly, else single tiles
  const int gmax = a.nmax <= (int)tma::kBufCols / 4 ? 2 : (a.nmax <= (int)tma::kBufCols / 2 ? 1 : 0);
  int g = gmax;
  if (var == kTmaBalancedVariant)
    while (g > 0 && (long long)st.nunits[dir][g] * ksplit * a.nrhs_tiles < 8LL * num_sms()) --g;
  if (gsel >= 0) g = std::min(g, gsel);
  a.ksplit = ksplit;
  a.part = part;
  a.prow = (long long)st.nblk * a.rows_per_blk;
  a.units = st.units[dir][g];
  a.nunits = st.nunits[dir][g];
  a.x = x;
  a.xrs = xrs;
  a.y = y;
  a.yrs = yrs;
  a.ycs = ycs;
  if (!a.units) return false;
  const long long total = (long long)a.nunits * a.ksplit * a.nrhs_tiles;
  if (total == 0) return true;
  const int grid = (int)std::min<long long>(total, num_sms());
  // shared memory (227 KB, minus the kernel's static barriers): the deepest x staging (gathers
  // that miss L2 wait on HBM under the factor stream) that leaves at least six A slots, then as
  // many 16 KB A slots as fit (at least the split mode's tail ring of three)
  // split mode also keeps a tail ring: 3 slots, or 6 with variant 33 (a six-slot A ring otherwise)
  constexpr int kSmemMax = 227 * 1024 - 1024;
  const bool x3 = g_tc_mode == kTcX3;
  a.sl = x3 ? (var == kTmaShallowVariant ? 6 : 3) : 2;
  const int xs = tma::xslot_bytes(g_tc_mode, a.nmax);
  const int fixed = tma::smem_fixed(g_tc_mode, a.nmax) + (x3 ? a.sl * 16384 : 0);
  const int amax = (var == kTmaShallowVariant && !x3) ? 6 : tma::kMaxSA;
  a.sx = x3 ? 4 : tma::kMaxSX;
  while (a.sx > 3 && fixed + a.sx * xs + 6 * 16384 > kSmemMax) --a.sx;
  a.sa = std::min(amax, (kSmemMax - fixed - a.sx * xs) / 16384);
  if (a.sa < 3) return false;
  const int need = tma::smem_bytes(g_tc_mode, a.nmax, a.sa, a.sx, a.sl);
  const CUtensorMap& map = st.tmap[dir][bf ? 1 : 0];
  switch (g_tc_mode * 2 + dir) {
#define FIO_TMA_CASE(MODE, ADJ)                                                                   \
  case 2 * MODE + ADJ:                                                                            \
    if (!smem_opt_in((const void*)k_stage_tma<ADJ, MODE>, need)) return false;                   \
    pdl_launch(false, k_stage_tma<ADJ, MODE>, grid, tma::kThreads, need, s, a, map);                             \
    return true;
    FIO_TMA_CASE(kTcTF32, 0)
    FIO_TMA_CASE(kTcTF32, 1)
    FIO_TMA_CASE(kTcBF16, 0)
    FIO_TMA_CASE(kTcBF16, 1)
    FIO_TMA_CASE(kTcX3, 0)
    FIO_TMA_CASE(kTcX3, 1)
#undef FIO_TMA_CASE
    default: return false;
  }
}

// false when variant `var` does not apply (the caller then uses variant 0)
bool launch_tc(const Stage& st, bool adj, const float2* x, long long xrs, long long xcs, float2* y,
               long long yrs, long long ycs, int b, cudaStream_t s, int var) {
  const bool bf = g_tc_mode == kTcBF16;
  TcArgs a;
  if (!adj) {
    a.A = bf ? (const void*)st.Mbf : (const void*)st.M32;
    a.lda = bf ? st.ldbf : (int)st.C;
    a.bstride = (long long)st.R * a.lda;
  } else {
    a.A = bf ? (const void*)st.Mbft : (const void*)st.M32t;
    a.lda = bf ? st.ldbft : (int)st.R;
    a.bstride = (long long)st.C * a.lda;
  }
  a.rowidx = adj ? st.in : st.out;
  a.colidx = adj ? st.out : st.in;
  a.ldr = (int)st.R;
  a.ldc = (int)st.C;
  a.dims = st.dims;
  a.tiles = adj ? st.t128_adj : st.t128_fwd;
  const int ncta = adj ? st.n128_adj : st.n128_fwd;
  a.x = x;
  a.xrs = xrs;
  a.xcs = xcs;
  a.y = y;
  a.yrs = yrs;
  a.ycs = ycs;
  a.b = b;
  a.nmax = 2 * ((std::min(b, kTcMaxRhs) + 7) & ~7);
  a.stage_x = (xcs == 1 && xrs % 2 == 0 && b % 2 == 0 && ((uintptr_t)x & 15) == 0) ? 1 : 0;
  a.ncmax = adj ? (int)st.R : (int)st.C;  // gather list length per block (forward: in, adjoint: out)
  if (is_tma_variant(var)) return launch_tma(st, adj, x, xrs, xcs, y, yrs, ycs, b, s, var);
  if (ncta == 0) return true;
  switch (g_tc_mode * 2 + (adj ? 1 : 0)) {
    case 2 * kTcTF32: return launch_tc_var<false, kTcTF32>(a, ncta, s, var);
    case 2 * kTcTF32 + 1: return launch_tc_var<true, kTcTF32>(a, ncta, s, var);
    case 2 * kTcBF16: return launch_tc_var<false, kTcBF16>(a, ncta, s, var);
    case 2 * kTcBF16 + 1: return launch_tc_var<true, kTcBF16>(a, ncta, s, var);
    case 2 * kTcX3: return launch_tc_var<false, kTcX3>(a, ncta, s, var);
    default: return launch_tc_var<true, kTcX3>(a, ncta, s, var);
  }
}

template <typename V>
bool use_tc(const Stage& st, int b, bool adj) {
  return false;
}
// the tensor-core kernels copy operand rows in 16-byte pieces: the stage's A operand (forward: the
// complex64 or bf16 blocks, adjoint: their transposed copies) must have 16-byte aligned rows and
// base (the builder pads widths to even; a hand-packed odd width keeps the FP32 CUDA cores)
template <>
bool use_tc<float2>(const Stage& st, int b, bool adj) {
  if (g_tc_mode == 0 || b < 8 || st.M32t == nullptr) return false;
  if (g_tc_mode == kTcBF16) return true;  // bf16 rows padded to a multiple of 4 complex, 256-byte bases
  const void* A = adj ? (const void*)st.M32t : (const void*)st.M32;
  const uint32_t ld = adj ? st.R : st.C;
  return (ld & 1) == 0 && ((uintptr_t)A & 15) == 0;
}

template <typename V> constexpr int type_index();
template <> constexpr int type_index<double2>() { return 0; }
template <> constexpr int type_index<float2>() { return 1; }
template <> constexpr int type_index<dfc>() { return 2; }

// FIO_PDF running in FP64 (df_as_fp64): its choices are kept apart from FIO_P64's
thread_local bool g_for_df = false;
struct ForDf {
  bool prev;
  explicit ForDf(bool on) : prev(g_for_df) { g_for_df = on; }
  ~ForDf() { g_for_df = prev; }
};
template <typename V>
int var_table() { return std::is_same<V, double2>::value && g_for_df ? 6 : type_index<V>(); }

template <typename V>
StageArgs<V> stage_args(const Stage& st, bool adj, const V* x, long long xrs, long long xcs, V* y,
                        long long yrs, long long ycs, int b) {
  StageArgs<V> a;
  a.M = stage_M<V>(st);
  a.in = st.in;
  a.out = st.out;
  a.nblk = (int)st.nblk;
  a.R = (int)st.R;
  a.C = (int)st.C;
  a.x = x;
  a.xrs = xrs;
  a.xcs = xcs;
  a.y = y;
  a.yrs = yrs;
  a.ycs = ycs;
  a.b = b;
  a.ntiles = 1;
  a.dims = st.dims;
  a.tiles = adj ? st.tiles_adj : st.tiles_fwd;
  a.ntiles_list = adj ? st.ntiles_adj : st.ntiles_fwd;
  a.tiles128 = adj ? st.t128_adj : st.t128_fwd;
  a.ntiles128 = adj ? st.n128_adj : st.n128_fwd;
  return a;
}

// ---- fixed-point tensor-core kernel (fio_fx.cuh): variant 50, and the built-in choice of the
// stages it takes.  Its scratch is set for the duration of one public call (FxScratch); without
// one the CUDA-core kernels serve.
constexpr int kFxVariant = 50;
thread_local void* g_fx_scratch = nullptr;
thread_local size_t g_fx_bytes = 0;
thread_local bool g_fx_corrections = false;  // within fio_apply_correction
struct FxScratch {
  void* prev;
  size_t prev_bytes;
  FxScratch(void* p, size_t n) : prev(g_fx_scratch), prev_bytes(g_fx_bytes) {
    g_fx_scratch = p;
    g_fx_bytes = n;
  }
  ~FxScratch() {
    g_fx_scratch = prev;
    g_fx_bytes = prev_bytes;
  }
};
// whether the kernel can run this launch, and (pinned false) whether it is the built-in choice
template <typename V>
bool fx_rule(const Stage& st, bool adj, int b, bool pinned) {
  constexpr bool W = std::is_same<V, double2>::value;
  if (std::is_same<V, dfc>::value || !g_fx_scratch || (!W && g_tc_mode != 0 && !g_fx_corrections)) return false;
  // FP32 by the built-in rule in the solvers' split-TF32 corrections only.  Taken back for FP32 applies when
  // the factor's rows alone were scaled: 7.7e-6 off the FP64 apply on a real operator (generalized Radon
  // transform n = 256), lost in the HIF stages, against 1.4e-6 on the CUDA cores.  With column scales
  // 9.3e-7 (K-dot 1.9e-7 against 1.2e-6, G-dot 8.8e-7 against 7.3e-7; split TF32 3.2e-5)
  if (!W && !pinned && !g_fx_corrections) return false;
  return st.fx_ok[W ? 0 : 1] && (pinned || fx_takes(st, adj, W, b));
}
// device address of the timeout flag (the kernel is in another translation unit), cached per device
int* timeout_flag() {
  static std::mutex mu;
  static std::map<int, int*> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return nullptr;
  }
  std::lock_guard<std::mutex> lock(mu);
  int*& p = cache[dev];
  void* q = nullptr;
  if (!p && cudaGetSymbolAddress(&q, g_tc_timeout) == cudaSuccess) p = (int*)q;
  if (!p) cudaGetLastError();
  return p;
}
template <typename V>
bool launch_fx(const Stage& st, bool adj, const V* x, long long xrs, long long xcs, V* y, long long yrs, long long ycs,
               int b, cudaStream_t s, bool pinned) {
  if (!fx_rule<V>(st, adj, b, pinned)) return false;
  int* flag = timeout_flag();
  return flag && fx_launch(st, adj, std::is_same<V, double2>::value, x, xrs, xcs, y, yrs, ycs, b, g_fx_scratch, g_fx_bytes,
                           flag, s);
}

// a stage of a correction that was asked for in split TF32 (fio_apply_correction)
template <typename V>
bool launch_correction(const Stage& st, bool adj, const V* x, long long xrs, long long xcs, V* y, long long yrs, long long ycs,
                       int b, cudaStream_t s) {
  return g_fx_corrections && std::is_same<V, float2>::value && !st.x3_pinned[rhs_bucket(b)] &&
         launch_fx<V>(st, adj, x, xrs, xcs, y, yrs, ycs, b, s, false);
}

// Whether the tensor-core precision's own kernels run a stage.  In a correction not where nothing is tuned or
// pinned for split TF32: the FP32 CUDA cores are closer there, and faster than the untuned split-TF32 kernel
// (refinement 2D n = 128: b = 32 5.0 ms against 5.5, b = 8 3.3 against 4.8; tuned split TF32 4.8 and 2.9).
template <typename V>
bool tc_serves(const Stage& st, int b, bool adj) {
  return use_tc<V>(st, b, adj) && !(g_fx_corrections && st.var[2 + g_tc_mode][adj ? 1 : 0][rhs_bucket(b)] == 0);
}

template <typename V>
void launch_stage(const Stage& st, bool adj, const V* x, long long xrs, long long xcs, V* y,
                  long long yrs, long long ycs, int b, cudaStream_t s) {
  if (st.nblk == 0 || launch_correction<V>(st, adj, x, xrs, xcs, y, yrs, ycs, b, s)) return;
  if (tc_serves<V>(st, b, adj)) {
    const int tv = st.var[2 + g_tc_mode][adj ? 1 : 0][rhs_bucket(b)];
    if (tv != kFp32CoresVariant) {
      if (!launch_tc(st, adj, (const float2*)x, xrs, xcs, (float2*)y, yrs, ycs, b, s, tv))
        launch_tc(st, adj, (const float2*)x, xrs, xcs, (float2*)y, yrs, ycs, b, s, 0);
      return;
    }
  }
  const StageArgs<V> a = stage_args<V>(st, adj, x, xrs, xcs, y, yrs, ycs, b);
  int var = st.var[var_table<V>()][adj ? 1 : 0][rhs_bucket(b)];
  if ((var == 0 || var == kFxVariant) && launch_fx<V>(st, adj, x, xrs, xcs, y, yrs, ycs, b, s, var == kFxVariant)) return;
  if (st.kind == 1) var = four_product_of(var);  // in-place stages keep four products
  if (adj) launch_stage_dir<V, true>(a, s, var);
  else launch_stage_dir<V, false>(a, s, var);
}

// In-place stage split over K (variant 31 on the tensor cores): slices of every block's chunks as
// separate work units of the TMA kernel (enough of them to fill the GPU: the root and the top HIF
// levels have few, large blocks), partial sums into P, then k_partial_reduce adds the slices in a
// fixed order straight into W (the stage's copy-back).  False when it does not apply.
template <typename V>
bool inplace_split(const Stage&, bool, V*, V*, long long, int, int, cudaStream_t) {
  return false;
}
constexpr int kFp32SplitVariant = 12;

// the FP32 CUDA-core split (variant 12): 128-row tiles of 8 x 4 thread tiles, about two CTAs per
// SM slot, at least four 16-column chunks per slice
bool inplace_split_fp32(const Stage& st, bool adj, float2* W, float2* P, long long pcap, int b, int rs, cudaStream_t s) {
  StageArgs<float2> a = stage_args<float2>(st, adj, W, rs, 1, W, rs, 1, b);
  if (!pipe_ok(a) || !a.tiles128 || a.ntiles128 <= 0) return false;
  const long long prow = (long long)st.nblk * (adj ? st.C : st.R);
  if (prow <= 0 || prow > pcap) return false;
  const int dir = adj ? 1 : 0;
  const long long ctas = (long long)a.ntiles128 * ((b + 31) / 32);
  const int nch = (st.maxcols[dir] + 15) / 16;
  long long ks = (8LL * num_sms() + ctas - 1) / ctas;
  ks = std::min<long long>(ks, std::max(1, nch / 4));
  ks = std::min<long long>(ks, pcap / prow);
  a.ksplit = (int)std::max<long long>(1, std::min<long long>(ks, 64));
  a.part = P;
  a.prow = prow;
  const bool ok = adj ? launch_vt<true, 8, 4, 8, 128, 16>(a, s) : launch_vt<false, 8, 4, 8, 128, 16>(a, s);
  if (!ok) return false;
  const long long tot = prow * b;
  pdl_launch(true, k_partial_reduce, (unsigned)((tot + 255) / 256), 256, 0, s, P, a.ksplit, prow, b, st.out, W, rs);
  return true;
}

// Untuned, the split is the choice for the few large blocks of an operator above 4096 unknowns (the
// root and the top HIF levels): fewer 128-row tiles than a third of the SMs (2D n = 128, the root of
// 1346 rows at b = 32: FP32 0.125 ms whole, 0.035 split; split TF32 0.225 whole, 0.041 split; 64
// blocks of 390 rows keep the whole form, 0.067 against 0.083).
bool split_by_default(const Stage& st, bool adj, int b) {
  const int tiles = adj ? st.n128_adj : st.n128_fwd;
  return st.in_len > 4096 && b >= 17 && (long long)tiles * ((b + 31) / 32) * 3 < num_sms() &&
         std::max(st.maxcols[0], st.maxcols[1]) >= 128;
}

template <>
bool inplace_split<float2>(const Stage& st, bool adj, float2* W, float2* P, long long pcap, int b, int rs, cudaStream_t s) {
  if (!P) return false;
  const int bk = rhs_bucket(b), dir = adj ? 1 : 0;
  const bool tc = tc_serves<float2>(st, b, adj);
  const bool dflt = split_by_default(st, adj, b);
  if (!tc || st.var[2 + g_tc_mode][dir][bk] == kFp32CoresVariant) {
    const int v = st.var[1][dir][bk];
    return (v == kFp32SplitVariant || (v == 0 && dflt)) && inplace_split_fp32(st, adj, W, P, pcap, b, rs, s);
  }
  const int v = st.var[2 + g_tc_mode][dir][bk];
  if (v != kTmaSplitVariant && !(v == 0 && dflt)) return false;
  const long long prow = (long long)st.nblk * (adj ? st.C : st.R);
  const int units = st.nunits[dir][0];
  if (prow <= 0 || units <= 0 || prow > pcap) return false;
  const int kc = g_tc_mode == kTcBF16 ? 32 : 16;
  const int nch = (st.maxcols[dir] + kc - 1) / kc;
  // slices: about two units per SM, at least 4 chunks per slice, all slices fit in P
  int ks = (2 * num_sms() + units - 1) / units;
  ks = std::min<long long>(ks, std::max(1, nch / 4));
  ks = (int)std::min<long long>(ks, pcap / prow);
  ks = std::max(1, std::min(ks, 64));
  if (!launch_tma(st, adj, W, rs, 1, nullptr, 0, 0, b, s, kTmaVariant, ks, P, 0)) return false;
  const long long tot = prow * b;
  pdl_launch(true, k_partial_reduce, (unsigned)((tot + 255) / 256), 256, 0, s, P, ks, prow, b, st.out, W, rs);
  return true;
}

// Rows of a block up to which an in-place stage is written straight into the work vector: a block is
// then one row tile of every stage kernel, whose CTA (or warp) has read all of the block's entries of
// its right-hand sides before it writes any, and no other block reads them.  (Before, every HIF level
// computed into scratch and copied back: 9 more launches of 2.5 us each in the 27 of the direct solve
// at N = 1024.)
constexpr int kDirectRows = kTileRows;

// one INPLACE stage on the row-major work vector W (scratch S has the same shape; P, when not
// null, is free scratch of pcap rows for the split variant)
template <typename V>
void inplace_stage(const Stage& st, bool adj, V* W, V* S, int b, int rs, cudaStream_t s, V* P = nullptr,
                   long long pcap = 0) {
  if (st.nblk == 0) return;
  // the fixed-point kernel reads W in a launch of its own (the gather), so it may write W
  if (launch_correction<V>(st, adj, W, rs, 1, W, rs, 1, b, s) || inplace_split<V>(st, adj, W, P, pcap, b, rs, s)) {
    mark(s);
    return;
  }
  const int var = st.var[var_table<V>()][adj ? 1 : 0][rhs_bucket(b)];
  if ((var == 0 || var == kFxVariant) && launch_fx<V>(st, adj, W, rs, 1, W, rs, 1, b, s, var == kFxVariant)) {
    mark(s);
    return;
  }
  const bool direct = std::max(st.maxcols[0], st.maxcols[1]) <= kDirectRows;
  launch_stage<V>(st, adj, W, rs, 1, direct ? W : S, rs, 1, b, s);
  if (!direct) {
    const long long nidx = (long long)st.nblk * st.R;
    const long long tot = nidx * b;
    pdl_launch(true, k_scatter_back<V>, (unsigned)((tot + 255) / 256), 256, 0, s, st.out, nidx, S, W, b, rs);
  }
  mark(s);
}

template <typename V>
void to_row(const V* X, long long ld, V* W, long long N, int b, int rs, cudaStream_t s) {
  dim3 grid((unsigned)((N + 31) / 32), (unsigned)((b + 31) / 32));
  pdl_launch(true, k_col_to_row<V>, grid, dim3(32, 8), 0, s, X, ld, W, N, b, rs);
  mark(s);
}
template <typename V>
void to_col(const V* W, V* Y, long long ld, long long N, int b, int rs, cudaStream_t s) {
  dim3 grid((unsigned)((N + 31) / 32), (unsigned)((b + 31) / 32));
  pdl_launch(true, k_row_to_col<V>, grid, dim3(32, 8), 0, s, W, Y, ld, N, b, rs);
  mark(s);
}

// K-dot (adj = false) or K-dot* (adj = true): x (xrs, xcs) -> y (yrs, ycs); A, B ping-pong
template <typename V>
void bf_chain(fio_op op, bool adj, const V* x, long long xrs, long long xcs, V* y, long long yrs,
              long long ycs, int b, V* A, V* B, int rs, cudaStream_t s) {
  const int n = op->n_bf;
  const V* cur = x;
  long long crs = xrs, ccs = xcs;
  if (b >= 5 && xrs == 1 && n > 1) {
    // caller's column-major input -> row-major work array, so every stage streams whole rows
    to_row<V>(x, xcs, B, op->N, b, rs, s);
    cur = B;
    crs = rs;
    ccs = 1;
  }
  for (int k = 0; k < n; ++k) {
    const Stage& st = op->st[adj ? n - 1 - k : k];
    const bool last = k == n - 1;
    V* dst = last ? y : ((k & 1) ? B : A);
    const long long drs = last ? yrs : rs, dcs = last ? ycs : 1;
    launch_stage<V>(st, adj, cur, crs, ccs, dst, drs, dcs, b, s);
    mark(s);
    cur = dst;
    crs = drs;
    ccs = dcs;
  }
}

// G-dot on the row-major work vector W in place; S scratch; P (max_len rows) free scratch for the
// split in-place stages
template <typename V>
void g_sweep(fio_op op, V* W, V* S, int b, int rs, cudaStream_t s, V* P = nullptr) {
  const int h0 = op->n_bf, nh = op->n_hif;
  const long long pc = op->max_len;
  for (int t = 0; t < nh; ++t) inplace_stage<V>(op->st[h0 + t], false, W, S, b, rs, s, P, pc);
  for (int t = 0; t < op->n_root; ++t) inplace_stage<V>(op->st[h0 + nh + t], false, W, S, b, rs, s, P, pc);
  for (int t = nh - 1; t >= 0; --t) inplace_stage<V>(op->st[h0 + t], true, W, S, b, rs, s, P, pc);
}

int check_args(fio_op op, const void* x, const void* y, int64_t ld, int b, int dtype, int prec) {
  if (!op || b < 0) return FIO_EINVAL;
  if (b > 0 && (!x || !y || x == y)) return FIO_EINVAL;
  if (ld < op->N) return FIO_EINVAL;
  const bool c64prec = prec == FIO_P32 || is_tc_precision(prec);
  const bool c128prec = prec == FIO_P64 || prec == FIO_PDF;
  if (!((dtype == FIO_C128 && c128prec) || (dtype == FIO_C64 && c64prec))) return FIO_EINVAL;
  if (c64prec && !op->arena32) return FIO_EINVAL;
  if (prec == FIO_PDF && !op->arena_df) return FIO_EINVAL;
  if (is_tc_precision(prec) && !op->arena_tc) return FIO_EINVAL;
  const size_t es = dtype == FIO_C128 ? 16 : 8;
  const uint8_t *xb = (const uint8_t*)x, *yb = (const uint8_t*)y;
  const size_t span = ((size_t)ld * (b > 0 ? b - 1 : 0) + op->N) * es;
  if (b > 0 && xb < yb + span && yb < xb + span) return FIO_EINVAL;  // overlap
  return FIO_OK;
}

int finish(cudaStream_t) {
  const cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) return FIO_OK;
  if (getenv("FIO_DEBUG")) fprintf(stderr, "libfio: %s\n", cudaGetErrorString(e));
  return FIO_ECUDA;
}

enum Which { W_K = 0, W_KADJ = 1, W_G = 2, W_INV = 3 };

// the apply `w` from x to y (both column-major, leading dimension ld) with work arrays A, B, W
template <typename V>
void apply_core(fio_op op, Which w, const V* x, V* y, int64_t ld, int b, V* A, V* B, V* W, cudaStream_t s) {
  const int rs = row_stride<V>(b);
  switch (w) {
    case W_K: bf_chain<V>(op, false, x, 1, ld, y, 1, ld, b, A, B, rs, s); break;
    case W_KADJ: bf_chain<V>(op, true, x, 1, ld, y, 1, ld, b, A, B, rs, s); break;
    case W_G:
      to_row<V>(x, ld, W, op->N, b, rs, s);
      g_sweep<V>(op, W, A, b, rs, s, B);
      to_col<V>(W, y, ld, op->N, b, rs, s);
      break;
    case W_INV:
      bf_chain<V>(op, true, x, 1, ld, W, rs, 1, b, A, B, rs, s);
      g_sweep<V>(op, W, A, b, rs, s, B);
      to_col<V>(W, y, ld, op->N, b, rs, s);
      break;
  }
}

// whether a call may launch the fixed-point kernel, and takes its scratch
bool fx_may_run(fio_op op, int b, size_t elem) {
  if (elem != sizeof(float2) || g_fx_corrections) return true;
  for (const auto& st : op->st)
    for (int dir = 0; dir < 2; ++dir)
      if (st.var[1][dir][rhs_bucket(b)] == kFxVariant) return true;
  return false;
}

constexpr int kNoRoom = 1;  // FIO_PDF in FP64: no room for the fixed-point scratch (never returned to a caller)

template <typename V>
int apply_t(fio_op op, Which w, const void* xv, void* yv, int64_t ld, int b, cudaStream_t s) {
  void *bufs[5], *fxb = nullptr;
  size_t fxn = 0;
  int rc = fx_may_run(op, b, sizeof(V)) ? fio_scratch(op, b, sizeof(V), s, bufs, &fxb, &fxn) : fio_scratch(op, b, sizeof(V), s, bufs);
  if (rc) return rc;
  if (g_for_df && !fxb) return kNoRoom;
  FxScratch fxs(fxb, fxn);
  apply_core<V>(op, w, (const V*)xv, (V*)yv, ld, b, (V*)bufs[0], (V*)bufs[1], (V*)bufs[2], s);
  return finish(s);
}

// FIO_PDF: complex128 vectors in and out, every stage in double-float arithmetic; the vectors are
// split into double-floats on entry (work array X, leading dimension N) and summed back on exit
int apply_df(fio_op op, Which w, const void* xv, void* yv, int64_t ld, int b, cudaStream_t s) {
  void* bufs[5];
  int rc = fio_scratch(op, b, sizeof(dfc), s, bufs);
  if (rc) return rc;
  dfc *X = (dfc*)bufs[3], *Y = (dfc*)bufs[4];
  const long long n = op->N * (long long)b;
  const unsigned g = (unsigned)((n + 255) / 256);
  pdl_launch(true, k_c128_to_df, g, 256, 0, s, (const double2*)xv, ld, X, op->N, b);
  apply_core<dfc>(op, w, X, Y, op->N, b, (dfc*)bufs[0], (dfc*)bufs[1], (dfc*)bufs[2], s);
  pdl_launch(true, k_df_to_c128, g, 256, 0, s, Y, op->N, (double2*)yv, ld, b);
  return finish(s);
}

// Whether FIO_PDF runs as FIO_P64: when every stage has the fixed-point kernel's FP64 copy, that
// kernel is both faster than double-float arithmetic on the FP32 pipes (2D n = 256, K-dot at b = 16:
// 3.1 ms against 15) and more accurate (exact sums of 62-bit operands against 48-bit ones).  A
// double-float variant pinned by fio_set_variant keeps the double-float kernels, as does a call that
// has no room for the fixed-point scratch.
bool df_as_fp64(fio_op op, int b) {
  if (!fx_all_wide(op)) return false;
  const int k = rhs_bucket(b);
  for (const auto& st : op->st)
    if (st.var[2][0][k] || st.var[2][1][k]) return false;
  return true;
}

int apply_prec(fio_op op, Which w, const void* x, void* y, int64_t ld, int b, int prec, cudaStream_t s) {
  if (prec == FIO_P64) return apply_t<double2>(op, w, x, y, ld, b, s);
  if (prec == FIO_PDF && df_as_fp64(op, b)) {
    ForDf in_fp64(true);
    const int rc = apply_t<double2>(op, w, x, y, ld, b, s);
    if (rc != kNoRoom) return rc;
  }
  if (prec == FIO_PDF) return apply_df(op, w, x, y, ld, b, s);
  TcMode m(tc_mode_of(prec));
  return apply_t<float2>(op, w, x, y, ld, b, s);
}

int apply_any(fio_op op, Which w, const void* x, void* y, int64_t ld, int b, int dtype, int prec,
              void* stream) {
  int rc = check_args(op, x, y, ld, b, dtype, prec);
  if (rc) return rc;
  if ((w == W_G || w == W_INV) && op->n_root == 0) return FIO_ENOTSUP;
  if (b == 0) return FIO_OK;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaGetLastError() != cudaSuccess) return FIO_ECUDA;
  return apply_prec(op, w, x, y, ld, b, prec, s);
}

}  // namespace

// internal entry used by the solvers (same semantics as the public applies)
int fio_apply_internal(fio_op op, int which, const void* x, void* y, int64_t ld, int b, int prec,
                       cudaStream_t s) {
  if (b == 0) return FIO_OK;
  return apply_prec(op, (Which)which, x, y, ld, b, prec, s);
}

int fio_tc_timeout_reset() {
  int v = 0, zero = 0;
  if (cudaMemcpyFromSymbol(&v, g_tc_timeout, sizeof(int)) != cudaSuccess) return -1;
  if (v) cudaMemcpyToSymbol(g_tc_timeout, &zero, sizeof(int));
  return v;
}

int fio_apply_correction(fio_op op, int which, const void* x, void* y, int64_t ld, int b, cudaStream_t s) {
  g_fx_corrections = true;
  const int rc = fio_apply_internal(op, which, x, y, ld, b, FIO_PTF32X3, s);
  g_fx_corrections = false;
  return rc;
}

int fio_sync_flag(fio_op op, cudaStream_t s) {
  if (!op->flag_host) {
    if (cudaMallocHost(&op->flag_host, sizeof(int)) != cudaSuccess) {
      cudaGetLastError();
      op->flag_host = nullptr;
    }
  }
  if (!op->flag_host) return cudaStreamSynchronize(s) == cudaSuccess ? fio_tc_timeout_reset() : -1;
  if (cudaMemcpyFromSymbolAsync(op->flag_host, g_tc_timeout, sizeof(int), 0, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return -1;
  return *op->flag_host ? fio_tc_timeout_reset() : 0;
}

extern "C" int fio_apply_K(fio_op op, const void* x, void* y, int64_t ld, int b, int dtype,
                           int precision, void* stream) {
  return apply_any(op, W_K, x, y, ld, b, dtype, precision, stream);
}
extern "C" int fio_apply_Kadj(fio_op op, const void* x, void* y, int64_t ld, int b, int dtype,
                              int precision, void* stream) {
  return apply_any(op, W_KADJ, x, y, ld, b, dtype, precision, stream);
}
extern "C" int fio_apply_G(fio_op op, const void* x, void* y, int64_t ld, int b, int dtype,
                           int precision, void* stream) {
  return apply_any(op, W_G, x, y, ld, b, dtype, precision, stream);
}
extern "C" int fio_apply_inv(fio_op op, const void* u, void* f, int64_t ld, int b, int dtype,
                             int precision, void* stream) {
  return apply_any(op, W_INV, u, f, ld, b, dtype, precision, stream);
}

extern "C" int fio_apply_inv_host(fio_op op, const void* u_host, void* f_host, int64_t ld, int b,
                                  int dtype, int precision, void* stream) {
  if (!op || !u_host || !f_host || b < 0 || ld < op->N) return FIO_EINVAL;
  if (!((dtype == FIO_C128 && (precision == FIO_P64 || precision == FIO_PDF)) ||
        (dtype == FIO_C64 && (precision == FIO_P32 || is_tc_precision(precision)))))
    return FIO_EINVAL;
  if (is_tc_precision(precision) && !op->arena_tc) return FIO_EINVAL;
  if (precision == FIO_PDF && !op->arena_df) return FIO_EINVAL;
  if (op->n_root == 0) return FIO_ENOTSUP;
  if (b == 0) return FIO_OK;
  cudaStream_t s = (cudaStream_t)stream;
  const size_t es = dtype == FIO_C128 ? 16 : 8;
  void *bufs[5], *fxb;  // asked for with its scratch, so that the apply below does not grow it again
  int rc = fio_scratch(op, b, es, s, bufs, fx_may_run(op, b, es) ? &fxb : nullptr);
  if (rc) return rc;
  void *U = bufs[3], *F = bufs[4];
  const size_t w = (size_t)op->N * es;
  // one contiguous copy each way when the caller's columns are packed (ld == N)
  const cudaError_t e_in = ld == op->N
      ? cudaMemcpyAsync(U, u_host, w * (size_t)b, cudaMemcpyHostToDevice, s)
      : cudaMemcpy2DAsync(U, w, u_host, (size_t)ld * es, w, (size_t)b, cudaMemcpyHostToDevice, s);
  if (e_in != cudaSuccess) return FIO_ECUDA;
  rc = fio_apply_internal(op, W_INV, U, F, op->N, b, precision, s);
  if (rc) return rc;
  const cudaError_t e_out = ld == op->N
      ? cudaMemcpyAsync(f_host, F, w * (size_t)b, cudaMemcpyDeviceToHost, s)
      : cudaMemcpy2DAsync(f_host, (size_t)ld * es, F, w, w, (size_t)b, cudaMemcpyDeviceToHost, s);
  if (e_out != cudaSuccess) return FIO_ECUDA;
  // a tensor-core bounded wait that gave up left part of f unwritten: report it here, at the
  // call that produced the result, not at some later synchronising call
  const int to = fio_sync_flag(op, s);
  return to < 0 ? FIO_ECUDA : (to > 0 ? FIO_ETIMEOUT : FIO_OK);
}

extern "C" int fio_sync(void* stream) {
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) {
    cudaGetLastError();
    return FIO_ECUDA;
  }
  const int to = fio_tc_timeout_reset();
  return to < 0 ? FIO_ECUDA : (to > 0 ? FIO_ETIMEOUT : FIO_OK);
}

extern "C" int fio_launch_count(fio_op op, int which, int b, int* launches) {
  if (!op || !launches || which < 0 || which > 3) return FIO_EINVAL;
  int bfl = 0, gl = 0;
  for (int k = 0; k < op->n_bf; ++k) bfl += op->st[k].nblk ? 1 : 0;
  // an in-place stage is one launch per direction, and a copy-back (or reduction) for large blocks
  auto inplace = [&](int k) { return std::max(op->st[k].maxcols[0], op->st[k].maxcols[1]) <= kDirectRows ? 1 : 2; };
  for (int k = op->n_bf; k < op->n_bf + op->n_hif; ++k) gl += op->st[k].nblk ? 2 * inplace(k) : 0;
  for (int k = op->n_bf + op->n_hif; k < (int)op->st.size(); ++k) gl += op->st[k].nblk ? inplace(k) : 0;
  switch (which) {
    case 0:
    case 1: *launches = b ? bfl : 0; break;
    case 2: *launches = b ? gl + 2 : 0; break;
    case 3: *launches = b ? bfl + gl + 1 : 0; break;
  }
  return FIO_OK;
}

extern "C" int fio_apply_profiled(fio_op op, int which, const void* x, void* y, int64_t ld, int b,
                                  int dtype, int precision, void* stream, float* stage_ms, int cap,
                                  int* nmarks) {
  if (!stage_ms || cap <= 0 || !nmarks || which < 0 || which > 3) return FIO_EINVAL;
  int rc = check_args(op, x, y, ld, b, dtype, precision);
  if (rc) return rc;
  if ((which == 2 || which == 3) && op->n_root == 0) return FIO_ENOTSUP;
  if (b == 0) {
    *nmarks = 0;
    return FIO_OK;
  }
  cudaStream_t s = (cudaStream_t)stream;
  std::vector<cudaEvent_t> ev((size_t)cap + 1);
  for (auto& e : ev)
    if (cudaEventCreate(&e) != cudaSuccess) return FIO_ECUDA;
  Marks m{ev.data() + 1, cap, 0};
  cudaEventRecord(ev[0], s);
  g_marks = &m;
  rc = apply_prec(op, (Which)which, x, y, ld, b, precision, s);
  g_marks = nullptr;
  if (rc == FIO_OK) {
    const cudaError_t se = cudaStreamSynchronize(s);
    if (se != cudaSuccess) {
      if (getenv("FIO_DEBUG")) fprintf(stderr, "libfio: %s\n", cudaGetErrorString(se));
      rc = FIO_ECUDA;
    }
    for (int k = 0; rc == FIO_OK && k < m.n; ++k)
      if (cudaEventElapsedTime(&stage_ms[k], ev[k], ev[k + 1]) != cudaSuccess) rc = FIO_ECUDA;
    *nmarks = m.n;
    if (rc == FIO_OK && fio_tc_timeout_reset() > 0) rc = FIO_ETIMEOUT;
  }
  for (auto& e : ev) cudaEventDestroy(e);
  return rc;
}

// ---------------------------------------------------------------------------------------------
// fio_autotune: per-stage choice of the kernel variant by timing the candidates (see fio.h)
// ---------------------------------------------------------------------------------------------
namespace {

// L2 flush of the autotuner: a write larger than the 129 MB L2 before every timed launch, so that
// a stage is timed with its factor coming from HBM, as in an apply (where the stages before it
// have streamed the rest of the factors through L2); small stages would otherwise be timed on
// L2-resident data and the choice between close variants would follow a regime the apply never
// sees
constexpr size_t kTuneFlushBytes = 256ull << 20;
thread_local void* g_tune_flush = nullptr;  // set by fio_autotune for the duration of the call

// time a launcher (best of 3 after one warm-up): the launcher returns false when its variant does
// not apply (-1); -2 on a CUDA error
template <typename F>
float time_launch(F&& launch, cudaStream_t s, cudaEvent_t e0, cudaEvent_t e1) {
  if (!launch()) return -1.f;
  float best = -1.f;
  for (int rep = 0; rep < 3; ++rep) {
    if (g_tune_flush) cudaMemsetAsync(g_tune_flush, rep, kTuneFlushBytes, s);
    cudaEventRecord(e0, s);
    launch();
    cudaEventRecord(e1, s);
    float ms = 0.f;
    if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&ms, e0, e1) != cudaSuccess) return -2.f;
    if (best < 0.f || ms < best) best = ms;
  }
  return best;
}

constexpr int kTcCand[9] = {0,  20, 21, 22, kTmaVariant, kTmaSplitVariant, kTmaBalancedVariant, kTmaShallowVariant,
                            kFp32CoresVariant};

// tune every stage launch of one vector type at b right-hand sides; choices[] gets the variant
// per (stage, direction) in stage order, forward before adjoint
template <typename V>
int tune_type(fio_op op, int b, cudaStream_t s, int* choices, int cap, int* nch) {
  void *bufs[5], *fxb = nullptr;
  size_t fxn = 0;
  int rc = fio_scratch(op, b, sizeof(V), s, bufs, sizeof(V) == sizeof(float2) ? nullptr : &fxb, &fxn);
  if (rc) return rc;
  if (g_for_df && !fxb) return kNoRoom;
  FxScratch fxs(fxb, fxn);
  const int rs = row_stride<V>(b);
  const size_t bytes = (size_t)op->max_len * rs * sizeof(V);
  V* X = (V*)bufs[0];
  V* Y = (V*)bufs[1];
  if (cudaMemsetAsync(X, 0, bytes, s) != cudaSuccess || cudaMemsetAsync(Y, 0, bytes, s) != cudaSuccess)
    return FIO_ECUDA;
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess) return FIO_ECUDA;
  if (cudaEventCreate(&e1) != cudaSuccess) {
    cudaEventDestroy(e0);
    return FIO_ECUDA;
  }
  const int bucket = rhs_bucket(b);
  int n = 0;
  rc = FIO_OK;
  for (int si = 0; si < (int)op->st.size() && rc == FIO_OK; ++si) {
    Stage& st = op->st[si];
    const bool root = si >= op->n_bf + op->n_hif;
    for (int dir = 0; dir < (root ? 1 : 2) && rc == FIO_OK; ++dir) {
      const bool adj = dir == 1;
      const bool tc = use_tc<V>(st, b, adj);
      const int ti = tc ? 2 + g_tc_mode : var_table<V>();
      int best = 0;
      // FIO_PDF runs in FP64 for the fixed-point kernel, several times as fast as the CUDA-core tiles where its rule
      // takes the stage: against it only the warp kernel is timed there (16-point leaf stages at wide batches)
      const bool fx_or_small = g_for_df && fx_takes(st, adj, true, b);
      if (st.nblk > 0) {
        const StageArgs<V> a = stage_args<V>(st, adj, X, rs, 1, Y, rs, 1, b);
        float tbest = -1.f;
        const int ncand = tc ? 9 : kNCand + 1;
        for (int k = 0; k < ncand; ++k) {
          const int var = tc ? kTcCand[k] : (k == kNCand ? kFxVariant : kCand[bucket][k]);
          if ((var <= 0 && !tc) || (fx_or_small && var != kFxVariant && var != kSmallVariant)) continue;
          if (var == kFxVariant && (ti == 1 || !fx_rule<V>(st, adj, b, true))) continue;
          float t;
          if (st.kind == 1) {
            // in-place stages: the whole stage (compute and copy-back, or split compute and
            // reduction), so that the split variant is weighed with its reduction
            t = time_launch(
                [&] {
                  if (!tc && var != kFxVariant && (!variant_applies<V>(a, var) || is_3m_variant(var))) return false;
                  st.var[ti][dir][bucket] = (int8_t)var;
                  inplace_stage<V>(st, adj, X, Y, b, rs, s, (V*)bufs[2], op->max_len);
                  return true;
                },
                s, e0, e1);
          } else if (tc && var == kFp32CoresVariant) {
            // the FP32 CUDA-core launch with its own tuned (or built-in) tile shape
            t = time_launch(
                [&] {
                  if (adj) launch_stage_dir<V, true>(a, s, st.var[1][1][bucket]);
                  else launch_stage_dir<V, false>(a, s, st.var[1][0][bucket]);
                  return true;
                },
                s, e0, e1);
          } else if (tc) {
            t = time_launch([&] { return launch_tc(st, adj, (const float2*)X, rs, 1, (float2*)Y, rs, 1, b, s, var); },
                            s, e0, e1);
          } else if (var == kFxVariant) {
            t = time_launch([&] { return launch_fx<V>(st, adj, X, rs, 1, Y, rs, 1, b, s, true); }, s, e0, e1);
          } else if (adj) {
            t = time_launch([&] { return launch_variant<V, true>(a, s, var); }, s, e0, e1);
          } else {
            t = time_launch([&] { return launch_variant<V, false>(a, s, var); }, s, e0, e1);
          }
          if (t == -2.f || cudaGetLastError() != cudaSuccess) {
            rc = FIO_ECUDA;
            break;
          }
          if (t >= 0.f && (tbest < 0.f || t < tbest)) {
            tbest = t;
            best = var;
          }
        }
        if (rc == FIO_OK && (tc || best == kFxVariant) && fio_tc_timeout_reset() != 0) rc = FIO_ETIMEOUT;
      }
      st.var[ti][dir][bucket] = (int8_t)best;
      if (tc && g_tc_mode == kTcX3) st.x3_pinned[bucket] = false;
      if (choices && n < cap) choices[n] = best;
      ++n;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (nch) *nch = n;
  return rc;
}

}  // namespace

extern "C" int fio_set_variant(fio_op op, int b, int precision, int variant) {
  if (!op || b <= 0 || precision < FIO_P64 || precision > FIO_PDF) return FIO_EINVAL;
  const int bucket = rhs_bucket(b);
  const int mode = tc_mode_of(precision);
  const bool tc = mode != 0 && b >= 8;
  int ti;
  if (tc) {
    if (variant != 0 && (variant < 20 || variant > 22) && !is_tma_variant(variant) && variant != kFp32CoresVariant)
      return FIO_EINVAL;
    ti = 2 + mode;
  } else {
    ti = precision == FIO_P64 ? 0 : (precision == FIO_PDF ? 2 : 1);
    if (variant == kFxVariant && ti != 2) {
      // the fixed-point kernel where it takes the stage (also the built-in choice there)
    } else if (variant < 0 || variant > kMaxCudaCoreVariant || (variant == 8 && b > kVecMaxRhs) ||
        (is_fp32_tile_variant(variant) && ti != 1) || (variant == kSmallVariant && ti == 2) ||
        (is_3m_variant(variant) && ti == 1))
      return FIO_EINVAL;
  }
  for (auto& st : op->st) {
    st.var[ti][0][bucket] = st.var[ti][1][bucket] = (int8_t)variant;
    if (ti == 2) st.var[6][0][bucket] = st.var[6][1][bucket] = 0;
    if (tc && mode == kTcX3) st.x3_pinned[bucket] = variant != 0;
  }
  return FIO_OK;
}

extern "C" int fio_autotune(fio_op op, int b, int precision, void* stream, int* choices, int cap, int* nchoices) {
  if (!op || b < 0 || cap < 0 || (cap > 0 && !choices)) return FIO_EINVAL;
  if (precision < FIO_P64 || precision > FIO_PDF) return FIO_EINVAL;
  if (precision == FIO_P64 && !op->arena) return FIO_EINVAL;
  if ((precision == FIO_P32 || is_tc_precision(precision)) && !op->arena32) return FIO_EINVAL;
  if (is_tc_precision(precision) && !op->arena_tc) return FIO_EINVAL;
  if (precision == FIO_PDF && !op->arena_df) return FIO_EINVAL;
  if (nchoices) *nchoices = 0;
  if (b == 0) return FIO_OK;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaGetLastError() != cudaSuccess) return FIO_ECUDA;
  // the L2 flush target (without device memory for it, the launches are timed unflushed)
  void* flush = nullptr;
  if (cudaMalloc(&flush, kTuneFlushBytes) != cudaSuccess) {
    cudaGetLastError();
    flush = nullptr;
  }
  g_tune_flush = flush;
  int rc;
  if (precision == FIO_P64) {
    rc = tune_type<double2>(op, b, s, choices, cap, nchoices);
  } else if (precision == FIO_PDF) {
    rc = kNoRoom;
    if (df_as_fp64(op, b)) {
      ForDf in_fp64(true);
      rc = tune_type<double2>(op, b, s, choices, cap, nchoices);
    }
    if (rc == kNoRoom) rc = tune_type<dfc>(op, b, s, choices, cap, nchoices);
  } else {
    TcMode m(tc_mode_of(precision));
    rc = tune_type<float2>(op, b, s, choices, cap, nchoices);
  }
  g_tune_flush = nullptr;
  if (cudaStreamSynchronize(s) != cudaSuccess && rc == FIO_OK) rc = FIO_ECUDA;
  if (flush) cudaFree(flush);
  return rc;
}

// ---------------------------------------------------------------------------------------------
// fio_stage_errors: per-stage error of a precision against the FP64 path (see fio.h)
// ---------------------------------------------------------------------------------------------
namespace {

__device__ __forceinline__ double2 to_d2(double2 v) { return v; }
__device__ __forceinline__ double2 to_d2(float2 v) { return make_double2(v.x, v.y); }
__device__ __forceinline__ double2 to_d2(dfc v) { return make_double2((double)v.rh + v.rl, (double)v.ih + v.il); }

// acc[0] += sum |a - ref|^2, acc[1] += sum |ref|^2 over n values
template <typename V>
__global__ void k_diff_norm(const V* a, const double2* ref, long long n, double* acc) {
  double d = 0.0, r = 0.0;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const double2 u = to_d2(a[i]), v = ref[i];
    const double ex = u.x - v.x, ey = u.y - v.y;
    d += ex * ex + ey * ey;
    r += v.x * v.x + v.y * v.y;
  }
  for (int o = 16; o > 0; o >>= 1) {
    d += __shfl_xor_sync(0xffffffffu, d, o);
    r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&acc[0], d);
    atomicAdd(&acc[1], r);
  }
}

__global__ void k_to_c64(const double2* a, float2* b, long long n) {
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n) b[t] = make_float2((float)a[t].x, (float)a[t].y);
}
void convert_in(const double2* a, float2* b, long long n, cudaStream_t s) {
  k_to_c64<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, b, n);
}
void convert_in(const double2* a, double2* b, long long n, cudaStream_t s) {
  cudaMemcpyAsync(b, a, (size_t)n * sizeof(double2), cudaMemcpyDeviceToDevice, s);
}
void convert_in(const double2* a, dfc* b, long long n, cudaStream_t s) {
  k_split_df<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(a, b, (size_t)n);
}

template <typename V>
int stage_errors_t(fio_op op, int which, const void* x, int64_t ld, int b, cudaStream_t s, double* errs, int cap,
                   int* nerr) {
  const size_t len = (size_t)op->max_len * b;
  double2 *A64 = nullptr, *B64 = nullptr, *W64 = nullptr;
  V *A = nullptr, *B = nullptr, *W = nullptr;
  double* acc = nullptr;
  bool ok = cudaMalloc(&A64, len * sizeof(double2)) == cudaSuccess &&
            cudaMalloc(&B64, len * sizeof(double2)) == cudaSuccess &&
            cudaMalloc(&W64, len * sizeof(double2)) == cudaSuccess && cudaMalloc(&A, len * sizeof(V)) == cudaSuccess &&
            cudaMalloc(&B, len * sizeof(V)) == cudaSuccess && cudaMalloc(&W, len * sizeof(V)) == cudaSuccess &&
            cudaMalloc(&acc, 2 * sizeof(double)) == cudaSuccess;
  const size_t fxn = std::max(fx_scratch_bytes(op, b, sizeof(double2)), fx_scratch_bytes(op, b, sizeof(float2)));
  void* fxb = nullptr;
  if (ok && fxn && cudaMalloc(&fxb, fxn) != cudaSuccess) {  // no room: the CUDA cores serve
    cudaGetLastError();
    fxb = nullptr;
  }
  FxScratch fxs(fxb, fxn);
  int rc = ok ? FIO_OK : FIO_ENOMEM;
  int k = 0;
  auto record = [&](const double2* ref, const V* val, long long n) {
    if (rc) return;
    double h[2] = {0.0, 0.0};
    cudaMemsetAsync(acc, 0, 2 * sizeof(double), s);
    k_diff_norm<V><<<1024, 256, 0, s>>>(val, ref, n, acc);
    if (cudaMemcpyAsync(h, acc, sizeof(h), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess) {
      rc = FIO_ECUDA;
      return;
    }
    if (k < cap) errs[k] = h[1] > 0.0 ? sqrt(h[0] / h[1]) : sqrt(h[0]);
    ++k;
  };
  // the FP64 chain beside FIO_PDF in FP64 runs on the CUDA cores: not the kernel that is measured
  auto reference = [&](auto&& launch) {
    const bool other = std::is_same<V, double2>::value;
    ForDf plain(g_for_df && !other);
    FxScratch cores(other ? nullptr : g_fx_scratch, other ? 0 : g_fx_bytes);
    launch();
  };
  if (rc == FIO_OK) {
    const long long N = op->N;
    to_row<double2>((const double2*)x, ld, W64, N, b, b, s);  // both chains start from the same values
    convert_in(W64, W, N * b, s);
    if (which != 2) {
      const bool adj = which != 0;
      const double2* c64 = W64;
      const V* c = W;
      for (int kk = 0; kk < op->n_bf && rc == FIO_OK; ++kk) {
        const Stage& st = op->st[adj ? op->n_bf - 1 - kk : kk];
        double2* d64 = (kk & 1) ? B64 : A64;
        V* d = (kk & 1) ? B : A;
        reference([&] { launch_stage<double2>(st, adj, c64, b, 1, d64, b, 1, b, s); });
        launch_stage<V>(st, adj, c, b, 1, d, b, 1, b, s);
        record(d64, d, (adj ? st.in_len : st.out_len) * (long long)b);
        c64 = d64;
        c = d;
      }
      if (which == 3 && rc == FIO_OK && op->n_bf > 0) {
        cudaMemcpyAsync(W64, c64, (size_t)N * b * sizeof(double2), cudaMemcpyDeviceToDevice, s);
        cudaMemcpyAsync(W, c, (size_t)N * b * sizeof(V), cudaMemcpyDeviceToDevice, s);
      }
    }
    if (which >= 2) {
      const int h0 = op->n_bf, nh = op->n_hif;
      auto step = [&](const Stage& st, bool adj) {
        reference([&] { inplace_stage<double2>(st, adj, W64, A64, b, b, s); });
        inplace_stage<V>(st, adj, W, A, b, b, s, B, op->max_len);
        record(W64, W, N * b);
      };
      for (int t = 0; t < nh && rc == FIO_OK; ++t) step(op->st[h0 + t], false);
      for (int t = 0; t < op->n_root && rc == FIO_OK; ++t) step(op->st[h0 + nh + t], false);
      for (int t = nh - 1; t >= 0 && rc == FIO_OK; --t) step(op->st[h0 + t], true);
    }
    if (rc == FIO_OK && cudaGetLastError() != cudaSuccess) rc = FIO_ECUDA;
  }
  cudaStreamSynchronize(s);
  cudaFree(A64);
  cudaFree(B64);
  cudaFree(W64);
  cudaFree(A);
  cudaFree(B);
  cudaFree(W);
  cudaFree(acc);
  if (fxb) cudaFree(fxb);
  cudaGetLastError();
  if (nerr) *nerr = k;
  if (rc == FIO_OK && fio_tc_timeout_reset() > 0) rc = FIO_ETIMEOUT;
  return rc;
}

}  // namespace

extern "C" int fio_stage_errors(fio_op op, int which, const void* x, int64_t ld, int b, int precision, void* stream,
                                double* errs, int cap, int* nerr) {
  if (!op || !x || which < 0 || which > 3 || b <= 0 || ld < op->N || cap < 0 || (cap > 0 && !errs)) return FIO_EINVAL;
  if (precision == FIO_P64 || precision < FIO_P64 || precision > FIO_PDF) return FIO_EINVAL;
  if (precision == FIO_PDF ? !op->arena_df : !op->arena32) return FIO_EINVAL;
  if (is_tc_precision(precision) && !op->arena_tc) return FIO_EINVAL;
  if (which >= 2 && op->n_root == 0) return FIO_ENOTSUP;
  cudaStream_t s = (cudaStream_t)stream;
  if (cudaGetLastError() != cudaSuccess) return FIO_ECUDA;
  if (precision == FIO_PDF && df_as_fp64(op, b)) {
    ForDf in_fp64(true);
    return stage_errors_t<double2>(op, which, x, ld, b, s, errs, cap, nerr);
  }
  if (precision == FIO_PDF) return stage_errors_t<dfc>(op, which, x, ld, b, s, errs, cap, nerr);
  TcMode m(tc_mode_of(precision));
  return stage_errors_t<float2>(op, which, x, ld, b, s, errs, cap, nerr);
}

// ---------------------------------------------------------------------------------------------
// fio_apply_inv_noalloc: the direct solve with scratch in a static device array
// ---------------------------------------------------------------------------------------------
// For callers that must not allocate device memory during a solve (see fio.h).  The scratch is
// this file-scope array; every device that loads the library holds one copy until the process
// exits.  Host code must not use the array's name as a device address: its address on the
// current device comes from cudaGetSymbolAddress, taken once per device on the first call there.
static __device__ __align__(256) unsigned char g_noalloc_scratch[FIO_NOALLOC_SCRATCH_BYTES];
// the fixed-point kernel's scratch beside it: a gathered vector, at most 1.5 times a work vector but
// for blocks of a few columns (a stage that does not fit runs on the CUDA cores)
constexpr size_t kNoallocFxBytes = FIO_NOALLOC_SCRATCH_BYTES / 2;
static __device__ __align__(256) unsigned char g_noalloc_fx[kNoallocFxBytes];

namespace {
constexpr int kNoallocMaxDevices = 64;
void* g_noalloc_addr[kNoallocMaxDevices];
void* g_noalloc_fx_addr[kNoallocMaxDevices];
std::mutex g_noalloc_mu;

int noalloc_scratch(void** out, void** fx) {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return FIO_ECUDA;
  }
  if (dev < 0 || dev >= kNoallocMaxDevices) return FIO_EINVAL;
  std::lock_guard<std::mutex> lock(g_noalloc_mu);
  if (!g_noalloc_addr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p) {
      cudaGetLastError();
      return FIO_ECUDA;
    }
    void* q = nullptr;
    if (cudaGetSymbolAddress(&q, g_noalloc_fx) != cudaSuccess || !q) {
      cudaGetLastError();
      return FIO_ECUDA;
    }
    g_noalloc_addr[dev] = p;
    g_noalloc_fx_addr[dev] = q;
  }
  *out = g_noalloc_addr[dev];
  *fx = g_noalloc_fx_addr[dev];
  return FIO_OK;
}

template <typename V>
void inv_with_buffers(fio_op op, const V* u, V* f, int64_t ld, int b, int rs, V* A, V* B, V* W,
                      cudaStream_t s) {
  bf_chain<V>(op, true, u, 1, ld, W, rs, 1, b, A, B, rs, s);
  g_sweep<V>(op, W, A, b, rs, s, B);
  to_col<V>(W, f, ld, op->N, b, rs, s);
}
}  // namespace

extern "C" int fio_apply_inv_noalloc(fio_op op, const void* u, void* f, int64_t ld, int b,
                                     int dtype, int precision, void* stream) {
  int rc = check_args(op, u, f, ld, b, dtype, precision);
  if (rc) return rc;
  if (precision == FIO_PDF) return FIO_EINVAL;  // the static scratch serves P64, P32 and tensor cores
  if (op->n_root == 0) return FIO_ENOTSUP;
  if (b == 0) return FIO_OK;
  const size_t es = precision == FIO_P64 ? sizeof(double2) : sizeof(float2);
  auto per_of = [&](int rs) { return (((size_t)op->max_len * (size_t)rs * es) + 255) & ~(size_t)255; };
  if (per_of(b) > FIO_NOALLOC_SCRATCH_BYTES / 3) return FIO_EINVAL;  // does not fit the static scratch
  int rs = precision == FIO_P64 ? row_stride<double2>(b) : row_stride<float2>(b);
  if (per_of(rs) > FIO_NOALLOC_SCRATCH_BYTES / 3) rs = b;  // the padded rows do not: unpadded
  const size_t per = per_of(rs);
  void *base = nullptr, *fxb = nullptr;
  rc = noalloc_scratch(&base, &fxb);
  if (rc) return rc;
  FxScratch fxs(fxb, kNoallocFxBytes);
  if (cudaGetLastError() != cudaSuccess) return FIO_ECUDA;
  uint8_t* p = (uint8_t*)base;
  cudaStream_t s = (cudaStream_t)stream;
  // Nothing here needs clearing: every stage writes all of its outputs before a later stage
  // reads them, so contents left by an earlier call are never read.
  if (precision == FIO_P64) {
    inv_with_buffers<double2>(op, (const double2*)u, (double2*)f, ld, b, rs, (double2*)p,
                              (double2*)(p + per), (double2*)(p + 2 * per), s);
  } else {
    // the stage arithmetic of the complex64 path (FP32 CUDA cores or a tensor-core mode), as in
    // fio_apply_inv
    TcMode m(tc_mode_of(precision));
    inv_with_buffers<float2>(op, (const float2*)u, (float2*)f, ld, b, rs, (float2*)p,
                             (float2*)(p + per), (float2*)(p + 2 * per), s);
  }
  return finish(s);
}

// ---------------------------------------------------------------------------------------------
// fio_probe_fp32: measured FP32 FMA throughput of the device (the roofline of the CUDA-core path)
// ---------------------------------------------------------------------------------------------
namespace {
// every thread runs 8 independent FMA chains of `iters` steps (enough independent work to fill
// the FMA pipes: 8 chains x 8 warps per scheduler); the sum is stored so nothing is removed
__global__ void __launch_bounds__(256) k_fma_probe(float* out, int iters, float a, float b) {
  float x[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) x[k] = (float)(threadIdx.x + k) * 1e-3f;
  for (int i = 0; i < iters; ++i) {
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = fmaf(x[k], a, b);
  }
  float t = 0.f;
#pragma unroll
  for (int k = 0; k < 8; ++k) t += x[k];
  if (t == 12345.678f) out[blockIdx.x] = t;  // (practically) never taken, but not removable
}
}  // namespace

extern "C" int fio_probe_fp32(int iters, double* tflops, float* ms, int* sms, void* stream) {
  if (iters <= 0 || iters > (1 << 24) || !tflops) return FIO_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  const int nsm = num_sms();
  const int blocks = nsm * 8;  // 8 CTAs of 256 threads per SM: 64 warps, full occupancy
  float* d = nullptr;
  if (cudaMalloc(&d, sizeof(float) * blocks) != cudaSuccess) {
    cudaGetLastError();
    return FIO_ENOMEM;
  }
  cudaEvent_t e0, e1;
  int rc = FIO_OK;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) rc = FIO_ECUDA;
  float best = -1.f;
  for (int rep = 0; rc == FIO_OK && rep < 4; ++rep) {  // first launch warms up; best of the rest
    cudaEventRecord(e0, s);
    k_fma_probe<<<blocks, 256, 0, s>>>(d, iters, 0.999f, 1e-3f);
    cudaEventRecord(e1, s);
    float t = 0.f;
    if (cudaEventSynchronize(e1) != cudaSuccess || cudaEventElapsedTime(&t, e0, e1) != cudaSuccess) rc = FIO_ECUDA;
    if (rep > 0 && (best < 0.f || t < best)) best = t;
  }
  if (rc == FIO_OK) {
    *tflops = 2.0 * 8.0 * iters * 256.0 * blocks / (best * 1e-3) / 1e12;
    if (ms) *ms = best;
    if (sms) *sms = nsm;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  cudaFree(d);
  cudaGetLastError();
  return rc;
}

// ---------------------------------------------------------------------------------------------
// fio_selftest_wait: exercises the bounded-wait path of the tensor-core kernel (see fio.h)
// ---------------------------------------------------------------------------------------------
extern "C" int fio_selftest_wait(int limit_us, int nblocks, int* gave_up, void* stream) {
  if (limit_us <= 0 || limit_us > 1000000 || nblocks <= 0 || nblocks > 4096 || !gave_up) return FIO_EINVAL;
  cudaStream_t s = (cudaStream_t)stream;
  int* d = nullptr;
  if (cudaMalloc(&d, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return FIO_ENOMEM;
  }
  cudaMemsetAsync(d, 0, sizeof(int), s);
  k_wait_selftest<<<nblocks, 32, 0, s>>>((uint64_t)limit_us * 1000ull, d);
  int rc = FIO_OK;
  if (cudaGetLastError() != cudaSuccess ||
      cudaMemcpyAsync(gave_up, d, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    rc = FIO_ECUDA;
  cudaFree(d);
  if (rc == FIO_OK && fio_tc_timeout_reset() > 0 && *gave_up > 0) rc = FIO_ETIMEOUT;
  return rc;
}
