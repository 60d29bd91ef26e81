// fio_internal.h -- operator object shared by the translation units of libfio (not installed).
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <utility>
#include <vector>

#include "fio.h"

namespace fio {

struct dfc;  // double-float complex (fio_kernels.cuh)

// work unit of the fixed-point kernel (fio_fx.cuh): one 128-row tile of a block in one direction
struct FxUnit {
  int blk, r0, nrows, ncols;  // block, first row of the tile, valid rows and columns of the block
  int a64, a32;               // where its digits start in the FP64 / FP32 copy (128-byte rows)
  int x64, x32;               // columns before the block in the gathered vector
};

struct Stage {
  uint32_t kind, nblk, R, C;
  int64_t in_len, out_len;
  uint64_t offM, offIn, offOut;
  uint32_t level, role;
  const double2* M64 = nullptr;  // device, complex128 blocks (inside the arena)
  const float2* M32 = nullptr;   // device, complex64 copy (inside arena32)
  const dfc* Mdf = nullptr;      // device, double-float copy (inside arena_df)
  const int* in = nullptr;       // device
  const int* out = nullptr;      // device
  long long launch_rows;
  // per block: valid rows / columns (the padded tail of a block is never touched), and the CTA
  // work lists of 64-row tiles for the forward (over rows) and adjoint (over columns) directions
  const int2* dims = nullptr;      // device, nblk x (rows, cols)
  const int2* tiles_fwd = nullptr;  // device, (block, tile) pairs
  const int2* tiles_adj = nullptr;
  int ntiles_fwd = 0, ntiles_adj = 0;
  int maxcols[2] = {0, 0};  // longest valid gather list of a block: forward (cols), adjoint (rows)
  // tensor-core copies (FIO_MASK_TC): block-transposed complex64 (C x R per block), bf16 in both
  // orientations with row strides padded to a multiple of 4; 128-row tile lists
  const float2* M32t = nullptr;
  const __nv_bfloat162* Mbf = nullptr;
  const __nv_bfloat162* Mbft = nullptr;
  int ldbf = 0, ldbft = 0;
  const int2* t128_fwd = nullptr;
  const int2* t128_adj = nullptr;
  int n128_fwd = 0, n128_adj = 0;
  // kernel variant chosen by fio_autotune per [arithmetic: c128, c64, double-float, TF32, BF16,
  // split TF32, c128 on behalf of FIO_PDF][direction: forward, adjoint][right-hand-side bucket]; 0 = the
  // built-in choice (see fio_capi.cu)
  bool x3_pinned[5] = {};  // per bucket: the split-TF32 variant was set by fio_set_variant, not by the autotuner
  int8_t var[7][2][5] = {};
  // TMA tensor maps of the tensor-core A operands per [direction: forward (M32 / Mbf), adjoint
  // (M32t / Mbft)][element: FP32, BF16]; tma_ok marks the maps that encoded (16-byte aligned
  // rows and base)
  CUtensorMap tmap[2][2];
  bool tma_ok[2][2] = {};
  // work units of the TMA kernel per [direction][at most 1, 2, 4 row tiles per unit]: (block,
  // first 128-row tile, tiles, 0), largest first
  const int4* units[2][3] = {};
  int nunits[2][3] = {};
  // fixed-point kernel per [forward, adjoint]: scale exponents of the product's rows and columns, work units,
  // column offsets of the blocks in the gathered vector and its columns, and the digit copies of
  // the factor per [FP64, FP32][direction]; fx_ok: the copies exist and every exponent is in range
  bool fx_ok[2] = {};
  const short *fx_exp[2] = {}, *fx_cexp[2] = {};
  const int2* fx_list[2] = {};  // rows gathered and their columns' scale exponents
  const FxUnit* fx_units[2] = {};
  int n_fx_units[2] = {};
  const int2* fx_xofs[2] = {};
  int2 fx_cols[2] = {};
  long long fx_steps[2] = {0, 0};  // K steps (8 columns) of all units
  long long nnz = 0;               // block entries, padding excluded
  const uint8_t* fxA[2][2] = {};
};

}  // namespace fio

struct fio_op_s {
  int d = 0;
  int64_t n = 0, N = 0;
  int n_bf = 0, n_hif = 0, n_root = 0;
  unsigned mask = 0;
  int64_t max_len = 0;            // longest vector between two stages (>= N)
  std::vector<fio::Stage> st;     // butterfly stages, HIF stages, root
  void* arena = nullptr;          // device copy of the packed buffer
  size_t arena_bytes = 0;
  void* arena32 = nullptr;        // complex64 copies of every stage's blocks
  size_t arena32_bytes = 0;
  void* scratch = nullptr;        // 5 work arrays of max_len x b (grown on demand)
  size_t scratch_bytes = 0;
  void* arena_tc = nullptr;       // tensor-core copies of every stage's blocks
  size_t arena_tc_bytes = 0;
  void* arena_df = nullptr;       // double-float copies of every stage's blocks
  size_t arena_df_bytes = 0;
  void* meta = nullptr;           // per-block dims and tile lists of every stage
  size_t meta_bytes = 0;
  void* units = nullptr;          // work-unit lists of the TMA kernel (every stage)
  size_t units_bytes = 0;
  void* fx = nullptr;             // digit copies, scale exponents and work units of the fixed-point kernel
  size_t fx_bytes = 0;
  long long fx_max_cols[2] = {0, 0};  // most columns of a gathered vector (FP64, FP32 chunking)
  long long fx_max_blk = 0;           // most blocks of a stage it takes
  void* fx_scratch = nullptr;         // its scratch, apart from the pool: a call runs without it where it has no room
  size_t fx_scratch_bytes = 0;
  void* fft_tw = nullptr;         // DFT twiddles: exp(2 pi i k / 2048), 2048 double2 then 2048 float2
  size_t fft_bytes = 0;
  void* solver = nullptr;         // solver work arrays (fio_solve.cu)
  size_t solver_bytes = 0;
  int* flag_host = nullptr;       // pinned copy of the timeout flag (fio_sync_flag)
  void* solver_host = nullptr;    // pinned scalars that the solver's kernels write and the host reads
  size_t solver_host_bytes = 0;
};

// Kernels of an apply or a solve are launched with programmatic stream serialisation where `early`:
// such a kernel may be scheduled once all CTAs of the kernel before it have started (pdl_go in that
// kernel), sets itself up and loads what no kernel of the chain writes (factors, index lists), and
// waits in pdl_wait, before its first access to a vector, until the kernel before it has completed.
// Every kernel that is ever launched so calls pdl_wait in all of its CTAs, or a kernel behind it could
// overtake the one before.  A chain of small launches is then as long as its dependent loads instead
// of its launch latencies (direct solve at N = 1024, b = 1, 18 launches: 91 us without, 46 with).
// Not `early`: a kernel of heavy CTAs that do not fill the chip several times over.  Started early, they
// pile up on the multiprocessors that the kernel before frees first (2D n = 128 FP32 b = 32, 288
// CTAs a stage: 440 us without, 530 with).
template <typename... P, typename... A>
inline void pdl_launch(bool early, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c = {};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = at;
  c.numAttrs = early ? 1 : 0;
  cudaLaunchKernelEx(&c, kernel, std::forward<A>(args)...);  // errors are found by the caller's cudaGetLastError
}
#ifdef __CUDACC__
namespace fio {
__device__ __forceinline__ void pdl_go() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
}  // namespace fio
#endif

// precisions whose stage products may run on the tensor cores (complex64 vectors)
inline bool is_tc_precision(int p) { return p == FIO_PTF32 || p == FIO_PBF16 || p == FIO_PTF32X3; }

// fixed-point tensor-core stage kernel (fio_fx.cu): its copies at upload (synchronises s); the
// scratch that its launches need for b right-hand sides of `elem` bytes; whether it takes a stage
// launch; the launch (false: not taken, nothing launched; *timeout is set by a bounded wait that gives up)
int fx_build(fio_op op, const std::vector<int2>& meta, const std::vector<size_t>& mdims, cudaStream_t s);
size_t fx_scratch_bytes(fio_op op, int b, size_t elem);
bool fx_takes(const fio::Stage& st, bool adj, bool wide, int b);
int fft_build(fio_op op, cudaStream_t s);  // the DFT's twiddle table (fio_fft.cu)
bool fx_all_wide(fio_op op);  // every stage of the operator has an FP64 digit copy
bool fx_launch(const fio::Stage& st, bool adj, bool wide, const void* x, long long xrs, long long xcs, void* y,
               long long yrs, long long ycs, int b, void* scratch, size_t scratch_bytes, int* timeout, cudaStream_t s);

// scratch work arrays (5 of max_len x b elements of `elem` bytes); grows with a stream sync;
// fxbuf (may be null) receives the fixed-point kernel's scratch, or null where there is no room, fxbytes its size
int fio_scratch(fio_op op, int b, size_t elem, cudaStream_t s, void** bufs, void** fxbuf = nullptr,
                size_t* fxbytes = nullptr);
// which: 0 K-dot, 1 K-dot*, 2 G-dot, 3 G-dot K-dot*; x, y column-major with leading dimension ld
int fio_apply_internal(fio_op op, int which, const void* x, void* y, int64_t ld, int b, int prec,
                       cudaStream_t s);
// the same for a correction asked for in split TF32: stages with work enough in 30-bit fixed point (closer
// than split TF32, and faster) unless a variant is pinned for split TF32, the others in what is tuned or pinned
// for split TF32, or else on the FP32 CUDA cores
int fio_apply_correction(fio_op op, int which, const void* x, void* y, int64_t ld, int b, cudaStream_t s);
void fio_solver_free(fio_op op);
// 1 when a tensor-core kernel's bounded wait gave up since the last call (and clear the flag),
// 0 otherwise, -1 on a CUDA error
int fio_tc_timeout_reset();
// synchronise s with the flag read back in the same wait (a copy of its own takes 8 us); as above
int fio_sync_flag(fio_op op, cudaStream_t s);
