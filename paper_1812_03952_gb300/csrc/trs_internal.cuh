// Internal declarations of libtrs (not part of the C ABI).
//
// Block matrices live in an "ELL-7 + tail" layout:
//   * the first nc rows are cells of an nx*ny*nz grid; their couplings to the
//     six 7-point neighbours and to themselves sit in seven slots ordered by
//     ascending column (-z, -y, -x, self, +x, +y, +z), stored structure-of-
//     arrays: ell[(slot * bb + e) * nc + row], e = r*b + c of the b x b block.
//     Columns are implicit (row + kSlotOff[slot]); emask[row] bit s says
//     whether slot s is stored (the caller's pattern), so coalesced
//     row-parallel loads need no column indices.
//   * every other block (well columns of perforated cells, all blocks of the
//     well rows, everything for unstructured matrices) is in a block-CSR tail
//     over all rows: tptr[n_rows+1], tcol[ntail], tval[t * bb + e].
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <mutex>
#include <stdexcept>
#include <string>
#include <tuple>
#include <utility>
#include <vector>

#include "../../include/trs.h"

namespace trs {

constexpr int kMaxB = 5;
constexpr int kSlots = 7;
constexpr int kSelf = 3;
// Bit 7 of a cell's slot mask (emask) and of a position's lower mask
// (lmask): the row also has entries in the tail, so that rows without any
// (almost all cells) never read their tail pointers.
constexpr unsigned kTailBit = 0x80u;
// Block ILU(1) keeps the level-1 fill of a cell row that falls on one of the
// 18 cells two 7-point steps away in fill slots next to the 7 stencil slots:
// (dx, dy, dz) of fill slot s, ordered by (dz, dy, dx).
constexpr int kFill = 18;
constexpr int kFillD[kFill][3] = {{0, 0, -2}, {0, -1, -1}, {-1, 0, -1}, {1, 0, -1}, {0, 1, -1}, {0, -2, 0},
                                  {-1, -1, 0}, {1, -1, 0}, {-2, 0, 0}, {2, 0, 0}, {-1, 1, 0}, {1, 1, 0},
                                  {0, 2, 0}, {0, -1, 1}, {-1, 0, 1}, {1, 0, 1}, {0, 1, 1}, {0, 0, 2}};
constexpr int kMaxLevels = 16;
constexpr int kDenseMax = 4096;
constexpr int kMaxColours = 64;
constexpr int kMaxRestart = 64;

struct Error : std::runtime_error {
  trs_status code;
  Error(trs_status c, const std::string &m) : std::runtime_error(m), code(c) {}
};

#define TRS_CUDA(call)                                                                         \
  do {                                                                                         \
    cudaError_t e_ = (call);                                                                   \
    if (e_ != cudaSuccess)                                                                     \
      throw ::trs::Error(e_ == cudaErrorMemoryAllocation ? TRS_ERR_OOM : TRS_ERR_CUDA,         \
                         std::string(#call) + ": " + cudaGetErrorString(e_));                  \
  } while (0)
// Every kernel launch is followed by TRS_LAUNCHED(), which checks the launch
// and counts it (trs_kernel_launches()).
void note_launch();
#define TRS_LAUNCHED()                                                                         \
  do {                                                                                         \
    ::trs::note_launch();                                                                      \
    TRS_CUDA(cudaGetLastError());                                                              \
  } while (0)
#define TRS_REQUIRE(cond, code, msg)                                                           \
  do {                                                                                         \
    if (!(cond)) throw ::trs::Error((code), (msg));                                            \
  } while (0)

// Owning device buffer (move-only).
template <class T>
struct DBuf {
  T *p = nullptr;
  size_t n = 0;
  DBuf() = default;
  explicit DBuf(size_t count) { alloc(count); }
  DBuf(const DBuf &) = delete;
  DBuf &operator=(const DBuf &) = delete;
  DBuf(DBuf &&o) noexcept : p(o.p), n(o.n) { o.p = nullptr; o.n = 0; }
  DBuf &operator=(DBuf &&o) noexcept {
    if (this != &o) { release(); p = o.p; n = o.n; o.p = nullptr; o.n = 0; }
    return *this;
  }
  ~DBuf() { release(); }
  void alloc(size_t count) {
    release();
    n = count;
    if (count) TRS_CUDA(cudaMalloc(reinterpret_cast<void **>(&p), count * sizeof(T)));
  }
  void release() {
    if (p) cudaFree(p);
    p = nullptr;
    n = 0;
  }
  void upload(const T *h, size_t count, cudaStream_t s) {
    if (count) TRS_CUDA(cudaMemcpyAsync(p, h, count * sizeof(T), cudaMemcpyHostToDevice, s));
  }
  void zero(cudaStream_t s) {
    if (n) TRS_CUDA(cudaMemsetAsync(p, 0, n * sizeof(T), s));
  }
  T *get() const { return p; }
};

// Stream-ordered temporary device buffer (cudaMallocAsync / cudaFreeAsync on
// the stream that uses it): no device-wide synchronisation on free.
template <class T>
struct TBuf {
  T *p = nullptr;
  size_t n = 0;
  cudaStream_t s = nullptr;
  TBuf(size_t count, cudaStream_t st) : n(count), s(st) {
    if (count) TRS_CUDA(cudaMallocAsync(reinterpret_cast<void **>(&p), count * sizeof(T), s));
  }
  TBuf(const TBuf &) = delete;
  TBuf &operator=(const TBuf &) = delete;
  ~TBuf() {
    if (p) cudaFreeAsync(p, s);
  }
  void zero() {
    if (n) TRS_CUDA(cudaMemsetAsync(p, 0, n * sizeof(T), s));
  }
};

// Page-locked host memory that kernels write directly: a result the host waits
// for needs no copy after the kernel.
template <class T>
struct HBuf {
  T *p = nullptr;
  HBuf() = default;
  HBuf(const HBuf &) = delete;
  HBuf &operator=(const HBuf &) = delete;
  ~HBuf() {
    if (p) cudaFreeHost(p);
  }
  void alloc(size_t count) {
    if (!p) TRS_CUDA(cudaHostAlloc(reinterpret_cast<void **>(&p), count * sizeof(T), cudaHostAllocMapped));
  }
};

// Keeps freed stream-ordered memory in the current device's pool.
void keep_pool_memory();

template <class T>
std::vector<T> download(const T *d, size_t count, cudaStream_t s) {
  std::vector<T> h(count);
  if (count) {
    TRS_CUDA(cudaMemcpyAsync(h.data(), d, count * sizeof(T), cudaMemcpyDeviceToHost, s));
    TRS_CUDA(cudaStreamSynchronize(s));
  }
  return h;
}

// Geometry of the structured part.
// Programmatic dependent launch (sm_90 and later): every kernel of the library
// is launched with programmatic stream serialisation, so that the next kernel
// in the stream is scheduled while this one drains instead of after it.  Each
// kernel waits (griddepcontrol.wait: the previous grid complete and its memory
// visible) before it touches anything that a kernel still in flight may write or
// read; which kernels read what before that, and why they may, stands at
// pdl_enter below.
template <class... KArgs, class... Args>
void launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args &&...args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  TRS_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(std::forward<Args>(args))...));
}

// Sets an attribute of a kernel, once per kernel, attribute and device.
template <class... KArgs>
void set_attribute(void (*kernel)(KArgs...), cudaFuncAttribute attr, int value) {
  static std::mutex mu;
  static std::vector<std::tuple<const void *, int, int>> done;
  int dev = 0;
  TRS_CUDA(cudaGetDevice(&dev));
  const std::tuple<const void *, int, int> key{reinterpret_cast<const void *>(kernel), (int)attr, dev};
  std::lock_guard<std::mutex> lock(mu);
  for (auto &e : done)
    if (e == key) return;
  TRS_CUDA(cudaFuncSetAttribute(kernel, attr, value));
  done.push_back(key);
}

__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" :::); }

// Most kernels touch no memory before the wait, and let the next one start after
// it: stream order holds for all that they do.
__device__ __forceinline__ void pdl_enter() {
  pdl_wait();
  pdl_trigger();
}
// The kernels of the preconditioner's application first read what no kernel of a
// solve writes (pattern, factors, level operators, D^-1: complete and synchronised
// with the host when the setup returns), and only then wait and touch the vectors;
// in FP32, and on large FP64 levels, they also trigger before that.  Such a kernel
// may be resident before its predecessor's predecessor has finished, but passes
// its wait only when its predecessor, which waited in its turn, is complete.  So
// whatever a new kernel writes for them has to be synchronised with the host, or
// at least two waits away.  k_ilu_factor_star alone writes before its wait: slots
// of its own rows that no kernel queued with it reads.

// Relative-permeability tables of the thermal model, passed by value.
constexpr int kThermalTableMax = 32;
struct ThermalTables {
  int nswt, nslt;
  double swt[3 * kThermalTableMax];   // S_w, k_rw, k_row
  double slt[3 * kThermalTableMax];   // S_l, k_rg, k_rog
  // per segment i, the slopes (y_{i+1} - y_i) / (x_{i+1} - x_i) of columns 1, 2
  double swt_slope[2 * kThermalTableMax];
  double slt_slope[2 * kThermalTableMax];
};

struct Geom {
  int64_t nc;       // cells
  int64_t n_rows;   // cells + other rows
  int64_t off[kSlots];
  int64_t off2[kFill];   // index offsets of the fill slots
  int nx, ny, nz;
};

inline Geom make_geom(int nx, int ny, int nz, int64_t n_rows) {
  Geom g;
  g.nx = nx; g.ny = ny; g.nz = nz;
  g.nc = (int64_t)nx * ny * nz;
  g.n_rows = n_rows;
  const int64_t sxy = (int64_t)nx * ny;
  int64_t o[kSlots] = {-sxy, -(int64_t)nx, -1, 0, 1, nx, sxy};
  for (int s = 0; s < kSlots; s++) g.off[s] = o[s];
  for (int s = 0; s < kFill; s++) g.off2[s] = kFillD[s][0] + kFillD[s][1] * (int64_t)nx + kFillD[s][2] * sxy;
  return g;
}

// Device view of a block (or scalar, bb = 1) matrix in ELL-7 + tail form.
template <class T>
struct MatView {
  Geom g;
  const uint8_t *emask;   // [nc]
  const int64_t *tptr;    // [n_rows + 1]
  const int32_t *tcol;    // [ntail]
  const T *ell;           // [7][bb][nc] (the decoupled matrix Ã: [7][nc][bb], blocks contiguous)
  const T *tval;          // [ntail][bb]
};

}  // namespace trs

// The handles of the C ABI.
struct trs_bsr {
  int b = 0;
  int64_t n = 0, nnzb = 0, ntail = 0;
  trs::Geom g{};
  bool structured = false;
  bool cell_tail = false;     // some cell is coupled to another outside its 7-point star
  trs::DBuf<uint8_t> emask;
  trs::DBuf<int64_t> tptr;
  trs::DBuf<int32_t> tcol;
  trs::DBuf<double> ell, tval;
  trs::DBuf<int64_t> tdiag;   // [n - nc] tail index of the diagonal block of each non-cell row
  // canonical BSR order: internal location of each block, row and column
  trs::DBuf<int64_t> map;
  trs::DBuf<int32_t> urow, ucol;
  std::vector<int64_t> h_rp;
  std::vector<int32_t> h_col;
  // for a matrix made by trs_bsr_transpose: canonical index in the source of
  // each canonical block (refresh with trs_bsr_transpose_values)
  trs::DBuf<int64_t> tsrc;
  trs::DBuf<int64_t> ttail;   // canonical index of each tail entry, in tail order
  // tail entries grouped by column (for the transposed product)
  trs::DBuf<int64_t> tc_ptr, tc_src;
  trs::DBuf<int32_t> tc_row;
  // synthetic assembly bookkeeping
  bool synthetic = false;
  int n_wells = 0;
  int64_t n_perf = 0;
  trs::DBuf<int64_t> cperf_ptr, cperf_idx, wperf_ptr, wperf_idx;   // perforations by cell / well
  trs::DBuf<int32_t> perf_cell, perf_well;
  trs::DBuf<int64_t> perf_cw, perf_wc, wdiag;                      // tail slots of (c,w), (w,c), (w,w)
  trs::DBuf<double> host_stage;   // device copy of host assembly inputs (trs_bsr_assemble_host)
  trs::DBuf<double> thermal_props;  // per-cell thermal properties with derivatives (trs_thermal_assemble)

  template <class T = double>
  trs::MatView<T> view() const {
    return trs::MatView<T>{g, emask.p, tptr.p, tcol.p, ell.p, tval.p};
  }
};
