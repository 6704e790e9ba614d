// Internal interfaces between the C-ABI layer (lbpc_api.cu) and the kernel files.
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>

#include <nvtx3/nvToolsExt.h>

#include "lbpc_device.cuh"

namespace lbpc {

// NVTX range over a host call of the library (NVTX v3 is header-only: without an attached profiler a
// range costs a check of a null function pointer). Profilers show and filter by these names.
struct TraceRange {
  explicit TraceRange(const char* name) { nvtxRangePushA(name); }
  ~TraceRange() { nvtxRangePop(); }
  TraceRange(const TraceRange&) = delete;
  TraceRange& operator=(const TraceRange&) = delete;
};

// Launch with programmatic stream serialization: the kernel is set up while the one before it on the stream
// ends. Every kernel launched so calls pdl_wait() first, which waits for the completion of everything before it
// on the stream. Ordinary launches leave about 2.5 us between dependent kernels on GB300, in steps of 2.05 us
// (chains of small kernels, 152 CTAs: 4.1 us each; 1.4 us launched this way), as much as the kernels of a small
// grid take. No kernel lets its successor start early (griddepcontrol.launch_dependents): the waiting blocks then
// fill whatever slots are free, unevenly over the SMs (binary64 256^2: 54 us a step instead of 40; 43 with
// ordinary launches).
template <class... P, class... A>
inline cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, A&&... args) {
  cudaLaunchConfig_t cfg = {};
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

// CTAs of a kernel that fit on the current device at once, queried once per device: the value cannot change while the
// process runs, so two first calls racing only store the same number twice. The dynamic shared-memory limit is set
// before the query; launches set it themselves (it is held per device context).
struct Residency {
  std::atomic<int> of[64];
};
template <class K> inline cudaError_t resident_ctas(Residency& cache, K* kernel, int threads, int smem, int* out) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 0 && dev < 64 && (*out = cache.of[dev].load(std::memory_order_relaxed)) > 0) return cudaSuccess;
  int sms = 0, occ = 0;
  if ((e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem)) != cudaSuccess) return e;
  if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
  if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, (size_t)smem)) != cudaSuccess) return e;
  *out = (occ > 0 ? occ : 1) * sms;
  if (dev >= 0 && dev < 64) cache.of[dev].store(*out, std::memory_order_relaxed);
  return cudaSuccess;
}

template <class S, int TX, int TY> struct TmaBox {
  static constexpr int XOFF = 16 / (int)sizeof(S) > 4 ? 16 / (int)sizeof(S) : 4;
  static constexpr int EPR = 16 / (int)sizeof(S);                // elements per 16 bytes
  static constexpr int BX = ((TX + XOFF + 3 + EPR - 1) / EPR) * EPR;
  static constexpr int BY = TY + 6;
  static constexpr int PLANE = BX * BY * (int)sizeof(S);                        // bytes
  static constexpr int SET = ((9 * PLANE + 127) / 128) * 128;                   // f or g: one copy of nine planes
  static constexpr int REFX = ((TX + XOFF + 3 + 3) / 4) * 4;                    // float reference planes
  static constexpr int RPLANE = ((REFX * BY * 4 + 127) / 128) * 128;
  static constexpr bool HALF = is_half_t<S>::value;
  static constexpr int BYTES = 2 * SET + (HALF ? 2 * RPLANE : 0) + 128;       // + the mbarrier
};

struct alignas(64) TmaMaps {
  CUtensorMap f, g, rf, rg;  // current buffer's populations (3D) and FP16 reference planes (2D)
};
// Those that a storage type has, for parameters that hold many.
template <class S> struct alignas(64) TmaMapsOf {
  CUtensorMap f, g;
};
template <> struct alignas(64) TmaMapsOf<__half> {
  CUtensorMap f, g, rf, rg;
};

// Most tiles a fused or batched step launches over an nx x ny domain (the 32 x 8 tile, the smallest
// shape). A step with the domain-mean buoyancy writes one partial sum per tile, so the partials array
// holds at least this many; on narrow domains (nx < 4) it exceeds the 2 * ceil(N / 64) of the split step.
inline size_t fused_max_tiles(int nx, int ny) { return (size_t)((nx + 31) / 32) * (size_t)((ny + 7) / 8); }

// Fused-step tile configuration a new context starts with: 32 x 8 tiles, one node per thread, in
// persistent CTAs that stage each next tile early (the fastest measured on GB300 at 2048^2 - 8192^2 in
// FP32 and FP16).
constexpr int kDefaultFusedTile = 4;

// Elements of a stored row of populations, phi and scratch planes. 4- and 2-byte rows are padded to whole 16-byte
// pieces, which the tensor copies of the fused step need (a 1023 x 1025 FP32 step 43 us without them, 37 with). Rows
// shorter than a tile with its rings, which no tensor copy serves, and a padding that would take a batch
// instance's 32-bit population indices past their range are left alone. Data that enters or leaves the library
// has no padding.
inline int row_pitch(int nx, int ny, size_t store) {
  if (store >= 8 || nx < 64) return nx;
  const int per = (int)(16 / store), pitch = (nx + per - 1) / per * per;
  return 9LL * pitch * ny > 2147483647LL && 9LL * nx * ny <= 2147483647LL ? nx : pitch;
}

// Device buffers of a context, carved from the caller's workspace.
struct SplitBuffers {
  void* f[2];        // populations f, post-collision layout, A/B (storage type)
  void* g[2];        // populations g
  float* ref_f[2];   // FP16 storage: per-node reference density of the stored f deviations (A/B)
  float* ref_g[2];   // FP16 storage: per-node reference temperature of the stored g deviations (A/B)
  double* wall[2] = {nullptr, nullptr};  // wall-row forces stored with f (A/B, wall_doubles(nx) each); null if y is periodic
  void* phi_prev;    // phi(t - dt), arithmetic type
  void* planes[16];  // scratch planes of the split kernels, arithmetic type
  double* partials;  // per-block (split) or per-tile (fused) partial sums: max(2 * nblocks, fused_max_tiles)
  double* scalars;   // [0] rho_ave, [1] mass, [2] heat
  long long* status; // [0] flag, [1] step, [2] x, [3] y, [4] code; [5] partial sums of rho written by the fused step, [6], [7] tile tickets and ended CTAs of the persistent fused step, zero between launches
  const TmaMaps* tma[2] = {nullptr, nullptr};  // tensor maps of buffer A / B for the TMA-staged fused step
  int fused_tile = 1;  // 0: 32x16, 1: 32x8, 2: 32x16 two nodes per thread, 3: 32x32 two per thread (maps match)
};

// ev: null, or split_kernel_count(P, prec) + 1 events recorded before the first and after each kernel.
cudaError_t split_step(const SplitBuffers& b, const DevParams& P, int prec, int cur, long long step, cudaStream_t st,
                       cudaEvent_t* ev = nullptr);
int split_kernel_count(const DevParams& P, int prec);
const char* split_kernel_name(int prec, int k);
cudaError_t split_init(const SplitBuffers& b, const DevParams& P, int prec, const double* rho, const double* T,
                       const double* ux, const double* uy, cudaStream_t st);
// Domain sums into scalars[1], scalars[2] and, unless null, out[0], out[1] (memory the device can write).
cudaError_t split_sums(const SplitBuffers& b, const DevParams& P, int prec, int cur, cudaStream_t st,
                       double* out = nullptr);
cudaError_t split_fields(const SplitBuffers& b, const DevParams& P, int prec, int cur, long long step, double* rho,
                         double* ux, double* uy, double* T, cudaStream_t st);
// which = 0: f, 1: g; only < 0: all 9 planes [9][ny][nx], else plane `only` into out[ny][nx].
cudaError_t split_export_pops(const SplitBuffers& b, const DevParams& P, int prec, int cur, int which, int only,
                              double* out, cudaStream_t st);
// Enqueue copies of rows of nx elements (2 or 4 bytes, at addresses that are multiples of it) from one stride, in
// elements, to another, between memory that the device reaches: several sets of rows in one launch.
struct RowSet {
  void* dst;
  const void* src;
  long long dst_stride, src_stride, rows;
  int elem;
};
struct RowSets {
  int n, nx;
  RowSet set[5];
};
cudaError_t repack_rows(const RowSets& s, cudaStream_t st);
int split_nplanes();
int split_block();

// ---- batched step (lbpc_fused.cu kernels, lbpc_batch.cu host) ----
// One instance of a batch as the device sees it; S is the storage type of the batch.
template <class S> struct alignas(16) BatchInst {
  DevParams P;
  PopBuf<S> f[2], g[2];
  void* phi_prev;      // arithmetic type
  double* scalars;     // [0] rho_ave, [1] mass, [2] heat
  double* partials;    // per-tile partial sums of rho (buoyancy) and per-block sums
  long long* status;   // first non-physical node of this instance
  long long step;      // steps taken
  int cur;             // buffer holding the current state
  int active;
  int ntiles;          // tiles of this instance in the current work list
  int pad_;
};
struct BatchTile {
  int inst, x0, y0, pslot;
};
struct BatchMeta {
  const BatchTile* tiles;
  int ntiles;
  int ninst;  // instance slots (active or not)
};
// Step-kernel variants of a batch (tile shape and nodes per thread): 0 = 32x8, 1 = 32x16, 2 = 64x8
// with one node per thread; 3 = 32x16, 4 = 64x16, 5 = 32x32 with two nodes per thread.
constexpr int kBatchVariants = 6;
inline void batch_tile_shape(int v, int& tx, int& ty) {
  static const int TXS[kBatchVariants] = {32, 32, 64, 32, 64, 32}, TYS[kBatchVariants] = {8, 16, 8, 16, 16, 32};
  const int k = (v >= 0 && v < kBatchVariants) ? v : 0;
  tx = TXS[k];
  ty = TYS[k];
}
inline int batch_nodes_per_thread(int v) { return v >= 3 && v < kBatchVariants ? 2 : 1; }
// Enqueue one batched step (persistent step kernel + per-instance advance) on st.
cudaError_t batch_step_launch(int prec, int variant, int ctas, const BatchMeta* d_meta, void* d_insts, int ninst,
                              cudaStream_t st);

// Per-tile launches of a batched step (the configuration with 0 CTAs per SM): one CTA per tile, and the
// instances of a launch in its kernel parameters, so that the tile body reads every per-instance value
// and buffer pointer as a uniform operand, as the single-instance kernel does. A step is a sequence of
// such launches over the active instances (up to seg_capacity each), then the per-instance advance.
template <class S> struct ArithOf { using type = float; };  // arithmetic of a storage type in a batch
template <> struct ArithOf<double> { using type = double; };
template <class S> struct alignas(16) SegInst {
  DevParamsOf<typename ArithOf<S>::type> P;  // header and the one coefficient set the kernel reads
  PopBuf<S> fs, gs, fd, gd;  // this launch's source and destination populations
  void* phi_prev;            // arithmetic type
  double* scalars;
  double* partials;
  long long* status;
  const long long* step;     // the instance's step counter (in its device descriptor), read to report
  int tiles_x;               // tiles per row
  int first;                 // the instance's first step (its source term starts from phi itself)
};
constexpr size_t kSegParamBytes = 32720;  // within the 32,764 bytes of kernel parameters
template <class S> constexpr int seg_capacity() {
  return (int)((kSegParamBytes - 32) / (sizeof(SegInst<S>) + sizeof(int))) & ~3;
}
// Launches of few instances take a kernel with smaller parameters (measured 4 % faster on one 2048^2
// instance than the full-size parameters, which every launch copies).
constexpr int kSegSmall = 16;
template <class S, int CAP> struct SegLaunch {
  int n;      // instances of this launch
  int tiles;  // its CTAs
  int waits;  // the first launch of its step: waits for the step before it
  int pad_;
  int first_tile[CAP];  // each instance's first CTA, ascending: kept together so that the search of a
                        // CTA's instance reads a few cache lines
  SegInst<S> in[CAP];
};
static_assert(sizeof(SegLaunch<double, seg_capacity<double>()>) <= kSegParamBytes &&
                  sizeof(SegLaunch<float, seg_capacity<float>()>) <= kSegParamBytes,
              "per-tile launch parameters");
// Enqueue one per-tile launch over the instances of L, a host SegLaunch<S, CAP> of the batch's storage
// type with CAP = kSegSmall (small) or seg_capacity<S>(). Unless L waits, the launch may begin while the previous
// kernel on st drains (its instances are others).
cudaError_t batch_seg_launch(int prec, int variant, bool small, const void* L, cudaStream_t st);

// The same launch walked by persistent CTAs (4- and 2-byte storage, 32 x 8 tiles). The tensor maps of the source
// buffers travel in the parameters beside their instances, which so many fewer fit. Maps in device memory would have to
// be acquired by each block that uses them, with a system-scope proxy fence per instance: the tiles a block takes are
// of ever other instances, and 64 uneven FP32 instances took 71.2 ms per 256 steps that way, 60.0 this way.
template <class S, int CAP> struct WalkLaunch {
  int n;      // instances of this launch
  int tiles;  // its tiles
  int waits;  // the first launch of its step: waits for the step before it
  int pad_;
  unsigned long long mapped;  // bit k: instance k has tensor maps
  int first_tile[CAP];
  SegInst<S> in[CAP];
  TmaMapsOf<S> maps[CAP];
};
template <class S> constexpr int walk_capacity() {
  return (int)((kSegParamBytes - 128) / (sizeof(SegInst<S>) + sizeof(TmaMapsOf<S>) + sizeof(int))) & ~3;
}
static_assert(sizeof(WalkLaunch<float, walk_capacity<float>()>) <= kSegParamBytes &&
                  sizeof(WalkLaunch<__half, walk_capacity<__half>()>) <= kSegParamBytes && walk_capacity<float>() <= 64,
              "walk launch parameters");
// Whether a launch of that many tiles, `staged` of which tensor copies can stage, is faster walked.
cudaError_t batch_walk_wanted(int prec, bool small, long long tiles, long long staged, bool* yes);
// Enqueue it; L: a host WalkLaunch<S, CAP>, CAP = kSegSmall (small) or walk_capacity<S>(). tickets: two zeroed words of
// this launch's own in device memory, left zero.
cudaError_t batch_walk_launch(int prec, bool small, const void* L, unsigned long long* tickets, cudaStream_t st);
// Enqueue the per-instance advance of a step (rho_ave, buffer parity, step count).
cudaError_t batch_advance_launch(int prec, void* d_insts, int ninst, cudaStream_t st);
// Largest resident CTAs per SM of the step kernel for (prec, variant).
int batch_max_ctas_per_sm(int prec, int variant);

// Fused single-kernel step (lbpc_fused.cu); same buffers, no scratch planes touched. ev: null, or fused_kernel_count + 1
// events as for split_step. The count is 2 where a staged step (tensor copies) with the domain-mean buoyancy leaves the
// mean to a kernel of its own.
int fused_kernel_count(const SplitBuffers& b, const DevParams& P, int prec, int cur);
cudaError_t fused_step(const SplitBuffers& b, const DevParams& P, int prec, int cur, long long step, cudaStream_t st,
                       cudaEvent_t* ev = nullptr);
// Encode the tensor maps of one buffer (populations f, g and, for FP16, the reference planes) for the
// TMA-staged fused step; false when the layout does not allow TMA (row stride not 16-byte aligned).
bool fused_tma_encode(TmaMaps* m, int prec, int tile, void* f, void* g, float* rf, float* rg, const DevParams& P);

// rho_ave <- sum of n per-tile partials / nodes (fixed order), on st.
void fused_finish(const SplitBuffers& b, const DevParams& P, int n, cudaStream_t st);

}  // namespace lbpc
