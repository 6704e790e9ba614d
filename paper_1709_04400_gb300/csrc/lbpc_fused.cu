// Fused step of one domain: one kernel per time step, one CTA per tile (tile body in lbpc_tile.cuh),
// with the interior tiles' populations staged in shared memory by TMA where the row stride allows.
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>

#include "lbpc_tile.cuh"

namespace lbpc {

template <class S, class R, int TX, int TY, int NPT>
__global__ void __launch_bounds__(TX* TY / NPT, fused_min_blocks<S, TX * TY / NPT, NPT>()) k_fused(PopBuf<S> fsrc, PopBuf<S> gsrc, PopBuf<S> fdst, PopBuf<S> gdst,
                                                   R* __restrict__ phi_prev, DevParams P, long long step, int first,
                                                   const MeanOf mean, double* __restrict__ partials,
                                                   long long* __restrict__ status) {
  __shared__ FusedSmem<R, TX, TY> sm;
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const bool interior = x0 >= 3 && x0 + TX + 3 <= P.nx && y0 >= 3 && y0 + TY + 3 <= P.ny;
  const int pslot = blockIdx.y * gridDim.x + blockIdx.x;
  const int t = pdl_wait<TX * TY / NPT>();
  if (interior)
    fused_body<1, S, R, TX, TY, NPT>(t, fsrc, gsrc, fdst, gdst, phi_prev, P, step, first, mean.out, partials, status, sm,
                                     x0, y0, pslot, TmaTile<S>{nullptr}, nullptr, NoStageHook{}, &mean);
  else if (rows_inside<TY>(P, y0))
    fused_body<4, S, R, TX, TY, NPT>(t, fsrc, gsrc, fdst, gdst, phi_prev, P, step, first, mean.out, partials, status, sm,
                                     x0, y0, pslot, TmaTile<S>{nullptr}, nullptr, NoStageHook{}, &mean);
  else
    fused_body<0, S, R, TX, TY, NPT>(t, fsrc, gsrc, fdst, gdst, phi_prev, P, step, first, mean.out, partials, status, sm,
                                     x0, y0, pslot, TmaTile<S>{nullptr}, nullptr, NoStageHook{}, &mean);
}

// Same step with the interior tiles' populations staged in shared memory by TMA (dynamic shared
// memory of TmaBox<S, TX, TY>::BYTES). Tiles that touch an edge take the general path.
template <class S, class R, int TX, int TY, int NPT>
__global__ void __launch_bounds__(TX* TY / NPT, fused_min_blocks<S, TX * TY / NPT, NPT>()) k_fused_tma(PopBuf<S> fsrc, PopBuf<S> gsrc, PopBuf<S> fdst, PopBuf<S> gdst,
                                                       R* __restrict__ phi_prev, DevParams P, long long step, int first,
                                                       const double* __restrict__ rho_ave,
                                                       double* __restrict__ partials, long long* __restrict__ status,
                                                       const __grid_constant__ TmaMaps maps) {
  using B = TmaBox<S, TX, TY>;
  __shared__ FusedSmem<R, TX, TY> sm;
  extern __shared__ __align__(128) unsigned char dyn[];
  const int x0 = blockIdx.x * TX, y0 = blockIdx.y * TY;
  const bool interior = x0 >= 3 && x0 + TX + 3 <= P.nx && y0 >= 3 && y0 + TY + 3 <= P.ny;
  const int pslot = blockIdx.y * gridDim.x + blockIdx.x;
  uint64_t* bar = (uint64_t*)(dyn + B::BYTES - 128);
  if (interior) {
    if (threadIdx.x == 0) mbar_init(bar, 1);
    __syncthreads();
  }
  const int t = pdl_wait<TX * TY / NPT>();
  if (!interior) {
    if (rows_inside<TY>(P, y0))
      fused_body<4, S, R, TX, TY, NPT>(t, fsrc, gsrc, fdst, gdst, phi_prev, P, step, first, rho_ave, partials, status, sm,
                                       x0, y0, pslot);
    else
      fused_body<0, S, R, TX, TY, NPT>(t, fsrc, gsrc, fdst, gdst, phi_prev, P, step, first, rho_ave, partials, status, sm,
                                       x0, y0, pslot);
    return;
  }
  if (threadIdx.x == 0) {
    mbar_expect_tx(bar, (unsigned)(18 * B::BX * B::BY * sizeof(S) + (B::HALF ? 2 * B::REFX * B::BY * 4 : 0)));
    tma_load_3d(dyn, &maps.f, x0 - B::XOFF, y0 - 3, 0, bar);
    tma_load_3d(dyn + B::SET, &maps.g, x0 - B::XOFF, y0 - 3, 0, bar);
    if (B::HALF) {
      tma_load_2d(dyn + 2 * B::SET, &maps.rf, x0 - B::XOFF, y0 - 3, bar);
      tma_load_2d(dyn + 2 * B::SET + B::RPLANE, &maps.rg, x0 - B::XOFF, y0 - 3, bar);
    }
  }
  // Every thread polls the barrier. Measured against one polling thread with the others parked at a block
  // barrier (820 instead of 888 instructions per node, but 1 % slower in FP32, also with two kernels
  // sharing the GPU) and against waits that sleep in the barrier with a suspend-time hint (slower, more
  // instructions): polling wakes the warps soonest.
  if (!mbar_wait_bounded(bar, 0)) {
    if (threadIdx.x == 0) report(status, step, x0, y0, ST_TIMEOUT);
    mbar_wait_bounded(bar, 0);  // let the copies in flight land before the block's shared memory goes away
    return;
  }
  fused_body<2, S, R, TX, TY, NPT>(threadIdx.x, fsrc, gsrc, fdst, gdst, phi_prev, P, step, first, rho_ave, partials, status, sm,
                                   x0, y0, pslot, TmaTile<S>{dyn});
}

// Persistent form of the TMA-staged step: resident CTAs take tiles in order from a ticket counter (so
// the tiles in flight stay one compact band of the grid, as with one CTA per tile, and the rings they
// re-read meet in L2), and each starts its next interior tile's copy as soon as the current tile has
// finished reading its staged populations (after stage 1). The copy then runs under stages 2 and 3
// instead of in front of the next tile. An edge tile reads nothing staged, so the next copy starts
// before it. One mbarrier serves every copy; the waits alternate its phase parity.
//
// Bound by HBM in FP32 (4096^2: 413 us, 91 % of the measured copy bandwidth at 152 B per node) and by issue in
// FP16. What the walk itself costs counts: with each ticket awaited where the next copy starts, one tensor copy
// per population plane, and tile origins divided out by every thread, 4096^2 took 469 us (FP16 528, then 470; now 455,
// see pitch_of).
template <class S, class R, int TX, int TY, int NPT>
__global__ void __launch_bounds__(TX* TY / NPT, fused_min_blocks<S, TX * TY / NPT, NPT>())
    k_fused_tma_loop(PopBuf<S> fsrc, PopBuf<S> gsrc, PopBuf<S> fdst, PopBuf<S> gdst, R* __restrict__ phi_prev,
                     DevParams P, long long step, int first, const double* __restrict__ rho_ave,
                     double* __restrict__ partials, long long* __restrict__ status,
                     unsigned long long* __restrict__ tickets, const __grid_constant__ TmaMaps maps) {
  using B = TmaBox<S, TX, TY>;
  __shared__ FusedSmem<R, TX, TY> sm;
  // walk state, double-buffered by iteration parity: this tile and the next one (being staged), each with its
  // origin (x < 0: no tile left); thread 0 fills the other slot during the tile, so one block barrier per tile
  // orders both
  struct Tile {
    int x, y, index;
  };
  __shared__ Tile s_tile[2], s_next[2];
  extern __shared__ __align__(128) unsigned char dyn[];
  uint64_t* bar = (uint64_t*)(dyn + B::BYTES - 128);
  const int ntx = (P.nx + TX - 1) / TX, ntiles = ntx * ((P.ny + TY - 1) / TY);
  auto tile_at = [&](unsigned long long k) {  // thread 0: the k-th tile in order
    const int i = (int)k;
    return k < (unsigned long long)ntiles ? Tile{(i % ntx) * TX, (i / ntx) * TY, i} : Tile{-1, 0, 0};
  };
  // whether a tile, its 2-ring and their pull sources stay inside the domain
  auto inside = [&](const Tile& t) { return t.x >= 3 && t.x + TX + 3 <= P.nx && t.y >= 3 && t.y + TY + 3 <= P.ny; };
  pdl_wait<TX * TY / NPT>();  // every address below depends on a ticket or a staged copy taken after it
  // the first tile of a CTA is its own number's, the later ones are tickets
  auto take = [&]() { return gridDim.x + atomicAdd(tickets, 1ull); };
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    const Tile t0 = tile_at(blockIdx.x);
    if (inside(t0)) tma_issue_tile<S, TX, TY>(dyn, bar, maps, t0.x, t0.y);
    s_tile[0] = t0;
    s_next[0] = tile_at(take());
  }
  __syncthreads();
  unsigned parity = 0;  // of the mbarrier phase awaited next
  for (int it = 0;; it ^= 1) {
    const Tile tile = s_tile[it];
    if (tile.x < 0) break;
    // Thread 0 takes the ticket of the tile after the next one here and turns it into a tile at the end of this
    // one: the counter's answer takes most of a microsecond, and waiting for it where the next copy starts held
    // the whole block at its next barrier.
    unsigned long long ticket = 0;
    if (threadIdx.x == 0) ticket = take();
    auto start_next = [&]() {  // thread 0 starts the copy of the next tile, if interior
      if (threadIdx.x != 0) return;
      const Tile next = s_next[it];
      if (inside(next)) tma_issue_tile<S, TX, TY>(dyn, bar, maps, next.x, next.y);
    };
    if (inside(tile)) {
      if (!mbar_wait_bounded(bar, parity)) {
        report(status, step, tile.x, tile.y, ST_TIMEOUT);
        mbar_wait_bounded(bar, parity);  // let the copy in flight land before the block's shared memory goes away
        // no tile is left for the threads whose wait did end, with or without thread 0
        s_tile[0].x = s_tile[1].x = s_next[0].x = s_next[1].x = -1;
        __threadfence();  // this tile's ticket is counted before the CTA's end is
        break;
      }
      parity ^= 1u;
      fused_body<2, S, R, TX, TY, NPT>(threadIdx.x, fsrc, gsrc, fdst, gdst, phi_prev, P, step, first, rho_ave, partials, status, sm,
                                       tile.x, tile.y, tile.index, TmaTile<S>{dyn}, nullptr, start_next);
    } else {
      start_next();
      if (is_half_t<S>::value && rows_inside<TY>(P, tile.y))  // in FP32 a third body costs every tile 4 %
        fused_body<4, S, R, TX, TY, NPT>(threadIdx.x, fsrc, gsrc, fdst, gdst, phi_prev, P, step, first, rho_ave, partials, status, sm,
                                         tile.x, tile.y, tile.index);
      else
        fused_body<0, S, R, TX, TY, NPT>(threadIdx.x, fsrc, gsrc, fdst, gdst, phi_prev, P, step, first, rho_ave, partials, status, sm,
                                         tile.x, tile.y, tile.index);
    }
    if (threadIdx.x == 0) {
      s_tile[it ^ 1] = s_next[it];
      s_next[it ^ 1] = tile_at(ticket);
    }
    __syncthreads();  // the tile body is done with the shared arrays; the next walk state has landed
  }
  // The last CTA to end puts the counter back to zero for the next launch (a CTA has its last ticket's answer
  // when it comes here); the count of ended CTAs wraps to zero by itself.
  if (threadIdx.x == 0 && atomicInc((unsigned*)(tickets + 1), gridDim.x - 1) == gridDim.x - 1)
    atomicExch(tickets, 0ull);
}

template <class S, class R, int TX, int TY, int NPT> static cudaError_t loop_residency(int smem, int* out) {
  static Residency cache;
  return resident_ctas(cache, k_fused_tma_loop<S, R, TX, TY, NPT>, TX * TY / NPT, smem, out);
}

// Whether a step's interior tiles are staged by tensor copies: wherever the buffers have tensor maps, but for small FP32
// grids of 32 x 8 tiles, which pull straight from L2 (below three tiles per four resident CTAs a copy has nothing to
// overlap with; with the domain-mean buoyancy the unstaged step also takes the mean in its last block, a launch less, and
// stays ahead up to two tiles per CTA). us a step, unstaged and staged, 608 resident CTAs: 224^2 (196 tiles) 5.3,
// 5.6; 288 x 352 (396) 6.57, 6.83; 320^2 (400) 6.25, 6.21; 352^2 (484) 7.24, 7.00; 384 x 400 (600) 7.37, 7.05; 512^2 (1024)
// 11.5, 11.4. Closed pools with the mean: 150 x 300 (190) 8.5, 9.1; 384 x 400 11.0, 11.5; 512^2 16.7, 17.6; 640 x 512 (1280)
// 20.9, 20.7. The other tile shapes do not differ by more than a few per cent either way, nor does FP16.
template <class S, class R, int TX, int TY, int NPT>
static cudaError_t takes_staging(const SplitBuffers& b, const DevParams& P, int cur, bool* yes) {
  *yes = false;
  if constexpr (sizeof(S) <= 4) {  // the staged kernels exist for FP32 and FP16 storage
    *yes = b.tma[cur] != nullptr;
    if (*yes && !is_half_t<S>::value && TX * TY == 32 * 8) {
      static Residency cache;
      int resident = 0;
      const cudaError_t e =
          resident_ctas(cache, k_fused_tma<S, R, TX, TY, NPT>, TX * TY / NPT, TmaBox<S, TX, TY>::BYTES, &resident);
      if (e != cudaSuccess) return e;
      const long long tiles = (long long)((P.nx + TX - 1) / TX) * ((P.ny + TY - 1) / TY);
      *yes = 4 * tiles >= (P.buoyancy == 1 ? 8LL : 3LL) * resident;
    }
  }
  return cudaSuccess;
}

// ------------------------------------------------------------------------------------------------
template <class S, class R, int TX, int TY, int NPT = 1, bool LOOP = false>
static cudaError_t fused_impl(const SplitBuffers& b, const DevParams& P, int cur, long long step, cudaStream_t st,
                              cudaEvent_t* ev) {
  dim3 grid((P.nx + TX - 1) / TX, (P.ny + TY - 1) / TY);
  const PopBuf<S> fs{(S*)b.f[cur], b.ref_f[cur], b.wall[cur]}, gs{(S*)b.g[cur], b.ref_g[cur]};
  const PopBuf<S> fd{(S*)b.f[cur ^ 1], b.ref_f[cur ^ 1], b.wall[cur ^ 1]}, gd{(S*)b.g[cur ^ 1], b.ref_g[cur ^ 1]};
  const MeanOf mean{b.scalars, (unsigned*)(b.status + 5), grid.x * grid.y, 1.0 / node_count(P)};
  if (ev) cudaEventRecord(ev[0], st);
  bool staged = false;
  {
    const cudaError_t e = takes_staging<S, R, TX, TY, NPT>(b, P, cur, &staged);
    if (e != cudaSuccess) return e;
  }
  if constexpr (sizeof(S) <= 4) {
    if (staged) {
      using B = TmaBox<S, TX, TY>;
      // The dynamic shared-memory limit is held per device context, so it is set before every launch:
      // the call is cheap, thread-safe, and right after a device reset or on a second device.
      bool persistent = false;
      if constexpr (LOOP) {
        cudaError_t e = cudaFuncSetAttribute(k_fused_tma_loop<S, R, TX, TY, NPT>,
                                             cudaFuncAttributeMaxDynamicSharedMemorySize, B::BYTES);
        if (e != cudaSuccess) return e;
        int resident = 0;  // CTAs of the persistent kernel that fit on the device at once
        if ((e = loop_residency<S, R, TX, TY, NPT>(B::BYTES, &resident)) != cudaSuccess) return e;
        // Persistent CTAs pay off where each walks several tiles. us, one CTA per tile against persistent, FP32: 768^2
        // (3.8 tiles per CTA) 21.6, 23.1; 896^2 (5.2) 30.7, 30.3; 1024^2 (6.7) 38.5, 36.6; 2048^2 130, 112. FP16: 25.3, 26.4;
        // 32.3, 32.2; 41.5, 40.1; 133, 124.
        if ((long long)grid.x * grid.y > 5LL * resident) {
          unsigned long long* tickets = (unsigned long long*)(b.status + 6);
          if ((e = launch_pdl(k_fused_tma_loop<S, R, TX, TY, NPT>, resident, TX * TY / NPT, B::BYTES, st, fs, gs, fd, gd,
                              (R*)b.phi_prev, P, step, step == 0, b.scalars, b.partials, b.status, tickets,
                              *b.tma[cur])) != cudaSuccess)
            return e;
          persistent = true;
        }
      }
      if (!persistent) {
        cudaError_t e =
            cudaFuncSetAttribute(k_fused_tma<S, R, TX, TY, NPT>, cudaFuncAttributeMaxDynamicSharedMemorySize, B::BYTES);
        if (e != cudaSuccess) return e;
        if ((e = launch_pdl(k_fused_tma<S, R, TX, TY, NPT>, grid, TX * TY / NPT, B::BYTES, st, fs, gs, fd, gd,
                            (R*)b.phi_prev, P, step, step == 0, b.scalars, b.partials, b.status, *b.tma[cur])) != cudaSuccess)
          return e;
      }
      // the mean as a kernel of its own: its code in the staged kernels costs every step of theirs 2 to 5 %
      if (P.buoyancy == 1) {
        if (ev) cudaEventRecord(ev[1], st);
        fused_finish(b, P, (int)(grid.x * grid.y), st);
      }
    }
  }
  if (!staged) {
    const cudaError_t e = launch_pdl(k_fused<S, R, TX, TY, NPT>, grid, TX * TY / NPT, 0, st, fs, gs, fd, gd, (R*)b.phi_prev,
                                     P, step, step == 0, mean, b.partials, b.status);
    if (e != cudaSuccess) return e;
  }
  if (ev) cudaEventRecord(ev[staged && P.buoyancy == 1 ? 2 : 1], st);
  return cudaGetLastError();
}

// ---- tensor maps of the TMA-staged path ----
static PFN_cuTensorMapEncodeTiled_v12000 query_encode_fn() {
  void* p = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
      q == cudaDriverEntryPointSuccess)
    return (PFN_cuTensorMapEncodeTiled_v12000)p;
  return nullptr;
}

// The driver's entry point is the same for every device and context; the function-local static is
// initialised once, thread-safely.
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static const PFN_cuTensorMapEncodeTiled_v12000 fn = query_encode_fn();
  return fn;
}

template <class S, int TX, int TY>
static bool encode_t(TmaMaps* m, void* f, void* g, float* rf, float* rg, const DevParams& P) {
  using B = TmaBox<S, TX, TY>;
  auto fn = encode_fn();
  if (!fn) return false;
  if (((size_t)P.pitch * sizeof(S)) % 16 != 0) return false;  // row stride must be a multiple of 16 bytes
  static_assert(sizeof(S) <= 4, "FP32 and FP16 storage");
  const CUtensorMapDataType dt = sizeof(S) == 2 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32;
  const cuuint64_t dims[3] = {(cuuint64_t)P.nx, (cuuint64_t)P.ny, 9};
  const cuuint64_t strides[2] = {(cuuint64_t)P.pitch * sizeof(S), (cuuint64_t)P.N * sizeof(S)};
  const cuuint32_t box[3] = {(cuuint32_t)B::BX, (cuuint32_t)B::BY, 9};
  const cuuint32_t es[3] = {1, 1, 1};
  auto enc3 = [&](CUtensorMap* t, void* base) {
    return fn(t, dt, 3, base, dims, strides, box, es, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
              CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  };
  if (!enc3(&m->f, f) || !enc3(&m->g, g)) return false;
  if (B::HALF) {
    const cuuint64_t d2[2] = {(cuuint64_t)P.nx, (cuuint64_t)P.ny};
    const cuuint64_t s2[1] = {(cuuint64_t)P.pitch * 4};
    const cuuint32_t b2[2] = {(cuuint32_t)B::REFX, (cuuint32_t)B::BY};
    auto enc2 = [&](CUtensorMap* t, void* base) {
      return fn(t, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, base, d2, s2, b2, es, CU_TENSOR_MAP_INTERLEAVE_NONE,
                CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
             CUDA_SUCCESS;
    };
    if (!enc2(&m->rf, rf) || !enc2(&m->rg, rg)) return false;
  }
  return true;
}

template <class S>
static bool encode_tile(TmaMaps* m, int tile, void* f, void* g, float* rf, float* rg, const DevParams& P) {
  if (tile == 1 || tile == 4) return encode_t<S, 32, 8>(m, f, g, rf, rg, P);
  if (tile == 3) return encode_t<S, 32, 32>(m, f, g, rf, rg, P);
  return encode_t<S, 32, 16>(m, f, g, rf, rg, P);  // tiles 0 and 2
}

bool fused_tma_encode(TmaMaps* m, int prec, int tile, void* f, void* g, float* rf, float* rg, const DevParams& P) {
  if (prec == 1) return encode_tile<float>(m, tile, f, g, rf, rg, P);
  if (prec == 2) return encode_tile<__half>(m, tile, f, g, rf, rg, P);
  return false;  // FP64 runs the split step by default; its fused form keeps per-thread loads
}

// Tile configurations of the FP32 / FP16 fused step: 0 = 32x16, 1 = 32x8, 2 = 32x16 with 2 nodes per
// thread, 3 = 32x32 with 2 nodes per thread, 4 = 32x8 in persistent CTAs that start each next tile's copy
// early. f is called with the shape.
template <int TX_, int TY_, int NPT_, bool LOOP_ = false> struct Shape {
  static constexpr int TX = TX_, TY = TY_, NPT = NPT_;
  static constexpr bool LOOP = LOOP_;
};
template <class F> static cudaError_t with_shape(int fused_tile, F f) {
  switch (fused_tile) {
    case 1: return f(Shape<32, 8, 1>());
    case 2: return f(Shape<32, 16, 2>());
    case 3: return f(Shape<32, 32, 2>());
    case 4: return f(Shape<32, 8, 1, true>());
    default: return f(Shape<32, 16, 1>());
  }
}
template <class S, class R>
static cudaError_t fused_tiles(const SplitBuffers& b, const DevParams& P, int cur, long long step, cudaStream_t st,
                               cudaEvent_t* ev) {
  return with_shape(b.fused_tile, [&](auto s) {
    using T = decltype(s);
    return fused_impl<S, R, T::TX, T::TY, T::NPT, T::LOOP>(b, P, cur, step, st, ev);
  });
}
template <class S> static int kernel_count(const SplitBuffers& b, const DevParams& P, int cur) {
  bool staged = false;
  with_shape(b.fused_tile, [&](auto s) {
    using T = decltype(s);
    return takes_staging<S, float, T::TX, T::TY, T::NPT>(b, P, cur, &staged);
  });
  return P.buoyancy == 1 && staged ? 2 : 1;
}

int fused_kernel_count(const SplitBuffers& b, const DevParams& P, int prec, int cur) {
  if (prec == 1) return kernel_count<float>(b, P, cur);
  if (prec == 2) return kernel_count<__half>(b, P, cur);
  return 1;
}

cudaError_t fused_step(const SplitBuffers& b, const DevParams& P, int prec, int cur, long long step, cudaStream_t st,
                       cudaEvent_t* ev) {
  if (prec == 0) {
    SplitBuffers nb = b;
    nb.tma[0] = nb.tma[1] = nullptr;
    return fused_impl<double, double, 32, 8>(nb, P, cur, step, st, ev);
  }
  if (prec == 3) {
    SplitBuffers nb = b;
    nb.tma[0] = nb.tma[1] = nullptr;
    return fused_impl<dw, dw, 32, 8>(nb, P, cur, step, st, ev);
  }
  if (prec == 1) return fused_tiles<float, float>(b, P, cur, step, st, ev);
  return fused_tiles<__half, float>(b, P, cur, step, st, ev);
}

}  // namespace lbpc
