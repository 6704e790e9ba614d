// Batched step as per-tile launches (the configuration with 0 CTAs per SM): the instances of a launch in its kernel
// parameters (tile body in lbpc_tile.cuh), and one CTA per tile or, in launches of many tiles of 4- and 2-byte storage,
// persistent CTAs that walk them.
#include "lbpc_tile.cuh"

namespace lbpc {

// Per-tile launch of a batched step: CTA b finds its instance by the launch's first-tile offsets (a
// uniform search over the kernel parameters) and runs the tile body on that instance's tile
// b - first_tile. Every value of the instance is then a parameter-space operand, as in the single-instance
// kernel, so the body has none of the work-list kernel's per-use shared-memory loads.
//
// The launches of one step cover disjoint instances, so each lets the next one start while its own
// last CTAs run (programmatic dependent launch). The last CTA of a launch waits, before it exits, for
// the launch before it to complete: a launch then completes only after every earlier launch of the step
// has, and the advance kernel, which waits for the last one, sees the whole step. The first launch of a
// step (waits) in turn waits for the advance kernel before it reads anything. The earlier launch's
// CTAs have all started when this one starts, so the waits always end.
template <class S, class R, int TX, int TY, int NPT, int CAP>
__global__ void __launch_bounds__(TX* TY / NPT, fused_min_blocks<S, TX * TY / NPT, NPT>())
    k_batch_tiles(const __grid_constant__ SegLaunch<S, CAP> L) {
  // The next launch of the step covers other instances: let it start as this one's last CTAs run.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ FusedSmem<R, TX, TY> sm;
  const int b = blockIdx.x;
  int k = 0, hi = L.n - 1;  // the last instance whose first CTA is at most b (a uniform binary search)
#pragma unroll 1
  while (k < hi) {
    const int mid = (k + hi + 1) >> 1;
    if (L.first_tile[mid] <= b) k = mid;
    else hi = mid - 1;
  }
  const SegInst<S>& I = L.in[k];
  const auto& P = I.P;
  const int t = b - L.first_tile[k];
  const int x0 = (t % I.tiles_x) * TX, y0 = (t / I.tiles_x) * TY;
  const bool interior = x0 >= 3 && x0 + TX + 3 <= P.nx && y0 >= 3 && y0 + TY + 3 <= P.ny;
  if (interior)
    fused_body<1, S, R, TX, TY, NPT>(threadIdx.x, I.fs, I.gs, I.fd, I.gd, (R*)I.phi_prev, P, 0, I.first, I.scalars, I.partials,
                                     I.status, sm, x0, y0, t, TmaTile<S>{nullptr}, I.step);
  else if (rows_inside<TY>(P, y0))
    fused_body<4, S, R, TX, TY, NPT, true>(threadIdx.x, I.fs, I.gs, I.fd, I.gd, (R*)I.phi_prev, P, 0, I.first, I.scalars,
                                           I.partials, I.status, sm, x0, y0, t, TmaTile<S>{nullptr}, I.step);
  else  // edge tiles wrap and clamp their indices: cheaper in 32 bits
    fused_body<0, S, R, TX, TY, NPT, true>(threadIdx.x, I.fs, I.gs, I.fd, I.gd, (R*)I.phi_prev, P, 0, I.first, I.scalars,
                                           I.partials, I.status, sm, x0, y0, t, TmaTile<S>{nullptr}, I.step);
  if (b == (int)gridDim.x - 1) asm volatile("griddepcontrol.wait;" ::: "memory");
}

// The same launch by persistent CTAs, for 4- and 2-byte storage: resident CTAs take the launch's tiles in order from a
// ticket counter and stage each next interior tile by tensor copies while they finish the current one, as the
// persistent single-instance step does. The walk is one tile deeper: a tile's number becomes its instance and
// origin (a search over the parameters) by a warp of its own while the tile before it pulls. The instance of the
// tile being worked on is broadcast from one lane, which lets the compiler keep its parameters in uniform registers.
template <class S, class R, int TX, int TY, int CAP>
__global__ void __launch_bounds__(TX* TY, fused_min_blocks<S, TX * TY, 1>())
    k_batch_walk(const __grid_constant__ WalkLaunch<S, CAP> L, unsigned long long* __restrict__ tickets) {
  using B = TmaBox<S, TX, TY>;
  constexpr int NTH = TX * TY;
  if (L.waits) pdl_wait<NTH>();  // every address below depends on shared memory written after it
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ FusedSmem<R, TX, TY> sm;
  struct Tile {
    int k, x, y, index;  // instance (-1: no tile left), origin, number within the instance
  };
  __shared__ Tile s_tile[2], s_next;
  __shared__ unsigned s_raw;  // number of the next tile
  extern __shared__ __align__(128) unsigned char dyn[];
  uint64_t* bar = (uint64_t*)(dyn + B::BYTES - 128);
  auto tile_at = [&](unsigned b) {
    if (b >= (unsigned)L.tiles) return Tile{-1, 0, 0, 0};
    int k = 0, hi = L.n - 1;  // the last instance whose first tile is at most b
#pragma unroll 1
    while (k < hi) {
      const int mid = (k + hi + 1) >> 1;
      if (L.first_tile[mid] <= (int)b) k = mid;
      else hi = mid - 1;
    }
    const int t = (int)b - L.first_tile[k], nx = L.in[k].tiles_x;
    return Tile{k, (t % nx) * TX, (t / nx) * TY, t};
  };
  // staged: the tile, its 2-ring and their pull sources lie inside a domain that has tensor maps
  auto staged = [&](const Tile& t) {
    if (t.k < 0) return false;
    const SegInst<S>& I = L.in[t.k];
    return ((L.mapped >> t.k) & 1) && t.x >= 3 && t.x + TX + 3 <= I.P.nx && t.y >= 3 && t.y + TY + 3 <= I.P.ny;
  };
  auto take = [&]() { return (unsigned)(gridDim.x + atomicAdd(tickets, 1ull)); };
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    const Tile t0 = tile_at(blockIdx.x);
    if (staged(t0)) tma_issue_tile<S, TX, TY>(dyn, bar, L.maps[t0.k], t0.x, t0.y);
    s_tile[0] = t0;
    s_raw = take();
  }
  __syncthreads();
  unsigned parity = 0;
  for (int it = 0;; it ^= 1) {
    const Tile tile = s_tile[it];
    if (tile.k < 0) break;
    unsigned ticket = 0;
    if (threadIdx.x == 0) ticket = take();            // used at the end of this tile
    if (threadIdx.x == NTH - 32) s_next = tile_at(s_raw);  // read after the body's first barrier
    auto start_next = [&]() {
      if (threadIdx.x != 0) return;
      const Tile next = s_next;
      if (staged(next)) tma_issue_tile<S, TX, TY>(dyn, bar, L.maps[next.k], next.x, next.y);
    };
    const int k = __shfl_sync(0xffffffffu, tile.k, 0);
    const int x0 = __shfl_sync(0xffffffffu, tile.x, 0), y0 = __shfl_sync(0xffffffffu, tile.y, 0);
    const SegInst<S>& I = L.in[k];
    const bool st = __shfl_sync(0xffffffffu, (int)staged(tile), 0) != 0;
    if (st) {
      if (!mbar_wait_bounded(bar, parity)) {
        report(I.status, *I.step, x0, y0, ST_TIMEOUT);
        mbar_wait_bounded(bar, parity);  // let the copy in flight land before the block's shared memory goes away
        // no tile is left for the threads whose wait did end, with or without thread 0
        s_tile[0].k = s_tile[1].k = s_next.k = -1;
        __threadfence();  // this tile's ticket is counted before the CTA's end is
        break;
      }
      parity ^= 1u;
      fused_body<2, S, R, TX, TY, 1>(threadIdx.x, I.fs, I.gs, I.fd, I.gd, (R*)I.phi_prev, I.P, 0, I.first, I.scalars, I.partials,
                                     I.status, sm, x0, y0, tile.index, TmaTile<S>{dyn}, I.step, start_next);
    } else if (rows_inside<TY>(I.P, y0)) {
      fused_body<4, S, R, TX, TY, 1, true>(threadIdx.x, I.fs, I.gs, I.fd, I.gd, (R*)I.phi_prev, I.P, 0, I.first, I.scalars,
                                           I.partials, I.status, sm, x0, y0, tile.index, TmaTile<S>{nullptr}, I.step, start_next);
    } else {
      fused_body<0, S, R, TX, TY, 1, true>(threadIdx.x, I.fs, I.gs, I.fd, I.gd, (R*)I.phi_prev, I.P, 0, I.first, I.scalars,
                                           I.partials, I.status, sm, x0, y0, tile.index, TmaTile<S>{nullptr}, I.step, start_next);
    }
    if (threadIdx.x == 0) {
      s_tile[it ^ 1] = s_next;
      s_raw = ticket;
    }
    __syncthreads();
  }
  // the counter goes back to zero for the next step's launch, as in the single-instance step
  if (threadIdx.x == 0 && atomicInc((unsigned*)(tickets + 1), gridDim.x - 1) == gridDim.x - 1) atomicExch(tickets, 0ull);
  if (blockIdx.x == gridDim.x - 1) asm volatile("griddepcontrol.wait;" ::: "memory");
}

template <class S, class R, int CAP> static cudaError_t walk_resident(int* out) {
  static Residency cache;
  return resident_ctas(cache, k_batch_walk<S, R, 32, 8, CAP>, 256, TmaBox<S, 32, 8>::BYTES, out);
}

// Where the walk is the faster form. Against one CTA per tile it gains on a staged tile, loses on an edge tile, whose own
// pulls leave the CTA's next copy waiting, and pays once per CTA for its first copy and the last, ragged wave: an
// edge tile costs what 2.3 staged tiles bring in FP32 and 1.9 in FP16, a CTA what 2.4 and 2.0 bring. The numbers are
// fitted to 240 batches of one launch, 1 to 40 instances of one size or of mixed ones, evaporation alone and half pools,
// 2.6 to 59 tiles per CTA, 44 to 92 % of them staged; the rule takes the slower form by more than 1 % in 4 of them, by
// 1.9 % at most. us a step by one CTA per tile and walked, FP32: 36 of 256^2 (15 tiles per CTA, 70 %) 91.7, 95.9;
// 12 of 64^2 to 512^2 (7.4, 78 %) 46.7, 49.5; 13 of 384^2 (12, 80 %) 72.9, 71.6; 4 of 512^2 (6.7, 85 %) 43.0, 42.1; 40 of
// 256^2 to 512^2 (35, 79 %) 191, 184. FP16: 28 of 256^2 (12, 70 %) 94.5, 94.8; 5 of 384^2 (4.7, 80 %) 37.9, 39.8; 7 of 384^2 (6.6)
// 53.1, 51.6; 6 of 512^2 (10, 85 %) 75.4, 66.0.
template <class S, class R, int CAP> static cudaError_t walk_wanted_c(long long tiles, long long staged, bool* yes) {
  constexpr bool kHalf = is_half_t<S>::value;
  int resident = 0;
  const cudaError_t e = walk_resident<S, R, CAP>(&resident);
  if (e != cudaSuccess) return e;
  *yes = 10 * staged - (kHalf ? 19LL : 23LL) * (tiles - staged) >= (kHalf ? 20LL : 24LL) * resident;
  return cudaSuccess;
}
cudaError_t batch_walk_wanted(int prec, bool small, long long tiles, long long staged, bool* yes) {
  if (prec == 1)
    return small ? walk_wanted_c<float, float, kSegSmall>(tiles, staged, yes)
                 : walk_wanted_c<float, float, walk_capacity<float>()>(tiles, staged, yes);
  return small ? walk_wanted_c<__half, float, kSegSmall>(tiles, staged, yes)
               : walk_wanted_c<__half, float, walk_capacity<__half>()>(tiles, staged, yes);
}

template <class S, class R, int CAP>
static cudaError_t walk_launch_c(const void* Lh, unsigned long long* tickets, cudaStream_t st) {
  using B = TmaBox<S, 32, 8>;
  const WalkLaunch<S, CAP>& L = *(const WalkLaunch<S, CAP>*)Lh;
  int resident = 0;
  cudaError_t e = walk_resident<S, R, CAP>(&resident);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_batch_walk<S, R, 32, 8, CAP>, cudaFuncAttributeMaxDynamicSharedMemorySize, B::BYTES);
  if (e != cudaSuccess) return e;
  return launch_pdl(k_batch_walk<S, R, 32, 8, CAP>, resident, 256, B::BYTES, st, L, tickets);
}
cudaError_t batch_walk_launch(int prec, bool small, const void* L, unsigned long long* tickets, cudaStream_t st) {
  if (prec == 1)
    return small ? walk_launch_c<float, float, kSegSmall>(L, tickets, st)
                 : walk_launch_c<float, float, walk_capacity<float>()>(L, tickets, st);
  return small ? walk_launch_c<__half, float, kSegSmall>(L, tickets, st)
               : walk_launch_c<__half, float, walk_capacity<__half>()>(L, tickets, st);
}

template <class S, class R, int TX, int TY, int NPT, int CAP>
static cudaError_t seg_launch_t(const void* Lh, cudaStream_t st) {
  const SegLaunch<S, CAP>& L = *(const SegLaunch<S, CAP>*)Lh;
  if (L.n <= 0 || L.tiles <= 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)L.tiles);
  cfg.blockDim = dim3(TX * TY / NPT);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  // a step's first launch is an ordinary one: a wait in the kernel costs every tile of it 1 %
  cfg.numAttrs = L.waits ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, k_batch_tiles<S, R, TX, TY, NPT, CAP>, L);
}

template <class S, class R, int CAP>
static cudaError_t seg_launch_c(int variant, const void* L, cudaStream_t st) {
  switch (variant) {
    case 1: return seg_launch_t<S, R, 32, 16, 1, CAP>(L, st);
    case 2: return seg_launch_t<S, R, 64, 8, 1, CAP>(L, st);
    case 3: return seg_launch_t<S, R, 32, 16, 2, CAP>(L, st);
    case 4: return seg_launch_t<S, R, 64, 16, 2, CAP>(L, st);
    case 5: return seg_launch_t<S, R, 32, 32, 2, CAP>(L, st);
    default: return seg_launch_t<S, R, 32, 8, 1, CAP>(L, st);
  }
}

template <class S, class R>
static cudaError_t seg_launch_p(int variant, bool small, const void* L, cudaStream_t st) {
  return small ? seg_launch_c<S, R, kSegSmall>(variant, L, st)
               : seg_launch_c<S, R, seg_capacity<S>()>(variant, L, st);
}

cudaError_t batch_seg_launch(int prec, int variant, bool small, const void* L, cudaStream_t st) {
  if (prec == 0) return seg_launch_p<double, double>(variant, small, L, st);
  if (prec == 1) return seg_launch_p<float, float>(variant, small, L, st);
  return seg_launch_p<__half, float>(variant, small, L, st);
}

}  // namespace lbpc
