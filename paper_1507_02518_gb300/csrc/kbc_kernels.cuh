// kbc_kernels.cuh -- CUDA kernels of the D3Q27 KBC step and their launchers.
//
// Included once per storage type by kbc_f64.cu / kbc_f32.cu / kbc_f16.cu, which instantiate
// kbc::Ops<S>. Hot path: fix_step_kernel (FP64), adj_*_kernel (FP32 and FP16, even nx; with the
// FP64 re-collision inside for small boxes), pair_*_kernel (odd nx) and step_kernel: one fused
// stream + KBC collide per node, eq:Egeneral; batch_*_kernel run the same update over a work
// list of boxes. Transfer, diagnostics and pre-solve kernels are in kbc_aux.cuh.
#pragma once

#include <type_traits>
#include <utility>

#include "kbc_device.cuh"
#include "kbc_ops.h"
#include "kbc_staged.cuh"
#include "kbc_tma.cuh"

namespace kbc {

// FP64 arithmetic needs more than 128 registers per thread: cap its blocks at 256 threads
template <typename S> struct MaxThreads { static constexpr int value = 512; };
template <> struct MaxThreads<double> { static constexpr int value = 256; };

// Step and pass kernels follow one another on the stream, each depending on all of the one
// before. They are launched with programmatic stream serialisation: a kernel's blocks may take
// their places while the one before drains, and wait in follow() until all of it has finished
// and its writes are visible; follow() lets the next kernel's blocks do the same. A kernel
// that waits has only such kernels before it that are resident or done, so the chain always
// ends. What it hides is the launch latency between kernels and the start of the next one behind
// the last blocks of this: 32^3 FP32 AA (step and pass) 9.2 -> 5.4 us a step with the node order
// below, 256^3 pull 542 -> 537 us. Launched without the attribute, follow() does nothing.
// Blocks that wait on an SM take places there and unbalance the next kernel over the SMs, so the
// adjacent-pair steps let the next kernel in at their end only (let_next(): 32^3 FP32 pull 3.9 ->
// 3.4 us, AA without a pass 4.6 -> 3.2), and the FP64 step, whose blocks fill an SM with three, when
// its blocks exit (32^3 11.2 -> 8.7 us).
// Populations are read by ordinary loads only: __ldg() and ld.global.nc are for memory that nothing
// writes while the kernel lives, and a kernel of the chain lives while the one before writes what
// it will read (with small grids also while the one before that still reads the same buffer).
__device__ __forceinline__ void wait_before() { cudaGridDependencySynchronize(); }
__device__ __forceinline__ void let_next() { cudaTriggerProgrammaticLaunchCompletion(); }
__device__ __forceinline__ void follow() {
  let_next();
  wait_before();
}
template <typename... P, typename... A>
static cudaError_t launch_following(void (*kernel)(P...), dim3 grid, dim3 block, cudaStream_t st,
                                    A&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = st;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

template <typename S, int MODE, bool RECORD, bool CENTRAL, bool EXACT = false,
          bool POLY = false>
__global__ void __launch_bounds__(MaxThreads<S>::value) step_kernel(const S* src, S* dst, Geo g, CollideParams cp,
                                                   float* gamma_out, StepCounters* ctr) {
  const uint32_t x = blockIdx.x * blockDim.x + threadIdx.x;
  const uint32_t y = blockIdx.y * blockDim.y + threadIdx.y;
  const uint32_t z = blockIdx.z + g.zb;
  if (x >= g.nx || y >= g.ny) return;
  node_update<S, MODE, RECORD, CENTRAL, EXACT, POLY>(src, dst, g, x, y, z, cp, gamma_out, ctr);
}

// The FP64 step with the fixed-point collision, one node per thread over the node order, so that
// rows of any length keep every lane busy (the two divisions are nothing beside the ~4000
// instructions of the collision): with 128-thread rows 22 % of a 100^3 box's lanes idled. 128
// registers give 16 warps per SM: 256^3 pull 3.20 ms, 3.58 at 168 (12 warps), 3.31 at 112 (all in one
// session; 3.27 in others); 100^3 AA 196, 218, 204 us; 32^3 pull 11.3, 11.0, 11.7.
template <int MODE, bool RECORD>
__global__ void __maxnreg__(128) fix_step_kernel(const double* src, double* dst, Geo g,
                                                         CollideParams cp, float* gamma_out,
                                                         StepCounters* ctr) {
  wait_before();
  const uint32_t n = g.zb * g.nxy + blockIdx.x * blockDim.x + threadIdx.x;  // P < 2^31
  if (n >= g.ze * g.nxy) return;
  const uint32_t row = n / g.nx;
  const uint32_t x = n - row * g.nx;
  const uint32_t z = row / g.ny;
  node_update<double, MODE, RECORD>(src, dst, g, x, row - z * g.ny, z, cp, gamma_out, ctr);
}

// Moves node (x, y, z) of a box with rows of nx nodes and planes of ny rows k nodes forward in
// the node order (x fastest); x may start at or beyond nx (it is reduced first).
__device__ __forceinline__ void advance_node(uint32_t& x, uint32_t& y, uint32_t& z, uint32_t k,
                                             uint32_t nx, uint32_t ny) {
  x += k;
  if (x >= nx) {
    const uint32_t r = x / nx;
    x -= r * nx;
    y += r;
    if (y >= ny) {
      const uint32_t p = y / ny;
      y -= p * ny;
      z += p;
    }
  }
}

// Brings into L2 what the blocks one wave ahead will load (kWave blocks are resident on the
// chip: 3 on each of 152 SMs): of each of the 27 planes the warp's share of the tile that starts
// kWave blocks after node n, moved by the plane's velocity as the step's loads are (ahead_node()), a
// 128-byte line per lane. With 12 warps per SM the loads' latency is what the step waits for. us a
// step without -> with: adjacent pairs FP16 256^3 AA 422 -> 387, pull 413 -> 384, FP32 AA 256^3 550 ->
// 540, 768^3 14722 -> 14336, 1536 x 768 x 192 7361 -> 7134; pairs (n, n + 32) FP32 201^3 AA 325 -> 304,
// pull 293 -> 289, central moments FP32 pull 192^3 271 -> 260, 384^3 2130 -> 2030. (Lines of the same
// node in every plane, without the move, are read after their use where a plane of the box is larger
// than a wave's nodes: 1536 x 768 x 192 FP32 AA 8146.) The adjacent-pair FP32 pull step, at the DRAM
// rate already, lost (256^3 537 -> 555) and does without. (200 or 912 blocks ahead: FP16 AA 391, 390
// where 456 took 378. Loading the next tile into registers instead takes 238 of them, 8 warps per SM:
// 438.)
constexpr uint32_t kWave = 456;
template <typename S, int MODE>
__device__ __forceinline__ void prefetch_ahead(const S* src, const Geo& g, uint32_t n) {
  const uint32_t lane = threadIdx.x & 31;
  n += kWave * 2 * blockDim.x + 2 * (threadIdx.x & ~31u);
  if (lane < 27 && n < (uint32_t)g.P) {
    n = ahead_node<MODE>(g, lane, n);
    const S* p = src + (uint64_t)lane * g.P + n;
    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
    // FP32: the second half of the warp's 64 nodes
    if (sizeof(S) == 4 && n + 32 < (uint32_t)g.P) asm volatile("prefetch.global.L2 [%0];" ::"l"(p + 32));
  }
}
// where it is worth its instructions: a step's populations (pull: both buffers) larger than L2
// (129 MB); FP16 pull 112^3 41.5 -> 38.4 us, 128^3 54.4 -> 50.8
template <typename S, int MODE> __host__ __device__ inline bool beyond_l2(const Geo& g) {
  return 27 * g.P * sizeof(S) * (MODE == MODE_PULL ? 2 : 1) > (129ull << 20);
}

// Two nodes per thread with packed FP32x2 arithmetic: a block of up to 128 threads covers
// 2 x blockDim.x consecutive x nodes of one row, each warp 64 of them as (x, x + 32) pairs.
template <typename S, int MODE, bool RECORD, bool CENTRAL, bool POLY, bool AHEAD>
__global__ void __launch_bounds__(128, 3) pair_step_kernel(const S* src, S* dst, Geo g,
                                                        CollideParams cp, float* gamma_out,
                                                        StepCounters* ctr) {
  follow();
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t xa = blockIdx.x * (2 * blockDim.x) + warp * 64 + lane;
  if (xa >= g.nx) return;
  if constexpr (AHEAD)
    prefetch_ahead<S, MODE>(src, g, (blockIdx.z + g.zb) * g.nxy + blockIdx.y * g.nx +
                                        blockIdx.x * (2 * blockDim.x));
  const bool vb = xa + 32 < g.nx;
  const uint32_t z = blockIdx.z + g.zb;
  node_update2<S, MODE, RECORD, CENTRAL, POLY>(src, dst, g, xa, blockIdx.y, z,
                                               vb ? xa + 32 : xa, blockIdx.y, z, vb,
                                               cp, gamma_out, ctr);
}

// Two adjacent nodes per thread, (x, x + 1) with x even: a block of blockDim.x threads covers
// 2 blockDim.x consecutive nodes of one row (nx even).
template <typename S, int MODE, bool RECORD, bool AHEAD>
__global__ void __launch_bounds__(128, 3) adj_step_kernel(const S* src, S* dst, Geo g,
                                                       CollideParams cp, float* gamma_out,
                                                       StepCounters* ctr) {
  wait_before();
  if constexpr (AHEAD)
    prefetch_ahead<S, MODE>(src, g, (blockIdx.z + g.zb) * g.nxy + blockIdx.y * g.nx +
                                        2 * blockIdx.x * blockDim.x);
  const uint32_t x = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  if (x >= g.nx) return;
  node_update_adj<S, MODE, RECORD>(src, dst, g, x, blockIdx.y, blockIdx.z + g.zb, cp,
                                   gamma_out, ctr);
  let_next();
}

// The same over the box's node order: pair k is nodes (2k, 2k + 1), which share a row as nx is
// even. For rows that are no multiple of 64 nodes this keeps every lane busy (at 32 nodes half of a
// warp idled), at the price of two divisions per thread: FP32 pull 48^3 11.3 -> 5.2 us, 200^3 303 ->
// 268, FP32 AA 96^3 41 -> 34 (with the overlapped launches).
template <typename S, int MODE, bool RECORD, bool AHEAD>
__global__ void __launch_bounds__(128, 3) adj_linear_kernel(const S* src, S* dst, Geo g,
                                                         CollideParams cp, float* gamma_out,
                                                         StepCounters* ctr) {
  wait_before();
  const uint32_t n = g.zb * g.nxy + 2 * (blockIdx.x * blockDim.x + threadIdx.x);  // P < 2^31
  if (n >= g.ze * g.nxy) return;
  if constexpr (AHEAD) prefetch_ahead<S, MODE>(src, g, n - 2 * threadIdx.x);
  const uint32_t row = n / g.nx;
  const uint32_t z = row / g.ny;
  node_update_adj<S, MODE, RECORD>(src, dst, g, n - row * g.nx, row - z * g.ny, z, cp, gamma_out,
                                   ctr);
  let_next();
}

// The adjacent-pair FP32 step of a small box, over the node order, with the FP64 re-collision in the
// kernel instead of in a pass after it: the launch of the pass costs as much as the step there.
// node_update_adj<..., true> hands back the flagged lanes (their FP32 results are stored by the pull
// step, not by AA); a lane's FP64 collision needs its own inputs only, which are still in place.
// Rule: up to 2^18 nodes. us a step with the pass -> without: FP32 pull 16^3 3.5 -> 2.6 (the rate at
// which the host launches), 32^3 3.6 -> 2.7, 48^3 5.1 -> 4.2, 64^3 9.0 -> 8.3, AA 32^3 5.2 -> 3.2, 64^3
// 9.6 -> 9.3; beyond, the call in the step kernel costs more than the pass (128^3 AA 69.8 -> 77.3).
// That is with nothing flagged; with flagged nodes the pass, a few blocks on a small box, is the slower
// one by more (pull, with the pass -> here): every node flagged (uniform flow) 32^3 375 -> 18, 64^3 398
// -> 67 us a step; the first 20 steps of a Taylor-Green field 32^3 25.9 -> 4.8, 64^3 31 -> 12, of a Kida
// field 27.3 -> 6.2, 34 -> 15.
constexpr uint64_t kSmallNodes = 1ull << 18;
template <int MODE>
__device__ __noinline__ void recollide_here(const float* src, float* dst, Geo g, uint32_t n,
                                            CollideParams cp, float* gamma_out,
                                            StepCounters* ctr) {
  const uint32_t row = n / g.nx, z = row / g.ny;
  int gd = 0;
  const float gam = fix_node_update<float, MODE>(src, dst, g, n - row * g.nx, row - z * g.ny, z, cp,
                                                 &gd);
  if (gamma_out) {
    gamma_out[n] = gam;
    if (gd) atomicAdd(&ctr->guarded, 1ull);
  }
}
template <int MODE, bool RECORD>
__global__ void __launch_bounds__(128, 3) adj_small_kernel(const float* src, float* dst, Geo g,
                                                        CollideParams cp, float* gamma_out,
                                                        StepCounters* ctr) {
  wait_before();
  const uint32_t n = g.zb * g.nxy + 2 * (blockIdx.x * blockDim.x + threadIdx.x);  // P < 2^31
  if (n >= g.ze * g.nxy) return;
  const uint32_t row = n / g.nx;
  const uint32_t z = row / g.ny;
  int flagged = 0;
  node_update_adj<float, MODE, RECORD, true>(src, dst, g, n - row * g.nx, row - z * g.ny, z, cp,
                                             gamma_out, ctr, &flagged);
  if (flagged & 1) recollide_here<MODE>(src, dst, g, n, cp, RECORD ? gamma_out : nullptr, ctr);
  if (flagged & 2) recollide_here<MODE>(src, dst, g, n + 1, cp, RECORD ? gamma_out : nullptr, ctr);
  let_next();
}
// whether the step of this box re-collides its flagged nodes itself (no pass follows)
template <typename S, bool CENTRAL, bool POLY>
inline bool small_step(const Geo& g, const CollideParams& cp, const StepOpts& o) {
  return std::is_same<S, float>::value && !CENTRAL && !POLY && g.nx % 2 == 0 && g.P <= kSmallNodes &&
         cp.gamma_mode == GAMMA_ESTIMATE && (o.kernel == KERNEL_ADJ || o.kernel == KERNEL_AUTO);
}

// Rows of a multiple of 64 nodes: blocks of whole row segments; other rows: the node order.
template <typename S, int MODE, bool RECORD>
static cudaError_t launch_adj(const S* src, S* dst, const Geo& g, const CollideParams& cp,
                              float* gamma_out, StepCounters* ctr, bool small, cudaStream_t st) {
  const uint32_t pairs = g.nx / 2;
  if constexpr (std::is_same<S, float>::value) {
    if (small) {
      const uint32_t all = pairs * g.ny * (g.ze - g.zb);
      return launch_following(adj_small_kernel<MODE, RECORD>, (all + 127) / 128, 128, st, src, dst,
                              g, cp, gamma_out, ctr);
    }
  }
  auto run = [&](auto ahead) {
    constexpr bool A = decltype(ahead)::value;
    if (pairs % 32 != 0) {
      const uint32_t all = pairs * g.ny * (g.ze - g.zb);
      return launch_following(adj_linear_kernel<S, MODE, RECORD, A>, (all + 127) / 128, 128, st,
                              src, dst, g, cp, gamma_out, ctr);
    }
    const uint32_t threads = pairs >= 128 ? 128 : pairs;
    const dim3 grid((pairs + threads - 1) / threads, g.ny, g.ze - g.zb);
    return launch_following(adj_step_kernel<S, MODE, RECORD, A>, grid, threads, st, src, dst, g, cp,
                            gamma_out, ctr);
  };
  if constexpr (sizeof(S) == 2 || MODE != MODE_PULL) {
    if (beyond_l2<S, MODE>(g)) return run(std::true_type{});
  }
  return run(std::false_type{});
}

// The same update over the box's node order instead of rows: block k covers nodes
// [256 k, 256 k + 256), each warp 64 of them as pairs (n, n + 32), which may straddle rows.
// For row lengths that are not a multiple of 64 this keeps every lane busy, at the price of
// two divisions per thread for the coordinates and of two coordinate triples kept live.
template <typename S, int MODE, bool RECORD, bool CENTRAL, bool POLY = false>
__global__ void __launch_bounds__(128, 3) pair_linear_kernel(const S* src, S* dst, Geo g,
                                                          CollideParams cp, float* gamma_out,
                                                          StepCounters* ctr) {
  follow();
  const uint32_t warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t nend = g.ze * g.nxy;  // P < 2^31
  const uint32_t n = g.zb * g.nxy + blockIdx.x * 256 + warp * 64 + lane;
  if (n >= nend) return;
  if (beyond_l2<S, MODE>(g)) prefetch_ahead<S, MODE>(src, g, g.zb * g.nxy + blockIdx.x * 256);
  const uint32_t row = n / g.nx;
  const uint32_t xa = n - row * g.nx;
  const uint32_t za = row / g.ny;
  const uint32_t ya = row - za * g.ny;
  uint32_t xb = xa, yb = ya, zb = za;
  const bool vb = n + 32 < nend;
  if (vb) advance_node(xb, yb, zb, 32, g.nx, g.ny);
  node_update2<S, MODE, RECORD, CENTRAL, POLY, false>(src, dst, g, xa, ya, za, xb, yb, zb, vb,
                                                      cp, gamma_out, ctr);
}

// Warps per block of the pair kernel: a row needs ceil(nx / 64) warps; blocks of w <= 4 warps
// launch ceil(rows' warps / w) w warps per row, so take the w with the fewest warps left
// without nodes (the larger w on a tie): nx = 100 -> 2, 256 -> 4, 400 -> 1, 600 -> 2.
inline uint32_t pair_block_warps(uint32_t nx) {
  const uint32_t need = (nx + 63) / 64;
  uint32_t best = 4, best_idle = (need + 3) / 4 * 4 - need;
  for (uint32_t w = 3; w >= 1; --w) {
    const uint32_t idle = (need + w - 1) / w * w - need;
    if (idle < best_idle) {
      best = w;
      best_idle = idle;
    }
  }
  return best;
}

// Blocks of whole row segments (a persistent grid measured slower on GB300), sized by
// pair_block_warps; when that leaves more than 5 % of the lanes without a node (rows that are
// not close to a multiple of 64 nodes long), blocks of 256 consecutive nodes instead.
template <typename S, int MODE, bool RECORD, bool CENTRAL, bool POLY = false>
static cudaError_t launch_pair(const S* src, S* dst, const Geo& g, const CollideParams& cp,
                               float* gamma_out, StepCounters* ctr, cudaStream_t st) {
  const uint32_t warps = pair_block_warps(g.nx);
  const uint32_t row_blocks = (g.nx + 64 * warps - 1) / (64 * warps);
  const uint64_t nodes = (uint64_t)(g.ze - g.zb) * g.nxy;
  if (20 * (uint64_t)g.nx < 19 * (uint64_t)row_blocks * 64 * warps) {
    return launch_following(pair_linear_kernel<S, MODE, RECORD, CENTRAL, POLY>,
                            (unsigned)((nodes + 255) / 256), 128, st, src, dst, g, cp, gamma_out,
                            ctr);
  }
  const dim3 grid(row_blocks, g.ny, g.ze - g.zb);
  auto run = [&](auto ahead) {
    return launch_following(
        pair_step_kernel<S, MODE, RECORD, CENTRAL, POLY, decltype(ahead)::value>, grid, 32 * warps,
        st, src, dst, g, cp, gamma_out, ctr);
  };
  if (beyond_l2<S, MODE>(g)) return run(std::true_type{});
  return run(std::false_type{});
}

// the geometry and collision parameters of box `bd` of a batch (the whole box is stepped;
// flagged nodes also set the batch-wide flag fb_batch)
__device__ __forceinline__ Geo box_geo(const BoxDesc& bd, unsigned int* fb_batch) {
  Geo g;
  g.nx = bd.nx;
  g.ny = bd.ny;
  g.nz = bd.nz;
  g.nxy = bd.nxy;
  g.P = (uint64_t)bd.nxy * bd.nz;
  g.zb = 0;
  g.ze = bd.nz;
  g.fbmask = bd.fbmask;
  g.fb_any = &bd.ctr->fb_any;
  g.fb_batch = fb_batch;
  return g;
}

__device__ __forceinline__ CollideParams box_cp(const BoxDesc& bd, int with_t, int with_q,
                                                int gamma_mode) {
  CollideParams cp;
  cp.beta = bd.beta;
  cp.two_beta = bd.two_beta;
  cp.inv_beta = bd.inv_beta;
  cp.betaf = (float)bd.beta;
  cp.two_betaf = (float)bd.two_beta;
  cp.inv_betaf = (float)bd.inv_beta;
  cp.quarter_beta = bd.quarter_beta;
  cp.two_beta_1 = bd.two_beta_1;
  cp.with_t = with_t;
  cp.with_q = with_q;
  cp.gamma_mode = gamma_mode;
  return cp;
}

// Batched ensemble: a persistent grid walks the work list; item k covers rows
// [row0, row0 + nrows) (row = y + ny z) of one box. (This kernel: FP64 storage, and one node per
// thread; 24 FP64 boxes of 32^3 to 128^3, 14.3 ms a step in FP64 instructions, 3.74 in fixed point.)
template <typename S, int MODE, bool RECORD, bool CENTRAL>
__global__ void __launch_bounds__(MaxThreads<S>::value) batch_kernel(const BoxDesc* __restrict__ boxes,
                                                    const WorkItem* __restrict__ items,
                                                    int nitems, BatchFlags* flags, int parity,
                                                    int with_t, int with_q, int gamma_mode) {
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const WorkItem w = items[it];
    const BoxDesc bd = boxes[w.box];
    const Geo g = box_geo(bd, &flags->any);
    const CollideParams cp = box_cp(bd, with_t, with_q, gamma_mode);
    const S* src = (const S*)bd.pop[MODE == MODE_PULL ? parity : 0];
    S* dst = (S*)bd.pop[MODE == MODE_PULL ? (parity ^ 1) : 0];
    const uint32_t nodes = bd.nx * (uint32_t)w.nrows;
    for (uint32_t k = threadIdx.x; k < nodes; k += blockDim.x) {
      const uint32_t row = (uint32_t)w.row0 + k / bd.nx;
      const uint32_t x = k - (k / bd.nx) * bd.nx;
      const uint32_t z = row / bd.ny;
      const uint32_t y = row - z * bd.ny;
      node_update<S, MODE, RECORD, CENTRAL>(src, dst, g, x, y, z, cp, bd.gamma, bd.ctr);
    }
  }
}

// The packed form of batch_kernel: 128 threads, each item's rows cut into 64-node chunks,
// each thread two nodes (x, x + 32) of a chunk with the FP32x2 collision.
template <typename S, int MODE, bool RECORD, bool CENTRAL>
__global__ void __launch_bounds__(128, 3) batch_pair_kernel(const BoxDesc* __restrict__ boxes,
                                                           const WorkItem* __restrict__ items,
                                                           int nitems, BatchFlags* flags, int parity,
                                                           int with_t, int with_q, int gamma_mode) {
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const WorkItem w = items[it];
    const BoxDesc bd = boxes[w.box];
    const Geo g = box_geo(bd, &flags->any);
    const CollideParams cp = box_cp(bd, with_t, with_q, gamma_mode);
    const S* src = (const S*)bd.pop[MODE == MODE_PULL ? parity : 0];
    S* dst = (S*)bd.pop[MODE == MODE_PULL ? (parity ^ 1) : 0];
    // The item's rows are one contiguous range of nodes: warp q handles its nodes
    // [64 q, 64 q + 64) as pairs (n, n + 32), so rows of any length keep every lane busy
    // (rows shorter or longer than a multiple of 64 nodes share warps). The coordinates of
    // a advance by the block's 256 nodes per iteration, those of b are a's plus 32; a row
    // crossing costs one division, none otherwise. blockDim.x is 128 for this kernel.
    const uint32_t nodes = bd.nx * (uint32_t)w.nrows;
    const uint32_t wstep = blockDim.x >> 5, slot = threadIdx.x & 31;
    const uint32_t stride = 64 * wstep;
    uint32_t la = 64 * (threadIdx.x >> 5) + slot;
    uint32_t za = (uint32_t)w.row0 / bd.ny;
    uint32_t ya = (uint32_t)w.row0 - za * bd.ny, xa = 0;
    advance_node(xa, ya, za, la, bd.nx, bd.ny);
    for (; la < nodes; la += stride) {
      uint32_t xb = xa, yb = ya, zb = za;
      const bool vb = la + 32 < nodes;
      if (vb) advance_node(xb, yb, zb, 32, bd.nx, bd.ny);
      node_update2<S, MODE, RECORD, CENTRAL, false, false>(src, dst, g, xa, ya, za, xb, yb, zb,
                                                           vb, cp, bd.gamma, bd.ctr);
      advance_node(xa, ya, za, stride, bd.nx, bd.ny);
    }
  }
}

// The adjacent-pair form of the batched step (every box of the batch has an even nx; product
// form, natural moments): each thread takes nodes (x, x + 1) of a row, x even, walking the
// item's node range 256 nodes per block pass (coordinates advance incrementally).
template <typename S, int MODE, bool RECORD>
__global__ void __launch_bounds__(128, 3) batch_adj_kernel(const BoxDesc* __restrict__ boxes,
                                                          const WorkItem* __restrict__ items,
                                                          int nitems, BatchFlags* flags, int parity,
                                                          int with_t, int with_q, int gamma_mode) {
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    const WorkItem w = items[it];
    const BoxDesc bd = boxes[w.box];
    const Geo g = box_geo(bd, &flags->any);
    const CollideParams cp = box_cp(bd, with_t, with_q, gamma_mode);
    const S* src = (const S*)bd.pop[MODE == MODE_PULL ? parity : 0];
    S* dst = (S*)bd.pop[MODE == MODE_PULL ? (parity ^ 1) : 0];
    const uint32_t nodes = bd.nx * (uint32_t)w.nrows;
    const uint32_t stride = 2 * blockDim.x;
    uint32_t n = 2 * threadIdx.x;
    uint32_t z = (uint32_t)w.row0 / bd.ny;
    uint32_t y = (uint32_t)w.row0 - z * bd.ny, x = 0;
    advance_node(x, y, z, n, bd.nx, bd.ny);
    for (; n < nodes; n += stride) {
      node_update_adj<S, MODE, RECORD>(src, dst, g, x, y, z, cp, bd.gamma, bd.ctr);
      advance_node(x, y, z, stride, bd.nx, bd.ny);
    }
  }
}

// ------------------------------------------------------------------ FP64 re-collision pass
// A step kernel (FP32 storage) that meets a node whose FP32 <dh|dh> fell under kDenFp64 sets
// its bit in the box's mask (flag_fp64) and, in AA, does not store it. The pass launched
// after it collides every flagged node again in FP64 from its inputs (fix_node_update) and
// clears the mask. When nothing was flagged (the usual case) it
// reads one flag and exits. The last of its blocks to finish clears the flags; all blocks
// have read them by then.
constexpr int kPassThreads = 384;  // 12 warps at 168 registers
constexpr int kPassBlocks = 152;   // one wave: the pass kernels run one block per SM

// the flagged nodes among the mask words of warps w0, w0 + stride, ... (32 words a warp);
// returns the guard events. A warp takes its words' flagged nodes 32 at a time in the node order,
// a node per lane, so that runs of flagged nodes are read and written coalesced; a node per word
// and thread (words in a loop over their bits) touched a sector per value: a full 256^3 box took
// 20 ms, 4.2 now (3.7 with a fixed unit and products rounded down throughout, see kbc_fix.cuh).
template <typename S, int MODE, bool CENTRAL, bool POLY>
__device__ unsigned long long fp64_pass_words(const S* src, S* dst, const Geo& g,
                                              const CollideParams& cp,
                                              float* gamma_out, int record, uint32_t w0,
                                              uint32_t stride) {
  const uint32_t words = (uint32_t)((g.P + 31) >> 5), lane = threadIdx.x & 31;
  unsigned long long guards = 0;
  for (uint32_t base = 32 * w0; base < words; base += 32 * stride) {
    const uint32_t w = base + lane;
    const uint32_t mine = w < words ? g.fbmask[w] : 0;
    if (!__any_sync(0xffffffffu, mine != 0)) continue;
    if (mine) g.fbmask[w] = 0;
    uint32_t end = __popc(mine);  // flagged nodes up to and including this lane's word
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += up;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, end, 31);
    for (uint32_t k0 = 0; k0 < total; k0 += 32) {
      const uint32_t k = k0 + lane;
      uint32_t slot = 0;  // the word that holds the k-th flagged node: the first with end > k
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const uint32_t e = __shfl_sync(0xffffffffu, end, slot + o - 1);
        if (e <= k) slot += o;
      }
      slot = slot > 31 ? 31 : slot;
      const uint32_t m = __shfl_sync(0xffffffffu, mine, slot);
      const uint32_t e = __shfl_sync(0xffffffffu, end, slot);
      if (k >= total) continue;
      const uint32_t bit = __fns(m, 0, (int)(k - (e - __popc(m))) + 1);
      const uint32_t n = 32 * (base + slot) + bit;
      const uint32_t z = n / g.nxy, r = n - z * g.nxy;
      const uint32_t y = r / g.nx, x = r - y * g.nx;
      int gd = 0;
      float gam;
      if constexpr (!CENTRAL && !POLY)
        gam = fix_node_update<S, MODE>(src, dst, g, x, y, z, cp, &gd);
      else
        gam = fp64_node_native<S, MODE, CENTRAL, POLY>(src, dst, g, x, y, z, cp, &gd);
      if (record) {
        gamma_out[n] = gam;
        guards += (unsigned long long)gd;
      }
    }
  }
  return guards;
}

// true in thread 0 of the last block of the grid to get here (after __syncthreads)
__device__ __forceinline__ bool pass_last_block(unsigned int* done) {
  __syncthreads();
  if (threadIdx.x != 0) return false;
  __threadfence();
  return atomicAdd(done, 1u) == gridDim.x - 1;
}

template <typename S, int MODE, bool CENTRAL, bool POLY>
__global__ void __launch_bounds__(kPassThreads) fp64_pass_kernel(const S* src, S* dst, Geo g,
                                                                 CollideParams cp,
                                                                 float* gamma_out,
                                                                 StepCounters* ctr, int record) {
  follow();
  if (*(volatile unsigned int*)&ctr->fb_any == 0) return;
  const unsigned long long guards =
      fp64_pass_words<S, MODE, CENTRAL, POLY>(src, dst, g, cp, gamma_out, record,
                                              (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                                              (gridDim.x * blockDim.x) >> 5);
  if (guards) atomicAdd(&ctr->guarded, guards);
  if (pass_last_block(&ctr->fb_done)) {
    ctr->fb_any = 0;
    ctr->fb_done = 0;
  }
}

// the same over the boxes of a batch (boxes that flagged nothing are skipped)
template <typename S, int MODE, bool CENTRAL>
__global__ void __launch_bounds__(kPassThreads) batch_fp64_pass_kernel(
    const BoxDesc* __restrict__ boxes, int nbox, BatchFlags* flags, int parity, int with_t,
    int with_q, int gamma_mode, int record) {
  if (*(volatile unsigned int*)&flags->any == 0) return;
  for (int k = 0; k < nbox; ++k) {
    const BoxDesc bd = boxes[k];
    if (*(volatile unsigned int*)&bd.ctr->fb_any == 0) continue;
    const Geo g = box_geo(bd, nullptr);
    const CollideParams cp = box_cp(bd, with_t, with_q, gamma_mode);
    const S* src = (const S*)bd.pop[MODE == MODE_PULL ? parity : 0];
    S* dst = (S*)bd.pop[MODE == MODE_PULL ? (parity ^ 1) : 0];
    const unsigned long long guards =
        fp64_pass_words<S, MODE, CENTRAL, false>(src, dst, g, cp, bd.gamma, record,
                                                 (blockIdx.x * blockDim.x + threadIdx.x) >> 5,
                                                 (gridDim.x * blockDim.x) >> 5);
    if (guards) atomicAdd(&bd.ctr->guarded, guards);
  }
  if (pass_last_block(&flags->done)) {
    for (int k = 0; k < nbox; ++k) boxes[k].ctr->fb_any = 0;
    flags->any = 0;
    flags->done = 0;
  }
}

// ------------------------------------------------------------------ host launchers
inline Geo make_geo(const BoxView& b) {
  Geo g;
  g.nx = b.nx;
  g.ny = b.ny;
  g.nz = b.nz;
  g.nxy = b.nx * b.ny;
  g.P = b.P;
  g.zb = b.zb;
  g.ze = b.ze;
  g.fbmask = b.fbmask;
  g.fb_any = nullptr;
  g.fb_batch = nullptr;
  return g;
}

inline CollideParams make_cp(double beta, int with_t, int with_q, int gamma_mode) {
  CollideParams cp;
  cp.beta = beta;
  cp.two_beta = 2.0 * beta;
  cp.inv_beta = 1.0 / beta;
  cp.betaf = (float)cp.beta;
  cp.two_betaf = (float)cp.two_beta;
  cp.inv_betaf = (float)cp.inv_beta;
  cp.quarter_beta = fix::quarter_beta(beta);
  cp.two_beta_1 = fix::two_beta_1(beta);
  cp.with_t = with_t;
  cp.with_q = with_q;
  cp.gamma_mode = gamma_mode;
  return cp;
}

inline int grid_for(uint64_t cnt, int threads) {
  uint64_t blocks = (cnt + threads - 1) / threads;
  const uint64_t cap = 152ull * 16;
  if (blocks > cap) blocks = cap;
  if (blocks < 1) blocks = 1;
  return (int)blocks;
}

template <typename S, int MODE, bool RECORD, bool CENTRAL, bool POLY>
static cudaError_t launch_step_c(const BoxView& b, const S* src, S* dst, const Geo& g,
                                 const CollideParams& cp, const StepOpts& o, StepCounters* ctr,
                                 cudaStream_t st) {
  if constexpr (!POLY) {
    if (cp.gamma_mode == GAMMA_EXACT) {  // one node per thread, whatever kernel was chosen
      const dim3 block(o.bx, o.by, 1);
      const dim3 grid((b.nx + o.bx - 1) / o.bx, (b.ny + o.by - 1) / o.by, g.ze - g.zb);
      step_kernel<S, MODE, RECORD, CENTRAL, true><<<grid, block, 0, st>>>(src, dst, g, cp,
                                                                          b.gamma, ctr);
      return cudaGetLastError();
    }
  }
  if constexpr (!CENTRAL && !POLY) {
    if (o.kernel == KERNEL_STAGED)
      return launch_staged<S, MODE, RECORD>(src, dst, g, cp, b.gamma, ctr, o.budget, o.stall, st);
    if (o.kernel == KERNEL_PERSISTENT)
      return launch_persistent<S, MODE, RECORD>(src, dst, g, cp, b.gamma, ctr,
                                                (uint32_t)o.prefetch, st);
  }
  if constexpr (!std::is_same<S, double>::value) {
    if constexpr (!CENTRAL && !POLY) {
      if (o.kernel == KERNEL_ROWS)
        return launch_rows<S, MODE, RECORD>(src, dst, g, cp, b.gamma, ctr, o.budget, o.stall, st);
      // the default for even rows: adjacent pairs (measured faster than (x, x + 32) pairs at
      // 256^3: FP32 AA 0.549 vs 0.630 ms, FP16 AA 0.446 vs 0.504 ms, pull equal or better)
      if ((o.kernel == KERNEL_ADJ || o.kernel == KERNEL_AUTO) && g.nx % 2 == 0)
        return launch_adj<S, MODE, RECORD>(src, dst, g, cp, b.gamma, ctr,
                                           small_step<S, CENTRAL, POLY>(g, cp, o), st);
    }
    if (o.kernel == KERNEL_PACKED || o.kernel == KERNEL_AUTO || o.kernel == KERNEL_ROWS)
      return launch_pair<S, MODE, RECORD, CENTRAL, POLY>(src, dst, g, cp, b.gamma, ctr, st);
  }
  if constexpr (std::is_same<S, double>::value && !CENTRAL && !POLY) {
    const uint32_t threads = o.bx * o.by;
    const uint32_t nodes = (g.ze - g.zb) * g.nxy;
    return launch_following(fix_step_kernel<MODE, RECORD>, (nodes + threads - 1) / threads, threads,
                            st, src, dst, g, cp, b.gamma, ctr);
  }
  const dim3 block(o.bx, o.by, 1);
  const dim3 grid((b.nx + o.bx - 1) / o.bx, (b.ny + o.by - 1) / o.by, g.ze - g.zb);
  step_kernel<S, MODE, RECORD, CENTRAL, false, POLY><<<grid, block, 0, st>>>(src, dst, g, cp,
                                                                             b.gamma, ctr);
  return cudaGetLastError();
}

// the step kernel, then (FP32 storage, the estimate of eq:result21: the only case that
// flags nodes) the FP64 re-collision pass over the nodes it flagged
template <typename S, int MODE, bool RECORD, bool CENTRAL, bool POLY>
static cudaError_t launch_step_p(const BoxView& b, const S* src, S* dst, const Geo& g,
                                 const CollideParams& cp, const StepOpts& o, StepCounters* ctr,
                                 cudaStream_t st) {
  cudaError_t e = launch_step_c<S, MODE, RECORD, CENTRAL, POLY>(b, src, dst, g, cp, o, ctr, st);
  if constexpr (std::is_same<S, float>::value) {
    if (e == cudaSuccess && cp.gamma_mode == GAMMA_ESTIMATE &&
        !small_step<S, CENTRAL, POLY>(g, cp, o)) {
      const uint64_t warps = (g.P + 1023) / 1024;  // a warp takes 32 mask words
      uint64_t blocks = (32 * warps + kPassThreads - 1) / kPassThreads;
      if (blocks > (uint64_t)kPassBlocks) blocks = kPassBlocks;
      e = launch_following(fp64_pass_kernel<S, MODE, CENTRAL, POLY>, (unsigned)blocks, kPassThreads,
                           st, src, dst, g, cp, b.gamma, ctr, RECORD ? 1 : 0);
    }
  }
  return e;
}

template <typename S, int MODE, bool RECORD>
static cudaError_t launch_step(const BoxView& b, const S* src, S* dst, const Geo& g,
                               const CollideParams& cp, const StepOpts& o, StepCounters* ctr,
                               cudaStream_t st) {
  if (b.poly) {
    if (b.central)
      return launch_step_p<S, MODE, RECORD, true, true>(b, src, dst, g, cp, o, ctr, st);
    return launch_step_p<S, MODE, RECORD, false, true>(b, src, dst, g, cp, o, ctr, st);
  }
  if (b.central)
    return launch_step_p<S, MODE, RECORD, true, false>(b, src, dst, g, cp, o, ctr, st);
  return launch_step_p<S, MODE, RECORD, false, false>(b, src, dst, g, cp, o, ctr, st);
}

template <typename S>
bool Ops<S>::staged_ok(uint32_t nx) {
  return staged_supported<S>(nx);
}

template <typename S>
bool Ops<S>::rows_ok(uint32_t nx, uint32_t ny, uint32_t nz) {
  if constexpr (std::is_same<S, double>::value) {
    return false;
  } else {
    Geo g;
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.nxy = nx * ny;
    g.P = (uint64_t)nx * ny * nz;
    g.zb = 0;
    g.ze = nz;
    g.fbmask = nullptr;
    g.fb_any = g.fb_batch = nullptr;
    RowsArgs a;
    return rows_shape<S>(g, &a);
  }
}

template <typename S>
cudaError_t Ops<S>::step(const BoxView& b, int64_t t, bool record, const StepOpts& o,
                         StepCounters* counters, cudaStream_t st) {
  Geo g = make_geo(b);
  g.fb_any = &counters->fb_any;
  const CollideParams cp = make_cp(b.beta, b.with_t, b.with_q, b.gamma_mode);
  const int parity = (int)(t & 1);
  if (b.scheme == 0) {
    const S* src = (const S*)b.pop[parity];
    S* dst = (S*)b.pop[parity ^ 1];
    return record ? launch_step<S, MODE_PULL, true>(b, src, dst, g, cp, o, counters, st)
                  : launch_step<S, MODE_PULL, false>(b, src, dst, g, cp, o, counters, st);
  }
  S* buf = (S*)b.pop[0];
  if (parity == 0)
    return record ? launch_step<S, MODE_AA_EVEN, true>(b, buf, buf, g, cp, o, counters, st)
                  : launch_step<S, MODE_AA_EVEN, false>(b, buf, buf, g, cp, o, counters, st);
  return record ? launch_step<S, MODE_AA_ODD, true>(b, buf, buf, g, cp, o, counters, st)
                : launch_step<S, MODE_AA_ODD, false>(b, buf, buf, g, cp, o, counters, st);
}

// Launch arguments shared by the batch kernels.
struct BatchArgs {
  const BoxDesc* boxes;
  int nbox;
  BatchFlags* flags;
  const WorkItem* items;
  int nitems, parity, with_t, with_q, gamma_mode, threads, grid;
};

template <typename S, int MODE, bool CENTRAL>
static void launch_batch_c(const BatchArgs& a, bool record, int packed, cudaStream_t st) {
  if constexpr (!std::is_same<S, double>::value) {
    if constexpr (!CENTRAL) {
      if (packed == 2) {
        if (record)
          batch_adj_kernel<S, MODE, true><<<a.grid, 128, 0, st>>>(
              a.boxes, a.items, a.nitems, a.flags, a.parity, a.with_t, a.with_q, a.gamma_mode);
        else
          batch_adj_kernel<S, MODE, false><<<a.grid, 128, 0, st>>>(
              a.boxes, a.items, a.nitems, a.flags, a.parity, a.with_t, a.with_q, a.gamma_mode);
        return;
      }
    }
    if (packed) {
      if (record)
        batch_pair_kernel<S, MODE, true, CENTRAL><<<a.grid, 128, 0, st>>>(
            a.boxes, a.items, a.nitems, a.flags, a.parity, a.with_t, a.with_q, a.gamma_mode);
      else
        batch_pair_kernel<S, MODE, false, CENTRAL><<<a.grid, 128, 0, st>>>(
            a.boxes, a.items, a.nitems, a.flags, a.parity, a.with_t, a.with_q, a.gamma_mode);
      return;
    }
  }
  if (record)
    batch_kernel<S, MODE, true, CENTRAL><<<a.grid, a.threads, 0, st>>>(
        a.boxes, a.items, a.nitems, a.flags, a.parity, a.with_t, a.with_q, a.gamma_mode);
  else
    batch_kernel<S, MODE, false, CENTRAL><<<a.grid, a.threads, 0, st>>>(
        a.boxes, a.items, a.nitems, a.flags, a.parity, a.with_t, a.with_q, a.gamma_mode);
}

template <typename S, int MODE>
static void launch_batch(const BatchArgs& a, bool record, int packed, bool central,
                         cudaStream_t st) {
  if (central)
    launch_batch_c<S, MODE, true>(a, record, packed, st);
  else
    launch_batch_c<S, MODE, false>(a, record, packed, st);
  if constexpr (std::is_same<S, float>::value) {
    if (a.gamma_mode == GAMMA_ESTIMATE) {  // the FP32 kernels' flagged nodes, in FP64
      if (central)
        batch_fp64_pass_kernel<S, MODE, true><<<kPassBlocks, kPassThreads, 0, st>>>(
            a.boxes, a.nbox, a.flags, a.parity, a.with_t, a.with_q, a.gamma_mode, record);
      else
        batch_fp64_pass_kernel<S, MODE, false><<<kPassBlocks, kPassThreads, 0, st>>>(
            a.boxes, a.nbox, a.flags, a.parity, a.with_t, a.with_q, a.gamma_mode, record);
    }
  }
}

template <typename S>
cudaError_t Ops<S>::batch_step(const BoxDesc* boxes, int nbox, BatchFlags* flags,
                               const WorkItem* items, int nitems, int64_t t, bool record,
                               int packed, int scheme, int with_t, int with_q, int central,
                               int gamma_mode, int threads, int grid, cudaStream_t st) {
  BatchArgs a;
  a.boxes = boxes;
  a.nbox = nbox;
  a.flags = flags;
  a.items = items;
  a.nitems = nitems;
  a.parity = (int)(t & 1);
  a.with_t = with_t;
  a.with_q = with_q;
  a.gamma_mode = gamma_mode;
  a.threads = threads;
  a.grid = grid;
  if (scheme == 0)
    launch_batch<S, MODE_PULL>(a, record, packed, central != 0, st);
  else if (a.parity == 0)
    launch_batch<S, MODE_AA_EVEN>(a, record, packed, central != 0, st);
  else
    launch_batch<S, MODE_AA_ODD>(a, record, packed, central != 0, st);
  return cudaGetLastError();
}

template <typename S>
int Ops<S>::batch_occupancy(int threads, int scheme, int packed) {
  int blocks = 0;
  cudaError_t e = cudaErrorInvalidValue;
  if constexpr (!std::is_same<S, double>::value) {
    if (packed == 2) {
      if (scheme == 0)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &blocks, batch_adj_kernel<S, MODE_PULL, false>, 128, 0);
      else
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &blocks, batch_adj_kernel<S, MODE_AA_ODD, false>, 128, 0);
      if (e != cudaSuccess || blocks < 1) blocks = 1;
      return blocks;
    }
    if (packed) {
      if (scheme == 0)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &blocks, batch_pair_kernel<S, MODE_PULL, false, false>, 128, 0);
      else
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &blocks, batch_pair_kernel<S, MODE_AA_ODD, false, false>, 128, 0);
      if (e != cudaSuccess || blocks < 1) blocks = 1;
      return blocks;
    }
  }
  if (scheme == 0)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks, batch_kernel<S, MODE_PULL, false, false>,
                                                      threads, 0);
  else
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&blocks,
                                                      batch_kernel<S, MODE_AA_ODD, false, false>,
                                                      threads, 0);
  if (e != cudaSuccess || blocks < 1) blocks = 1;
  return blocks;
}

}  // namespace kbc

#include "kbc_aux.cuh"
