// k_pd_tma.cu -- primal-dual iterations (Eq. 11, 13) on the large levels
// with every footprint's inputs staged in shared memory by the tensor memory
// accelerator (TMA).  The per-pixel arithmetic and the iteration loop are
// those of k_pd (pd_math.cuh, pd_tile.cuh), so the results are the same bits.
//
// Why: a 64 x 64 footprint of 1024 threads holds all 64K registers of an
// SM, so in k_pd nothing covers the start of a footprint, when every thread
// waits for its 44 loads (11 planes x 4 rows).  Here each CTA stays resident
// and takes footprints blockIdx.x, + gridDim.x, ... in turn; while it
// iterates on one, the TMA copies the next one's planes into shared memory,
// so only the first footprint of a CTA waits on L2.
//
// Geometry.  Footprints of 64 x 64 pixels, 1024 threads of 4 rows (as
// PD_TILE_64_T1024).  A tiled TMA copy must start on a 16-byte boundary, so
// footprints start at column 48 bx - 8 (a multiple of 8 elements: 16 bytes
// of a 2-byte plane, 32 of a 4-byte one) and own the 48 interior columns
// 48 bx .. 48 bx + 47; the 8-column margins allow up to 8 iterations per
// launch.  Rows have no alignment rule and keep the margin B of the blocking
// depth (origin by (64 - 2B) - B).  After n <= B iterations the interior is
// exact (its dependency cone stays inside the footprint), so every footprint
// geometry computes the same values.  The mask (1 byte per pixel, 16-element
// rule) comes as an 80-column box from 48 bx - 16.  Copies that reach
// outside the level are filled with zeros, which are the inputs k_pd gives
// such pixels (no mask bit, all constants and state 0).
//
// Synchronisation.  One mbarrier: the leader thread arms it with the bytes
// of a footprint (arrive.expect_tx), twelve warps issue a copy each; every
// thread waits on its phase (try_wait.parity) before reading the planes.
// The planes of the next footprint are requested only after the CTA barrier
// that follows every thread's reads of the current one.  Every wait is
// bounded by wait_ns of global time; a wait that runs out sets *status to
// FS_ETIMEOUT and the CTA returns, one thread of it only once the copies it
// has under way have landed (or two seconds later).
#include <algorithm>
#include <atomic>

#include "fs.h"
#include "fs_kernels.h"
#include "pd_tile.cuh"

namespace fs {

namespace {

constexpr int kFW = 64, kNY = 16, kR = 4, kFH = kNY * kR;   // 64 x 64, 1024 threads
constexpr int kIW = 48, kXM = 8;                             // interior columns, column margin
constexpr int kMaskW = 80, kMaskOff = 16;                    // mask box: 80 columns from 48 bx - 16
constexpr unsigned long long kDrainNs = 2000000000ull;       // a CTA's last wait for its own copies

// Offsets (bytes) of the staged planes, the exchange planes of pd_iterate
// and the mbarrier in dynamic shared memory; all multiples of 128.
template <int S>
struct TmaLayout {
  static constexpr size_t f32 = (size_t)kFW * kFH * 4;                   // an FP32 plane
  static constexpr size_t sp = (size_t)kFW * kFH * storage_size(S);      // a storage plane
  // FP32: tau and the per-warp constants dinv, sd, step, c0, then u, ubar;
  // storage type: s_x, s_y, p1, p2
  static constexpr size_t tau = 0, dinv = f32, sd = 2 * f32, step = 3 * f32, c0 = 4 * f32;
  static constexpr size_t u = 5 * f32, ub = 6 * f32;
  static constexpr size_t sx = 7 * f32, sy = sx + sp, p1 = sy + sp, p2 = p1 + sp;
  static constexpr size_t mask = p2 + sp;                                // kMaskW x kFH bytes
  static constexpr size_t x_ub = mask + (size_t)kMaskW * kFH;            // kFH x kFW floats
  static constexpr size_t x_t1 = x_ub + f32;                             // kFH x kFW floats
  static constexpr size_t x_t2 = x_t1 + f32;                             // kNY x kFW floats
  static constexpr size_t bar = x_t2 + (size_t)kNY * kFW * 4;
  static constexpr size_t bytes = bar + 128;
  // bytes one footprint's copies deliver (boxes count whole, zero fill included)
  static constexpr unsigned tx = (unsigned)(7 * f32 + 4 * sp + (size_t)kMaskW * kFH);
};

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ void mbar_init(uint32_t bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
  // make the initialised barrier visible to the TMA unit (the async proxy)
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, unsigned parity) {
  unsigned done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}

// One 2-D tiled copy of the box at column x, row y of the tensor `map` into
// shared memory at dst, completing on the mbarrier bar.
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap* map, int x, int y,
                                         uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar)
      : "memory");
}

// The twelve copies of a footprint, in the order of PdTmaMaps and of the
// shared-memory planes; one warp requests each.
constexpr int kCopies = 12;
__device__ __forceinline__ bool is_state(int k) { return k == 5 || k == 6 || k == 9 || k == 10; }

template <int S>
__device__ __forceinline__ void request(const PdTmaMaps& m, unsigned char* smem, uint32_t bar,
                                        int k, int bx, int by, int IH, int B) {
  using Lay = TmaLayout<S>;
  const size_t dst = k < 7 ? k * Lay::f32 : Lay::sx + (k - 7) * Lay::sp;   // the mask follows p2
  tma_load(smem_addr(smem + dst), reinterpret_cast<const CUtensorMap*>(&m) + k,
           bx * kIW - (k == 11 ? kMaskOff : kXM), by * IH - B, bar);
}

// A staged storage-typed value (FP16 / BF16 converted to float).
template <int S>
__device__ __forceinline__ float sval(const unsigned char* plane, int k) {
  if constexpr (S == ST_F16) return __half2float(reinterpret_cast<const __half*>(plane)[k]);
  else if constexpr (S == ST_BF16)
    return __bfloat162float(reinterpret_cast<const __nv_bfloat16*>(plane)[k]);
  else return reinterpret_cast<const float*>(plane)[k];
}

}  // namespace

// n_iters (<= B <= 8) iterations on the level's footprints --
// those of `rows` where rows.n > 0 (the others hold no FOV pixel; pp.idle),
// else all; the state is read (through the copies in `maps`) from the buffer
// set `in` and written to `out`.  chained (pd_tile): PD_CHAINED requests the
// first footprint's constants before the wait for the preceding launch and
// its state after, PD_CHAIN_START waits first.  stall: testing aid, the
// first wait's barrier expects an arrival that only comes when it is given up.
//
// Bound by the iterations, 1450-1700 clock cycles each, and by what lies
// between two footprints: 3800 cycles, the 1400 shared-memory wavefronts of
// the reads among them, against 7000 when one thread requested all the copies
// and four barriers kept the stores, the reads and the requests apart.  2048
// x 2048, 100 iterations: 14.9 us each against 16.4, 12.2 without the
// footprints outside a 180-degree FOV (19.3 on 64 x 64 footprints of k_pd).
template <int S, bool ACC>
__global__ void __launch_bounds__(kFW * kNY, 1)
k_pd_tma(LevelView L, PDState in, PDState out, PDParams pp, int B, int n_iters, int chained,
         const __grid_constant__ PdTmaMaps maps, const __grid_constant__ PdTmaRows rows,
         int* status, unsigned long long wait_ns, int stall) {
  using Lay = TmaLayout<S>;
  extern __shared__ __align__(128) unsigned char smem[];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const bool leader = tx == 0 && ty == 0;
  // the copy this thread requests, -1: none
  const int copy = (tx & 31) == 0 && 2 * ty + (tx >> 5) < kCopies ? 2 * ty + (tx >> 5) : -1;
  const int IH = kFH - 2 * B;
  const int tiles_x = (L.W + kIW - 1) / kIW;
  const int all_tiles = tiles_x * ((L.H + IH - 1) / IH);
  const int ntiles = rows.n > 0 ? rows.start[rows.n] : all_tiles;
  float(*s_ub)[kFW] = reinterpret_cast<float(*)[kFW]>(smem + Lay::x_ub);
  float(*s_t1)[kFW] = reinterpret_cast<float(*)[kFW]>(smem + Lay::x_t1);
  float(*s_t2)[kFW] = reinterpret_cast<float(*)[kFW]>(smem + Lay::x_t2);
  const uint32_t bar = smem_addr(smem + Lay::bar);
  volatile int* s_late = reinterpret_cast<volatile int*>(smem + Lay::bar + 16);

  // footprint t's place; by: a row at or before it (only ever moves down)
  auto column = [&](int t, int& by) {
    if (rows.n == 0) {
      by = t / tiles_x;
      return t - by * tiles_x;
    }
    while (t >= rows.start[by + 1]) ++by;
    return rows.lo[by] + t - rows.start[by];
  };

  // the next launch of the chain may be scheduled once every CTA of this one
  // is resident (it waits for this grid's completion before its state); for
  // the first of a chain once the constants are complete
  if (chained >= PD_CHAIN_START) cudaGridDependencySynchronize();
  if (chained) cudaTriggerProgrammaticLaunchCompletion();
  int tile = blockIdx.x, by = 0, bx = tile < ntiles ? column(tile, by) : 0;
  if (leader) {
    mbar_init(bar, stall ? 2 : 1);
    *s_late = 0;
    if (tile < ntiles) mbar_expect_tx(bar, Lay::tx);
  }
  __syncthreads();
  if (copy >= 0 && tile < ntiles && !is_state(copy))
    request<S>(maps, smem, bar, copy, bx, by, IH, B);
  if (chained == PD_CHAINED) cudaGridDependencySynchronize();
  if (copy >= 0 && tile < ntiles && is_state(copy))
    request<S>(maps, smem, bar, copy, bx, by, IH, B);

  unsigned parity = 0;
  while (tile < ntiles) {
    const unsigned long long t0 = global_ns();
    while (!mbar_try_wait(bar, parity)) {
      if (global_ns() - t0 > wait_ns) {
        *s_late = 1 + (int)parity;
        break;
      }
    }
    parity ^= 1u;

    // this thread's 4 rows of column tx from the staged planes
    float u[kR], ub[kR], p1[kR], p2[kR];
    PxConst c[kR];
    unsigned mb = 0;
    // (outside the level the copies read zeros: the constants of k_pd's
    // all-zero inputs, except dinv = 0 instead of 1, which only scales a
    // dual that is 0 there and stays 0)
#pragma unroll
    for (int r = 0; r < kR; ++r) {
      const int k = (ty * kR + r) * kFW + tx;
      auto f32 = [&](size_t plane) { return reinterpret_cast<const float*>(smem + plane)[k]; };
      c[r].tau = f32(Lay::tau);
      c[r].dinv = f32(Lay::dinv);
      c[r].sd = f32(Lay::sd);
      c[r].step = f32(Lay::step);
      c[r].c0 = f32(Lay::c0);
      c[r].sx = sval<S>(smem + Lay::sx, k);
      c[r].sy = sval<S>(smem + Lay::sy, k);
      u[r] = f32(Lay::u);
      ub[r] = f32(Lay::ub);
      p1[r] = sval<S>(smem + Lay::p1, k);
      p2[r] = sval<S>(smem + Lay::p2, k);
      mb |= (unsigned)smem[Lay::mask + (ty * kR + r) * kMaskW + tx + (kMaskOff - kXM)]
            << (3 * r);
    }
#pragma unroll
    for (int r = 0; r < kR; ++r) s_ub[ty * kR + r][tx] = ub[r];
    // one barrier: every thread has read the staged planes, ubar is in place
    // for the neighbours, and whether every pixel of the footprint lies in
    // the level with all three mask bits set (outside it the mask reads 0).
    // (s_ub: the last footprint's iterations ended with a barrier.)
    const bool full = __syncthreads_and(mb == 07777u);
    if (*s_late) break;
    if (n_iters == 0) __syncthreads();   // s_late and s_ub as if iterations followed
    const int next = tile + (int)gridDim.x;
    int nby = by;
    const int nbx = next < ntiles ? column(next, nby) : 0;
    if (copy >= 0 && next < ntiles) {
      if (leader) mbar_expect_tx(bar, Lay::tx);
      // order the reads above before the copies that overwrite the planes
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      request<S>(maps, smem, bar, copy, nbx, nby, IH, B);
    }

    float theta = pp.theta;
    if (full)
      pd_iterate_rows<kFW, kNY, kR, ACC, false>(pp, n_iters, tx, ty, mb, c, u, ub, p1, p2,
                                                theta, s_ub, s_t1, s_t2);
    else
      pd_iterate_rows<kFW, kNY, kR, ACC, true>(pp, n_iters, tx, ty, mb, c, u, ub, p1, p2,
                                               theta, s_ub, s_t1, s_t2);

    // the interior back to global memory
    const int gx = bx * kIW - kXM + tx;
    if (tx >= kXM && tx < kXM + kIW && gx < L.W) {
#pragma unroll
      for (int r = 0; r < kR; ++r) {
        const int fy = ty * kR + r;
        const int gy = by * IH - B + fy;
        if (fy < B || fy >= kFH - B || gy >= L.H) continue;
        const size_t i = (size_t)gy * L.P + gx;
        out.u[i] = u[r];
        out.ubar[i] = ub[r];
        sst<S>(out.p1, i, p1[r]);
        sst<S>(out.p2, i, p2[r]);
      }
    }
    tile = next;
    bx = nbx;
    by = nby;
  }

  if (*s_late) {
    // the footprint's copies may still be under way (the limit can be as short
    // as a caller likes), and the shared memory they write is another CTA's
    // once this one has left: one thread stays for them
    if (threadIdx.x == 0 && threadIdx.y == 0) {
      atomicCAS(status, 0, (int)FS_ETIMEOUT);
      const uint32_t b = smem_addr(smem + Lay::bar);
      if (stall) mbar_arrive(b);
      const unsigned long long t1 = global_ns();
      while (!mbar_try_wait(b, (unsigned)(*s_late - 1)) && global_ns() - t1 <= kDrainNs) {
      }
    }
    return;
  }

  // the first launch of a warp: all its iterations on the footprints left out
  if (rows.n == 0 || pp.idle <= 0) return;
  for (int t = blockIdx.x; t < all_tiles; t += (int)gridDim.x) {
    const int y = t / tiles_x, x = t - y * tiles_x;
    const int k = x - rows.lo[y];
    if (k >= 0 && k < rows.start[y + 1] - rows.start[y]) continue;
    pd_idle<kFW, kNY, kR, S, ACC>(L, in, pp, kXM, B, x * kIW - kXM, y * IH - B, tx, ty);
  }
}

namespace {

template <int S, bool ACC>
cudaError_t launch_tma_t(const LevelView& L, const PDState& in, const PDState& out,
                         const PDParams& pp, int B, int n, int chained, const PdTmaMaps& maps,
                         int* status, unsigned long long wait_ns, int stall, cudaStream_t st) {
  using Lay = TmaLayout<S>;
  // the SMs of each device the kernel's shared memory is opted in on (0: not
  // yet): handles of any device and thread come here
  constexpr int kDevices = 64;
  static std::atomic<int> sms_of[kDevices] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int sms = dev < kDevices ? sms_of[dev].load() : 0;
  if (sms == 0) {
    e = cudaFuncSetAttribute(k_pd_tma<S, ACC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)Lay::bytes);
    if (e != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
      return e;
    if (dev < kDevices) sms_of[dev].store(sms);
  }
  const int IH = kFH - 2 * B;
  const int tiles_x = (L.W + kIW - 1) / kIW, tiles_y = (L.H + IH - 1) / IH;
  PdTmaRows rows{};
  int ntiles = tiles_x * tiles_y;
  if (pp.idle >= 0 && tiles_y <= PdTmaRows::kMax) {
    rows.n = tiles_y;
    for (int y = 0; y < tiles_y; ++y) {
      int lo = 0, hi = 0;
      fov_columns(L, kIW, -kXM, kFW, kFH, tiles_x, y * IH - B, lo, hi);
      rows.lo[y] = (unsigned short)lo;
      rows.start[y + 1] = rows.start[y] + (hi - lo);
    }
    ntiles = std::max(rows.start[tiles_y], 1);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)std::min(ntiles, sms), 1, 1);
  cfg.blockDim = dim3(kFW, kNY, 1);
  cfg.dynamicSmemBytes = Lay::bytes;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_pd_tma<S, ACC>, L, in, out, pp, B, n, chained, maps, rows,
                            status, wait_ns, stall);
}

}  // namespace

size_t pd_tma_smem_bytes(int storage) {
  switch (storage) {
    case ST_F16: return TmaLayout<ST_F16>::bytes;
    case ST_BF16: return TmaLayout<ST_BF16>::bytes;
    default: return TmaLayout<ST_F32>::bytes;
  }
}

cudaError_t launch_pd_tma(const LevelView& L, const PDState& in, const PDState& out,
                          const PDParams& pp, int B, int n, int chained, const PdTmaMaps& maps,
                          int* status, unsigned long long wait_ns, int stall, cudaStream_t st) {
  if (B < 1 || B > kXM || n < 0 || n > B || L.W < 1 || L.H < 1) return cudaErrorInvalidValue;
  if (pp.sched) {
    if (L.st != ST_F32) return cudaErrorInvalidValue;
    return launch_tma_t<ST_F32, true>(L, in, out, pp, B, n, chained, maps, status, wait_ns, stall, st);
  }
  switch (L.st) {
    case ST_F16:
      return launch_tma_t<ST_F16, false>(L, in, out, pp, B, n, chained, maps, status, wait_ns, stall,
                                         st);
    case ST_BF16:
      return launch_tma_t<ST_BF16, false>(L, in, out, pp, B, n, chained, maps, status, wait_ns,
                                          stall, st);
    default:
      return launch_tma_t<ST_F32, false>(L, in, out, pp, B, n, chained, maps, status, wait_ns, stall,
                                         st);
  }
}

}  // namespace fs
