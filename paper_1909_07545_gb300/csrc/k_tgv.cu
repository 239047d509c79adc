// k_tgv.cu -- primal-dual iterations of the tensor-guided TGV-L1 energy
// (Sec. III-C, Eq. 10-11):
//
//   E(u, v) = lam |rho_bar(u)| + alpha1 |T^1/2 grad u - v| + alpha0 |grad v|
//
// The per-pixel steps are in pd_tgv_math.cuh.  Two schedules compute them
// with identical arithmetic:
//   * launch per step: a dual launch then a primal launch per iteration,
//     state in place (each pixel reads its right / lower neighbours in the
//     dual and its left / upper ones in the primal, so the launch boundary is
//     the only synchronisation needed);
//   * temporal blocking (k_tgv_blocked): a CTA keeps a footprint's (32 x 16
//     to 64 x 32 pixels; tgv_auto or the tuner picks one per level) whole state (u, ubar, v, vbar, p, q: 12 values per pixel) in registers
//     for n <= B iterations, exchanging ubar, vbar and the masked products
//     T^1/2 p and q with its neighbours through shared memory; the outer B
//     pixels of the footprint are halo, recomputed by the neighbouring CTAs.
//     State ping-pongs between the level's planes and an alternate set, and
//     a warp runs an even number of launches so that it ends in the level's
//     planes.
// Steps (Pock-Chambolle 2011 diagonal preconditioning of the block operator
// (T^1/2 grad u - v, grad v), in tgv_const): tau_u the Huber-TV tau; sigma_p
// = 1 / (max row sum of |T^1/2| |grad| + 1) from the stored Huber-TV sigma;
// sigma_q = 1/2; tau_v = 1 / (1 + the active differences touching the
// pixel); all 0 off the FOV mask, where nothing moves.
#include <atomic>

#include "fs_kernels.h"
#include "pd_tgv_math.cuh"
#include "pd_tile.cuh"

namespace fs {

namespace {

__device__ __forceinline__ void load_const(const LevelView& L, size_t i, int x, int y,
                                           const TgvParams& tp, TgvConst& c) {
  const unsigned m = L.mask[i];
  const unsigned ml = x > 0 ? L.mask[i - 1] : 0u;
  const unsigned mu = y > 0 ? L.mask[i - L.P] : 0u;
  tgv_const(m, ml, mu, sld<ST_F32>(L.sx, i), sld<ST_F32>(L.sy, i), L.sig[i], L.tau[i],
            sld<ST_F32>(L.Iu, i), sld<ST_F32>(L.rho0, i), L.uw[i], tp, c);
}

// t = T^1/2 p and the masked q of pixel k (what tgv_px_dual returns).
__device__ __forceinline__ void masked_products(const LevelView& L, size_t k, unsigned m,
                                                float& t1, float& t2, float& qx1, float& qx2,
                                                float& qy1, float& qy2) {
  const float sx = sld<ST_F32>(L.sx, k), sy = sld<ST_F32>(L.sy, k);
  const float p1 = sld<ST_F32>(L.p1, k), p2 = sld<ST_F32>(L.p2, k);
  const float dp = fmaf(sx, p1, __fmul_rn(sy, p2));
  const bool gx = m & MASK_GX, gy = m & MASK_GY;
  t1 = gx ? fmaf(-sx, dp, p1) : 0.f;
  t2 = gy ? fmaf(-sy, dp, p2) : 0.f;
  qx1 = gx ? L.q11[k] : 0.f;
  qx2 = gx ? L.q21[k] : 0.f;
  qy1 = gy ? L.q12[k] : 0.f;
  qy2 = gy ? L.q22[k] : 0.f;
}

}  // namespace

__global__ void k_tgv_dual(LevelView L, TgvParams tp) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  const size_t i = (size_t)y * L.P + x;
  const unsigned m = L.mask[i];
  if (!(m & MASK_IN)) return;
  TgvConst c;
  load_const(L, i, x, y, tp, c);
  const bool gx = m & MASK_GX, gy = m & MASK_GY;
  const size_t r = gx ? i + 1 : i, b = gy ? i + L.P : i;   // unread when masked
  float p1 = sld<ST_F32>(L.p1, i), p2 = sld<ST_F32>(L.p2, i);
  float q11 = L.q11[i], q12 = L.q12[i], q21 = L.q21[i], q22 = L.q22[i];
  float t1, t2, qx1, qx2, qy1, qy2;
  tgv_px_dual<false>(m, L.ubar[i], L.ubar[r], L.ubar[b], L.vb1[i], L.vb1[r], L.vb1[b], L.vb2[i],
              L.vb2[r], L.vb2[b], c, tp, p1, p2, q11, q12, q21, q22, t1, t2, qx1, qx2, qy1,
              qy2);
  sst<ST_F32>(L.p1, i, p1);
  sst<ST_F32>(L.p2, i, p2);
  L.q11[i] = q11;
  L.q12[i] = q12;
  L.q21[i] = q21;
  L.q22[i] = q22;
}

__global__ void k_tgv_primal(LevelView L, TgvParams tp) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  const size_t i = (size_t)y * L.P + x;
  const unsigned m = L.mask[i];
  if (!(m & MASK_IN)) return;
  TgvConst c;
  load_const(L, i, x, y, tp, c);
  float t1, t2, qx1, qx2, qy1, qy2;
  float t1_l = 0.f, t2_l, qx1_l = 0.f, qx2_l = 0.f, qy1_l, qy2_l;
  float t1_u, t2_u = 0.f, qx1_u, qx2_u, qy1_u = 0.f, qy2_u = 0.f;
  masked_products(L, i, m, t1, t2, qx1, qx2, qy1, qy2);
  if (x > 0) masked_products(L, i - 1, L.mask[i - 1], t1_l, t2_l, qx1_l, qx2_l, qy1_l, qy2_l);
  if (y > 0)
    masked_products(L, i - L.P, L.mask[i - L.P], t1_u, t2_u, qx1_u, qx2_u, qy1_u, qy2_u);
  float u = L.u[i], ub, v1 = L.v1[i], v2 = L.v2[i], vb1, vb2;
  tgv_px_primal(t1, t1_l, t2, t2_u, qx1, qx1_l, qy1, qy1_u, qx2, qx2_l, qy2, qy2_u,
                sld<ST_F32>(L.p1, i), sld<ST_F32>(L.p2, i), c, tp.theta, u, ub, v1, v2, vb1,
                vb2);
  L.u[i] = u;
  L.ubar[i] = ub;
  L.v1[i] = v1;
  L.v2[i] = v2;
  L.vb1[i] = vb1;
  L.vb2[i] = vb2;
}

// One set of the 12 state planes of a TGV level.
struct TgvState {
  float* s[12];   // u, ubar, v1, v2, vb1, vb2, p1, p2, q11, q12, q21, q22
};

// Shared memory of a footprint: what neighbours read of each other.  ubar,
// vbar (the dual reads them from the right and from below) and t1, qx (the
// primal reads them from the left) for every pixel; t2, qy (read from above)
// only for the last row of each thread, as a thread keeps its other rows.
template <int FW, int NY, int R>
struct TgvShared {
  float ub[NY * R][FW], vb1[NY * R][FW], vb2[NY * R][FW];
  float t1[NY * R][FW], qx1[NY * R][FW], qx2[NY * R][FW];
  float t2[NY][FW], qy1[NY][FW], qy2[NY][FW];
};

// A thread's R rows: u, ubar, v, vbar, p, q.
template <int R>
struct TgvRows {
  float u[R], ub[R], v1[R], v2[R], vb1[R], vb2[R], p1[R], p2[R], q11[R], q12[R], q21[R], q22[R];
};

// n_iters iterations on a thread's rows (neighbours through sm); FTZ as in
// tgv_ball, MASKED as in tgv_px_dual.  Rows in pairs (j, j + H) on the packed
// FP32 operations, as in pd_iterate2: the rows below pair j are pair j + 1,
// those above it pair j - 1; the same values in the same order, so the same
// bits.
template <int FW, int NY, int R, bool FTZ, bool MASKED>
__device__ __forceinline__ void tgv_iterate(const TgvParams& tp, int n_iters, int tx, int ty,
                                            unsigned mb, const TgvConst (&c)[R], TgvRows<R>& s,
                                            TgvShared<FW, NY, R>& sm) {
  constexpr int FH = NY * R;
  const int txr = min(tx + 1, FW - 1), txl = max(tx - 1, 0);
  const int fnext = min(ty * R + R, FH - 1);     // the thread below's first row
  if constexpr (R % 2 == 0) {
    constexpr int H = R / 2;
    TgvConst2 c2[H];
    float2 u2[H], ub2[H], v12[H], v22[H], vb12[H], vb22[H], p12[H], p22[H];
    float2 q112[H], q122[H], q212[H], q222[H];
#pragma unroll
    for (int j = 0; j < H; ++j) {
      c2[j] = tgv_pair(c[j], c[j + H]);
      u2[j] = make_float2(s.u[j], s.u[j + H]);
      ub2[j] = make_float2(s.ub[j], s.ub[j + H]);
      v12[j] = make_float2(s.v1[j], s.v1[j + H]);
      v22[j] = make_float2(s.v2[j], s.v2[j + H]);
      vb12[j] = make_float2(s.vb1[j], s.vb1[j + H]);
      vb22[j] = make_float2(s.vb2[j], s.vb2[j + H]);
      p12[j] = make_float2(s.p1[j], s.p1[j + H]);
      p22[j] = make_float2(s.p2[j], s.p2[j + H]);
      q112[j] = make_float2(s.q11[j], s.q11[j + H]);
      q122[j] = make_float2(s.q12[j], s.q12[j + H]);
      q212[j] = make_float2(s.q21[j], s.q21[j + H]);
      q222[j] = make_float2(s.q22[j], s.q22[j + H]);
    }
    const float2 th2 = make_float2(tp.theta, tp.theta);
    float2 t12[H], t22[H], qx12[H], qx22[H], qy12[H], qy22[H];
#pragma unroll 1
    for (int it = 0; it < n_iters; ++it) {
#pragma unroll
      for (int j = 0; j < H; ++j) {
        const int f0 = ty * R + j, f1 = f0 + H;
        const bool last = j + 1 == H;
        const int k = last ? j : j + 1;
        const float2 ub_b = last ? make_float2(ub2[0].y, sm.ub[fnext][tx]) : ub2[k];
        const float2 vb1_b = last ? make_float2(vb12[0].y, sm.vb1[fnext][tx]) : vb12[k];
        const float2 vb2_b = last ? make_float2(vb22[0].y, sm.vb2[fnext][tx]) : vb22[k];
        tgv_px_dual2<FTZ, MASKED>(
            mb >> (3 * j), mb >> (3 * (j + H)), ub2[j],
            make_float2(sm.ub[f0][txr], sm.ub[f1][txr]), ub_b, vb12[j],
            make_float2(sm.vb1[f0][txr], sm.vb1[f1][txr]), vb1_b, vb22[j],
            make_float2(sm.vb2[f0][txr], sm.vb2[f1][txr]), vb2_b, c2[j], tp, p12[j], p22[j],
            q112[j], q122[j], q212[j], q222[j], t12[j], t22[j], qx12[j], qx22[j], qy12[j],
            qy22[j]);
        sm.t1[f0][tx] = t12[j].x;   sm.t1[f1][tx] = t12[j].y;
        sm.qx1[f0][tx] = qx12[j].x; sm.qx1[f1][tx] = qx12[j].y;
        sm.qx2[f0][tx] = qx22[j].x; sm.qx2[f1][tx] = qx22[j].y;
        if (last) {                                    // row R - 1
          sm.t2[ty][tx] = t22[j].y;
          sm.qy1[ty][tx] = qy12[j].y;
          sm.qy2[ty][tx] = qy22[j].y;
        }
      }
      __syncthreads();
#pragma unroll
      for (int j = 0; j < H; ++j) {
        const int f0 = ty * R + j, f1 = f0 + H;
        // above: the previous pair, or for the first pair the thread above's
        // last row (the footprint's top row, halo, reads its own) and row H - 1
        float2 t2_u, qy1_u, qy2_u;
        if (j > 0) {
          t2_u = t22[j > 0 ? j - 1 : 0];
          qy1_u = qy12[j > 0 ? j - 1 : 0];
          qy2_u = qy22[j > 0 ? j - 1 : 0];
        } else {
          t2_u = make_float2(ty > 0 ? sm.t2[ty - 1][tx] : t22[0].x, t22[H - 1].x);
          qy1_u = make_float2(ty > 0 ? sm.qy1[ty - 1][tx] : qy12[0].x, qy12[H - 1].x);
          qy2_u = make_float2(ty > 0 ? sm.qy2[ty - 1][tx] : qy22[0].x, qy22[H - 1].x);
        }
        tgv_px_primal2(t12[j], make_float2(sm.t1[f0][txl], sm.t1[f1][txl]), t22[j], t2_u,
                       qx12[j], make_float2(sm.qx1[f0][txl], sm.qx1[f1][txl]), qy12[j], qy1_u,
                       qx22[j], make_float2(sm.qx2[f0][txl], sm.qx2[f1][txl]), qy22[j], qy2_u,
                       p12[j], p22[j], c2[j], th2, u2[j], ub2[j], v12[j], v22[j], vb12[j],
                       vb22[j]);
        sm.ub[f0][tx] = ub2[j].x;   sm.ub[f1][tx] = ub2[j].y;
        sm.vb1[f0][tx] = vb12[j].x; sm.vb1[f1][tx] = vb12[j].y;
        sm.vb2[f0][tx] = vb22[j].x; sm.vb2[f1][tx] = vb22[j].y;
      }
      __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < H; ++j) {
      s.u[j] = u2[j].x;     s.u[j + H] = u2[j].y;
      s.ub[j] = ub2[j].x;   s.ub[j + H] = ub2[j].y;
      s.v1[j] = v12[j].x;   s.v1[j + H] = v12[j].y;
      s.v2[j] = v22[j].x;   s.v2[j + H] = v22[j].y;
      s.vb1[j] = vb12[j].x; s.vb1[j + H] = vb12[j].y;
      s.vb2[j] = vb22[j].x; s.vb2[j + H] = vb22[j].y;
      s.p1[j] = p12[j].x;   s.p1[j + H] = p12[j].y;
      s.p2[j] = p22[j].x;   s.p2[j + H] = p22[j].y;
      s.q11[j] = q112[j].x; s.q11[j + H] = q112[j].y;
      s.q12[j] = q122[j].x; s.q12[j + H] = q122[j].y;
      s.q21[j] = q212[j].x; s.q21[j + H] = q212[j].y;
      s.q22[j] = q222[j].x; s.q22[j + H] = q222[j].y;
    }
  } else {
    float t1[R], t2[R], qx1[R], qx2[R], qy1[R], qy2[R];
#pragma unroll 1
    for (int it = 0; it < n_iters; ++it) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int fy = ty * R + r;
        const int k = r + 1 < R ? r + 1 : r;
        const float ub_b = (r + 1 < R) ? s.ub[k] : sm.ub[fnext][tx];
        const float vb1_b = (r + 1 < R) ? s.vb1[k] : sm.vb1[fnext][tx];
        const float vb2_b = (r + 1 < R) ? s.vb2[k] : sm.vb2[fnext][tx];
        tgv_px_dual<FTZ, MASKED>(mb >> (3 * r), s.ub[r], sm.ub[fy][txr], ub_b, s.vb1[r],
                                 sm.vb1[fy][txr], vb1_b, s.vb2[r], sm.vb2[fy][txr], vb2_b, c[r],
                                 tp, s.p1[r], s.p2[r], s.q11[r], s.q12[r], s.q21[r], s.q22[r],
                                 t1[r], t2[r], qx1[r], qx2[r], qy1[r], qy2[r]);
        sm.t1[fy][tx] = t1[r];
        sm.qx1[fy][tx] = qx1[r];
        sm.qx2[fy][tx] = qx2[r];
        if (r + 1 == R) {
          sm.t2[ty][tx] = t2[r];
          sm.qy1[ty][tx] = qy1[r];
          sm.qy2[ty][tx] = qy2[r];
        }
      }
      __syncthreads();
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int fy = ty * R + r;
        const int k = r > 0 ? r - 1 : 0;
        const float t2_u = r > 0 ? t2[k] : (ty > 0 ? sm.t2[ty - 1][tx] : t2[0]);
        const float qy1_u = r > 0 ? qy1[k] : (ty > 0 ? sm.qy1[ty - 1][tx] : qy1[0]);
        const float qy2_u = r > 0 ? qy2[k] : (ty > 0 ? sm.qy2[ty - 1][tx] : qy2[0]);
        tgv_px_primal(t1[r], sm.t1[fy][txl], t2[r], t2_u, qx1[r], sm.qx1[fy][txl], qy1[r], qy1_u,
                      qx2[r], sm.qx2[fy][txl], qy2[r], qy2_u, s.p1[r], s.p2[r], c[r], tp.theta,
                      s.u[r], s.ub[r], s.v1[r], s.v2[r], s.vb1[r], s.vb2[r]);
        sm.ub[fy][tx] = s.ub[r];
        sm.vb1[fy][tx] = s.vb1[r];
        sm.vb2[fy][tx] = s.vb2[r];
      }
      __syncthreads();
    }
  }
}

// n iterations, in place, on the interior pixels of a footprint without a FOV
// pixel: they move on their own (every step size is 0 there), and not at all
// where p = q = 0, ubar = u and vbar = v, as every warp of a solve starts.
template <int FW, int NY, int R, bool FTZ>
__device__ __forceinline__ void tgv_idle(const LevelView& L, const TgvState& io,
                                         const TgvParams& tp, int B, int n, int ox, int oy,
                                         int tx, int ty) {
  const int gx = ox + tx;
  if (gx < 0 || gx >= L.W || tx < B || tx >= FW - B) return;
#pragma unroll 1
  for (int r = 0; r < R; ++r) {
    const int fy = ty * R + r, gy = oy + fy;
    if (gy < 0 || gy >= L.H || fy < B || fy >= NY * R - B) continue;
    const size_t i = (size_t)gy * L.P + gx;
    float a[12];
    bool rest = true;
#pragma unroll
    for (int j = 0; j < 12; ++j) a[j] = __ldcg(io.s[j] + i);
#pragma unroll
    for (int j = 6; j < 12; ++j) rest = rest && a[j] == 0.f;
    if (rest && a[0] == a[1] && a[2] == a[4] && a[3] == a[5]) continue;
    TgvConst c;
    tgv_const(0u, 0u, 0u, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, tp, c);
    for (int it = 0; it < n; ++it) {
      float t1, t2, x1, x2, y1, y2;
      tgv_px_dual<FTZ>(0u, a[1], 0.f, 0.f, a[4], 0.f, 0.f, a[5], 0.f, 0.f, c, tp, a[6], a[7],
                       a[8], a[9], a[10], a[11], t1, t2, x1, x2, y1, y2);
      tgv_px_primal(t1, 0.f, t2, 0.f, x1, 0.f, y1, 0.f, x2, 0.f, y2, 0.f, a[6], a[7], c, tp.theta,
                    a[0], a[1], a[2], a[3], a[4], a[5]);
    }
#pragma unroll
    for (int j = 0; j < 12; ++j) io.s[j][i] = a[j];
  }
}

// One launch of n_iters <= B iterations on FW x (NY R) footprints with halo
// B; MB: CTAs per SM the registers have to allow.  IDLE: footprints without
// a FOV pixel are left out, after `idle` iterations on their pixels in place
// (the warp's iterations at its first launch, 0 at the others).
template <int FW, int NY, int R, int MB, bool FTZ, bool IDLE>
__global__ void __launch_bounds__(FW * NY, MB)
k_tgv_blocked(LevelView L, TgvState in, TgvState out, TgvParams tp, int B, int n_iters,
              int chained, int idle) {
  constexpr int FH = NY * R;
  extern __shared__ float tgv_smem[];
  TgvShared<FW, NY, R>& sm = *reinterpret_cast<TgvShared<FW, NY, R>*>(tgv_smem);

  const int tx = threadIdx.x, ty = threadIdx.y;
  const int IW = FW - 2 * B, IH = FH - 2 * B;
  const int ox = (int)blockIdx.x * IW - B;
  const int oy = (int)blockIdx.y * IH - B;
  const int gx = ox + tx;
  const bool col_in = gx >= 0 && gx < L.W;

  if constexpr (IDLE) {              // as in pd_tile
    if (outside_fov(L, ox, oy, FW, FH)) {
      if (chained && blockIdx.x == 0 && blockIdx.y == 0) cudaGridDependencySynchronize();
      if (idle > 0) tgv_idle<FW, NY, R, FTZ>(L, in, tp, B, idle, ox, oy, tx, ty);
      return;
    }
  }
  if (chained) cudaTriggerProgrammaticLaunchCompletion();

  // constants (written before the chain; unconditional loads from clamped
  // addresses, rows off the level made inert)
  const int gxc = min(max(gx, 0), L.W - 1);
  unsigned idx[R];
  bool ok[R];
  TgvConst c[R];
  unsigned mb = 0;
  {
    // every load first, from clamped addresses, then the selection: a
    // thread's loads are all in flight together
    float sx[R], sy[R], sp[R], ta[R], st[R], c0[R], tv[R];
    unsigned m[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const int gy = oy + ty * R + r;
      ok[r] = col_in && gy >= 0 && gy < L.H;
      idx[r] = (unsigned)(min(max(gy, 0), L.H - 1) * L.P + gxc);
      sx[r] = sld<ST_F32>(L.sx, idx[r]);
      sy[r] = sld<ST_F32>(L.sy, idx[r]);
      sp[r] = L.dinv[idx[r]];
      ta[r] = L.tau[idx[r]];
      st[r] = L.step[idx[r]];
      c0[r] = L.c0[idx[r]];
      tv[r] = L.sd[idx[r]];
      m[r] = L.mask[idx[r]];
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const unsigned mm = ok[r] ? m[r] : 0u;
      const bool in_fov = mm & MASK_IN;          // off the FOV nothing moves
      c[r].sx = in_fov ? sx[r] : 0.f;
      c[r].sy = in_fov ? sy[r] : 0.f;
      c[r].sp = in_fov ? sp[r] : 0.f;
      c[r].sq = in_fov ? (tp.precond ? 0.5f : kTgvScalarStep) : 0.f;
      c[r].tau = in_fov ? (tp.precond ? ta[r] : kTgvScalarStep) : 0.f;
      c[r].step = in_fov ? st[r] : 0.f;
      c[r].c0 = in_fov ? c0[r] : 0.f;
      c[r].tv = in_fov ? tv[r] : 0.f;
      mb |= mm << (3 * r);
    }
  }
  // the state is the preceding launch's output, read through L2 (a chained
  // launch may start while the launch two before it still caches lines of
  // this buffer set in L1)
  if (chained) cudaGridDependencySynchronize();
  TgvRows<R> s;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const unsigned k = idx[r];
    float a[12];
#pragma unroll
    for (int j = 0; j < 12; ++j) a[j] = __ldcg(in.s[j] + k);
    const float z = ok[r] ? 1.f : 0.f;   // off the level: inert zeros
    s.u[r] = a[0] * z; s.ub[r] = a[1] * z; s.v1[r] = a[2] * z; s.v2[r] = a[3] * z;
    s.vb1[r] = a[4] * z; s.vb2[r] = a[5] * z; s.p1[r] = a[6] * z; s.p2[r] = a[7] * z;
    s.q11[r] = a[8] * z; s.q12[r] = a[9] * z; s.q21[r] = a[10] * z; s.q22[r] = a[11] * z;
    const int fy = ty * R + r;
    sm.ub[fy][tx] = s.ub[r];
    sm.vb1[fy][tx] = s.vb1[r];
    sm.vb2[fy][tx] = s.vb2[r];
  }
  // every pixel of the footprint in the FOV with both forward neighbours: the
  // loop without the mask selects gives the same bits
  const bool full = mb == (R == 1 ? 7u : R == 2 ? 077u : 07777u);
  if (__syncthreads_and(full))
    tgv_iterate<FW, NY, R, FTZ, false>(tp, n_iters, tx, ty, mb, c, s, sm);
  else
    tgv_iterate<FW, NY, R, FTZ, true>(tp, n_iters, tx, ty, mb, c, s, sm);

  if (!col_in || tx < B || tx >= FW - B) return;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int fy = ty * R + r;
    if (fy < B || fy >= FH - B || !ok[r]) continue;
    const unsigned k = idx[r];
    const float a[12] = {s.u[r],  s.ub[r], s.v1[r],  s.v2[r],  s.vb1[r], s.vb2[r],
                         s.p1[r], s.p2[r], s.q11[r], s.q12[r], s.q21[r], s.q22[r]};
#pragma unroll
    for (int j = 0; j < 12; ++j) out.s[j][k] = a[j];
  }
}

// v, vbar, q <- 0 on a new level (and before a warm start), like p.
__global__ void k_tgv_reset(LevelView L) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  const size_t i = (size_t)y * L.P + x;
  L.v1[i] = L.v2[i] = L.vb1[i] = L.vb2[i] = 0.f;
  L.q11[i] = L.q12[i] = L.q21[i] = L.q22[i] = 0.f;
}

namespace {

dim3 tgrid(int W, int H) { return dim3((W + 31) / 32, (H + 7) / 8); }

TgvState primary(const LevelView& L) {
  return TgvState{{L.u, L.ubar, L.v1, L.v2, L.vb1, L.vb2, (float*)L.p1.p, (float*)L.p2.p,
                   L.q11, L.q12, L.q21, L.q22}};
}

TgvState alternate(const LevelView& L) {
  TgvState s;
  for (int j = 0; j < 12; ++j) s.s[j] = L.tgv_alt[j];
  return s;
}

template <int FW, int NY, int R, int MB, bool FTZ, bool IDLE>
cudaError_t launch_blocked_f(const LevelView& L, const TgvState& in, const TgvState& out,
                             const TgvParams& tp, int B, int n, bool chained, int idle,
                             cudaStream_t st) {
  const int IW = FW - 2 * B, IH = NY * R - 2 * B;
  if (IW <= 0 || IH <= 0 || n < 0 || n > B) return cudaErrorInvalidValue;
  constexpr size_t smem = sizeof(TgvShared<FW, NY, R>);
  if constexpr (smem > 48 * 1024) {      // above the default limit: opt in once per device
    static std::atomic<unsigned long long> opted{0};
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const unsigned long long bit = 1ull << (dev & 63);
    if (!(opted.load() & bit)) {
      e = cudaFuncSetAttribute(k_tgv_blocked<FW, NY, R, MB, FTZ, IDLE>,
                               cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
      if (e != cudaSuccess) return e;
      opted.fetch_or(bit);
    }
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((L.W + IW - 1) / IW, (L.H + IH - 1) / IH, 1);
  cfg.blockDim = dim3(FW, NY, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, k_tgv_blocked<FW, NY, R, MB, FTZ, IDLE>, L, in, out, tp, B, n,
                            chained ? 1 : 0, idle);
}

// SKIP: also instantiated without the footprints outside the FOV.
template <int FW, int NY, int R, int MB = (FW * NY >= 512 ? 1 : 2), bool SKIP = false>
cudaError_t launch_blocked_t(const LevelView& L, const TgvState& in, const TgvState& out,
                             const TgvParams& tp, int B, int n, bool chained, int idle,
                             cudaStream_t st) {
  const bool ftz = tgv_normal_radii(tp);
  if constexpr (SKIP) {
    if (idle >= 0)
      return ftz ? launch_blocked_f<FW, NY, R, MB, true, true>(L, in, out, tp, B, n, chained, idle, st)
                 : launch_blocked_f<FW, NY, R, MB, false, true>(L, in, out, tp, B, n, chained, idle, st);
  }
  return ftz ? launch_blocked_f<FW, NY, R, MB, true, false>(L, in, out, tp, B, n, chained, idle, st)
             : launch_blocked_f<FW, NY, R, MB, false, false>(L, in, out, tp, B, n, chained, idle, st);
}

// The 32 x 32 footprint on 256 threads of 4 rows (variant 0), 1024 threads
// of 1 row (1) or 512 threads of 2 rows (2): more threads shorten each
// thread's dependent chain per iteration on the latency-bound levels.  The
// 64 x 32 footprint on 512 threads of 4 rows (3) or 1024 threads of 2 rows
// (4): less halo recomputed per interior pixel on the large levels.  Only
// the automatic schedule uses 32 x 16 on 512 threads (5), 32 x 24 on 768 (6)
// and 32 x 48 on 768 of 2 rows (7).
cudaError_t launch_blocked(int variant, const LevelView& L, const TgvState& in,
                           const TgvState& out, const TgvParams& tp, int B, int n, bool chained,
                           int idle, cudaStream_t st) {
#define FS_TGV(...) return launch_blocked_t<__VA_ARGS__>(L, in, out, tp, B, n, chained, idle, st)
  switch (variant) {
    case 0: FS_TGV(32, 8, 4, 2, true);
    case 1: FS_TGV(32, 32, 1);
    case 2: FS_TGV(32, 16, 2);
    case 3: FS_TGV(64, 8, 4, 1, true);
    case 4: FS_TGV(64, 16, 2);
    case 5: FS_TGV(32, 16, 1);
    case 6: FS_TGV(32, 24, 1);
    case 7: FS_TGV(32, 24, 2, 1, true);
    default: return cudaErrorInvalidValue;
  }
#undef FS_TGV
}

}  // namespace

// Fitted as pd_auto's table.  What it picks against the fixed choice it
// replaces (32 x 32 footprints of 256 threads at depth 4), us per 10 / 100
// iterations: 50 x 50 9.5 / 58.6 against 18.2 / 118.7, 200 x 200 11.2 / 89.9
// against 18.7 / 138.5, 512 x 512 35.6 / 309 against 45.4 / 339.
PdSchedule tgv_auto(const LevelView& L, int iters, int launches, int sms) {
  static const BlockFit kFit[] = {
      {5, 32, 16, 1, 2.3f, 0.24f, false}, {6, 32, 24, 1, 2.7f, 0.36f, false},
      {2, 32, 32, 1, 3.0f, 0.46f, false}, {7, 32, 48, 1, 3.3f, 0.70f, true},
      {3, 64, 32, 1, 5.3f, 0.78f, true},  {0, 32, 32, 2, 3.3f, 0.95f, true},
  };
  return block_schedule(kFit, (int)(sizeof(kFit) / sizeof(kFit[0])), L, iters, launches, sms);
}

cudaError_t launch_tgv_iterations(const LevelView& L, const TgvParams& tp, const PdSchedule& ps,
                                  int n, cudaStream_t st) {
  if (ps.launches <= 0) {             // a dual and a primal launch per iteration
    const dim3 g = tgrid(L.W, L.H), b(32, 8);
    for (int k = 0; k < n; ++k) {
      k_tgv_dual<<<g, b, 0, st>>>(L, tp);
      k_tgv_primal<<<g, b, 0, st>>>(L, tp);
    }
    return cudaGetLastError();
  }
  // temporal blocking: an even number of launches (when n >= 2), so that the
  // state ends in the level's planes
  const int nl = ps.launches;
  const TgvState A = primary(L), Bs = alternate(L);
  for (int k = 0, done = 0; k < nl; ++k) {
    int m = (n - done) / (nl - k);
    if ((n - done) % (nl - k)) ++m;
    cudaError_t e = launch_blocked(ps.variant, L, (k % 2 == 0) ? A : Bs, (k % 2 == 0) ? Bs : A,
                                   tp, ps.depth, m, k > 0, !ps.skip ? -1 : k == 0 ? n : 0, st);
    if (e != cudaSuccess) return e;
    done += m;
  }
  if (nl % 2 == 1) {                  // a single launch: copy the state back
    const size_t bytes = (size_t)L.P * L.H * sizeof(float);
    for (int j = 0; j < 12; ++j) {
      cudaError_t e = cudaMemcpyAsync(A.s[j], Bs.s[j], bytes, cudaMemcpyDeviceToDevice, st);
      if (e != cudaSuccess) return e;
    }
  }
  return cudaGetLastError();
}

cudaError_t launch_tgv_reset(const LevelView& L, cudaStream_t st) {
  k_tgv_reset<<<tgrid(L.W, L.H), dim3(32, 8), 0, st>>>(L);
  return cudaGetLastError();
}

}  // namespace fs
