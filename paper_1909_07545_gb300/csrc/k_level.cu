// k_level.cu -- per-level kernels of the fisheye stereo path other than the
// primal-dual iteration: trajectory field, calibration field and
// pre-rotation, pyramid down/up-sampling, tensor and step sizes,
// warp + linearisation, clip + update, triangulation.
#include "fs_kernels.h"
#include "level_px.cuh"
#include "pd_math.cuh"
#include "pd_tgv_math.cuh"

namespace fs {

// ------------------------------------------------------------ float-float stores
// A plane value in storage S (rounded to nearest) and, in lo, the part of
// the float-float value v that the stored value leaves out.
template <int S>
__device__ __forceinline__ void sst_df(const SPlane& pl, float* __restrict__ lo, size_t i, df v) {
  const float s = round_storage<S>(v.hi);
  sst<S>(pl, i, s);
  lo[i] = __fadd_rn(__fsub_rn(v.hi, s), v.lo);
}

template <int S>
__device__ __forceinline__ df sld_df(const SPlane& pl, const float* __restrict__ lo, size_t i) {
  return df{sld<S>(pl, i), lo[i]};
}

// ------------------------------------------------------------ fields of a pose
// gamma'(x) = normalise(d/ds pi(pi^-1(x) + s t')) at s -> 0 (Sec. III-B,
// Eq. 6-7), evaluated as the analytic image-plane velocity of a point on the
// pixel's ray under the (pre-rotated) translation t' (unit vector).  The
// velocity and its normalisation are computed in float-float and rounded
// once.  Zero outside the mask and where the velocity vanishes (epipoles).
__device__ __forceinline__ float2 trajectory_df(const DevCamDF& cam, const RayDF& r, df tx,
                                                df ty, df tz) {
  df vx, vy;
  cam_velocity_df(cam, r, tx, ty, tz, vx, vy);
  const df n = dd_sqrt(dd_add(dd_mul(vx, vx), dd_mul(vy, vy)));
  return n.hi >= 1e-3f ? make_float2(dd_div(vx, n).hi, dd_div(vy, n).hi) : make_float2(0.f, 0.f);
}

// c(x) = pi_1(R X) - x, X = pi_0^-1(x) the ray r, at the level-0 FOV pixels
// (Sec. IV-A, the pre-rotation: t = 0), 0 elsewhere; in float-float, stored as
// the float pair (hi x, hi y, lo x, lo y).  x stands for pi_0(X), which it
// equals to about 1e-13 px.  (Two identical cameras with R = I have the field
// exactly 0; the host writes that one without a kernel.)
__device__ __forceinline__ float4 calib_df(const DevCamDF& c1, const RotDF& R, const RayDF& r,
                                           int x, int y) {
  const df X[3] = {dd_mul(r.s, r.ux), dd_mul(r.s, r.uy), r.c};
  df Y[3];
#pragma unroll
  for (int k = 0; k < 3; ++k)
    Y[k] = dd_add(dd_add(dd_mul(R.r[3 * k], X[0]), dd_mul(R.r[3 * k + 1], X[1])),
                  dd_mul(R.r[3 * k + 2], X[2]));
  df px, py;
  cam_project_df(c1, Y[0], Y[1], Y[2], px, py);
  const df dx = dd_sub(px, df_f((float)x)), dy = dd_sub(py, df_f((float)y));
  return make_float4(dx.hi, dy.hi, dx.lo, dy.lo);
}

// gamma' of every level and the calibration field of the first, in one launch
// over all levels' 32 x 8 blocks: the finest level's ray, most of the work,
// serves both fields, and the coarse levels fill the SMs beside it.  A pose
// change of a 1024 x 1024 rig (5 levels, Kannala-Brandt), with the
// pre-rotation of an image behind it and both read back, went from 317 to 223
// us.  MODEL: camera 0's lens, a constant for the compiler.  Bound by
// instruction issue: about 5000 FP32 instructions a pixel, 12 float-float
// divisions and 2 sine-cosine series among them.
template <int MODEL>
__global__ void __launch_bounds__(256) k_pose_fields(const __grid_constant__ PoseFields F) {
  int l = 0;
  while (l + 1 < F.n && (int)blockIdx.x >= F.lv[l + 1].first_block) ++l;
  const PoseLevel& L = F.lv[l];
  const int b = (int)blockIdx.x - L.first_block, nbx = (L.W + 31) / 32;
  const int x = b % nbx * 32 + (int)threadIdx.x, y = b / nbx * 8 + (int)threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  const size_t i = (size_t)y * L.P + x;
  float2 g = make_float2(0.f, 0.f);
  float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
  if (L.mask[i] & MASK_IN) {
    DevCamDF cam = L.cam;
    cam.model = cam.f32.model = MODEL;
    const RayDF r = cam_unproject_df(cam, x, y);
    g = trajectory_df(cam, r, F.tx, F.ty, F.tz);
    if (l == 0 && F.field) c = calib_df(F.cam1, F.R, r, x, y);
  }
  L.gamma[i] = g;
  if (l == 0 && F.field) F.field[i] = c;
}

cudaError_t launch_pose_fields(const PoseFields& F, int blocks, cudaStream_t st) {
  const dim3 blk(32, 8);
  switch (F.lv[0].cam.model) {
    case 0: k_pose_fields<0><<<blocks, blk, 0, st>>>(F); break;
    case 1: k_pose_fields<1><<<blocks, blk, 0, st>>>(F); break;
    case 3: k_pose_fields<3><<<blocks, blk, 0, st>>>(F); break;
    case 4: k_pose_fields<4><<<blocks, blk, 0, st>>>(F); break;
    default: k_pose_fields<2><<<blocks, blk, 0, st>>>(F); break;
  }
  return cudaGetLastError();
}

// ------------------------------------------------------------ pre-rotation
// I1'(x) = I1(x + c(x)), bilinear, position clamped to the image (Sec.
// IV-A); I1 dense FP32 (pitch W), output pitch P in the level's storage.
// The sample position and the interpolation are float-float; the result is
// stored rounded, its low part in lo (the start of the pyramid's carry).
struct TapDF {
  int i0, i1;   // the two neighbouring samples
  df a;         // weight of i1
};

__device__ __forceinline__ TapDF tap_linear_df(int x, df d, int n) {
  float fl;
  df f;
  dd_floor_frac(d, fl, f);
  const int b = x + (int)fl;
  TapDF t;
  if (b < 0) { t.i0 = 0; t.a = df_f(0.f); }
  else if (b >= n - 1) { t.i0 = max(n - 2, 0); t.a = df_f(n >= 2 ? 1.f : 0.f); }
  else { t.i0 = b; t.a = f; }
  t.i1 = min(t.i0 + 1, n - 1);
  return t;
}

// I0, when given, is copied in beside it (the finest level of I0: k_copy_in_s).
__device__ __forceinline__ df prerotate_px(const float* __restrict__ I1,
                                           const float4* __restrict__ field, int x, int y, int W,
                                           int H, int P) {
  const float4 c = field[(size_t)y * P + x];
  const TapDF tx = tap_linear_df(x, df{c.x, c.z}, W), ty = tap_linear_df(y, df{c.y, c.w}, H);
  const float* r0 = I1 + (size_t)ty.i0 * W;
  const float* r1 = I1 + (size_t)ty.i1 * W;
  const float v00 = __ldg(r0 + tx.i0), v01 = __ldg(r0 + tx.i1);
  const float v10 = __ldg(r1 + tx.i0), v11 = __ldg(r1 + tx.i1);
  const df top = dd_add(df_f(v00), dd_mul(tx.a, two_sum(v01, -v00)));
  const df bot = dd_add(df_f(v10), dd_mul(tx.a, two_sum(v11, -v10)));
  return dd_add(top, dd_mul(ty.a, dd_sub(bot, top)));
}

template <int S>
__global__ void k_prerotate(const float* __restrict__ I0, SPlane out0, float* __restrict__ lo0,
                            const float* __restrict__ I1, const float4* __restrict__ field,
                            SPlane out, float* __restrict__ lo, int W, int H, int P) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= W || y >= H) return;
  size_t i = (size_t)y * P + x;
  if (I0) sst_df<S>(out0, lo0, i, df_f(I0[(size_t)y * W + x]));
  sst_df<S>(out, lo, i, prerotate_px(I1, field, x, y, W, H, P));
}

// Dense FP32 (pitch W) -> pitched plane in the level's storage, with the
// low part of the rounding in lo (0 for FP32 storage): the finest level of
// I0, or a level image written through fs_buffer_write.
template <int S>
__global__ void k_copy_in_s(const float* __restrict__ src, SPlane dst, float* __restrict__ lo,
                            int W, int H, int P) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= W || y >= H) return;
  sst_df<S>(dst, lo, (size_t)y * P + x, df_f(src[(size_t)y * W + x]));
}

// Dense (pitch W) -> pitched FP32 copy, used for the warm-start input.
__global__ void k_copy_in(const float* __restrict__ src, float* __restrict__ dst, int W, int H,
                          int P) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= W || y >= H) return;
  dst[(size_t)y * P + x] = src[(size_t)y * W + x];
}

// ------------------------------------------------------------ pyramid
// 2x2 box mean over the children inside the finer mask (all existing
// children when none is inside), for I0 and I1 together (Sec. IV-B).  The
// children are float-float (stored value + low part), the mean is formed in
// float-float and stored rounded with its own low part, so each level is
// the exact mean of the exact finer level, rounded once.
template <int S>
__global__ void k_downsample(LevelView F, LevelView C) {
  int X = blockIdx.x * blockDim.x + threadIdx.x;
  int Y = blockIdx.y * blockDim.y + threadIdx.y;
  if (X >= C.W || Y >= C.H) return;
  df s0 = df_f(0.f), s1 = df_f(0.f), a0 = df_f(0.f), a1 = df_f(0.f);
  int nin = 0, nall = 0;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      int x = 2 * X + i, y = 2 * Y + j;
      if (x < F.W && y < F.H) {
        size_t k = (size_t)y * F.P + x;
        const df v0 = sld_df<S>(F.I0, F.I0lo, k), v1 = sld_df<S>(F.I1, F.I1lo, k);
        a0 = dd_add(a0, v0); a1 = dd_add(a1, v1); ++nall;
        if (F.mask[k] & MASK_IN) { s0 = dd_add(s0, v0); s1 = dd_add(s1, v1); ++nin; }
      }
    }
  }
  size_t o = (size_t)Y * C.P + X;
  if (nin > 0) {
    sst_df<S>(C.I0, C.I0lo, o, dd_div_f(s0, (float)nin));
    sst_df<S>(C.I1, C.I1lo, o, dd_div_f(s1, (float)nin));
  } else {
    sst_df<S>(C.I0, C.I0lo, o, dd_div_f(a0, (float)nall));
    sst_df<S>(C.I1, C.I1lo, o, dd_div_f(a1, (float)nall));
  }
}

// The start of a frame of a small image: k_prerotate of both images and
// k_downsample down to the n-th level in one
// launch: a CTA takes 16 x 16 pixels of the finest level, whose means down to
// one pixel need nothing of its neighbours', and carries each level to the
// next in shared memory.  Launches of their own took 2 to 4 us each, most of
// it start and drain: a 128 x 128 frame of 3 levels went from 133.1 to 124.9
// us, a 333 x 257 one of 4 from 534.2 to 529.9.
struct PyramidLevel {
  int W, H, P;
  const uint8_t* mask;
  SPlane I0, I1;
  float *I0lo, *I1lo;
};
struct Pyramid {
  int n;
  PyramidLevel lv[kPyramidLevels];
};
constexpr int kPyrTile = 1 << (kPyramidLevels - 1);

// Store both images' values at o; what the next level reads of them.
template <int S>
__device__ __forceinline__ float4 pyramid_store(const PyramidLevel& L, size_t o, df v0, df v1) {
  const float s0 = round_storage<S>(v0.hi), s1 = round_storage<S>(v1.hi);
  const float l0 = __fadd_rn(__fsub_rn(v0.hi, s0), v0.lo);
  const float l1 = __fadd_rn(__fsub_rn(v1.hi, s1), v1.lo);
  sst<S>(L.I0, o, s0);
  sst<S>(L.I1, o, s1);
  L.I0lo[o] = l0;
  L.I1lo[o] = l1;
  return make_float4(s0, l0, s1, l1);
}

template <int S>
__global__ void __launch_bounds__(kPyrTile * kPyrTile)
k_pyramid(const float* __restrict__ I0, const float* __restrict__ I1,
          const float4* __restrict__ field, const __grid_constant__ Pyramid py) {
  __shared__ float4 s[kPyrTile * kPyrTile * 4 / 3];     // every level's tile
  const int t = threadIdx.y * kPyrTile + threadIdx.x;
  {
    const PyramidLevel& L = py.lv[0];
    const int x = blockIdx.x * kPyrTile + threadIdx.x, y = blockIdx.y * kPyrTile + threadIdx.y;
    if (x < L.W && y < L.H)
      s[t] = pyramid_store<S>(L, (size_t)y * L.P + x, df_f(I0[(size_t)y * L.W + x]),
                              prerotate_px(I1, field, x, y, L.W, L.H, L.P));
  }
  int n = kPyrTile, from = 0;
  for (int l = 1; l < py.n; ++l) {
    __syncthreads();
    const PyramidLevel &F = py.lv[l - 1], &C = py.lv[l];
    const int m = n / 2, to = from + n * n, cx = t % m, cy = t / m;
    const int X = blockIdx.x * m + cx, Y = blockIdx.y * m + cy;
    if (t < m * m && X < C.W && Y < C.H) {
      df s0 = df_f(0.f), s1 = df_f(0.f), a0 = df_f(0.f), a1 = df_f(0.f);
      int nin = 0, nall = 0;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const int x = 2 * X + i, y = 2 * Y + j;
          if (x < F.W && y < F.H) {
            const float4 v = s[from + (2 * cy + j) * n + 2 * cx + i];
            const df v0{v.x, v.y}, v1{v.z, v.w};
            a0 = dd_add(a0, v0); a1 = dd_add(a1, v1); ++nall;
            if (F.mask[(size_t)y * F.P + x] & MASK_IN) {
              s0 = dd_add(s0, v0); s1 = dd_add(s1, v1); ++nin;
            }
          }
        }
      }
      const size_t o = (size_t)Y * C.P + X;
      s[to + t] = nin > 0 ? pyramid_store<S>(C, o, dd_div_f(s0, (float)nin), dd_div_f(s1, (float)nin))
                          : pyramid_store<S>(C, o, dd_div_f(a0, (float)nall),
                                             dd_div_f(a1, (float)nall));
    }
    from = to;
    n = m;
  }
}

// u, w of level C (coarse) -> level F (fine): upsample_px at every pixel.
template <int S>
__global__ void k_upsample(LevelView C, LevelView F) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= F.W || y >= F.H) return;
  float2 w;
  upsample_px<S, false>(C, F, x, y, w);
}

// Warm start at the finest level from a disparity already in L.u: w is
// rebuilt by walking along the trajectory field in n = ceil(|d| / du_max)
// equal steps of d / n, each along the renormalised bicubic gamma' at the
// current point; ubar = u_w = u, p = 0.  Non-finite disparities count as 0
// and n is capped at kMaxWarmSteps.
constexpr int kMaxWarmSteps = 16384;
template <int S>
__global__ void k_warm_start(LevelView L, float du_max) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  size_t i = (size_t)y * L.P + x;
  float d = L.u[i];
  if (!(L.mask[i] & MASK_IN) || !isfinite(d)) d = 0.f;
  float2 w = make_float2(0.f, 0.f);
  int n = (int)fminf(ceilf(fabsf(d) / du_max), (float)kMaxWarmSteps);
  if (n > 0) {
    float step = d / (float)n;
    for (int k = 0; k < n; ++k) {
      float2 gr = sample_bicubic2(L.gamma, L.W, L.H, L.P, x, w.x, y, w.y);
      float nr = sqrtf(gr.x * gr.x + gr.y * gr.y);
      if (nr >= 1e-6f) {
        w.x = fmaf(step, gr.x / nr, w.x);
        w.y = fmaf(step, gr.y / nr, w.y);
      }
    }
  }
  L.u[i] = d; L.ubar[i] = d; L.uw[i] = d;
  L.w[i] = w;
  sst<S>(L.p1, i, 0.f); sst<S>(L.p2, i, 0.f);
}

// Warm start at the finest level from its own last u and w (a video
// stream's next frame): ubar = u_w = u, p = 0, w kept.  Non-finite
// disparities count as 0 (with w = 0).
template <int S>
__device__ __forceinline__ float continue_px(const LevelView& L, size_t i, bool in, float2& w) {
  float d = ldf<true>(L.u + i);
  w = ldf2<true>(L.w + i);
  if (!in || !isfinite(d)) {
    d = 0.f;
    w = make_float2(0.f, 0.f);
    L.w[i] = w;
  }
  L.u[i] = d; L.ubar[i] = d; L.uw[i] = d;
  sst<S>(L.p1, i, 0.f); sst<S>(L.p2, i, 0.f);
  return d;
}

// ------------------------------------------------------------ tensor + steps
template <int S>
__global__ void k_tensor(LevelView L, float beta, float eta, int precond) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  tensor_px<S>(L, x, y, beta, eta, precond);
}

// ------------------------------------------------------------ warp + linearise
// The per-warp constants of the primal-dual iterations at pixel i
// (launch_pd_consts' values: px_make of the stored sigma, tau, I_u, rho0
// and u_w), written by the kernels that start a warp while they hold
// I_u, rho0 and u_w.  keep: dinv and sd, which follow from sigma alone, stand
// from the level's last warp.
template <int S>
__device__ __forceinline__ void pd_consts_px(const LevelView& L, size_t i, float tau, float Iu,
                                             float rho0, float uw, float lam, float eps,
                                             bool keep) {
  PxRaw raw;
  raw.sx = raw.sy = 0.f;                     // not used by px_make's outputs below
  raw.sig = keep ? 0.f : L.sig[i];
  raw.tau = tau;
  raw.Iu = round_storage<S>(Iu);
  raw.rho0 = round_storage<S>(rho0);
  raw.uw = uw;
  PxConst c;
  px_make(raw, lam, eps, c);
  if (!keep) {
    L.dinv[i] = c.dinv;
    L.sd[i] = c.sd;
  }
  L.step[i] = c.step;
  L.c0[i] = c.c0;
}

// The same for the TGV iterations (tgv_const of the stored values): sigma_p in
// L.dinv, tau_v in L.sd, the L1 step and c0 in their planes; and vbar <- v.
__device__ __forceinline__ void tgv_consts_px(const LevelView& L, int x, int y, size_t i,
                                              float Iu, float rho0, float uw, float lam,
                                              int precond) {
  const unsigned ml = x > 0 ? L.mask[i - 1] : 0u, mu = y > 0 ? L.mask[i - L.P] : 0u;
  const TgvParams tp{lam, 0.f, 0.f, 0.f, precond};
  TgvConst c;
  tgv_const(L.mask[i], ml, mu, 0.f, 0.f, L.sig[i], L.tau[i], Iu, rho0, uw, tp, c);
  L.dinv[i] = c.sp;
  L.sd[i] = c.tv;
  L.step[i] = c.step;
  L.c0[i] = c.c0;
}

// What a warp start writes for the iterations (enum WarpConsts; TGV: one of
// its two).
template <int S, bool TGV>
__device__ __forceinline__ void warp_consts_px(const LevelView& L, int x, int y, size_t i,
                                               float tau, float Iu, float rho0, float u,
                                               float lam, float eps, int consts, bool keep) {
  if constexpr (!TGV) {
    pd_consts_px<S>(L, i, tau, Iu, rho0, u, lam, eps, keep);
  } else {
    tgv_consts_px(L, x, y, i, Iu, rho0, u, lam, consts == WARP_CONSTS_TGV);
    L.vb1[i] = L.v1[i];
    L.vb2[i] = L.v2[i];
  }
}

__global__ void k_tgv_consts(LevelView L, float lam, int precond) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  size_t i = (size_t)y * L.P + x;
  tgv_consts_px(L, x, y, i, sld<ST_F32>(L.Iu, i), sld<ST_F32>(L.rho0, i), L.uw[i], lam, precond);
}

template <int S, bool TGV>
__global__ void k_warp(LevelView L, int central, float lam, float eps, int consts) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  size_t i = (size_t)y * L.P + x;
  float Iu = 0.f, rho0 = 0.f;
  float2 g = make_float2(0.f, 0.f);
  if (L.mask[i] & MASK_IN) warp_px<S>(L, x, y, i, L.w[i], central, Iu, rho0, g);
  sst<S>(L.Iu, i, Iu);
  sst<S>(L.rho0, i, rho0);
  L.g[i] = g;
  float u = L.u[i];
  L.ubar[i] = u;
  L.uw[i] = u;
  warp_consts_px<S, TGV>(L, x, y, i, L.tau[i], Iu, rho0, u, lam, eps, consts, false);
}

constexpr int kBlkX = 32, kBlkY = 8;     // the CTAs of the per-pixel kernels

// The start of a level in one pass: tensor and step sizes, the start state
// (MODE), and the first warp's linearisation and constants: k_tensor, the
// start state and k_warp, whose results a pixel only needs of itself.  A level started with three to five launches,
// each of a few microseconds on the small levels: a 128 x 128 frame of 3
// levels, all in all, went from 169 to 141 us, an 800 x 800 frame of 5 from 1707
// to 1684.  A programmatic dependent launch that waits first, which starts
// sooner than an ordinary one; so what the launch before wrote besides images
// is read through L2: 128 x 128 126.4 -> 120.8 us.
// The step sizes need the tensor at the left and the upper pixel too: a CTA
// evaluates each once and shares it (640 x 640 frame 302.6 -> 301.0 us, 1024 x
// 1024 6980 -> 6961).
template <int S, int MODE, bool TGV>
__global__ void k_level_start(LevelView C, LevelView L, float beta, float eta, int precond,
                              int central, float lam, float eps, int consts) {
  // the sums of |T^1/2| that the pixels to the right and below need too, with
  // those of the column and the row before the block
  __shared__ float s_h[kBlkY][kBlkX + 1], s_v[kBlkY + 1][kBlkX];
  cudaGridDependencySynchronize();
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int x0 = blockIdx.x * kBlkX, y0 = blockIdx.y * kBlkY;
  const int x = x0 + tx, y = y0 + ty;
  const bool inside = x < L.W && y < L.H;
  TensorAt t{};
  if (inside) {
    t = tensor_at<S>(L, x, y, beta, eta);
    s_h[ty][tx + 1] = t.aa + t.bb;
    s_v[ty + 1][tx] = t.bb + t.cc;
  }
  if (precond) {
    const int k = ty * kBlkX + tx - kBlkX;            // the second warp: the column
    if (ty == 0 && y0 > 0 && x < L.W) {
      const TensorAt a = tensor_at<S>(L, x, y0 - 1, beta, eta);
      s_v[0][tx] = a.bb + a.cc;
    } else if (k >= 0 && k < kBlkY && x0 > 0 && y0 + k < L.H) {
      const TensorAt a = tensor_at<S>(L, x0 - 1, y0 + k, beta, eta);
      s_h[k][0] = a.aa + a.bb;
    }
  }
  __syncthreads();
  if (!inside) return;
  size_t i = (size_t)y * L.P + x;
  const bool in = L.mask[i] & MASK_IN;
  tensor_store_px<S>(
      L, x, y, t, precond, L.mask[i], x > 0 && (L.mask[i - 1] & MASK_GX),
      y > 0 && (L.mask[i - L.P] & MASK_GY), [&] { return s_h[ty][tx]; }, [&] { return s_v[ty][tx]; });
  float u = 0.f;
  float2 w = make_float2(0.f, 0.f);
  if constexpr (MODE == START_ZERO) {
    zero_px<S>(L, i);
  } else if constexpr (MODE == START_UPSAMPLE) {
    u = upsample_px<S, true>(C, L, x, y, w);
  } else if constexpr (MODE == START_CONTINUE) {
    u = continue_px<S>(L, i, in, w);
  } else {
    u = ldf<true>(L.u + i);
    w = ldf2<true>(L.w + i);
  }
  if constexpr (TGV && MODE != START_GIVEN) {
    L.v1[i] = L.v2[i] = 0.f;
    L.q11[i] = L.q12[i] = L.q21[i] = L.q22[i] = 0.f;
  }
  float Iu = 0.f, rho0 = 0.f;
  float2 g = make_float2(0.f, 0.f);
  if (in) warp_px<S>(L, x, y, i, w, central, Iu, rho0, g);
  sst<S>(L.Iu, i, Iu);
  sst<S>(L.rho0, i, rho0);
  L.g[i] = g;
  L.ubar[i] = u;
  L.uw[i] = u;
  warp_consts_px<S, TGV>(L, x, y, i, L.tau[i], Iu, rho0, u, lam, eps, consts, false);
}

// ------------------------------------------------------------ clip + update
// CHAIN (k_clip_warp too): launched behind the warp's iterations as a
// programmatic dependent launch.  The wait comes first, then the trigger that
// lets the next launch be scheduled, and what those iterations or the last
// warp start wrote is read through L2 (launches of a chain overlap, so an
// SM's L1 may hold older lines).
template <bool CHAIN>
__global__ void k_clip(LevelView L, float du_max) {
  if constexpr (CHAIN) {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
  }
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  size_t i = (size_t)y * L.P + x;
  if (!(L.mask[i] & MASK_IN)) return;
  float2 w;
  float un = clip_px<CHAIN>(L, i, du_max, w);
  L.u[i] = un;
  L.ubar[i] = un;
  L.uw[i] = un;
  L.w[i] = w;
}

// *p after a programmatic dependent launch's wait, through L2.
__device__ __forceinline__ float ld_after(const float* p) {
  float v;
  asm volatile("ld.global.cg.f32 %0, [%1];" : "=f"(v) : "l"(p) : "memory");
  return v;
}

// The end of one warp and the start of the next in one pass: k_clip then
// k_warp at every pixel, with the updated w and u kept in registers (each
// pixel's clip and linearisation read only that pixel's state; the gathers
// read I1 and gamma', which neither writes).  keep: pd_consts_px.
//
// On the small levels bound by its chain of dependent loads.  So the loads
// that need nothing of one another come first, and in a chain (CHAIN) those
// of what the level's start or the last warp start wrote before the wait:
// the chain's first primal-dual launch waited for that kernel before it let
// any launch behind it begin.  800 x 800, 5 levels,
// 20 warps of 10 iterations: 1682 -> 1602 us a frame; 128 x 128: 139 -> 137.
template <int S, bool CHAIN, bool TGV>
__global__ void k_clip_warp(LevelView L, float du_max, int central, float lam, float eps,
                            int consts, int keep) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  const bool inside = x < L.W && y < L.H;
  const size_t i = inside ? (size_t)y * L.P + x : 0;
  const bool in = L.mask[i] & MASK_IN;
  const float uw = ldf<CHAIN>(L.uw + i), tau = ldf<CHAIN>(L.tau + i);
  const float2 g0 = ldf2<CHAIN>(L.g + i);
  float2 w = ldf2<CHAIN>(L.w + i);
  if constexpr (CHAIN) {
    cudaGridDependencySynchronize();
    cudaTriggerProgrammaticLaunchCompletion();
  }
  float u;
  if constexpr (CHAIN) u = ld_after(L.u + i);
  else u = L.u[i];
  if (!inside) return;
  float Iu = 0.f, rho0 = 0.f;
  float2 g = make_float2(0.f, 0.f);
  if (in) {
    u = clip_u(u, uw, g0, du_max, w);
    L.w[i] = w;
    L.u[i] = u;
    warp_px<S>(L, x, y, i, w, central, Iu, rho0, g);
  }
  sst<S>(L.Iu, i, Iu);
  sst<S>(L.rho0, i, rho0);
  L.g[i] = g;
  L.ubar[i] = u;
  L.uw[i] = u;
  warp_consts_px<S, TGV>(L, x, y, i, tau, Iu, rho0, u, lam, eps, consts, keep);
}

// ------------------------------------------------------------ triangulation
// Range along the camera-0 ray of x from the rays pi^-1(x) and pi^-1(x + w)
// of the pre-rotated pair (virtual camera-1 centre C = -t'), closest point
// of the two lines: l0 = ((C x r1) . (r0 x r1)) / |r0 x r1|^2 (Sec. III-D).
// Disparity u and the range of a pixel with warp vector w; either output may
// be null.
__device__ __forceinline__ void depth_px(const LevelView& L, const DevCam& cam, float Cx,
                                         float Cy, float Cz, int x, int y, bool in, float u,
                                         float2 w, float* __restrict__ disp,
                                         float* __restrict__ depth) {
  const size_t o = (size_t)y * L.W + x;
  if (disp) disp[o] = in ? u : 0.f;
  if (!depth) return;
  if (!in) { depth[o] = __int_as_float(0x7fc00000); return; }
  if (w.x == 0.f && w.y == 0.f) {   // no displacement: the rays coincide, range +inf
    depth[o] = __int_as_float(0x7f800000);
    return;
  }
  Ray r0 = cam_unproject(cam, (float)x, (float)y);
  Ray r1 = cam_unproject(cam, (float)x + w.x, (float)y + w.y);
  float nx = r0.y * r1.z - r0.z * r1.y;
  float ny = r0.z * r1.x - r0.x * r1.z;
  float nz = r0.x * r1.y - r0.y * r1.x;
  float mx = Cy * r1.z - Cz * r1.y;
  float my = Cz * r1.x - Cx * r1.z;
  float mz = Cx * r1.y - Cy * r1.x;
  float den = nx * nx + ny * ny + nz * nz;
  depth[o] = den > 0.f ? (mx * nx + my * ny + mz * nz) / den : __int_as_float(0x7f800000);
}

__global__ void k_depth(LevelView L, DevCam cam, float Cx, float Cy, float Cz,
                        float* __restrict__ disp, float* __restrict__ depth) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  size_t i = (size_t)y * L.P + x;
  const bool in = L.mask[i] & MASK_IN;
  depth_px(L, cam, Cx, Cy, Cz, x, y, in, L.u[i], L.w[i], disp, depth);
}

// The end of a frame in one pass: k_clip of the last warp and k_depth, 3 us
// less of a frame up to 256 x 256.  CHAIN as in k_clip.
template <bool CHAIN>
__global__ void k_clip_depth(LevelView L, float du_max, DevCam cam, float Cx, float Cy, float Cz,
                             float* __restrict__ disp, float* __restrict__ depth) {
  if constexpr (CHAIN) cudaGridDependencySynchronize();
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  size_t i = (size_t)y * L.P + x;
  const bool in = L.mask[i] & MASK_IN;
  float2 w = make_float2(0.f, 0.f);
  float un = 0.f;
  if (in) {
    un = clip_px<CHAIN>(L, i, du_max, w);
    L.u[i] = un;
    L.ubar[i] = un;
    L.uw[i] = un;
    L.w[i] = w;
  }
  asm volatile("" : "+f"(w.x), "+f"(w.y));   // depth_px rounds as it does in k_depth
  depth_px(L, cam, Cx, Cy, Cz, x, y, in, un, w, disp, depth);
}

// ------------------------------------------------------------ buffer access
__global__ void k_pack(const float* __restrict__ src, int stride, float* __restrict__ dst, int W,
                       int H, int P) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= W || y >= H) return;
  dst[(size_t)y * W + x] = src[((size_t)y * P + x) * stride];
}

__global__ void k_unpack(const float* __restrict__ src, float* __restrict__ dst, int stride,
                         int W, int H, int P) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= W || y >= H) return;
  dst[((size_t)y * P + x) * stride] = src[(size_t)y * W + x];
}

// Stored plane <-> dense FP32 (buffer access to the storage-typed fields).
template <int S>
__global__ void k_pack_s(SPlane src, float* __restrict__ dst, int W, int H, int P) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= W || y >= H) return;
  dst[(size_t)y * W + x] = sld<S>(src, (size_t)y * P + x);
}

template <int S>
__global__ void k_unpack_s(const float* __restrict__ src, SPlane dst, int W, int H, int P) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= W || y >= H) return;
  sst<S>(dst, (size_t)y * P + x, src[(size_t)y * W + x]);
}

__global__ void k_mask_to_float(const uint8_t* __restrict__ m, float* __restrict__ dst, int W,
                                int H, int P) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= W || y >= H) return;
  dst[(size_t)y * W + x] = (m[(size_t)y * P + x] & MASK_IN) ? 1.f : 0.f;
}

// T^1/2 entries a, b, c from s: a = 1 - sx^2, b = -sx sy, c = 1 - sy^2.
template <int S>
__global__ void k_tensor_abc(LevelView L, float* __restrict__ dst) {
  int x = blockIdx.x * blockDim.x + threadIdx.x;
  int y = blockIdx.y * blockDim.y + threadIdx.y;
  if (x >= L.W || y >= L.H) return;
  size_t i = (size_t)y * L.P + x, o = (size_t)y * L.W + x, n = (size_t)L.W * L.H;
  float sx = sld<S>(L.sx, i), sy = sld<S>(L.sy, i);
  dst[o] = 1.f - sx * sx;
  dst[n + o] = -sx * sy;
  dst[2 * n + o] = 1.f - sy * sy;
}

// ---------------------------------------------------------------- launchers
// Host launch of the storage-typed kernels: the level's storage picks the
// compiled instantiation.
namespace {
dim3 grid_of(int W, int H) { return dim3((W + 31) / 32, (H + 7) / 8); }
const dim3 kBlk(kBlkX, kBlkY);

// One thread per pixel of level L; chained: as a programmatic dependent
// launch of the kernel before it on the stream.
template <typename K, typename... A>
cudaError_t launch_chained(K kernel, const LevelView& L, bool chained, cudaStream_t st, A... a) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid_of(L.W, L.H);
  cfg.blockDim = kBlk;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, a...);
}
}  // namespace

#define FS_STORAGE_SWITCH(st, CALL)                           \
  switch (st) {                                               \
    case ST_F16: { constexpr int S = ST_F16; CALL; } break;   \
    case ST_BF16: { constexpr int S = ST_BF16; CALL; } break; \
    default: { constexpr int S = ST_F32; CALL; } break;       \
  }                                                           \
  return cudaGetLastError();

cudaError_t launch_prerotate(const float* I0, const float* I1, const float4* field,
                             const LevelView& L0, cudaStream_t st) {
  FS_STORAGE_SWITCH(L0.st, (k_prerotate<S><<<grid_of(L0.W, L0.H), kBlk, 0, st>>>(
                               I0, L0.I0, L0.I0lo, I1, field, L0.I1, L0.I1lo, L0.W, L0.H, L0.P)))
}
int pyramid_blocks(const LevelView& L0) {
  return ((L0.W + kPyrTile - 1) / kPyrTile) * ((L0.H + kPyrTile - 1) / kPyrTile);
}
cudaError_t launch_pyramid(const float* I0, const float* I1, const float4* field,
                           const LevelView* const* levels, int n, cudaStream_t st) {
  if (n < 1 || n > kPyramidLevels) return cudaErrorInvalidValue;
  Pyramid py{};
  py.n = n;
  for (int l = 0; l < n; ++l) {
    const LevelView& v = *levels[l];
    py.lv[l] = PyramidLevel{v.W, v.H, v.P, v.mask, v.I0, v.I1, v.I0lo, v.I1lo};
  }
  const LevelView& L0 = *levels[0];
  const dim3 g((L0.W + kPyrTile - 1) / kPyrTile, (L0.H + kPyrTile - 1) / kPyrTile);
  FS_STORAGE_SWITCH(L0.st, (k_pyramid<S><<<g, dim3(kPyrTile, kPyrTile), 0, st>>>(I0, I1, field, py)))
}
cudaError_t launch_copy_in_image(const float* src, const LevelView& L, int which,
                                 cudaStream_t st) {
  const SPlane& dst = which == 0 ? L.I0 : L.I1;
  float* lo = which == 0 ? L.I0lo : L.I1lo;
  FS_STORAGE_SWITCH(L.st, (k_copy_in_s<S><<<grid_of(L.W, L.H), kBlk, 0, st>>>(
                              src, dst, lo, L.W, L.H, L.P)))
}
cudaError_t launch_downsample(const LevelView& F, const LevelView& C, cudaStream_t st) {
  FS_STORAGE_SWITCH(F.st, (k_downsample<S><<<grid_of(C.W, C.H), kBlk, 0, st>>>(F, C)))
}
cudaError_t launch_upsample(const LevelView& C, const LevelView& F, cudaStream_t st) {
  FS_STORAGE_SWITCH(F.st, (k_upsample<S><<<grid_of(F.W, F.H), kBlk, 0, st>>>(C, F)))
}
cudaError_t launch_warm_start(const LevelView& L, float du_max, cudaStream_t st) {
  FS_STORAGE_SWITCH(L.st, (k_warm_start<S><<<grid_of(L.W, L.H), kBlk, 0, st>>>(L, du_max)))
}
cudaError_t launch_tensor(const LevelView& L, float beta, float eta, int precond,
                          cudaStream_t st) {
  FS_STORAGE_SWITCH(L.st, (k_tensor<S><<<grid_of(L.W, L.H), kBlk, 0, st>>>(L, beta, eta,
                                                                          precond)))
}
cudaError_t launch_warp(const LevelView& L, int central, float lam, float eps, int consts,
                        cudaStream_t st) {
  if (consts != WARP_CONSTS_HUBER) {            // TGV: FP32 storage only
    k_warp<ST_F32, true><<<grid_of(L.W, L.H), kBlk, 0, st>>>(L, central, lam, eps, consts);
    return cudaGetLastError();
  }
  FS_STORAGE_SWITCH(L.st, (k_warp<S, false><<<grid_of(L.W, L.H), kBlk, 0, st>>>(
                              L, central, lam, eps, consts)))
}

template <int S, bool TGV>
static auto level_start_kernel(int mode) {
  return mode == START_ZERO       ? k_level_start<S, START_ZERO, TGV>
         : mode == START_UPSAMPLE ? k_level_start<S, START_UPSAMPLE, TGV>
         : mode == START_CONTINUE ? k_level_start<S, START_CONTINUE, TGV>
                                  : k_level_start<S, START_GIVEN, TGV>;
}

cudaError_t launch_level_start(int mode, const LevelView& C, const LevelView& L, float beta,
                               float eta, int precond, int central, float lam, float eps,
                               int consts, cudaStream_t st) {
  if (consts != WARP_CONSTS_HUBER)
    return launch_chained(level_start_kernel<ST_F32, true>(mode), L, true, st, C, L, beta, eta,
                          precond, central, lam, eps, consts);
  FS_STORAGE_SWITCH(L.st, return launch_chained(level_start_kernel<S, false>(mode), L, true, st,
                                                C, L, beta, eta, precond, central, lam, eps,
                                                consts))
}

cudaError_t launch_clip_depth(const LevelView& L, float du_max, const DevCam& cam, float Cx,
                              float Cy, float Cz, float* disp, float* depth, bool chained,
                              cudaStream_t st) {
  return launch_chained(chained ? k_clip_depth<true> : k_clip_depth<false>, L, chained, st, L,
                        du_max, cam, Cx, Cy, Cz, disp, depth);
}

cudaError_t launch_tgv_consts(const LevelView& L, float lam, int precond, cudaStream_t st) {
  k_tgv_consts<<<grid_of(L.W, L.H), kBlk, 0, st>>>(L, lam, precond);
  return cudaGetLastError();
}

cudaError_t launch_clip_warp(const LevelView& L, float du_max, int central, float lam, float eps,
                             int consts, bool keep, bool chained, cudaStream_t st) {
  if (consts != WARP_CONSTS_HUBER)
    return launch_chained(k_clip_warp<ST_F32, false, true>, L, false, st, L, du_max, central, lam,
                          eps, consts, (int)keep);
  FS_STORAGE_SWITCH(L.st, return launch_chained(chained ? k_clip_warp<S, true, false>
                                                        : k_clip_warp<S, false, false>,
                                                L, chained, st, L, du_max, central, lam, eps,
                                                consts, (int)keep))
}
cudaError_t launch_clip(const LevelView& L, float du_max, bool chained, cudaStream_t st) {
  return chained ? launch_chained(k_clip<true>, L, true, st, L, du_max)
                 : launch_chained(k_clip<false>, L, false, st, L, du_max);
}
cudaError_t launch_tensor_abc(const LevelView& L, float* dst, cudaStream_t st) {
  FS_STORAGE_SWITCH(L.st, (k_tensor_abc<S><<<grid_of(L.W, L.H), kBlk, 0, st>>>(L, dst)))
}
cudaError_t launch_pack_s(const SPlane& src, int storage, float* dst, int W, int H, int P,
                          cudaStream_t st) {
  FS_STORAGE_SWITCH(storage, (k_pack_s<S><<<grid_of(W, H), kBlk, 0, st>>>(src, dst, W, H, P)))
}
cudaError_t launch_unpack_s(const float* src, const SPlane& dst, int storage, int W, int H,
                            int P, cudaStream_t st) {
  FS_STORAGE_SWITCH(storage, (k_unpack_s<S><<<grid_of(W, H), kBlk, 0, st>>>(src, dst, W, H, P)))
}

}  // namespace fs
