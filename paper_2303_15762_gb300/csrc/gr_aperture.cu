// Footprint-resolved generalized rays through an aperture (the paper's
// double-slit validation, Sec. 5.1-5.2, in a 2D world, and its extension to a
// plane aperture in a 3D world below): a detector element is
// a coherent state of width beta at the screen (Eq. wdf_coherent_states); each
// of its directions theta is a generalized ray propagated back to the aperture
// plane in closed form (Eq. K_free_space_propagation over the oblique length
// z / cos(theta)), truncated to the ball of radius rho_cut beta' (Sec. 6), and
// overlapped with the sampled aperture field; the element's intensity is
// int dkappa / (2 pi) |<U_ap, psi_kappa>|^2 with kappa = k sin(theta).
//
// One lane takes two neighbouring directions.  A block takes every n_split-th
// group of 2 kApertureThreads directions of one detector element, so that a
// screen of a few elements still fills the chip, and writes one partial sum;
// k_reduce adds an element's partial sums in block order, so the result does
// not depend on scheduling.
//
// What bounds it: the FP32 work of a (direction, sample) pair inside the
// truncation radius, ~20 operations on the FMA pipe beside an exponential, a
// sine and a cosine on the special-function unit.  The two directions of a
// lane ride in packed FP32 (fma.rn.f32x2: half the issue slots; each
// direction's sums keep their order and rounding), the rounding to whole turns
// is an addition of 1.5 * 2^23 instead of a conversion on the special-function
// unit, and samples are skipped 64 at a time when their interval or box lies
// outside the truncation radius of all 64 directions of a warp.  The terms of
// a direction are formed in FP64, of which the chip does 1/64 of the FP32
// rate: sine and cosine come from the previous direction's by rotation (at most
// kApertureRotations in a row), and reciprocals and square roots from an FP32
// seed and Newton steps, ~30 FP64 operations per direction instead of several
// hundred.
// Measured (kernel time, before -> after): double slit, 4001 elements x ~8900
// directions x 800 samples 12.74 -> 4.66 ms; 13 elements 1192 -> 73 us (13
// blocks before, 455 now); disk of 1152 samples, 400 elements x 61,009
// directions 30.9 -> 18.9 ms (FMA pipe 67% busy, issue slots 70%).  The second
// Newton steps cost 4.63 -> 4.64 ms there, and where FP64 weighs most, 5000
// elements x 445,000 directions x 4 samples, 129 -> 161 ms (547 with FP64
// divisions, roots and sines).  One
// direction per lane with two samples packed took 4.9 and 17.8 ms, but sums
// the samples in another order; sine and cosine as polynomials on the FMA pipe
// 6.3 and 22.2 ms.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "gr_build.h"

namespace gr {

namespace {

constexpr int kApertureThreads = 128;
constexpr int kApertureChunk = 64;  // samples with one bounding box
// blocks per SM the split of an element's directions aims at: several waves
// of the 5-7 resident blocks, so that the last, partly filled one is short
// (24 and 48 per SM: 5.28 and 5.06 ms on 4001 elements, but 208 and 261 us on
// 301 elements of half the samples and directions, where a block's start
// weighs more)
constexpr int kApertureBlocksPerSM = 32;

// groups of directions a lane walks by rotation: each adds up to an FP64
// rounding to sine and cosine, so an element of more directions takes more
// blocks (up to kApertureBlocks of them in all)
constexpr long long kApertureRotations = 256;
constexpr long long kApertureBlocks = 1 << 24;

// 2 pi split as hi + lo with hi the nearest float (Cody & Waite's additive
// range reduction): x - n (2 pi) is formed as (x - n hi) - n lo with one
// rounding per step, accurate to a few 1e-7 rad for |x| up to ~1e4.
constexpr float kTwoPiHi = 6.28318548202514648f;
constexpr float kTwoPiLo = -1.7484555314695172e-7f;
constexpr float kInvTwoPi = 0.159154943091895336f;
constexpr float kNegLog2e = -1.44269504088896340736f;
constexpr float kRound = 12582912.0f;  // 1.5 * 2^23: adding it rounds to an integer (|x| < 2^22)

// Hardware approximations with subnormal results and arguments as zero.  The
// exponential without .ftz spends three more instructions on results below
// 2^-126, which lie beyond sqrt(2 ln 2^126) = 13.2 widths: a truncation radius
// beyond kFlushRadius takes it (FAR, which also masks phases; 1001 elements x
// ~8900 directions x 800 samples, every sample inside: 4.26 -> 5.07 ms).
constexpr double kFlushRadius = 13.0;
template <bool FAR>
__device__ __forceinline__ float ex2_approx(float x) {
  float r;
  if (FAR) asm("ex2.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  else asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float sin_ftz(float x) {
  float r;
  asm("sin.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float cos_ftz(float x) {
  float r;
  asm("cos.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Adds w e^-u2 cis(phase) of one sample to the sums of two directions; `in`:
// the sample lies inside that direction's truncation radius.  The phase is
// reduced to [-pi, pi], where the hardware sine and cosine have an absolute
// error of ~1e-6, below the ~6e-5 rad to which the FP32 phase is known.  FAR:
// the phase of a sample outside the radius may be infinite or not a number,
// and must not reach the sums through 0 x NaN.
template <bool FAR>
__device__ __forceinline__ void add_sample(float w, f32x2 u2, f32x2 phase, bool in0, bool in1, f32x2& re, f32x2& im) {
  const f32x2 mag = add2(mul2(phase, dup2(kInvTwoPi)), dup2(kRound));
  const f32x2 neg_n = fma2(mag, dup2(-1.0f), dup2(kRound));
  const f32x2 r = fma2(neg_n, dup2(kTwoPiLo), fma2(neg_n, dup2(kTwoPiHi), phase));
  float e0, e1, r0, r1;
  unpack2(mul2(u2, dup2(kNegLog2e)), e0, e1);
  unpack2(r, r0, r1);
  if (FAR) {
    r0 = in0 ? r0 : 0.0f;
    r1 = in1 ? r1 : 0.0f;
  }
  const f32x2 g = pack2(in0 ? w * ex2_approx<FAR>(e0) : 0.0f, in1 ? w * ex2_approx<FAR>(e1) : 0.0f);
  re = fma2(g, pack2(cos_ftz(r0), cos_ftz(r1)), re);
  im = fma2(g, pack2(sin_ftz(r0), sin_ftz(r1)), im);
}

// 1 / a and 1 / sqrt(a) of a positive normal a: FP32 seed, one Newton step in
// FP64 (relative error ~1e-14, for what is rounded to FP32 next), and a second
// one to FP64's own accuracy (for the FP64 weights).
__device__ __forceinline__ double rcp_step(double a, double r) { return fma(r, fma(-a, r, 1.0), r); }
__device__ __forceinline__ double rsqrt_step(double a, double r) { return fma(0.5 * r, fma(-a * r, r, 1.0), r); }
__device__ __forceinline__ double rcp_d(double a) { return rcp_step(a, (double)__frcp_rn((float)a)); }
__device__ __forceinline__ double rsqrt_d(double a) { return rsqrt_step(a, (double)__frsqrt_rn((float)a)); }

// Block sum in a fixed order (warp shuffles, then the warps in turn).
__device__ __forceinline__ void block_partial(double acc, double* out) {
  __shared__ double s_red[kApertureThreads / 32];
  for (int off = 16; off > 0; off >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, off);
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kApertureThreads / 32; ++w) t += s_red[w];
    *out = t;
  }
}

// Distance from x to the interval [lo, hi].
__device__ __forceinline__ float gap(float x, float lo, float hi) { return fmaxf(fmaxf(lo - x, x - hi), 0.0f); }
// slack of the skip tests against FP32 rounding
constexpr float kSkipSlack = 0.9999f;

// Aperture samples in shared memory as (x, w); then the interval of each
// chunk and the interval of all samples.  rot1, rot: cosine and sine of the
// step to the lane's second direction and to its next pair.
template <bool FAR>
__global__ void __launch_bounds__(kApertureThreads, 7)
    k_aperture_backward(int n_split, const double* __restrict__ x0s, int n_ap, const float2* __restrict__ ap,
                        double beta, double z, double k, double reach, double dtheta, double rho_cut, double2 rot1,
                        double2 rot, double* __restrict__ part) {
  extern __shared__ float2 s_ap[];
  __shared__ double s_th[2];
  const int n_chunk = (n_ap + kApertureChunk - 1) / kApertureChunk;
  for (int i = threadIdx.x; i < n_ap + n_chunk + 1; i += blockDim.x) s_ap[i] = ap[i];
  const float2* s_box = s_ap + n_ap;
  const int det = blockIdx.x / n_split, split = blockIdx.x - det * n_split;
  const int stride = 2 * kApertureThreads * n_split;
  const double x0 = x0s[det];
  // two warps, one bound each: an FP64 arc tangent takes microseconds
  if (threadIdx.x == 0) s_th[0] = atan((x0 - reach) / z);
  if (threadIdx.x == 32) s_th[1] = atan((x0 + reach) / z);
  __syncthreads();
  const double th_lo = s_th[0];
  const long long n_th = (long long)ceil((s_th[1] - th_lo) / dtheta);
  const double pi = 3.14159265358979323846;
  const double beta2 = beta * beta, ib = 1.0 / beta2, zk = z / k;
  const double wk = k * dtheta / sqrt(pi);
  const float2 all = s_box[n_chunk];
  double acc = 0.0, sn = 0.0, c = 1.0;
  long long i = 2 * ((long long)split * kApertureThreads + threadIdx.x);
  long long iw = i - 2 * (threadIdx.x & 31);
  if (iw < n_th) sincos(th_lo + (double)i * dtheta, &sn, &c);
  // whole warps walk together: directions past the last one take part in the
  // votes with nothing to add
  for (; iw < n_th; iw += stride, i += stride) {
    float kap[2], cf[2], xcf[2], inv2b2[2], nrho[2], cut[2];
    double wgt[2];
    bool out[2];
    double s1 = sn, c1 = c;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const double r = rcp_step(c1, rcp_d(c1));
      const double t = zk * r;               // oblique path length over |k|
      const double rho = t * ib;             // Eq. K_free_space_propagation from rho = 0
      const double b2 = fma(rho, t, beta2);
      const double y = rsqrt_d(b2);
      kap[j] = (float)(k * s1);
      cf[j] = (float)c1;
      xcf[j] = (float)fma(-z, s1 * r, x0);   // where the ray meets the aperture plane
      inv2b2[j] = (float)(0.5 * y * y);
      nrho[j] = -(float)rho;
      cut[j] = (float)(rho_cut * (b2 * y));
      wgt[j] = c1 * c1 * wk * rsqrt_step(b2, y);  // cos(theta) (pi b'^2)^(-1/2) dkappa
      out[j] = i + j >= n_th || kSkipSlack * cf[j] * gap(xcf[j], all.x, all.y) > cut[j];
      if (j == 0) {
        s1 = fma(sn, rot1.x, c * rot1.y);
        c1 = fma(c, rot1.x, -(sn * rot1.y));
      }
    }
    s1 = sn;  // the lane's next directions: a rotation by stride * dtheta
    sn = fma(s1, rot.x, c * rot.y);
    c = fma(c, rot.x, -(s1 * rot.y));
    if (__all_sync(0xffffffffu, out[0] && out[1])) continue;
    const f32x2 kap2 = pack2(kap[0], kap[1]), cf2 = pack2(cf[0], cf[1]), inv2 = pack2(inv2b2[0], inv2b2[1]);
    const f32x2 nrho2 = pack2(nrho[0], nrho[1]);
    f32x2 re = 0ull, im = 0ull;
    for (int ch = 0; ch < n_chunk; ++ch) {
      const float2 bx = s_box[ch];
      if (__all_sync(0xffffffffu, (out[0] || kSkipSlack * cf[0] * gap(xcf[0], bx.x, bx.y) > cut[0]) &&
                                      (out[1] || kSkipSlack * cf[1] * gap(xcf[1], bx.x, bx.y) > cut[1])))
        continue;
      const int q1 = min((ch + 1) * kApertureChunk, n_ap);
#pragma unroll 4
      for (int q = ch * kApertureChunk; q < q1; ++q) {
        const float2 v = s_ap[q];
        const f32x2 dx = pack2(v.x - xcf[0], v.x - xcf[1]);
        const f32x2 u = mul2(dx, cf2);
        float u0, u1;
        unpack2(u, u0, u1);
        const f32x2 u2 = mul2(mul2(u, u), inv2);
        add_sample<FAR>(v.y, u2, fma2(kap2, dx, mul2(nrho2, u2)), !(fabsf(u0) > cut[0]), !(fabsf(u1) > cut[1]), re, im);
      }
    }
    float r[2], m[2];
    unpack2(re, r[0], r[1]);
    unpack2(im, m[0], m[1]);
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (i + j < n_th) acc = fma(fma((double)r[j], r[j], (double)m[j] * m[j]), wgt[j], acc);
  }
  block_partial(acc, part + blockIdx.x);
}

// The same computation for a plane aperture in a 3D world: a detector element
// at (x0, y0) on the screen, directions on the tangent-plane grid t = (s_x,
// s_y) / s_z (landing points x_c = x0 - z t, one grid step apart), each a
// generalized ray propagated back over z / s_z in closed form, its footprint
// projected obliquely onto the aperture plane (|P d|^2 = |d|^2 - s_z^2 (t.d)^2)
// and truncated at rho_cut beta'; the element's intensity is
// sum_t |A|^2 s_z / (pi beta'^2) k^2 s_z^4 dt^2 / (2 pi)^2.  Aperture samples
// are (x, y, weight, 0) in shared memory, then the chunks' boxes (x lo, x hi,
// y lo, y hi) and the box of all samples.
template <bool FAR>
__global__ void __launch_bounds__(kApertureThreads, 5)
    k_aperture_backward_3d(int n_split, const double2* __restrict__ x0s, int n_ap, const float4* __restrict__ ap,
                           double beta, double z, double k, double reach, double dt, double rho_cut, int n_t,
                           double* __restrict__ part) {
  extern __shared__ float4 s_ap4[];
  const int n_chunk = (n_ap + kApertureChunk - 1) / kApertureChunk;
  for (int i = threadIdx.x; i < n_ap + n_chunk + 1; i += blockDim.x) s_ap4[i] = ap[i];
  __syncthreads();
  const float4* s_box = s_ap4 + n_ap;
  const int det = blockIdx.x / n_split, split = blockIdx.x - det * n_split;
  const int stride = 2 * kApertureThreads * n_split;
  const double pi = 3.14159265358979323846;
  const double2 x0 = x0s[det];
  const double tx0 = (x0.x - reach) / z, ty0 = (x0.y - reach) / z;
  const double beta2 = beta * beta, ib = 1.0 / beta2, zk = z / k, Q = zk * zk * ib;
  const double wk = k * k * dt * dt / pi, rc2 = rho_cut * rho_cut;
  const float4 all = s_box[n_chunk];
  double acc = 0.0;
  const int n_dir = n_t * n_t;
  int i = 2 * (split * kApertureThreads + (int)threadIdx.x);
  for (int iw = i - 2 * (threadIdx.x & 31); iw < n_dir; iw += stride, i += stride) {
    float cx[2], cy[2], kx[2], ky[2], txf[2], tyf[2], nsz2[2], inv2b2[2], nrho[2], cut2[2], gz[2];
    double wgt[2];
    bool out[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int ix = (i + j) / n_t, iy = (i + j) - ix * n_t;
      const double tx = tx0 + (double)ix * dt, ty = ty0 + (double)iy * dt;
      const double q2 = fma(tx, tx, fma(ty, ty, 1.0));  // 1 / s_z^2
      const double sz = rsqrt_d(q2), s2 = sz * sz;
      const double b2 = fma(Q, q2, beta2);              // Eq. K_free_space_propagation from rho = 0
      const double ib2 = rcp_d(b2);
      cx[j] = (float)fma(-z, tx, x0.x);
      cy[j] = (float)fma(-z, ty, x0.y);
      kx[j] = (float)(k * sz * tx);
      ky[j] = (float)(k * sz * ty);
      txf[j] = (float)tx;
      tyf[j] = (float)ty;
      nsz2[j] = -(float)s2;
      inv2b2[j] = (float)(0.5 * ib2);
      nrho[j] = -(float)(zk * ib * q2 * sz);
      cut2[j] = (float)(rc2 * b2);
      const double szw = rsqrt_step(q2, sz), szw2 = szw * szw;
      wgt[j] = szw2 * szw2 * szw * rcp_step(b2, ib2) * wk;
      gz[j] = kSkipSlack * -nsz2[j];  // |P d|^2 >= s_z^2 |d|^2
      const float hx = gap(cx[j], all.x, all.y), hy = gap(cy[j], all.z, all.w);
      out[j] = i + j >= n_dir || gz[j] * fmaf(hx, hx, hy * hy) > cut2[j];
    }
    if (__all_sync(0xffffffffu, out[0] && out[1])) continue;
    const f32x2 kx2 = pack2(kx[0], kx[1]), ky2 = pack2(ky[0], ky[1]), tx2 = pack2(txf[0], txf[1]);
    const f32x2 ty2 = pack2(tyf[0], tyf[1]), ns2 = pack2(nsz2[0], nsz2[1]), inv2 = pack2(inv2b2[0], inv2b2[1]);
    const f32x2 nrho2 = pack2(nrho[0], nrho[1]);
    f32x2 re = 0ull, im = 0ull;
    for (int ch = 0; ch < n_chunk; ++ch) {
      const float4 bx = s_box[ch];
      const float hx0 = gap(cx[0], bx.x, bx.y), hy0 = gap(cy[0], bx.z, bx.w);
      const float hx1 = gap(cx[1], bx.x, bx.y), hy1 = gap(cy[1], bx.z, bx.w);
      if (__all_sync(0xffffffffu, (out[0] || gz[0] * fmaf(hx0, hx0, hy0 * hy0) > cut2[0]) &&
                                      (out[1] || gz[1] * fmaf(hx1, hx1, hy1 * hy1) > cut2[1])))
        continue;
      const int q1 = min((ch + 1) * kApertureChunk, n_ap);
#pragma unroll 4
      for (int q = ch * kApertureChunk; q < q1; ++q) {
        const float4 v = s_ap4[q];
        const f32x2 dx = pack2(v.x - cx[0], v.x - cx[1]), dy = pack2(v.y - cy[0], v.y - cy[1]);
        const f32x2 td = fma2(tx2, dx, mul2(ty2, dy));
        const f32x2 p2 = fma2(mul2(ns2, td), td, fma2(dx, dx, mul2(dy, dy)));
        float p0, p1;
        unpack2(p2, p0, p1);
        const f32x2 u2 = mul2(p2, inv2);
        add_sample<FAR>(v.z, u2, fma2(nrho2, u2, fma2(kx2, dx, mul2(ky2, dy))), !(p0 > cut2[0]), !(p1 > cut2[1]), re, im);
      }
    }
    float r[2], m[2];
    unpack2(re, r[0], r[1]);
    unpack2(im, m[0], m[1]);
#pragma unroll
    for (int j = 0; j < 2; ++j)
      if (i + j < n_dir) acc = fma(fma((double)r[j], r[j], (double)m[j] * m[j]), wgt[j], acc);
  }
  block_partial(acc, part + blockIdx.x);
}

// out[det] = scale * the sum of the element's partial sums in block order.
__global__ void k_reduce(int n_det, int n_split, const double* __restrict__ part, double scale,
                         double* __restrict__ out) {
  const int d = blockIdx.x * blockDim.x + threadIdx.x;
  if (d >= n_det) return;
  double t = 0.0;
  for (int s = 0; s < n_split; ++s) t += part[(size_t)d * n_split + s];
  out[d] = t * scale;
}

// Blocks per detector element of at most n_dir directions: as many as it takes
// to give the chip kApertureBlocksPerSM blocks per SM and a lane at most
// kApertureRotations groups of directions, each block the same number of them.
int split_of(long long n_det, double n_dir, int sms) {
  const long long groups = std::max(1LL, (long long)std::ceil(n_dir / (2 * kApertureThreads)));
  const long long fill = ((long long)kApertureBlocksPerSM * sms + n_det - 1) / n_det;
  const long long rotations = std::min((groups + kApertureRotations - 1) / kApertureRotations, kApertureBlocks / n_det);
  const long long want = std::min(groups, std::max(fill, rotations));
  const long long per = (groups + want - 1) / want;
  return (int)((groups + per - 1) / per);
}

// The samples' layout of the kernels: (x, w) or (x, y, w, 0), then the
// interval or box of every chunk, then that of all samples.  A sample that is
// not finite makes its boxes unbounded, so that it is never skipped.
std::vector<float> pack_samples(int dim, int n_ap, const double* xa, const double* wa) {
  const int n_chunk = (n_ap + kApertureChunk - 1) / kApertureChunk, f = 2 * dim;
  std::vector<float> v((size_t)f * (n_ap + n_chunk + 1), 0.0f);
  float* all = v.data() + (size_t)f * (n_ap + n_chunk);
  for (int a = 0; a < dim; ++a) {
    all[2 * a] = INFINITY;
    all[2 * a + 1] = -INFINITY;
  }
  for (int c = 0; c < n_chunk; ++c) {
    float* b = v.data() + (size_t)f * (n_ap + c);
    for (int a = 0; a < dim; ++a) {
      b[2 * a] = INFINITY;
      b[2 * a + 1] = -INFINITY;
    }
    bool finite = true;
    for (int i = c * kApertureChunk; i < std::min(n_ap, (c + 1) * kApertureChunk); ++i) {
      float* q = v.data() + (size_t)f * i;
      for (int a = 0; a < dim; ++a) {
        q[a] = (float)xa[(size_t)dim * i + a];
        finite = finite && std::isfinite(q[a]);
        b[2 * a] = std::min(b[2 * a], q[a]);
        b[2 * a + 1] = std::max(b[2 * a + 1], q[a]);
      }
      q[dim] = (float)wa[i];
      finite = finite && std::isfinite(q[dim]);
    }
    for (int a = 0; a < dim; ++a) {
      if (!finite) {
        b[2 * a] = -INFINITY;
        b[2 * a + 1] = INFINITY;
      }
      all[2 * a] = std::min(all[2 * a], b[2 * a]);
      all[2 * a + 1] = std::max(all[2 * a + 1], b[2 * a + 1]);
    }
  }
  return v;
}

// Both entry points: one device allocation for the centres, samples, partial
// sums and results; launch(grid, shared bytes, centres, samples, partials)
// starts the kernel.
template <class Launch>
cudaError_t run_aperture(int dim, const void* kernel, int n_det, const double* x0_host, int n_ap, const double* xa_host,
                         const double* wa_host, double n_dir, double scale, double* out_host, cudaStream_t st,
                         float* ms, Launch&& launch) {
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int n_split = split_of(n_det, n_dir, sms);
  const std::vector<float> h = pack_samples(dim, n_ap, xa_host, wa_host);
  const size_t smem = sizeof(float) * h.size(), b_x0 = sizeof(double) * dim * (size_t)n_det;
  const size_t o_ap = (b_x0 + 255) / 256 * 256, o_part = o_ap + (smem + 255) / 256 * 256;
  const size_t o_out = o_part + (sizeof(double) * (size_t)n_det * n_split + 255) / 256 * 256;
  unsigned char* d = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t e = dev_alloc((void**)&d, o_out + sizeof(double) * (size_t)n_det, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d, x0_host, b_x0, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(d + o_ap, h.data(), smem, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && ms) e = cudaEventCreate(&e0);
  if (e == cudaSuccess && ms) e = cudaEventCreate(&e1);
  if (e == cudaSuccess && smem > 48 * 1024)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) {
    if (ms) cudaEventRecord(e0, st);
    launch((unsigned)(n_det * n_split), n_split, smem, d, d + o_ap, (double*)(d + o_part));
    k_reduce<<<(n_det + 127) / 128, 128, 0, st>>>(n_det, n_split, (const double*)(d + o_part), scale,
                                                  (double*)(d + o_out));
    if (ms) cudaEventRecord(e1, st);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(out_host, d + o_out, sizeof(double) * (size_t)n_det, cudaMemcpyDeviceToHost, st);
  if (d) cudaFreeAsync(d, st);
  const cudaError_t es = cudaStreamSynchronize(st);  // the host arrays are pageable
  if (e == cudaSuccess) e = es;
  if (e == cudaSuccess && ms) e = cudaEventElapsedTime(ms, e0, e1);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  return e;
}

// Whether a sample's phase in some direction may not be finite, so that the
// kernels must mask it (FAR): D bounds the distance of
// a sample from a landing point per axis, tan2 the directions' squared tangent.
// The bounds are far above what the kernels form, and what is not a number
// fails them.
constexpr double kPhaseMax = 1e36;
bool phases_far(double D, double tan2, double beta, double z, double k) {
  const double ib = 1.0 / (beta * beta), q = 1.0 + tan2, d2 = 4.0 * D * D;
  return !(k * D < kPhaseMax && q * d2 < kPhaseMax && d2 * ib < kPhaseMax &&
           d2 * ib * (z / k) * ib * q < kPhaseMax);
}
// The largest magnitude of n values (infinity if one is not a number).
double max_abs(const double* v, size_t n) {
  double m = 0.0;
  for (size_t i = 0; i < n; ++i) m = std::fabs(v[i]) <= m ? m : v[i] == v[i] ? std::fabs(v[i]) : INFINITY;
  return m;
}

}  // namespace

cudaError_t aperture_backward_3d_impl(int n_det, const double* x0_host, int n_ap, const double* xa_host,
                                      const double* wa_host, double beta, double z, double k, double reach,
                                      double dt, double rho_cut, double* out_host, cudaStream_t st, float* ms) {
  const int n_t = (int)std::ceil(2.0 * reach / (z * dt));  // at most 2^13 (checked at the entry)
  const double pi = 3.14159265358979323846;
  const double t = (max_abs(x0_host, 2 * (size_t)n_det) + reach) / z;
  const bool far = rho_cut > kFlushRadius || phases_far(max_abs(xa_host, 2 * (size_t)n_ap) + reach, 2.0 * t * t, beta, z, k);
  const auto kernel = far ? k_aperture_backward_3d<true> : k_aperture_backward_3d<false>;
  return run_aperture(2, (const void*)kernel, n_det, x0_host, n_ap, xa_host, wa_host, (double)n_t * n_t,
                      1.0 / (4.0 * pi * pi), out_host, st, ms,
                      [&](unsigned grid, int n_split, size_t smem, const void* x0, const void* ap, double* part) {
                        kernel<<<grid, kApertureThreads, smem, st>>>(n_split, (const double2*)x0, n_ap, (const float4*)ap,
                                                                     beta, z, k, reach, dt, rho_cut, n_t, part);
                      });
}

cudaError_t aperture_backward_impl(int n_det, const double* x0_host, int n_ap, const double* xa_host,
                                   const double* wa_host, double beta, double z, double k, double reach,
                                   double dtheta, double rho_cut, double* out_host, cudaStream_t st, float* ms) {
  const double pi = 3.14159265358979323846;
  const double t = (max_abs(x0_host, (size_t)n_det) + reach) / z;
  const bool far = rho_cut > kFlushRadius || phases_far(max_abs(xa_host, (size_t)n_ap) + reach, t * t, beta, z, k);
  const auto kernel = far ? k_aperture_backward<true> : k_aperture_backward<false>;
  return run_aperture(1, (const void*)kernel, n_det, x0_host, n_ap, xa_host, wa_host,
                      2.0 * std::atan(reach / z) / dtheta + 1.0, 1.0 / (2.0 * pi), out_host, st, ms,
                      [&](unsigned grid, int n_split, size_t smem, const void* x0, const void* ap, double* part) {
                        const double step = 2.0 * kApertureThreads * n_split * dtheta;
                        kernel<<<grid, kApertureThreads, smem, st>>>(
                            n_split, (const double*)x0, n_ap, (const float2*)ap, beta, z, k, reach, dtheta, rho_cut,
                            make_double2(std::cos(dtheta), std::sin(dtheta)),
                            make_double2(std::cos(step), std::sin(step)), part);
                      });
}

}  // namespace gr
