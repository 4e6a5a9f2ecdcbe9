// k_pho.cu -- photometric loss of Eq. 8 (L1 + D-SSIM) with the depth term of Eq. 9-10, fused
// with its gradient w.r.t. the rendered colour and depth images.
//
// Per view:  loss = (1 - lambda) sum|C - Cbar| / 3HW + lambda (1 - sum SSIM / 3HW)
//                   + lambda_dep sum_{Dbar > 0} |D - Dbar| / HW.
// SSIM (Wang et al. 2004) of one channel at pixel p uses the local statistics mu_x, mu_y,
// e_xx, e_yy, e_xy: sums of x, y, x^2, y^2, xy under the 11 x 11 Gaussian window (sigma 1.5,
// normalised) centred on p, with zeros outside the image; C1 = 0.01^2, C2 = 0.03^2.  Its gradient
// is dSSIM_sum/dx(q) = (G * m0)(q) + 2 x(q) (G * m1)(q) + y(q) (G * m2)(q), where m0, m1, m2 are
// the partials of SSIM(p) w.r.t. mu_x, e_xx and e_xy (zero outside the image) and G * the same
// symmetric window sum.
//
// SSIM and its partials need e_xx and e_yy only as their sum, and the differences B1 - A1 = (mu_x - mu_y)^2
// and B2 - A2 = e_dd - (mu_x - mu_y)^2, with e_dd the window's mean of (x - y)^2, without cancellation where
// the images agree: so four moments are filtered (mu_x, mu_y, e_dd, e_xy), not five.  dL/dC came closer to its
// 64-bit value (3.3e-6 -> 1.8e-6 of its largest for 20 views of 1200 x 680), equal images still give SSIM = 1,
// and 714 us became 668.  (Filtering x^2 + y^2 instead is as fast, but leaves rounding noise of the moments
// in the gradient of images that agree.)  In FP32 the covariance e_xy - mu_x mu_y, and with it A2 and B2, still
// loses digits where the window is nearly constant at a non-zero value; the error of dL/dC stays below ~1e-7 of
// the magnitude of its terms weighted by (moments) / (sigma_x^2 + sigma_y^2 + C2).  (A shift of the data by one
// constant per tile does not help: it moves the cancellation to flat regions at other values, such as the zeros
// of a clamped or black background.)
//
// One CTA owns a strip of 64 output columns and HS output rows of one channel of one view and walks down
// it 16 rows at a time.  x and y arrive as interleaved pairs (asynchronous copies two steps ahead) over
// the strip widened by 10 pixels (the window of a window).  Per step: the four moments along columns
// (of x, y and the products formed in registers), along rows, SSIM and m0..m2; m0..m2 along rows into a
// ring of 32 rows; along columns out of the ring, and dL/dC.  Walking down, only the strip's sides and
// ends recompute neighbours' values.  Every filter pass is register-blocked (R consecutive outputs
// along the filter direction from R + 10 loads), and quantities that share a weight are filtered as
// pairs with two-element FMAs (fma.rn.f32x2: (mu_x, mu_y), (e_dd, e_xy), (m0, m1)), which halves the
// instructions of a pass that is bound by issue.  A row pass takes two rows
// per warp, so its warps go from the moments to the filtered partials without a CTA barrier (two per
// step); five outputs per lane put the 16 lanes of a row on distinct banks.  Issue-bound (60 % issue active; FMA
// pipe half busy): 689 us for 20 views of 1200 x 680 where 32 x 32 tiles with scalar FMAs, each recomputing its
// halo on all sides, took 1259; 823 us for 64 views of 640 x 480 (1466).  (An approximate reciprocal and one
// Newton-Raphson step for 1 / (B1 B2) save 3 % and lose its values where it leaves the normal range.)
// Loss partial sums go to one slot per CTA and are reduced per view in a fixed order: the loss is
// deterministic.  dL/dC of a pixel does not depend on the strips' heights; the last bits of a view's loss do, and
// the heights follow from all of the plan's views.
#include <algorithm>
#include <cmath>

#include "ts_internal.cuh"

namespace {

constexpr int PT = 256;          // threads per CTA
constexpr int OW = 64;           // output columns of a strip
constexpr int RAD = 5;           // window radius
constexpr int NT = 2 * RAD + 1;  // taps
constexpr int RB = 16;           // rows per step
constexpr int IN = OW + 4 * RAD, IS = IN + 1;   // staged columns: 84, stride 85
constexpr int MO = OW + 2 * RAD, MS = MO + 1;   // moment columns: 74, stride 75
constexpr int OS = OW + 1;                      // row-filtered partials: 64, stride 65
constexpr int XY_ROWS = 4 * RB;  // staged rows: the two blocks a step reads, one arriving, one still read
constexpr int H_ROWS = 2 * RB;   // ring of row-filtered partials
constexpr int R_V1 = 8, R_H1 = 5, R_H2 = 5, R_V2 = 4;  // outputs per thread and pass
constexpr int V1_THREADS = (IN * (RB / R_V1) + 31) / 32 * 32;  // six warps; the other two stage
static_assert(V1_THREADS < PT && RB == 2 * (PT / 32) && (MO + R_H1 - 1) / R_H1 <= 16 && (OW + R_H2 - 1) / R_H2 <= 16 &&
                  OW * (RB / R_V2) == PT && (MO + R_H1 - 1) / R_H1 * R_H1 + 2 * RAD <= IS &&
                  (OW + R_H2 - 1) / R_H2 * R_H2 + 2 * RAD <= MS,
              "one item per thread and pass; the row passes take two rows per warp, half a warp each");
// shared memory in floats: (x, y) pairs; moments along columns as two pairs and one value; (m0, m1) and
// m2; their row-filtered ring
constexpr int SM_XY = 0, SM_MU = SM_XY + 2 * XY_ROWS * IS, SM_EE = SM_MU + 2 * RB * IS,
              SM_MA = SM_EE + 2 * RB * IS, SM_MB = SM_MA + 2 * RB * MS, SM_HA = SM_MB + RB * MS,
              SM_HB = SM_HA + 2 * H_ROWS * OS, SM_FLOATS = SM_HB + H_ROWS * OS;
static_assert(SM_MA % 2 == 0 && SM_HA % 2 == 0, "pairs are 8-byte aligned");
constexpr size_t PHO_SMEM = (size_t)SM_FLOATS * 4;
static_assert(2 * (PHO_SMEM + 1024) <= 227 * 1024, "two CTAs per SM");

// Two floats in a 64-bit register, and the two-element operations on them (each element rounded as the
// scalar operation rounds it).
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

struct Taps {
  float w[RAD + 1];  // of the symmetric window: tap t weighs w[min(t, 10 - t)]
};

// 4-byte asynchronous global-to-shared copy; valid == false writes a zero and reads nothing.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(d), "l"(src), "r"(valid ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

// One of n warps issues its share of the copies of a block of RB staged rows, image rows gy0.. and columns
// gx0.. (zeros outside the image; rows from `rows` on are not needed).
__device__ __forceinline__ void stage_block(float* xy, const float* xc, const float* yc, int gx0, int gy0, int rows,
                                            int W, int H, int warp, int n) {
  const int lane = threadIdx.x & 31;
  for (int r = warp; r < min(rows, RB); r += n) {  // a row per warp: its place and validity are uniform
    const int gy = gy0 + r;
    const bool rowin = gy >= 0 && gy < H;
    const float* xr = xc + (rowin ? (long long)gy * W : 0);
    const float* yr = yc + (rowin ? (long long)gy * W : 0);
    float* d = xy + 2 * (r * IS + lane);
#pragma unroll
    for (int c0 = 0; c0 < IN; c0 += 32) {
      const int gx = gx0 + c0 + lane;
      if (c0 + 32 <= IN || c0 + lane < IN) {
        const bool in = rowin && gx >= 0 && gx < W;
        const int o = in ? gx : 0;
        cp_async4(d + 2 * c0, xr + o, in);
        cp_async4(d + 2 * c0 + 1, yr + o, in);
      }
    }
  }
  cp_async_commit();
}

// The weight of distance t along a window (both sides alike), or -1 outside it.
__host__ __device__ constexpr int tap(int t) { return t < 0 || t >= NT ? -1 : (t <= RAD ? t : NT - 1 - t); }

__device__ __forceinline__ float block_sum(float v, float* red) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  float s = 0.f;
#pragma unroll
  for (int i = 0; i < PT / 32; ++i) s += red[i];
  return s;
}

// blockIdx.x: (segment of HS rows, strip) of the view; blockIdx.y: view * 3 + channel.
__global__ void __launch_bounds__(PT, 2)
    k_pho_strip(const TsImageTable tab, const float* __restrict__ C, const float* __restrict__ D,
                const float* __restrict__ tC, const float* __restrict__ tD, float lambda, float lambda_dep, Taps tp,
                float* __restrict__ dC, float* __restrict__ dD, float* __restrict__ part, int nblk, int HS) {
  extern __shared__ __align__(16) float sm[];
  __shared__ float red[PT / 32];
  const int v = blockIdx.y / 3, ch = blockIdx.y - 3 * v;
  const int W = tab.W[v], H = tab.H[v];
  const long long pix_off = tab.pix_off[v];
  const int strips = (W + OW - 1) / OW;
  const int X0 = (blockIdx.x % strips) * OW, Y0 = (blockIdx.x / strips) * HS;
  if (Y0 >= H) return;  // uniform over the CTA
  const int rows = min(HS, H - Y0);
  const int steps = (rows + 2 * RAD + RB - 1) / RB;
  const long long HW = (long long)W * H;
  const float* xc = C + 3 * pix_off + ch * HW;
  const float* yc = tC + 3 * pix_off + ch * HW;
  const float inv3 = 1.0f / (3.0f * (float)HW), id = lambda_dep / (float)HW;
  const float C1 = 0.01f * 0.01f, C2 = 0.03f * 0.03f;
  f32x2* xy = reinterpret_cast<f32x2*>(sm + SM_XY);
  f32x2* vmu = reinterpret_cast<f32x2*>(sm + SM_MU);
  f32x2* vee = reinterpret_cast<f32x2*>(sm + SM_EE);
  f32x2* ma = reinterpret_cast<f32x2*>(sm + SM_MA);
  float* mb = sm + SM_MB;
  f32x2* ha = reinterpret_cast<f32x2*>(sm + SM_HA);
  float* hb = sm + SM_HB;
  f32x2 w2[RAD + 1];
#pragma unroll
  for (int t = 0; t <= RAD; ++t) w2[t] = pack2(tp.w[t], tp.w[t]);
  float l1 = 0.f, ss = 0.f, dep = 0.f;
  const int tid = threadIdx.x;

  // staged row q is image row Y0 - 10 + q, moment row i image row Y0 - 5 + i, output row o image row Y0 + o
  stage_block(sm + SM_XY, xc, yc, X0 - 2 * RAD, Y0 - 2 * RAD, rows + 4 * RAD, W, H, tid >> 5, PT / 32);
  stage_block(sm + SM_XY + 2 * RB * IS, xc, yc, X0 - 2 * RAD, Y0 - 2 * RAD + RB, rows + 4 * RAD - RB, W, H, tid >> 5,
              PT / 32);
  cp_async_wait<0>();
  __syncthreads();
  for (int s = 0; s < steps; ++s) {
    if (tid >= V1_THREADS) {
      // the block after next (its place was last read two steps ago), by the warps that have no columns
      stage_block(sm + SM_XY + 2 * ((s + 2) & 3) * RB * IS, xc, yc, X0 - 2 * RAD, Y0 - 2 * RAD + (s + 2) * RB,
                  rows + 4 * RAD - (s + 2) * RB, W, H, (tid - V1_THREADS) >> 5, (PT - V1_THREADS) / 32);
    } else if (tid < IN * (RB / R_V1)) {  // columns: moment rows RB s + 8 rg + j at staged column c
      const int rg = tid / IN, c = tid - rg * IN;
      f32x2 mu[R_V1], ee[R_V1];
#pragma unroll
      for (int k8 = 0; k8 < R_V1 + 2 * RAD; k8 += 8) {
        const f32x2* src = xy + ((s * RB + rg * R_V1 + k8) & (XY_ROWS - 1)) * IS + c;  // 8 rows without a wrap
#pragma unroll
        for (int k = k8; k < k8 + 8 && k < R_V1 + 2 * RAD; ++k) {
          const f32x2 q = src[(k - k8) * IS];
          float x, y;
          unpack2(q, x, y);
          const float d = x - y;
          const f32x2 qq = pack2(d * d, x * y);
#pragma unroll
          for (int j = 0; j < R_V1; ++j) {
            const int t = tap(k - j);
            if (t >= 0) {
              mu[j] = j == k ? mul2(w2[t], q) : fma2(w2[t], q, mu[j]);
              ee[j] = j == k ? mul2(w2[t], qq) : fma2(w2[t], qq, ee[j]);
            }
          }
        }
      }
#pragma unroll
      for (int j = 0; j < R_V1; ++j) {
        const int o = (rg * R_V1 + j) * IS + c;
        vmu[o] = mu[j];
        vee[o] = ee[j];
      }
    }
    __syncthreads();
    // rows: the moments of moment row i at columns cm, image (Y0 - 5 + i, X0 - 5 + cm), and the partials
    {
      const int r = tid >> 4, c0 = (tid & 15) * R_H1;
      if (c0 < MO) {
        f32x2 mu[R_H1], ee[R_H1];
#pragma unroll
        for (int k = 0; k < R_H1 + 2 * RAD; ++k) {
          const f32x2 a = vmu[r * IS + c0 + k], e = vee[r * IS + c0 + k];
#pragma unroll
          for (int j = 0; j < R_H1; ++j) {
            const int t = tap(k - j);
            if (t >= 0) {
              mu[j] = j == k ? mul2(w2[t], a) : fma2(w2[t], a, mu[j]);
              ee[j] = j == k ? mul2(w2[t], e) : fma2(w2[t], e, ee[j]);
            }
          }
        }
        const int i = s * RB + r, gy = Y0 - RAD + i;
        const bool rowin = gy >= 0 && gy < H, rowinner = i >= RAD && i < RAD + rows;
        const bool edge = X0 < RAD || X0 + OW + RAD > W || Y0 + s * RB < RAD || Y0 - RAD + (s + 1) * RB > H;  // uniform
#pragma unroll
        for (int j = 0; j < R_H1; ++j) {
          const int cm = c0 + j, gx = X0 - RAD + cm;
          float mx, my, edd, exy;
          unpack2(mu[j], mx, my);
          unpack2(ee[j], edd, exy);
          const float A1 = 2.f * mx * my + C1, A2 = 2.f * (exy - mx * my) + C2;
          const float dm = mx - my;
          const float B1 = fmaf(dm, dm, A1), B2 = A2 + fmaf(-dm, dm, edd);
          const float iB = 1.f / (B1 * B2);  // (0 where the product overflows: such a pixel's terms vanish)
          const float ssim = A1 * A2 * iB;
          // partials w.r.t. mu_x, e_xx and e_xy: zero outside the image
          float m0 = 2.f * (my * (A2 - A1) - mx * ssim * (B2 - B1)) * iB;
          float m1 = -ssim * B1 * iB;
          float m2 = 2.f * A1 * iB;
          const bool in = !edge || (rowin && gx >= 0 && gx < W);
          if (!in) m0 = m1 = m2 = 0.f;
          if (in && rowinner && cm >= RAD && cm < RAD + OW) ss += ssim;
          if (cm < MO) {
            ma[r * MS + cm] = pack2(m0, m1);
            mb[r * MS + cm] = m2;
          }
        }
      }
    }
    __syncwarp();  // the next pass reads the rows that this warp has just written
    // rows: partials of moment row i filtered to output columns co
    if ((tid & 15) * R_H2 < OW) {
      const int r = tid >> 4, c0 = (tid & 15) * R_H2;
      f32x2 g01[R_H2];
      float g2[R_H2];
#pragma unroll
      for (int k = 0; k < R_H2 + 2 * RAD; ++k) {
        const f32x2 a = ma[r * MS + c0 + k];
        const float b = mb[r * MS + c0 + k];
#pragma unroll
        for (int j = 0; j < R_H2; ++j) {
          const int t = tap(k - j);
          if (t >= 0) {
            g01[j] = j == k ? mul2(w2[t], a) : fma2(w2[t], a, g01[j]);
            g2[j] = j == k ? tp.w[t] * b : fmaf(tp.w[t], b, g2[j]);
          }
        }
      }
      const int o = ((s * RB + r) & (H_ROWS - 1)) * OS + c0;
#pragma unroll
      for (int j = 0; j < R_H2; ++j) {
        if (c0 + j < OW) {
          ha[o + j] = g01[j];
          hb[o + j] = g2[j];
        }
      }
    }
    cp_async_wait<0>();  // the next step's second block, published by the barrier
    __syncthreads();
    // columns: output rows o, whose moment rows o .. o + 10 the ring now holds
    {
      const int co = tid & (OW - 1), o0 = s * RB - 2 * RAD + (tid / OW) * R_V2;
      if (o0 + R_V2 > 0 && o0 < rows) {
        f32x2 g01[R_V2];
        float g2[R_V2];
#pragma unroll
        for (int k = 0; k < R_V2 + 2 * RAD; ++k) {
          const int h = ((o0 + k) & (H_ROWS - 1)) * OS + co;
          const f32x2 a = ha[h];
          const float b = hb[h];
#pragma unroll
          for (int j = 0; j < R_V2; ++j) {
            const int t = tap(k - j);
            if (t >= 0) {
              g01[j] = j == k ? mul2(w2[t], a) : fma2(w2[t], a, g01[j]);
              g2[j] = j == k ? tp.w[t] * b : fmaf(tp.w[t], b, g2[j]);
            }
          }
        }
        const int gx = X0 + co;
        float* out = dC + 3 * pix_off + ch * HW + (long long)(Y0 + o0) * W + gx;
        // (o0 + 10 is a multiple of 4: four rows without a wrap)
        const f32x2* own = xy + ((o0 + 2 * RAD) & (XY_ROWS - 1)) * IS + co + 2 * RAD;
#pragma unroll
        for (int j = 0; j < R_V2; ++j) {
          const int o = o0 + j;
          if (o >= 0 && o < rows && gx < W) {
            float x, y, g0, g1;
            unpack2(own[j * IS], x, y);
            unpack2(g01[j], g0, g1);
            const float d = x - y;
            l1 += fabsf(d);
            const float sg = d > 0.f ? 1.f : (d < 0.f ? -1.f : 0.f);
            const float gs = g0 + 2.f * x * g1 + y * g2[j];
            out[(long long)j * W] = ((1.f - lambda) * sg - lambda * gs) * inv3;
          }
        }
      }
    }
  }
  // depth term of Eq. 9: a third of the rows per channel's CTA, four rows' loads in flight
  {
    const int gx = X0 + (tid & (OW - 1)), r1 = rows * (ch + 1) / 3;
    if (gx < W) {
      for (int r0 = rows * ch / 3 + tid / OW; r0 < r1; r0 += 4 * (PT / OW)) {
        const long long at = pix_off + (long long)(Y0 + r0) * W + gx;
        float t[4], e[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const bool in = r0 + k * (PT / OW) < r1;
          t[k] = in ? tD[at + (long long)k * (PT / OW) * W] : 0.f;
          e[k] = in ? D[at + (long long)k * (PT / OW) * W] : 0.f;
        }
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (r0 + k * (PT / OW) >= r1) break;
          const float d = e[k] - t[k];
          const bool valid = t[k] > 0.f;
          if (valid) dep += fabsf(d);
          dD[at + (long long)k * (PT / OW) * W] = valid ? (d > 0.f ? id : (d < 0.f ? -id : 0.f)) : 0.f;
        }
      }
    }
  }
  l1 = block_sum(l1, red);
  ss = block_sum(ss, red);
  dep = block_sum(dep, red);
  if (tid == 0) {
    float* o = part + ((long long)blockIdx.y * nblk + blockIdx.x) * 3;
    o[0] = l1;
    o[1] = ss;
    o[2] = dep;
  }
}

__global__ void __launch_bounds__(PT) k_pho_final(const TsImageTable tab, const float* __restrict__ part, int nblk,
                                                   int HS, float lambda, float lambda_dep,
                                                   float* __restrict__ loss) {
  __shared__ double red[PT][3];
  const int v = blockIdx.x;
  const int n = ((tab.W[v] + OW - 1) / OW) * ((tab.H[v] + HS - 1) / HS);  // CTAs per channel
  double a = 0, b = 0, c = 0;
  for (int k = threadIdx.x; k < 3 * n; k += PT) {
    const int ch = k / n;
    const float* o = part + ((long long)(3 * v + ch) * nblk + (k - ch * n)) * 3;
    a += o[0];
    b += o[1];
    c += o[2];
  }
  red[threadIdx.x][0] = a;
  red[threadIdx.x][1] = b;
  red[threadIdx.x][2] = c;
  __syncthreads();
  for (int o = PT / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o)
#pragma unroll
      for (int i = 0; i < 3; ++i) red[threadIdx.x][i] += red[threadIdx.x + o][i];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const double HW = (double)tab.W[v] * tab.H[v];
    loss[v] = (float)((1.0 - lambda) * red[0][0] / (3.0 * HW) + lambda * (1.0 - red[0][1] / (3.0 * HW)) +
                      (double)lambda_dep * red[0][2] / HW);
  }
}

Taps gaussian_taps() {
  double g[NT], s = 0;
  for (int k = 0; k < NT; ++k) s += (g[k] = std::exp(-(double)((k - RAD) * (k - RAD)) / (2.0 * 1.5 * 1.5)));
  Taps t;
  for (int k = 0; k <= RAD; ++k) t.w[k] = (float)(g[k] / s);
  return t;
}

// Output rows per strip, 16 k - 10 for k steps: long strips recompute less at their ends (k = 16: 4 %), but
// a small batch is cut into at least four waves of two CTAs on every SM, down to k = 2.
int strip_rows(const TsView* views, int V) {
  long long total = 0;  // rows of all strips and channels
  for (int v = 0; v < V; ++v) total += 3ll * ((views[v].W + OW - 1) / OW) * views[v].H;
  const long long k = (total / (8 * TS_SMS) + 2 * RAD + RB - 1) / RB;
  return RB * (int)std::max(2ll, std::min(16ll, k)) - 2 * RAD;
}

}  // namespace

// CTAs of the largest view, over its three channels.
int64_t ts_pho_blocks(const TsView* views, int V) {
  const int HS = strip_rows(views, V);
  int64_t n = 1;
  for (int v = 0; v < V; ++v)
    n = std::max<int64_t>(n, (int64_t)((views[v].W + OW - 1) / OW) * ((views[v].H + HS - 1) / HS));
  return 3 * n;
}

cudaError_t ts_launch_pho_loss(const TsPlanImpl* p, const TsWs& w, const float* color, const float* depth,
                               const float* tc, const float* td, float lambda, float lambda_dep, float* loss,
                               float* dC, float* dD, cudaStream_t s) {
  cudaError_t e = ts_smem_limit((const void*)k_pho_strip, (int)PHO_SMEM);
  if (e != cudaSuccess) return e;
  const int nblk = (int)(p->n_pho_blocks / 3), HS = strip_rows(p->views, p->V);
  const TsImageTable tab = ts_image_table(p);
  k_pho_strip<<<dim3((unsigned)nblk, (unsigned)p->V * 3u), PT, PHO_SMEM, s>>>(
      tab, color, depth, tc, td, lambda, lambda_dep, gaussian_taps(), dC, dD, w.pho, nblk, HS);
  k_pho_final<<<p->V, PT, 0, s>>>(tab, w.pho, nblk, HS, lambda, lambda_dep, loss);
  return cudaGetLastError();
}
