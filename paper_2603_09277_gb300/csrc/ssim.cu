// ssim.cu -- the D-SSIM term of L_base (Sec. 3 Eq. base): D-SSIM = 1 - SSIM
// with an 11x11 Gaussian window (sigma 1.5, normalised), zero padding outside
// the image, C1 = 0.01^2, C2 = 0.03^2, SSIM = mean over the view's pixels and
// channels (the 3DGS reading; the paper does not define the term).
//
// Forward, one CTA per 32x32 block of output pixels of one view, one channel
// after the other: the block and its 5-pixel halo of image and target are
// staged in shared memory as pairs (x, y).  The window moments are taken about
// a constant per 16x16 quarter of the block and channel (the staged value at the
// quarter's centre, c): with d = s - c (padding samples s = 0), mu = c + E[d] and
// sigma^2 = E[d^2] - E[d]^2 hold exactly for any constant, and around a value of
// the quarter two large FP32 sums do not cancel in smooth regions.  Because c is
// constant over a quarter, the 11x11 window sums are separable: a horizontal pass
// over the 26 staged rows of each row of quarters and a vertical pass per output
// pixel.  Per pixel and channel the forward saves (mu_x, mu_y, dS/dmu_x,
// dS/dsigma_x^2, dS/dsigma_xy) (planar, one plane per quantity) and adds
// lambda (1 - S) / (3 M_v V) to the loss partials: a warp sums, in FP32, the 16
// columns and 8 rows of one quarter that it holds, everything above in FP64, so
// the loss does not depend on how blocks and channels are dealt to CTAs.
//
// Backward, blocks of 32x32 with one constant per block and channel:
//   dL/dx(p) -= lambda / (3 M_v V) sum_q G(q - p) [a(q)
//               + 2 (x(p) - mu_x(q)) b(q) + (y(p) - mu_y(q)) e(q)]
// over the window centres q inside the image, with a = dS/dmu_x, b =
// dS/dsigma_x^2, e = dS/dsigma_xy (dsigma_x^2(q)/dx(p) = 2 G(q-p)(x(p) -
// mu_x(q)) because the window weights sum to 1).  With the block constants c, c'
// of image and target the bracket splits into three separable correlations:
//   G*(a - 2 (mu_x - c) b - (mu_y - c') e) + 2 (x(p) - c) G*b + (y(p) - c') G*e.
// On smooth images the parts cancel the more the farther a pixel's values lie from
// the constants, so these are the values at the middle of the block's pixels.  Error
// of the gradient against 64 bits (FP32 restatement; a ramp / a sinusoid whose target
// differs by 1e-2): 1.9e-5 / 5.3e-5; with the first pixel's values 4.8e-5 / 6.5e-5;
// five correlations over 16x16 blocks about their first pixel 3.3e-5 / 7.8e-5.
//
// What bounds them: instruction issue (the window sums; about 60 FP32
// operations per pixel, channel and moment; 61 and 54 % issue active on a 1237x822
// view) and the latency of the staging loads.  Blocks of 32 instead of 16 pixels
// cut the halo rows of the backward's horizontal pass from 1.6 to 1.3 per output
// row and what both stage from 2.6 to 1.7 samples per pixel, one channel at a
// time keeps the shared memory of a CTA at 38 to 48 KB (4 to 5 CTAs per SM; three
// channels of 16x16 blocks took 67 KB in the backward, 33 % issue active), packed
// FP32 pairs halve the instructions of paired quantities, and the backward runs
// three correlations where it ran five.  The whole loss on two 1237x822 views: 204
// us against 315 with 16x16 blocks of three channels, 1920x1080: 202 against 317.
// (One constant per 32x32 block in the forward too is 3 % faster, but its moments
// about a farther constant move the loss of a small image by 1e-8.)
#include <cmath>

#include "gs_internal.cuh"

namespace gs {
namespace {

constexpr int kSsimR = 5;                   // window radius
constexpr int kSsimTaps = 2 * kSsimR + 1;
constexpr int kSsimB = 32;                  // output block side
constexpr int kSsimS = kSsimB + 2 * kSsimR; // staged side (42)
constexpr int kSsimP = 44;                  // staged row pitch (16-byte rows of 4 samples)
constexpr int kQ = 16;                      // side of the forward's quarters
constexpr int kQS = kQ + 2 * kSsimR;        // staged rows of a quarter (26)
constexpr int kSsimThreads = 256;
constexpr int kSsimSplitBlocks = 2 * 4 * 152;  // see ssim_parts
constexpr float kC1 = 0.01f * 0.01f;
constexpr float kC2 = 0.03f * 0.03f;

struct SsimViews {
  int V;
  long long pix_off[GS_MAX_VIEWS];
  int W[GS_MAX_VIEWS], H[GS_MAX_VIEWS], BX[GS_MAX_VIEWS];
  int block_off[GS_MAX_VIEWS + 1];
  float scale[GS_MAX_VIEWS];  // lambda / (3 M_v V)
  float2 win[kSsimTaps];      // normalised 1D Gaussian, sigma 1.5, each weight twice
};

__device__ __forceinline__ int view_of_block(const SsimViews& sv, int b) {
  int v = 0;
  while (v + 1 < sv.V && b >= sv.block_off[v + 1]) ++v;
  return v;
}

// Both passes of the separable window are register-blocked: a thread takes
// kRun consecutive outputs along the pass direction and reads the kRun + 10
// samples they share from shared memory once; each output's 11 taps are summed
// in tap order.
constexpr int kRun = 4;                              // outputs per thread and pass
constexpr int kSpan = kRun + 2 * kSsimR;             // samples per run (14)
constexpr int kHItems = kSsimS * (kSsimB / kRun);    // the backward's horizontal runs (336)
constexpr int kQItems = 2 * kQS * (kSsimB / kRun);   // the forward's (416)
constexpr int kXP = 36;                              // pitch of s_x: two rows of 16 columns
                                                     // four rows apart, no bank conflict
static_assert(kSsimB * (kSsimB / kRun) == kSsimThreads, "one vertical run per thread");
static_assert(kSsimB == 32, "a warp is a row of the block in the vertical pass");

// Sum of a warp's FP32 terms (every term is >= 0).
__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The block of CTA b: its view, origin, extents and first pixel.
struct SsimBlock {
  int v, W, H, bx, by;
  long long base;
};
__device__ __forceinline__ SsimBlock ssim_block(const SsimViews& sv, int b) {
  SsimBlock k;
  k.v = view_of_block(sv, b);
  const int lb = b - sv.block_off[k.v];
  k.W = sv.W[k.v];
  k.H = sv.H[k.v];
  k.bx = (lb % sv.BX[k.v]) * kSsimB;
  k.by = (lb / sv.BX[k.v]) * kSsimB;
  k.base = sv.pix_off[k.v];
  return k;
}

// The channels of a CTA: all three, or one where the grid has three CTAs per
// block (launch_ssim says when).
struct ChannelRange {
  int first, end;
};
__device__ __forceinline__ ChannelRange channels_of(unsigned parts, unsigned part) {
  return parts == 1 ? ChannelRange{0, 3} : ChannelRange{(int)part, (int)part + 1};
}

__global__ void __launch_bounds__(kSsimThreads, 4) ssim_fwd_kernel(
    const float* image, const float* target, const SsimViews sv,
    float* maps /* 15 planes of P */, long long P, double* partials) {
  behind_previous();
  __shared__ __align__(16) float2 s_xy[kSsimS][kSsimP];
  __shared__ __align__(16) float2 s_m[2 * kQS][kSsimB];  // horizontal sums of (x, y)
  __shared__ __align__(16) float2 s_q[2 * kQS][kSsimB];  // of (x^2, y^2)
  __shared__ __align__(16) float s_x[2 * kQS][kXP];      // of x y
  __shared__ double s_sum[kSsimThreads / 32];
  const SsimBlock k = ssim_block(sv, blockIdx.x);
  // a warp's outputs: 16 columns and two runs of 4 rows of quarter (qx, qy)
  const int warp = threadIdx.x >> 5, qx = (warp >> 1) & 1, qy = warp >> 2;
  const int col = qx * kQ + (threadIdx.x & 15);
  const int y0 = (2 * (warp & 1) + ((threadIdx.x >> 4) & 1)) * kRun;  // in the quarter
  const ChannelRange cr = channels_of(gridDim.y, blockIdx.y);
  double sum = 0.0;
#pragma unroll 1
  for (int ch = cr.first; ch < cr.end; ++ch) {
    for (int i = threadIdx.x; i < kSsimS * kSsimS; i += kSsimThreads) {
      const int r = i / kSsimS, c = i - r * kSsimS;
      const int yy = k.by - kSsimR + r, xx = k.bx - kSsimR + c;
      const bool in = xx >= 0 && xx < k.W && yy >= 0 && yy < k.H;
      const long long p = 3 * (k.base + (long long)yy * k.W + xx) + ch;
      s_xy[r][c] = in ? make_float2(image[p], target[p]) : make_float2(0.f, 0.f);
    }
    __syncthreads();
    // horizontal: run (row r of the row of quarters hq, columns x0 .. x0 + kRun - 1)
    for (int it = threadIdx.x; it < kQItems; it += kSsimThreads) {
      const int r = it / (kSsimB / kRun), x0 = (it % (kSsimB / kRun)) * kRun;
      const int hq = r >= kQS ? 1 : 0, sr = r - hq * (kQS - kQ);  // (its staged row)
      const float2 c =
          s_xy[kSsimR + hq * kQ + kQ / 2][kSsimR + (x0 & kQ) + kQ / 2];
      const float2 ncc = make_float2(-c.x, -c.y);
      float2 m[kRun], q[kRun];
      float x[kRun];
#pragma unroll
      for (int o = 0; o < kRun; ++o) {
        m[o] = q[o] = make_float2(0.f, 0.f);
        x[o] = 0.f;
      }
#pragma unroll
      for (int j = 0; j < kSpan; j += 2) {
        const float4 t = *reinterpret_cast<const float4*>(&s_xy[sr][x0 + j]);
        const float2 d[2] = {__fadd2_rn(make_float2(t.x, t.y), ncc),
                             __fadd2_rn(make_float2(t.z, t.w), ncc)};
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int o = 0; o < kRun; ++o) {
            const int tap = j + h - o;
            if (tap < 0 || tap >= kSsimTaps) continue;
            const float2 w = __fmul2_rn(sv.win[tap], d[h]);
            m[o] = __fadd2_rn(m[o], w);
            q[o] = __ffma2_rn(w, d[h], q[o]);
            x[o] = __fmaf_rn(w.x, d[h].y, x[o]);
          }
      }
      float4* pm = reinterpret_cast<float4*>(&s_m[r][x0]);
      float4* pq = reinterpret_cast<float4*>(&s_q[r][x0]);
      pm[0] = make_float4(m[0].x, m[0].y, m[1].x, m[1].y);
      pm[1] = make_float4(m[2].x, m[2].y, m[3].x, m[3].y);
      pq[0] = make_float4(q[0].x, q[0].y, q[1].x, q[1].y);
      pq[1] = make_float4(q[2].x, q[2].y, q[3].x, q[3].y);
      *reinterpret_cast<float4*>(&s_x[r][x0]) = make_float4(x[0], x[1], x[2], x[3]);
    }
    __syncthreads();
    // vertical: column col, output rows y0 .. y0 + kRun - 1 of the quarter
    const float2 cc = s_xy[kSsimR + qy * kQ + kQ / 2][kSsimR + qx * kQ + kQ / 2];
    const int r0 = qy * kQS + y0;
    float acc = 0.f;
    float2 m[kRun], q[kRun];
    float x[kRun];
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
      m[o] = q[o] = make_float2(0.f, 0.f);
      x[o] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < kSpan; ++j) {
      const float2 tm = s_m[r0 + j][col], tq = s_q[r0 + j][col];
      const float tx = s_x[r0 + j][col];
#pragma unroll
      for (int o = 0; o < kRun; ++o) {
        const int tap = j - o;
        if (tap < 0 || tap >= kSsimTaps) continue;
        m[o] = __ffma2_rn(sv.win[tap], tm, m[o]);
        q[o] = __ffma2_rn(sv.win[tap], tq, q[o]);
        x[o] = __fmaf_rn(sv.win[tap].x, tx, x[o]);
      }
    }
    const int px = k.bx + col;
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
      const int py = k.by + qy * kQ + y0 + o;
      if (px < k.W && py < k.H) {
        const long long p = k.base + (long long)py * k.W + px;
        const float m1 = m[o].x, n1 = m[o].y;
        const float mx = cc.x + m1, my = cc.y + n1;
        const float sxx = __fmaf_rn(-m1, m1, q[o].x), syy = __fmaf_rn(-n1, n1, q[o].y);
        const float sxy = __fmaf_rn(-m1, n1, x[o]);
        const float A1 = 2.f * mx * my + kC1, A2 = 2.f * sxy + kC2;
        const float B1 = mx * mx + my * my + kC1, B2 = sxx + syy + kC2;
        const float D = B1 * B2;
        const float S = A1 * A2 / D;
        acc += 1.f - S;
        float* mp = maps + (long long)(5 * ch) * P + p;
        mp[0] = mx;
        mp[P] = my;
        mp[2 * P] = (2.f * my * A2 - S * 2.f * mx * B2) / D;  // dS/dmu_x, sigmas fixed
        mp[3 * P] = -S / B2;                                   // dS/dsigma_x^2
        mp[4 * P] = 2.f * A1 / D;                              // dS/dsigma_xy
      }
    }
    sum += (double)warp_sum(acc);
    __syncthreads();  // (the staged channel is overwritten)
  }
  if ((threadIdx.x & 31) == 0) s_sum[warp] = sum;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < kSsimThreads / 32; ++w) t += s_sum[w];
    partials[blockIdx.x + gridDim.x * blockIdx.y] = t * (double)sv.scale[k.v];
  }
}

__global__ void __launch_bounds__(kSsimThreads, 5) ssim_bwd_kernel(
    const float* image, const float* target, const SsimViews sv,
    const float* maps, long long P, float* dimg) {
  behind_previous();
  __shared__ __align__(16) float2 s_ab[kSsimS][kSsimP];  // (a - 2 (mu_x - c) b - (mu_y - c') e, b)
  __shared__ __align__(16) float s_e[kSsimS][kSsimP];
  __shared__ __align__(16) float2 s_hab[kSsimS][kSsimB];  // horizontal sums
  __shared__ __align__(16) float s_he[kSsimS][kSsimB];
  const SsimBlock k = ssim_block(sv, blockIdx.x);
  const int col = threadIdx.x & 31, y0 = (threadIdx.x >> 5) * kRun;
  const int cy0 = k.by + min(kSsimB, k.H - k.by) / 2, cx0 = k.bx + min(kSsimB, k.W - k.bx) / 2;
  const long long p0 = 3 * (k.base + (long long)cy0 * k.W + cx0);
  const ChannelRange cr = channels_of(gridDim.y, blockIdx.y);
#pragma unroll 1
  for (int ch = cr.first; ch < cr.end; ++ch) {
    // block constants: the image and target at the middle pixel (0 in place of one
    // that is not finite, which would spread over the whole block)
    const float ix = image[p0 + ch], iy = target[p0 + ch];
    const float cx = isfinite(ix) ? ix : 0.f, cy = isfinite(iy) ? iy : 0.f;
    const float* mp = maps + (long long)(5 * ch) * P;
    for (int i = threadIdx.x; i < kSsimS * kSsimS; i += kSsimThreads) {
      const int r = i / kSsimS, c = i - r * kSsimS;
      const int yy = k.by - kSsimR + r, xx = k.bx - kSsimR + c;
      float a = 0.f, b = 0.f, e = 0.f;
      if (xx >= 0 && xx < k.W && yy >= 0 && yy < k.H) {  // window centres in the image
        const long long q = k.base + (long long)yy * k.W + xx;
        const float mx = mp[q] - cx, my = mp[P + q] - cy;
        b = mp[3 * P + q];
        e = mp[4 * P + q];
        a = __fmaf_rn(-2.f * mx, b, __fmaf_rn(-my, e, mp[2 * P + q]));
      }
      s_ab[r][c] = make_float2(a, b);
      s_e[r][c] = e;
    }
    __syncthreads();
    for (int it = threadIdx.x; it < kHItems; it += kSsimThreads) {
      const int r = it / (kSsimB / kRun), x0 = (it % (kSsimB / kRun)) * kRun;
      float2 h[kRun];
      float g[kRun];
#pragma unroll
      for (int o = 0; o < kRun; ++o) {
        h[o] = make_float2(0.f, 0.f);
        g[o] = 0.f;
      }
#pragma unroll
      for (int j = 0; j < kSpan; j += 2) {
        const float4 t = *reinterpret_cast<const float4*>(&s_ab[r][x0 + j]);
        const float2 u = *reinterpret_cast<const float2*>(&s_e[r][x0 + j]);
        const float2 d[2] = {make_float2(t.x, t.y), make_float2(t.z, t.w)};
        const float f[2] = {u.x, u.y};
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int o = 0; o < kRun; ++o) {
            const int tap = j + i - o;
            if (tap < 0 || tap >= kSsimTaps) continue;
            h[o] = __ffma2_rn(sv.win[tap], d[i], h[o]);
            g[o] = __fmaf_rn(sv.win[tap].x, f[i], g[o]);
          }
      }
      float4* ph = reinterpret_cast<float4*>(&s_hab[r][x0]);
      ph[0] = make_float4(h[0].x, h[0].y, h[1].x, h[1].y);
      ph[1] = make_float4(h[2].x, h[2].y, h[3].x, h[3].y);
      *reinterpret_cast<float4*>(&s_he[r][x0]) = make_float4(g[0], g[1], g[2], g[3]);
    }
    __syncthreads();
    float2 h[kRun];
    float g[kRun];
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
      h[o] = make_float2(0.f, 0.f);
      g[o] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < kSpan; ++j) {
      const float2 t = s_hab[y0 + j][col];
      const float u = s_he[y0 + j][col];
#pragma unroll
      for (int o = 0; o < kRun; ++o) {
        const int tap = j - o;
        if (tap < 0 || tap >= kSsimTaps) continue;
        h[o] = __ffma2_rn(sv.win[tap], t, h[o]);
        g[o] = __fmaf_rn(sv.win[tap].x, u, g[o]);
      }
    }
    const int px = k.bx + col;
#pragma unroll
    for (int o = 0; o < kRun; ++o) {
      const int py = k.by + y0 + o;
      if (px < k.W && py < k.H) {
        const long long p = 3 * (k.base + (long long)py * k.W + px) + ch;
        const float grad = h[o].x + 2.f * (image[p] - cx) * h[o].y + (target[p] - cy) * g[o];
        dimg[p] -= sv.scale[k.v] * grad;
      }
    }
    __syncthreads();  // (the staged channel is overwritten)
  }
}

}  // namespace

size_t ssim_workspace_bytes(long long total_pixels) {
  return sizeof(float) * 15 * (size_t)total_pixels;
}

namespace {
// CTAs per block of pixels: three, one per channel, up to two waves of 4 CTAs on
// 152 SMs; beyond, one CTA for all three, which reads a pixel's channels from the
// same lines.  Measured (whole loss, three CTAs against one): 8 blocks 16.3
// against 32.8 us, 70 blocks 20.8 against 37.6, 260 blocks 36.8 against 45.3,
// 1,014 blocks 105.8 against 111.8, 2,028 blocks 218 against 205.
int ssim_parts(long long blocks) { return blocks <= kSsimSplitBlocks ? 3 : 1; }
}  // namespace

// The partials that launch_ssim writes.
int ssim_blocks(const CamTable& ct) {
  long long n = 0;
  for (int v = 0; v < ct.V; ++v)
    n += (long long)((ct.c[v].W + kSsimB - 1) / kSsimB) * ((ct.c[v].H + kSsimB - 1) / kSsimB);
  return (int)n * ssim_parts(n);
}

// Adds lambda (1 - SSIM_v) / V per view to the partials (ssim_blocks of them) and
// the term's gradient to dimg; maps is ssim_workspace_bytes(P) of scratch.
int launch_ssim(const float* image, const float* target, const CamTable& ct, float lambda,
                float* maps, double* partials, float* dimg, cudaStream_t st) {
  SsimViews sv;
  {
    double g[2 * kSsimR + 1], sum = 0.0;
    for (int k = -kSsimR; k <= kSsimR; ++k) {
      g[k + kSsimR] = exp(-(double)(k * k) / (2.0 * 1.5 * 1.5));
      sum += g[k + kSsimR];
    }
    for (int k = 0; k < kSsimTaps; ++k)
      sv.win[k] = make_float2((float)(g[k] / sum), (float)(g[k] / sum));
  }
  sv.V = ct.V;
  sv.block_off[0] = 0;
  for (int v = 0; v < ct.V; ++v) {
    const CamInfo& c = ct.c[v];
    sv.pix_off[v] = c.pix_off;
    sv.W[v] = c.W;
    sv.H[v] = c.H;
    sv.BX[v] = (c.W + kSsimB - 1) / kSsimB;
    sv.block_off[v + 1] = sv.block_off[v] + sv.BX[v] * ((c.H + kSsimB - 1) / kSsimB);
    sv.scale[v] = (float)((double)lambda / (3.0 * (double)c.W * c.H * ct.V));
  }
  const int nb = sv.block_off[ct.V];
  if (nb == 0) return GS_OK;
  const long long P = ct.c[ct.V - 1].pix_off + (long long)ct.c[ct.V - 1].W * ct.c[ct.V - 1].H;
  const dim3 grid(nb, ssim_parts(nb));
  launch_behind(ssim_fwd_kernel, dim3(grid), kSsimThreads, st, image, target, sv, maps, P,
                partials);
  launch_behind(ssim_bwd_kernel, dim3(grid), kSsimThreads, st, image, target, sv, maps, P, dimg);
  count_launches(2);
  return check_launch();
}

}  // namespace gs
