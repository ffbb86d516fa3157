// Photometric loss with the structural term (Sec. 2, step 4: L = L_RGB + L_D-SSIM, read as
// L = (1 - lam) L1 + lam (1 - SSIM), lam = 0.2 in 3DGS practice) over the concatenated
// views of a batch, and its gradient with respect to the rendered images.
//
// SSIM per channel uses an 11 x 11 Gaussian window (sigma 1.5, weights w_i w_j) with zero
// padding, C1 = 0.01^2, C2 = 0.03^2; both terms are means over all pixels and channels.
// With the local means mx, my, E[x^2], E[y^2], E[xy] of the window,
//   S = (2 mx my + C1)(2 cov + C2) / ((mx^2 + my^2 + C1)(vx + vy + C2)).
// k_ssim_fwd computes S and its partial derivatives with respect to mx, E[x^2] and E[xy]
// per pixel; since every pixel's statistics are windowed sums of x, x^2 and x y, the
// gradient of sum S is  w * dS/dmx + 2 x (w * dS/dE[x^2]) + y (w * dS/dE[xy])  (the window
// is symmetric, so the adjoint of the windowed sum is itself), which k_ssim_bwd forms and
// adds to the L1 term.  Both kernels work on 32 x 32 output tiles with a 5-pixel halo in
// shared memory and separable passes.
//
// A plain two-pass filter is bound by shared-memory loads (one per tap and statistic, 84 per
// output in the forward), by the latency of staging its window load by load, and by its FP64
// sums (a 64th of the FP32 rate).  Here the window arrives by cp.async (zeros outside the
// image), a thread makes four outputs of a row and then four of a column, so that each staged
// value is loaded once for four, tap sums run in registers with two statistics to a packed
// instruction ((x, y) and (E[x^2], E[y^2]) sit side by side in shared memory for that), and
// the loss is summed in FP32 parts (Sum3) up to one FP64 add per CTA.  1920x1080x3: forward
// 128 -> 67 us, backward 102 -> 49 us (cold; with sums in two parts), the call 241 -> 128 us;
// the forward now issues on 79 % of the slots.
#include <cmath>
#include <cstring>

#include "common.cuh"

namespace splx {

namespace {

constexpr int kT = 32;                // output tile side
constexpr int kR = 5;                 // window radius
constexpr int kS = kT + 2 * kR;       // staged side (42)
constexpr int kH = kT + 2;            // row stride of the pairs' row sums (bank spread)
constexpr int kThreads = 256;         // four outputs of a column each
constexpr float kC1 = 0.01f * 0.01f, kC2 = 0.03f * 0.03f;

// Normalised 11-tap Gaussian, sigma 1.5 (weights computed once on the host).
__constant__ float c_w[2 * kR + 1];

// Work item = (view, channel, tile): decoded from the global block index.
struct SsimItem {
  int v, ch, x0, y0, W, H;
  int64_t base;  // offset of the channel plane in the concatenated images
};

__device__ __forceinline__ SsimItem decode(const LossImgs& L, int64_t blk) {
  SsimItem it;
  it.v = view_of(L.blk_off, L.V, blk);
  const int r = (int)(blk - L.blk_off[it.v]);
  it.W = L.W[it.v];
  it.H = L.H[it.v];
  const int tx = (it.W + kT - 1) / kT, ty = (it.H + kT - 1) / kT;
  const int per = tx * ty;
  it.ch = r / per;
  const int t = r - it.ch * per;
  it.x0 = t % tx * kT;
  it.y0 = t / tx * kT;
  it.base = 3 * L.pix_off[it.v] + (int64_t)it.ch * it.W * it.H;
  return it;
}

// Calls use(r, c, q, inside) for the pixels of the kS x kS window around the tile: row r and
// column c of the window, index q in the planes (0 outside the image).  A thread keeps its
// column and steps down kThreads / kS rows at a time.
template <typename F>
__device__ __forceinline__ void for_window(const SsimItem& it, F&& use) {
  constexpr int kRows = kThreads / kS;
  const int r0 = (int)threadIdx.x / kS, c = (int)threadIdx.x - r0 * kS;
  const int x = it.x0 + c - kR;
  const bool xin = r0 < kRows && x >= 0 && x < it.W;
  if (r0 < kRows) {
#pragma unroll
    for (int i = 0; i < (kS + kRows - 1) / kRows; ++i) {
      const int r = r0 + i * kRows;
      if (r < kS) {
        const int y = it.y0 + r - kR;
        const bool in = xin && y >= 0 && y < it.H;
        use(r, c, in ? it.base + (int64_t)y * it.W + x : 0, in);
      }
    }
  }
}

// The window's weights, twice each for the packed sums.
struct Taps {
  f32x2 w[2 * kR + 1];
  __device__ __forceinline__ void load() {
#pragma unroll
    for (int k = 0; k <= 2 * kR; ++k) w[k] = pack2(c_w[k], c_w[k]);
  }
};

// Vertical pass: the window sums of the packed pairs ha and (kSecond) hb and of hc for the
// kCol outputs of column c from row r0, taps in ascending order.
constexpr int kCol = kT * kT / kThreads;  // outputs per thread of a column
template <bool kSecond>
__device__ __forceinline__ void column_sums(const float2 (*ha)[kH], const float2 (*hb)[kH],
                                            const float (*hc)[kT], int r0, int c, const Taps& tp,
                                            f32x2 (&a)[kCol], f32x2 (&b)[kCol], float (&s)[kCol]) {
#pragma unroll
  for (int o = 0; o < kCol; ++o) { a[o] = 0; b[o] = 0; s[o] = 0.0f; }
#pragma unroll
  for (int r = 0; r < kCol + 2 * kR; ++r) {
    const float2 va = ha[r0 + r][c];
    const f32x2 pa = pack2(va.x, va.y);
    f32x2 pb = 0;
    if (kSecond) {
      const float2 vb = hb[r0 + r][c];
      pb = pack2(vb.x, vb.y);
    }
    const float vc = hc[r0 + r][c];
#pragma unroll
    for (int o = 0; o < kCol; ++o) {
      const int k = r - o;
      if (k < 0 || k > 2 * kR) continue;
      float wk, w1;
      unpack2(tp.w[k], wk, w1);
      a[o] = fma2(tp.w[k], pa, a[o]);
      if (kSecond) b[o] = fma2(tp.w[k], pb, b[o]);
      s[o] = fmaf(wk, vc, s[o]);
    }
  }
}

// A sum of FP32 values in three FP32 parts: Knuth's TwoSum carries every addition's rounding
// error into the second part and the errors of those into the third, some 70 bits, so that a
// CTA's thousand terms add up no worse than in FP64 (53 bits; a 64th of the FP32 rate, and two
// parts would keep 48).
struct Sum3 {
  float hi, mid, lo;
  __device__ __forceinline__ static float two_sum(float a, float b, float& err) {
    const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
    err = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
    return s;
  }
  __device__ __forceinline__ void add(float v) {
    float e1, e2;
    hi = two_sum(hi, v, e1);
    mid = two_sum(mid, e1, e2);
    lo = __fadd_rn(lo, e2);
  }
  __device__ __forceinline__ void add(const Sum3& o) {
    float e1, e2, e3;
    hi = two_sum(hi, o.hi, e1);
    mid = two_sum(mid, o.mid, e2);
    mid = two_sum(mid, e1, e3);
    lo = __fadd_rn(__fadd_rn(lo, o.lo), __fadd_rn(e2, e3));
  }
  // with the lanes `o` away, over 2 o lanes
  __device__ __forceinline__ void add_lane(int o) {
    Sum3 t;
    t.hi = __shfl_xor_sync(0xffffffffu, hi, o);
    t.mid = __shfl_xor_sync(0xffffffffu, mid, o);
    t.lo = __shfl_xor_sync(0xffffffffu, lo, o);
    add(t);
  }
  __device__ __forceinline__ double value() const {
    // (an infinite sum has no error terms)
    return isfinite(hi) ? (double)hi + ((double)mid + (double)lo) : (double)hi;
  }
};

// The CTA's sums of the threads' a and b, a's in thread 0 and b's in thread 16 (red: two
// entries per warp).  A warp's first step leaves the a's in its lower half and the b's in the
// upper one, so that the steps after it take one sum a lane.
__device__ __forceinline__ Sum3 block_sums(const Sum3& a, const Sum3& b, Sum3* red) {
  constexpr int kWarps = kThreads / 32;
  static_assert(kWarps == 8, "the last three steps reduce eight warps");
  const int lane = (int)(threadIdx.x & 31);
  const bool up = lane >= 16;
  Sum3 mine, t;
  mine.hi = up ? b.hi : a.hi;
  mine.mid = up ? b.mid : a.mid;
  mine.lo = up ? b.lo : a.lo;
  t.hi = __shfl_xor_sync(0xffffffffu, up ? a.hi : b.hi, 16);
  t.mid = __shfl_xor_sync(0xffffffffu, up ? a.mid : b.mid, 16);
  t.lo = __shfl_xor_sync(0xffffffffu, up ? a.lo : b.lo, 16);
  mine.add(t);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) mine.add_lane(o);
  if ((lane & 15) == 0) red[(up ? kWarps : 0) + (threadIdx.x >> 5)] = mine;
  __syncthreads();
  if (threadIdx.x < 32) {
    mine = red[(up ? kWarps : 0) + (lane & (kWarps - 1))];
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) mine.add_lane(o);
  }
  return mine;
}

}  // namespace

__global__ void __launch_bounds__(kThreads, 5) k_ssim_fwd(const LossImgs L, const float* __restrict__ x,
                                                       const float* __restrict__ y, float* __restrict__ dmx,
                                                       float* __restrict__ dexx, float* __restrict__ dexy,
                                                       double* __restrict__ sums) {
  __shared__ __align__(16) float2 sxy[kS][kS];               // (x, y)
  __shared__ __align__(16) float2 hm[kS][kH], hq[kS][kH];    // row sums of (x, y), (x^2, y^2)
  __shared__ __align__(16) float hc[kS][kT];                 // ... of x y
  __shared__ Sum3 red[2 * kThreads / 32];
  const SsimItem it = decode(L, blockIdx.x);
  Taps tp;
  tp.load();
  for_window(it, [&](int r, int c, int64_t q, bool in) {
    cp_async4_or_zero(&sxy[r][c].x, x + q, in);
    cp_async4_or_zero(&sxy[r][c].y, y + q, in);
  });
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  for (int t = threadIdx.x; t < kS * (kT / 4); t += kThreads) {
    // (eight lanes take four groups of columns in each of two rows: 16 different 16-byte banks)
    const int r = 2 * (t >> 4) + ((t >> 2) & 1), c = 4 * ((t & 3) | ((t >> 1) & 4));
    f32x2 m[4] = {0, 0, 0, 0}, q[4] = {0, 0, 0, 0};
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 4 + 2 * kR; i += 2) {
      const float4 v = *reinterpret_cast<const float4*>(&sxy[r][c + i]);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float xv = e ? v.z : v.x, yv = e ? v.w : v.y;
        const f32x2 p = pack2(xv, yv), pp = mul2(p, p);
        const float cv = xv * yv;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int k = i + e - o;
          if (k < 0 || k > 2 * kR) continue;
          float wk, w1;
          unpack2(tp.w[k], wk, w1);
          m[o] = fma2(tp.w[k], p, m[o]);
          q[o] = fma2(tp.w[k], pp, q[o]);
          s[o] = fmaf(wk, cv, s[o]);
        }
      }
    }
#pragma unroll
    for (int o = 0; o < 4; o += 2) {
      float4 a, b;
      unpack2(m[o], a.x, a.y);
      unpack2(m[o + 1], a.z, a.w);
      unpack2(q[o], b.x, b.y);
      unpack2(q[o + 1], b.z, b.w);
      *reinterpret_cast<float4*>(&hm[r][c + o]) = a;
      *reinterpret_cast<float4*>(&hq[r][c + o]) = b;
    }
    *reinterpret_cast<float4*>(&hc[r][c]) = make_float4(s[0], s[1], s[2], s[3]);
  }
  __syncthreads();
  const int c = (int)threadIdx.x % kT, r0 = (int)threadIdx.x / kT * kCol;
  f32x2 m2[kCol], q2[kCol];
  float cs[kCol];
  column_sums<true>(hm, hq, hc, r0, c, tp, m2, q2, cs);
  const int px = it.x0 + c;
  float ts[kCol], tl[kCol];  // S and |x - y| of the thread's pixels
#pragma unroll
  for (int o = 0; o < kCol; ++o) {
    const int r = r0 + o, py = it.y0 + r;
    ts[o] = tl[o] = 0.0f;
    if (px >= it.W || py >= it.H) continue;
    float mx, my, ex, ey;
    unpack2(m2[o], mx, my);
    unpack2(q2[o], ex, ey);
    const float vx = ex - mx * mx, vy = ey - my * my, cxy = cs[o] - mx * my;
    const float a1 = 2.0f * mx * my + kC1, a2 = 2.0f * cxy + kC2;
    const float b1 = mx * mx + my * my + kC1, b2 = vx + vy + kC2;
    const float rb1 = 1.0f / b1, rb2 = 1.0f / b2, ib = rb1 * rb2;
    const float S = a1 * a2 * ib;
    const int64_t q = it.base + (int64_t)py * it.W + px;
    dmx[q] = 2.0f * my * (a2 - a1) * ib + 2.0f * mx * S * (rb2 - rb1);
    dexx[q] = -S * rb2;
    dexy[q] = 2.0f * a1 * ib;
    const float2 v = sxy[r + kR][c + kR];
    ts[o] = S;
    tl[o] = fabsf(v.x - v.y);
  }
  Sum3 s_sum, l1_sum;
  s_sum.hi = Sum3::two_sum(ts[0], ts[1], s_sum.mid);
  l1_sum.hi = Sum3::two_sum(tl[0], tl[1], l1_sum.mid);
  s_sum.lo = l1_sum.lo = 0.0f;
#pragma unroll
  for (int o = 2; o < kCol; ++o) {
    s_sum.add(ts[o]);
    l1_sum.add(tl[o]);
  }
  const Sum3 sum = block_sums(s_sum, l1_sum, red);
  if (threadIdx.x == 0 || threadIdx.x == 16) atomicAdd(sums + (threadIdx.x >> 4), sum.value());
}

__global__ void __launch_bounds__(kThreads, 5) k_ssim_bwd(const LossImgs L, const float* __restrict__ x,
                                                       const float* __restrict__ y,
                                                       const float* __restrict__ dmx,
                                                       const float* __restrict__ dexx,
                                                       const float* __restrict__ dexy, float a,
                                                       float bcoef, float* __restrict__ dL) {
  __shared__ __align__(16) float2 sd[kS][kS];  // (dS/dmx, dS/dE[x^2])
  __shared__ __align__(16) float sc[kS][kS + 2];  // dS/dE[x y]
  __shared__ __align__(16) float2 hd[kS][kH];
  __shared__ __align__(16) float hc[kS][kT];
  const SsimItem it = decode(L, blockIdx.x);
  Taps tp;
  tp.load();
  for_window(it, [&](int r, int c, int64_t q, bool in) {
    cp_async4_or_zero(&sd[r][c].x, dmx + q, in);
    cp_async4_or_zero(&sd[r][c].y, dexx + q, in);
    cp_async4_or_zero(&sc[r][c], dexy + q, in);
  });
  cp_async_commit();
  cp_async_wait<0>();
  __syncthreads();
  for (int t = threadIdx.x; t < kS * (kT / 4); t += kThreads) {
    // (eight lanes take four groups of columns in each of two rows: 16 different 16-byte banks)
    const int r = 2 * (t >> 4) + ((t >> 2) & 1), c = 4 * ((t & 3) | ((t >> 1) & 4));
    f32x2 m[4] = {0, 0, 0, 0};
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 4 + 2 * kR; i += 2) {
      const float4 v = *reinterpret_cast<const float4*>(&sd[r][c + i]);
      const float2 u = *reinterpret_cast<const float2*>(&sc[r][c + i]);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const f32x2 p = e ? pack2(v.z, v.w) : pack2(v.x, v.y);
        const float cv = e ? u.y : u.x;
#pragma unroll
        for (int o = 0; o < 4; ++o) {
          const int k = i + e - o;
          if (k < 0 || k > 2 * kR) continue;
          float wk, w1;
          unpack2(tp.w[k], wk, w1);
          m[o] = fma2(tp.w[k], p, m[o]);
          s[o] = fmaf(wk, cv, s[o]);
        }
      }
    }
#pragma unroll
    for (int o = 0; o < 4; o += 2) {
      float4 a;
      unpack2(m[o], a.x, a.y);
      unpack2(m[o + 1], a.z, a.w);
      *reinterpret_cast<float4*>(&hd[r][c + o]) = a;
    }
    *reinterpret_cast<float4*>(&hc[r][c]) = make_float4(s[0], s[1], s[2], s[3]);
  }
  const int c = (int)threadIdx.x % kT, r0 = (int)threadIdx.x / kT * kCol;
  // (the pixels' own values, read while the others finish their rows)
  float xv[kCol], yv[kCol];
#pragma unroll
  for (int o = 0; o < kCol; ++o) {
    const int py = it.y0 + r0 + o;
    const bool in = it.x0 + c < it.W && py < it.H;
    const int64_t q = in ? it.base + (int64_t)py * it.W + it.x0 + c : 0;
    xv[o] = in ? x[q] : 0.0f;
    yv[o] = in ? y[q] : 0.0f;
  }
  __syncthreads();
  f32x2 d2[kCol], none[kCol];
  float cs[kCol];
  column_sums<false>(hd, nullptr, hc, r0, c, tp, d2, none, cs);
  const int px = it.x0 + c;
#pragma unroll
  for (int o = 0; o < kCol; ++o) {
    const int py = it.y0 + r0 + o;
    if (px >= it.W || py >= it.H) continue;
    float cv0, cv1;
    unpack2(d2[o], cv0, cv1);
    const int64_t q = it.base + (int64_t)py * it.W + px;
    const float d = xv[o] - yv[o];
    const float sgn = d > 0.0f ? 1.0f : (d < 0.0f ? -1.0f : 0.0f);
    dL[q] = a * sgn - bcoef * (cv0 + 2.0f * xv[o] * cv1 + yv[o] * cs[o]);
  }
}

__global__ void k_ssim_loss(const double* __restrict__ sums, double inv_n, float lam, float* loss) {
  *loss = (float)((1.0 - lam) * sums[1] * inv_n + lam * (1.0 - sums[0] * inv_n));
}

// Host side ----------------------------------------------------------------------
// Uploads the window weights to the current device (synchronous; called when a context is
// created, never inside a stream capture).
int ssim_init() {
  float w[2 * kR + 1];
  double sum = 0.0, wd[2 * kR + 1];
  for (int k = 0; k <= 2 * kR; ++k) {
    const double t = (double)(k - kR);
    wd[k] = std::exp(-t * t / (2.0 * 1.5 * 1.5));
    sum += wd[k];
  }
  for (int k = 0; k <= 2 * kR; ++k) w[k] = (float)(wd[k] / sum);
  return cudaMemcpyToSymbol(c_w, w, sizeof(w)) == cudaSuccess ? 0 : -1;
}

int64_t ssim_blocks(const LossImgs& L) { return L.blk_off[L.V]; }

void launch_loss_l1_dssim(const LossImgs& L, const float* x, const float* y, float lam,
                          float* dmx, float* dexx, float* dexy, double* sums, float* loss,
                          float* dL, cudaStream_t s) {
  const int64_t blocks = ssim_blocks(L);
  if (blocks == 0) return;
  const double inv_n = 1.0 / (3.0 * (double)L.pix_off[L.V]);
  cudaMemsetAsync(sums, 0, 2 * sizeof(double), s);
  k_ssim_fwd<<<(unsigned)blocks, kThreads, 0, s>>>(L, x, y, dmx, dexx, dexy, sums);
  k_ssim_bwd<<<(unsigned)blocks, kThreads, 0, s>>>(L, x, y, dmx, dexx, dexy,
                                                     (float)((1.0 - lam) * inv_n),
                                                     (float)(lam * inv_n), dL);
  k_ssim_loss<<<1, 1, 0, s>>>(sums, inv_n, lam, loss);
  count_launch();
  count_launch();
  count_launch();
}

LossImgs make_loss_imgs(int V, const int* W, const int* H) {
  LossImgs L;
  std::memset(&L, 0, sizeof(L));
  L.V = V;
  for (int v = 0; v < V; ++v) {
    L.W[v] = W[v];
    L.H[v] = H[v];
    L.pix_off[v + 1] = L.pix_off[v] + (int64_t)W[v] * H[v];
    L.blk_off[v + 1] = L.blk_off[v] + 3 * (int64_t)((W[v] + kT - 1) / kT) * ((H[v] + kT - 1) / kT);
  }
  return L;
}

}  // namespace splx
