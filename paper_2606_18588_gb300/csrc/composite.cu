// Global composition (Eq. 5) and its adjoint (Eq. 6-7), one thread per pixel of every
// view of the batch, plus the L1 photometric loss.
//
// Both are bound by HBM latency rather than bandwidth: their work per byte is a sort of a few
// keys.  With visible regions a warp takes a patch of one tile, so the subsets whose region
// misses the tile drop out for all its lanes at once, before anything is read; without them
// it takes 32 consecutive pixels, whole lines of every plane.  What is left is loaded, sorted
// and blended in registers, with the pointers of all planes in the lanes' registers and the
// colours of four subsets in flight.  Measured (composite, adjoint; before: a thread per
// pixel, keys and order in local memory): K = 32, 4 views 1920x1080 of the 20M-Gaussian city,
// where a tile has one or two subsets, 0.97 -> 0.14 and 1.64 -> 0.19 ms; K = 8, 16 views of
// 10M 0.64 -> 0.46 and 1.02 -> 0.66 ms; 16 partials of 1600x1064 from outside 212 -> 153 us
// (157 in patches of a tile).
//
// The thread per pixel stays where it is the better form.  One subset has no order (1M
// Gaussians, 2 views 1600x1064: composite 24 us, adjoint 23; a patch 24 and 42).  More than
// 16 subsets without regions go through local memory: 24 partials of 1600x1064, every pixel
// covered, 0.74 ms (0.88 by the patches' array form, which is the one for tiles with more
// than 8 subsets of a launch with regions: K = 24, all in every tile, two views 0.95 ms,
// adjoint 1.39; 1.15 and 1.58 before the patches).  Both are bound by the insertion's moves
// in local memory, which is why the order is a byte per subset (as ints, which leave L1:
// 0.90 ms, and 1.08 and 1.67).
//
// Order: subsets sorted per pixel by the normalised depth D^m / (1 - T^m), a convex
// combination of the subset's contributor depths (Eq. 4 read as D = sum d alpha T);
// ties go to the lower subset index and subsets with no contributor (T^m = 1) go last.
// Forward: C = sum_j C^{m_j} P_j + bg P_L with P_j = prod_{i<j} T^{m_i}, stopping once
// P_j < eps_comp (saturation, Sec. 4.2).  Adjoint per included subset m_j:
//   dL/dC^{m_j} = g P_j,  dL/dT^{m_j} = <g, P_j S_j> + gT P_j prod_{i>j} T^{m_i},
// with the suffix S_j = C^{m_{j+1}} + T^{m_{j+1}} S_{j+1}, S_{L-1} = bg.  Subsets after
// the cut get zero.
#include "common.cuh"

namespace splx {

namespace {

// A warp's 32 pixels: with visible regions a patch of one tile (32x1, 16x2 or 8x4 for tiles of
// 32, 16, 8), so that the subsets whose visible region holds the tile are the same for all of
// them; without (every subset everywhere) 32 consecutive pixels of a view, so that a plane is
// read and written by whole lines.
struct Patch {
  int v;
  bool in;          // the lane's pixel lies in the image
  int64_t p, HW;    // its index in the view's planes, pixels of the view
  uint64_t inside;  // bit m: subset m's visible region holds the tile
};

__device__ __forceinline__ Patch patch_of(const BatchDev& b, int64_t warp) {
  Patch q;
  const int lane = (int)(threadIdx.x & 31);
  if (!b.omega) {
    // view v's warps start at first_warp(v): room for a last warp of fewer pixels
    auto first_warp = [&](int v) { return (b.pix_off[v] >> 5) + v; };
    int lo = 0, hi = b.V - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (first_warp(mid) <= warp) lo = mid; else hi = mid - 1;
    }
    q.v = lo;
    q.HW = b.pix_off[lo + 1] - b.pix_off[lo];
    const int64_t p = ((warp - first_warp(lo)) << 5) + lane;
    q.in = p < q.HW;
    q.p = q.in ? p : 0;
    q.inside = ~0ull >> (64 - b.K);
    return q;
  }
  const int sh = __ffs(b.tile) - 1;  // the tile side is a power of two
  const int pp = 2 * sh - 5;         // log2 of the patches per tile
  const int64_t t = warp >> pp;
  q.v = view_of(b.tile_base, b.V, t * b.K);
  const ViewDev& cam = b.views[q.v];
  // (a view's tiles, and those before it, number fewer than 2^31)
  const uint32_t loc = (uint32_t)t - (uint32_t)b.tile_base[q.v] / (uint32_t)b.K;
  const int ty = (int)(loc / (uint32_t)cam.tiles_x), tx = (int)(loc - (uint32_t)ty * cam.tiles_x);
  const int rows = 5 - sh;  // log2 of the patch's rows
  const int x = (tx << sh) + (lane & (b.tile - 1));
  const int y = (ty << sh) + ((int)(warp & ((1 << pp) - 1)) << rows) + (lane >> sh);
  q.in = x < cam.W && y < cam.H;
  q.HW = (int64_t)cam.W * cam.H;
  q.p = q.in ? (int64_t)y * cam.W + x : 0;
  q.inside = 0;
  for (int m0 = 0; m0 < b.K; m0 += 32) {
    const int m = m0 + lane;
    const unsigned bits = __ballot_sync(0xffffffffu, m < b.K && in_omega(b, q.v, m, tx, ty));
    q.inside |= (uint64_t)bits << m0;
  }
  return q;
}

// One plane pointer of every subset, held by the warp's lanes (lane l: subsets l and l + 32):
// one table read for all subsets, then a shuffle per use instead of a dependent read.  get()
// is for the whole warp; m may differ from lane to lane.
template <bool kWide>
struct Planes {
  unsigned long long lo, hi;
  __device__ __forceinline__ void set(const void* a, const void* b) {
    lo = reinterpret_cast<unsigned long long>(a);
    hi = reinterpret_cast<unsigned long long>(b);
  }
  template <typename P>
  __device__ __forceinline__ P get(int m) const {
    unsigned long long r = __shfl_sync(0xffffffffu, lo, m & 31);
    if (kWide) {
      const unsigned long long h = __shfl_sync(0xffffffffu, hi, m & 31);
      r = m < 32 ? r : h;
    }
    return reinterpret_cast<P>(r);
  }
};
// The table rows of the lane's two subsets (any valid row beyond K).
__device__ __forceinline__ const ImgDev* lane_img(const BatchDev& b, const Patch& q, int half) {
  const int m = (int)(threadIdx.x & 31) + 32 * half;
  return b.imgs + q.v * b.K + (m < b.K ? m : 0);
}

// The inside subsets of the lane's pixel in composition order: by the normalised depth D / (1 -
// T), ties to the lower index, empty ones (T = 1) last.  n <= M of them (the same n for all
// lanes); everything stays in registers.  Subsets outside are empty and never written or
// read: they would stand among the last and add nothing.
template <int M, bool kWide>
struct PixOrder {
  float T[M], key[M];
  int idx[M];

  __device__ __forceinline__ void load(const BatchDev& b, const Patch& q, int n) {
    Planes<kWide> pt, pd;
    const ImgDev *a = lane_img(b, q, 0), *c = kWide ? lane_img(b, q, 1) : a;
    pt.set(a->T, c->T);
    pd.set(a->D, c->D);
    uint64_t rest = q.inside;
#pragma unroll
    for (int i = 0; i < M; ++i) {
      T[i] = 1.0f;
      key[i] = 0.0f;
      idx[i] = 0;
      if (i < n) {
        const int m = __ffsll((long long)rest) - 1;
        rest &= rest - 1;
        idx[i] = m;
        T[i] = pt.template get<const float*>(m)[q.p];
        key[i] = pd.template get<const float*>(m)[q.p];
      }
    }
#pragma unroll
    for (int i = 0; i < M; ++i)
      if (i < n) key[i] = T[i] < 1.0f ? key[i] / (1.0f - T[i]) : __int_as_float(0x7f800000);
    // insertion by exchanges of neighbours (stable)
#pragma unroll
    for (int i = 1; i < M; ++i) {
      if (i < n) {
#pragma unroll
        for (int j = i; j > 0; --j) {
          const bool sw = key[j - 1] > key[j];
          const float k = key[j], t = T[j];
          const int x = idx[j];
          key[j] = sw ? key[j - 1] : k;
          T[j] = sw ? T[j - 1] : t;
          idx[j] = sw ? idx[j - 1] : x;
          key[j - 1] = sw ? k : key[j - 1];
          T[j - 1] = sw ? t : T[j - 1];
          idx[j - 1] = sw ? x : idx[j - 1];
        }
      }
    }
  }
};

// How many subsets' colours are loaded ahead of their use.
constexpr int kAhead = 4;

template <int M, bool kWide>
__device__ __forceinline__ void composite_patch(const BatchDev& b, const Patch& q, int n) {
  PixOrder<M, kWide> po;
  po.load(b, q, n);
  Planes<kWide> pr;
  pr.set(lane_img(b, q, 0)->rgb, kWide ? lane_img(b, q, 1)->rgb : nullptr);
  float P = 1.0f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
#pragma unroll
  for (int j0 = 0; j0 < M; j0 += kAhead) {
    if (j0 < n) {
      // the colours of the next subsets up to the saturation cut, all in flight together
      float r[kAhead], g[kAhead], bl[kAhead], w[kAhead];
#pragma unroll
      for (int i = 0; i < kAhead; ++i) {
        const int j = j0 + i;
        r[i] = g[i] = bl[i] = w[i] = 0.0f;
        if (j < M && j < n) {
          const float* rgb = pr.template get<const float*>(po.idx[j < M ? j : 0]);
          if (!(P < b.eps_comp)) {
            r[i] = rgb[q.p];
            g[i] = rgb[q.HW + q.p];
            bl[i] = rgb[2 * q.HW + q.p];
            w[i] = P;
            P *= po.T[j < M ? j : 0];
          }
        }
      }
#pragma unroll
      for (int i = 0; i < kAhead; ++i) {
        c0 = fmaf(r[i], w[i], c0);
        c1 = fmaf(g[i], w[i], c1);
        c2 = fmaf(bl[i], w[i], c2);
      }
    }
  }
  if (!q.in) return;
  float* orgb = b.out_rgb + 3 * b.pix_off[q.v];
  orgb[q.p] = fmaf(b.bg[0], P, c0);
  orgb[q.HW + q.p] = fmaf(b.bg[1], P, c1);
  orgb[2 * q.HW + q.p] = fmaf(b.bg[2], P, c2);
  if (b.out_T) b.out_T[b.pix_off[q.v] + q.p] = P;
}

template <int M, bool kWide>
__device__ __forceinline__ void composite_bwd_patch(const BatchDev& b, const Patch& q, int n) {
  const float* dl = b.dL_drgb + 3 * b.pix_off[q.v];
  const float g0 = dl[q.p], g1 = dl[q.HW + q.p], g2 = dl[2 * q.HW + q.p];
  const float gT = b.dL_dT ? b.dL_dT[b.pix_off[q.v] + q.p] : 0.0f;
  PixOrder<M, kWide> po;
  po.load(b, q, n);
  Planes<kWide> pr, pg;
  const ImgDev *ia = lane_img(b, q, 0), *ib = kWide ? lane_img(b, q, 1) : ia;
  pr.set(ia->rgb, ib->rgb);
  pg.set(ia->gCT, ib->gCT);
  // key[j] becomes the prefix P_j; bit j of inc: included (before the saturation cut)
  float P = 1.0f;
  unsigned inc = 0;
#pragma unroll
  for (int j = 0; j < M; ++j) {
    po.key[j] = P;
    if (j < n && !(P < b.eps_comp)) {
      inc |= 1u << j;
      P *= po.T[j];
    }
  }
  float S0 = b.bg[0], S1 = b.bg[1], S2 = b.bg[2], Rt = 1.0f;
#pragma unroll
  for (int j1 = (M - 1) / kAhead * kAhead; j1 >= 0; j1 -= kAhead) {
    if (j1 < n) {
      // the colours of the next subsets back to front, all in flight together
      float r[kAhead], g[kAhead], bl[kAhead];
      float4* out[kAhead];
#pragma unroll
      for (int i = 0; i < kAhead; ++i) {
        const int j = j1 + i < M ? j1 + i : 0;
        r[i] = g[i] = bl[i] = 0.0f;
        out[i] = nullptr;
        if (j1 + i < M && j1 + i < n) {
          const float* rgb = pr.template get<const float*>(po.idx[j]);
          out[i] = pg.template get<float4*>(po.idx[j]) + q.p;
          if ((inc >> j) & 1u) {
            r[i] = rgb[q.p];
            g[i] = rgb[q.HW + q.p];
            bl[i] = rgb[2 * q.HW + q.p];
          }
        }
      }
#pragma unroll
      for (int i = kAhead - 1; i >= 0; --i) {
        const int j = j1 + i < M ? j1 + i : 0;
        if (j1 + i < M && j1 + i < n) {
          float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
          if ((inc >> j) & 1u) {
            const float Pm = po.key[j];
            const float gTm = (g0 * S0 + g1 * S1 + g2 * S2) * Pm + gT * Pm * Rt;
            o = make_float4(g0 * Pm, g1 * Pm, g2 * Pm, gTm);
            const float Tm = po.T[j];
            S0 = fmaf(Tm, S0, r[i]);
            S1 = fmaf(Tm, S1, g[i]);
            S2 = fmaf(Tm, S2, bl[i]);
            Rt *= Tm;
          }
          if (q.in) *out[i] = o;
        }
      }
    }
  }
}

// More inside subsets than the register forms hold: the same, through arrays indexed at run
// time (local memory; kept small, a key and a byte per subset, so that they stay in L1: the
// transmittances are read again where they are used).  All lanes run along (the planes'
// pointers come by shuffles).
struct PixOrderAny {
  float key[kMaxK];  // by subset
  uint8_t ord[kMaxK];
  Planes<true> pt;

  // kLoads: subsets whose planes are in flight together
  template <int kLoads>
  __device__ __forceinline__ int load(const BatchDev& b, const Patch& q) {
    Planes<true> pd;
    const ImgDev *a = lane_img(b, q, 0), *c = lane_img(b, q, 1);
    pt.set(a->T, c->T);
    pd.set(a->D, c->D);
    int n = 0;
    for (uint64_t rest = q.inside; rest;) {
      float t[kLoads], d[kLoads];
      int m[kLoads];
#pragma unroll
      for (int i = 0; i < kLoads; ++i) {
        m[i] = -1;
        if (rest) {
          m[i] = __ffsll((long long)rest) - 1;
          rest &= rest - 1;
          t[i] = pt.get<const float*>(m[i])[q.p];
          d[i] = pd.get<const float*>(m[i])[q.p];
        }
      }
#pragma unroll
      for (int i = 0; i < kLoads; ++i) {
        if (m[i] < 0) continue;
        const float km = t[i] < 1.0f ? d[i] / (1.0f - t[i]) : __int_as_float(0x7f800000);
        key[m[i]] = km;
        int j = n++;
        for (int o; j > 0 && key[o = ord[j - 1]] > km; --j) ord[j] = (uint8_t)o;
        ord[j] = (uint8_t)m[i];
      }
    }
    return n;
  }
};

__device__ __noinline__ void composite_any(const BatchDev& b, const Patch& q) {
  PixOrderAny po;
  const int n = po.load<4>(b, q);
  Planes<true> pr;
  pr.set(lane_img(b, q, 0)->rgb, lane_img(b, q, 1)->rgb);
  float P = 1.0f, c0 = 0.f, c1 = 0.f, c2 = 0.f;
  for (int j0 = 0; j0 < n; j0 += kAhead) {
    const bool open = !(P < b.eps_comp);
    if (!__any_sync(0xffffffffu, open)) break;
    float r[kAhead], g[kAhead], bl[kAhead], t[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      r[i] = g[i] = bl[i] = 0.0f;
      t[i] = 1.0f;
      if (j0 + i < n) {
        const int m = po.ord[j0 + i];
        const float* rgb = pr.get<const float*>(m);
        const float* Tm = po.pt.get<const float*>(m);
        if (open) {
          r[i] = rgb[q.p];
          g[i] = rgb[q.HW + q.p];
          bl[i] = rgb[2 * q.HW + q.p];
          t[i] = Tm[q.p];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      if (j0 + i < n && !(P < b.eps_comp)) {
        c0 = fmaf(r[i], P, c0);
        c1 = fmaf(g[i], P, c1);
        c2 = fmaf(bl[i], P, c2);
        P *= t[i];
      }
    }
  }
  if (!q.in) return;
  float* orgb = b.out_rgb + 3 * b.pix_off[q.v];
  orgb[q.p] = fmaf(b.bg[0], P, c0);
  orgb[q.HW + q.p] = fmaf(b.bg[1], P, c1);
  orgb[2 * q.HW + q.p] = fmaf(b.bg[2], P, c2);
  if (b.out_T) b.out_T[b.pix_off[q.v] + q.p] = P;
}

__device__ __noinline__ void composite_bwd_any(const BatchDev& b, const Patch& q) {
  PixOrderAny po;
  const int n = po.load<8>(b, q);
  Planes<true> pr, pg;
  const ImgDev *ia = lane_img(b, q, 0), *ib = lane_img(b, q, 1);
  pr.set(ia->rgb, ib->rgb);
  pg.set(ia->gCT, ib->gCT);
  // key[m] becomes the prefix P of the subsets before the cut, the first L in the order
  float P = 1.0f;
  int L = 0;
  for (int j0 = 0; j0 < n; j0 += kAhead) {
    if (!__any_sync(0xffffffffu, !(P < b.eps_comp))) break;
    float t[kAhead];
    int m[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      m[i] = j0 + i < n ? po.ord[j0 + i] : 0;
      const float* Tm = po.pt.get<const float*>(m[i]);
      t[i] = j0 + i < n ? Tm[q.p] : 1.0f;
    }
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      if (j0 + i < n && !(P < b.eps_comp)) {
        po.key[m[i]] = P;
        P *= t[i];
        ++L;
      }
    }
  }
  const float* dl = b.dL_drgb + 3 * b.pix_off[q.v];
  const float g0 = dl[q.p], g1 = dl[q.HW + q.p], g2 = dl[2 * q.HW + q.p];
  const float gT = b.dL_dT ? b.dL_dT[b.pix_off[q.v] + q.p] : 0.0f;
  float S0 = b.bg[0], S1 = b.bg[1], S2 = b.bg[2], Rt = 1.0f;
  for (int j1 = n - 1; j1 >= 0; j1 -= kAhead) {
    float r[kAhead], g[kAhead], bl[kAhead], t[kAhead];
    float4* out[kAhead];
    int m[kAhead];
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      const int j = j1 - i;
      r[i] = g[i] = bl[i] = t[i] = 0.0f;
      m[i] = 0;
      out[i] = nullptr;
      if (j >= 0) {
        m[i] = po.ord[j];
        const float* rgb = pr.get<const float*>(m[i]);
        const float* Tm = po.pt.get<const float*>(m[i]);
        out[i] = pg.get<float4*>(m[i]) + q.p;
        if (j < L) {
          r[i] = rgb[q.p];
          g[i] = rgb[q.HW + q.p];
          bl[i] = rgb[2 * q.HW + q.p];
          t[i] = Tm[q.p];
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kAhead; ++i) {
      const int j = j1 - i;
      if (j < 0) continue;
      float4 o = make_float4(0.f, 0.f, 0.f, 0.f);
      if (j < L) {
        const float Pm = po.key[m[i]];
        const float gTm = (g0 * S0 + g1 * S1 + g2 * S2) * Pm + gT * Pm * Rt;
        o = make_float4(g0 * Pm, g1 * Pm, g2 * Pm, gTm);
        S0 = fmaf(t[i], S0, r[i]);
        S1 = fmaf(t[i], S1, g[i]);
        S2 = fmaf(t[i], S2, bl[i]);
        Rt *= t[i];
      }
      if (q.in) *out[i] = o;
    }
  }
}

}  // namespace

// Resident CTAs of 256 threads that the register limits are set for.
template <int MK, bool kAny, bool kBwd>
constexpr int kCompositeCtas = kBwd ? (MK <= 2 ? 6 : MK <= 4 ? 5 : MK <= 8 ? 4 : 2)
                                    : (MK <= 2 ? 8 : MK <= 4 || kAny ? 6 : MK <= 8 ? 5 : 3);

// MK: the largest number of inside subsets taken in registers (2, 4, 8 or 16 by K); kAny: more
// are possible (K > 16 with visible regions; those kernels keep to 8 in registers, since few
// tiles have more: their 40 and 64 registers hold twice the warps of 16's 76 and 93).  A warp
// runs the form for its own tile's number of subsets.
template <int MK, bool kAny, bool kBwd>
__global__ void __launch_bounds__(256, kCompositeCtas<MK, kAny, kBwd>) k_composite(const BatchDev b, int64_t warps) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= warps) return;
  const Patch q = patch_of(b, w);
  const int n = __popcll(q.inside);
  if (MK > 4 && n > 4) {
    if (MK > 8 && n > 8) {
      if (kAny && n > MK) {
        if (kBwd) composite_bwd_any(b, q); else composite_any(b, q);
      } else {
        if (kBwd) composite_bwd_patch<MK, kAny>(b, q, n); else composite_patch<MK, kAny>(b, q, n);
      }
    } else if (kAny && MK <= 8 && n > MK) {
      if (kBwd) composite_bwd_any(b, q); else composite_any(b, q);
    } else {
      if (kBwd) composite_bwd_patch<8, kAny>(b, q, n); else composite_patch<8, kAny>(b, q, n);
    }
  } else {
    constexpr int M = MK < 4 ? MK : 4;
    if (kBwd) composite_bwd_patch<M, kAny>(b, q, n); else composite_patch<M, kAny>(b, q, n);
  }
}

// More than 16 subsets without visible regions (splx_composite): a thread takes a pixel, its
// order in local memory, MK subsets' planes unrolled.  32 registers: what bounds it is the
// latency of the insertion's moves, which only more warps hide.
template <int MK>
struct PixOrderMany {
  float T[MK], key[MK];
  uint8_t ord[MK];

  __device__ __forceinline__ void load(const BatchDev& b, int v, int64_t p) {
#pragma unroll
    for (int m = 0; m < MK; ++m) {
      if (m < b.K) {
        const ImgDev& im = b.imgs[v * b.K + m];
        const float t = im.T[p];
        const float d = im.D[p];
        T[m] = t;
        key[m] = t < 1.0f ? d / (1.0f - t) : __int_as_float(0x7f800000);
      }
    }
    for (int m = 0; m < b.K; ++m) {  // insertion by (key, index): stable
      int j = m;
      const float km = key[m];
      while (j > 0 && key[ord[j - 1]] > km) {
        ord[j] = ord[j - 1];
        --j;
      }
      ord[j] = (uint8_t)m;
    }
  }
};

template <int MK, bool kBwd>
__global__ void __launch_bounds__(256) k_composite_many(const BatchDev b, int64_t total) {
  const int64_t gp = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gp >= total) return;
  const int v = view_of(b.pix_off, b.V, gp);
  const ViewDev& cam = b.views[v];
  const int64_t HW = (int64_t)cam.W * cam.H;
  const int64_t p = gp - b.pix_off[v];
  PixOrderMany<MK> po;
  po.load(b, v, p);
  float P = 1.0f;
  if (!kBwd) {
    float c0 = 0.f, c1 = 0.f, c2 = 0.f;
    for (int j = 0; j < b.K; ++j) {
      if (P < b.eps_comp) break;
      const int m = po.ord[j];
      const float* rgb = b.imgs[v * b.K + m].rgb;
      c0 = fmaf(rgb[p], P, c0);
      c1 = fmaf(rgb[HW + p], P, c1);
      c2 = fmaf(rgb[2 * HW + p], P, c2);
      P *= po.T[m];
    }
    float* orgb = b.out_rgb + 3 * b.pix_off[v];
    orgb[p] = fmaf(b.bg[0], P, c0);
    orgb[HW + p] = fmaf(b.bg[1], P, c1);
    orgb[2 * HW + p] = fmaf(b.bg[2], P, c2);
    if (b.out_T) b.out_T[b.pix_off[v] + p] = P;
    return;
  }
  float Pj[MK];
  int L = 0;  // subsets before the cut
  for (int j = 0; j < b.K; ++j) {
    if (P < b.eps_comp) break;
    Pj[j] = P;
    P *= po.T[po.ord[j]];
    ++L;
  }
  const float* dl = b.dL_drgb + 3 * b.pix_off[v];
  const float g0 = dl[p], g1 = dl[HW + p], g2 = dl[2 * HW + p];
  const float gT = b.dL_dT ? b.dL_dT[b.pix_off[v] + p] : 0.0f;
  float S0 = b.bg[0], S1 = b.bg[1], S2 = b.bg[2], Rt = 1.0f;
  for (int j = b.K - 1; j >= 0; --j) {
    const int m = po.ord[j];
    const ImgDev& im = b.imgs[v * b.K + m];
    if (j >= L) {
      im.gCT[p] = make_float4(0.f, 0.f, 0.f, 0.f);
      continue;
    }
    const float Pm = Pj[j];
    const float gTm = (g0 * S0 + g1 * S1 + g2 * S2) * Pm + gT * Pm * Rt;
    im.gCT[p] = make_float4(g0 * Pm, g1 * Pm, g2 * Pm, gTm);
    const float Tm = po.T[m];
    S0 = fmaf(Tm, S0, im.rgb[p]);
    S1 = fmaf(Tm, S1, im.rgb[HW + p]);
    S2 = fmaf(Tm, S2, im.rgb[2 * HW + p]);
    Rt *= Tm;
  }
}

// One subset: nothing to sort, so a thread takes a pixel of its own, in the planes' order.
template <bool kBwd>
__global__ void __launch_bounds__(256) k_composite_one(const BatchDev b, int64_t total) {
  const int64_t gp = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gp >= total) return;
  const int v = view_of(b.pix_off, b.V, gp);
  const ViewDev& cam = b.views[v];
  const int64_t HW = (int64_t)cam.W * cam.H, p = gp - b.pix_off[v];
  bool inside = true;
  if (b.omega) {
    const int sh = __ffs(b.tile) - 1;  // the tile side is a power of two
    const uint32_t py = (uint32_t)p / (uint32_t)cam.W;
    inside = in_omega(b, v, 0, (int)(((uint32_t)p - py * (uint32_t)cam.W) >> sh), (int)(py >> sh));
  }
  const ImgDev& im = b.imgs[v];
  const bool take = inside && !(1.0f < b.eps_comp);
  if (kBwd) {
    if (!inside) return;  // never rendered
    const float* dl = b.dL_drgb + 3 * b.pix_off[v];
    const float g0 = dl[p], g1 = dl[HW + p], g2 = dl[2 * HW + p];
    const float gT = b.dL_dT ? b.dL_dT[gp] : 0.0f;
    im.gCT[p] = take ? make_float4(g0, g1, g2, g0 * b.bg[0] + g1 * b.bg[1] + g2 * b.bg[2] + gT)
                     : make_float4(0.f, 0.f, 0.f, 0.f);
    return;
  }
  float P = 1.0f, c[3] = {0.f, 0.f, 0.f};
  if (take) {
    P = im.T[p];
#pragma unroll
    for (int ch = 0; ch < 3; ++ch) c[ch] = im.rgb[ch * HW + p];
  }
  float* orgb = b.out_rgb + 3 * b.pix_off[v];
#pragma unroll
  for (int ch = 0; ch < 3; ++ch) orgb[ch * HW + p] = fmaf(b.bg[ch], P, c[ch]);
  if (b.out_T) b.out_T[gp] = P;
}

template <int MK, bool kAny>
static void launch_c(const BatchDev& b, int64_t total, bool bwd, cudaStream_t s) {
  const int64_t warps =
      b.omega ? b.n_tiles / b.K * (b.tile * b.tile / 32) : (total >> 5) + b.V;
  const unsigned blocks = (unsigned)((warps + 7) / 8);
  if (bwd) k_composite<MK, kAny, true><<<blocks, 256, 0, s>>>(b, warps);
  else k_composite<MK, kAny, false><<<blocks, 256, 0, s>>>(b, warps);
}
template <int MK>
static void launch_pixels(const BatchDev& b, int64_t total, bool bwd, cudaStream_t s) {
  const unsigned blocks = (unsigned)((total + 255) / 256);
  if constexpr (MK == 1) {
    if (bwd) k_composite_one<true><<<blocks, 256, 0, s>>>(b, total);
    else k_composite_one<false><<<blocks, 256, 0, s>>>(b, total);
  } else {
    if (bwd) k_composite_many<MK, true><<<blocks, 256, 0, s>>>(b, total);
    else k_composite_many<MK, false><<<blocks, 256, 0, s>>>(b, total);
  }
}

static void dispatch(const BatchDev& b, int64_t total, bool bwd, cudaStream_t s) {
  if (total <= 0) return;
  if (b.K == 1) launch_pixels<1>(b, total, bwd, s);
  else if (b.K <= 2) launch_c<2, false>(b, total, bwd, s);
  else if (b.K <= 4) launch_c<4, false>(b, total, bwd, s);
  else if (b.K <= 8) launch_c<8, false>(b, total, bwd, s);
  else if (b.K <= 16) launch_c<16, false>(b, total, bwd, s);
  else if (b.omega) launch_c<8, true>(b, total, bwd, s);
  else if (b.K <= 32) launch_pixels<32>(b, total, bwd, s);
  else launch_pixels<64>(b, total, bwd, s);
  count_launch();
}

void launch_composite(const BatchDev& b, int64_t total, cudaStream_t s) { dispatch(b, total, false, s); }
void launch_composite_bwd(const BatchDev& b, int64_t total, cudaStream_t s) { dispatch(b, total, true, s); }

// ---------------------------------------------------------------- stale saturation state
// Sec. 4.2 step 2: the composition of this visit finds the pixels where the subsets in
// front have saturated; in the view's next visit the subsets behind leave those pixels.
// Per pixel: the prefix product of the partial transmittances in the view's front-to-back
// order (FP32, multiplied in that order, as the exact waves do), over the ranks below the
// old state (ranks at or beyond it were left empty); the new state is the first rank whose
// prefix before it is below eps_comp, or 255 (none).  Ranks pruned by the old state count
// as transparent, so where the prefix no longer saturates they all come back.  Subsets
// whose visible region leaves the pixel's tile out have no partial there (transparent).
__global__ void __launch_bounds__(256) k_sat_update(const BatchDev b,
                                                    const int32_t* __restrict__ order,
                                                    int64_t total) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int v = view_of(b.pix_off, b.V, q);
    const int64_t p = q - b.pix_off[v];
    const ViewDev& cam = b.views[v];
    const int px = (int)(p % cam.W), py = (int)(p / cam.W);
    const int tx = px / b.tile, ty = py / b.tile;
    uint8_t* sp = b.sat[v];
    const int lim = min((int)sp[p], b.K);
    float prefix = 1.0f;
    int out = 255;
    for (int r = 0; r < lim; ++r) {
      const int k = order[v * b.K + r];
      if (!in_omega(b, v, k, tx, ty)) continue;
      prefix *= b.imgs[v * b.K + k].T[p];
      if (prefix < b.eps_comp) {
        out = r + 1 < b.K ? r + 1 : 255;
        break;
      }
    }
    sp[p] = (uint8_t)out;
  }
}

void launch_sat_update(const BatchDev& b, const int32_t* order, int64_t total, cudaStream_t s) {
  if (total <= 0 || !b.sat) return;
  int64_t blocks = (total + 255) / 256;
  const int64_t cap = (int64_t)device_sm_count() * 16;
  if (blocks > cap) blocks = cap;
  k_sat_update<<<(unsigned)blocks, 256, 0, s>>>(b, order, total);
  count_launch();
}

// ---------------------------------------------------------------- L1 loss
__global__ void __launch_bounds__(256) k_loss_l1(const float* __restrict__ img, const float* __restrict__ tgt,
                                                 int64_t n, float* loss, float* __restrict__ dL) {
  __shared__ float sw[8];
  const float inv = 1.0f / (float)n;
  float acc = 0.0f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float d = img[i] - tgt[i];
    acc += fabsf(d);
    if (dL) dL[i] = d > 0.0f ? inv : (d < 0.0f ? -inv : 0.0f);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sw[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sw[w];
    atomicAdd(loss, t * inv);
  }
}

void launch_loss_l1(const float* img, const float* target, int64_t n, float* loss, float* dL,
                    cudaStream_t s) {
  cudaMemsetAsync(loss, 0, sizeof(float), s);
  if (n <= 0) return;
  int64_t blocks = (n + 255) / 256;
  const int64_t cap = (int64_t)device_sm_count() * 16;
  if (blocks > cap) blocks = cap;
  k_loss_l1<<<(unsigned)blocks, 256, 0, s>>>(img, target, n, loss, dL);
  count_launch();
}

}  // namespace splx
