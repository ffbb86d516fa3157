// Local rendering of every (view, subset) tile: forward (Eq. 1-4) and backward.
//
// A warp owns a region of 8 x 8 pixels (16 x 8 in the forward at 32x32 tiles), a lane two of
// its pixels four rows apart (or four); a CTA holds the warps of one image tile.  Each warp
// picks, from the tile's sorted list, the entries that can reach alpha_min in its region.
// A pixel takes a Gaussian only inside its integer 3-sigma rectangle (so the result does
// not depend on TS), with alpha = min(alpha_max, o 2^(p2)) >= alpha_min, and stops before
// the Gaussian that would take its transmittance below eps_T.  The forward's CTA leaves the
// list once every pixel has stopped (__syncthreads_count).
//
// The backward walks the same list back to front from each pixel's last blended entry,
// recovering T_i = T_{i+1} / (1 - alpha_i) from the stored final T^m, and applies the
// adjoint of Eq. 3-4 with the composite adjoint (dL/dC^m, dL/dT^m of Eq. 6-7) as input:
//   dC^m/dc_i = alpha_i T_i,  dC^m/dalpha_i = c_i T_i - B_i / (1 - alpha_i),
//   dT^m/dalpha_i = -T^m / (1 - alpha_i),  B_i = sum_{j>i} c_j alpha_j T_j.
// Per-Gaussian sums over a warp's pixels are formed in shared memory and added to the
// per-(view, Gaussian) 2-D gradient with float4 atomics.  With gp = dL/dpower at a
// pixel, power = -(A dx^2 + 2 B dx dy + C dy^2) / 2 and (dx, dy) = pixel centre - (u, v),
// the record holds the conic-free moments of ge = gp / o = dL/dalpha e^power (0 where
// alpha is clamped), sum ge dx, ge dy, ge dx^2, ge dx dy, ge dy^2, and dL/do = sum ge;
// dL/du = o (A sum ge dx + B sum ge dy), dL/dA = -o sum ge dx^2 / 2 and the rest follow
// linearly in the projection adjoint, which knows the conic and the opacity.
#include "common.cuh"

namespace splx {

namespace {

// 2^x and 1/x as single special-function-unit instructions (relative error about 2^-22;
// subnormal results flush to zero, which the alpha threshold rejects anyway).
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Adds per-thread counts into counters[slot] with one atomic per warp.
__device__ __forceinline__ void flush_counter(unsigned long long* counters, int slot, unsigned v) {
  if (!counters) return;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0 && v) atomicAdd(counters + slot, (unsigned long long)v);
}

// Pixels of a forward thread: slot i of PPT is an 8 x 4 block of the tile, lanes laid out as
// 8 columns x 4 rows inside it; a warp's PPT blocks tile a 16 x 8 region (PPT = 4) or an
// 8 x 8 region (PPT = 2).  (x, y) is the thread's pixel in slot 0; slot i adds (8 (i & 1),
// 4 (i >> 1)) for PPT = 4 and (0, 4 i) for PPT = 2.
struct TileInfo {
  int v, k, x, y, W, H, tx, ty;
};

// ---- the forward's warp lists -----------------------------------------------------------
// A warp copies the staged entries that can reach a pixel of its region (8 x 8 pixels for
// PPT = 2, 16 x 8 for PPT = 4), in entry order, into a ring of kRingItems items of shared
// memory, laid out two entries side by side (kPairWords words per pair):
//   [u0 u1 v0 v1] [qa0 qa1 qb0 qb1] [qc0 qc1 o0 o1] [r0 g0 b0 d0] [r1 g1 b1 d1] [m0 m1 j0 j1]
// so that the conic of both entries is evaluated by packed FP32 instructions without moving
// a register.  m: the region's columns (bits 8 and up) and rows (bits 24 and up) that the
// entry's rectangle spans; j: the entry's position in the tile's list.
constexpr int kRingItems = 64;
constexpr int kPairWords = 28;  // 24 used; the stride spreads the pairs over the banks
constexpr uint32_t kDeadPixel = 1u;  // a pixel's mask once it takes nothing more (bit 0 of m is 0)

// Whether an entry with conic (qa, qb, qc), opacity o and centre (u, v) may reach alpha >=
// alpha_min in the box [X0, X1] x [Y0, Y1] (offsets from the centre): its exponent's maximum
// over the box, with a margin above the rounding of this evaluation and of pixel_alpha's
// (at most a few 1e-7 of the terms' sum, and |qb x y| <= |qa| x^2 + |qc| y^2), against
// lg_amin - log2(o).  The form is concave: its maximum over the box is 0 if that holds the
// centre and else lies on an edge facing the centre, at the edge's clamped stationary point;
// the other candidate is some point of the box and so never above it.  NaN keeps the entry.
__device__ __forceinline__ bool box_reached(float qa, float qb, float qc, float o, float X0,
                                            float X1, float Y0, float Y1, float lg_amin) {
  const float x1 = fminf(fmaxf(0.0f, X0), X1), y2 = fminf(fmaxf(0.0f, Y0), Y1);
  const float y1 = fminf(fmaxf(-0.5f * qb * rcp_approx(qc) * x1, Y0), Y1);
  const float x2 = fminf(fmaxf(-0.5f * qb * rcp_approx(qa) * y2, X0), X1);
  const float p1 = fmaf(fmaf(qa, x1, qb * y1), x1, qc * y1 * y1);
  const float p2 = fmaf(fmaf(qa, x2, qb * y2), x2, qc * y2 * y2);
  const float best = p1 > p2 ? p1 : p2;
  const float xm = fmaxf(fabsf(X0), fabsf(X1)), ym = fmaxf(fabsf(Y0), fabsf(Y1));
  const float margin = fmaf(-8e-6f, fmaf(qa * xm, xm, qc * ym * ym), 2e-3f);
  return !(best + margin < lg_amin - __log2f(o));
}

// Tests the staged entries e0 + lane (< cnt) of one group of 32 against the warp's region
// (its origin RX, RY on the image, rx0, ry0 in the tile) and appends those that may reach it
// at ring position `tail`; returns the new tail.  Staged: a, b, c of the record with the
// rectangle's words replaced by the tile's columns (b.w) and rows (c.w) that it spans.
// pos0: list position of staged entry 0.
template <int PPT>
__device__ __forceinline__ unsigned append_group(const float4* sA, const float4* sB,
                                                 const float4* sC, int e0, int cnt, int pos0,
                                                 int RX, int RY, int rx0, int ry0, int lane,
                                                 float lg_amin, float* ring, unsigned tail) {
  constexpr int RW = PPT == 4 ? 16 : 8;  // region width
  const int e = e0 + lane;
  uint32_t m = 0;
  float4 A, B, C;
  if (e < cnt) {
    B = sB[e];
    C = sC[e];
    const uint32_t cm = (__float_as_uint(B.w) >> rx0) & ((1u << RW) - 1u);
    const uint32_t rm = (__float_as_uint(C.w) >> ry0) << 24;
    if (cm != 0u && rm != 0u) {
      A = sA[e];
      const float X0 = ((float)RX + 0.5f) - A.x, Y0 = ((float)RY + 0.5f) - A.y;
      if (box_reached(A.z, A.w, B.x, B.y, X0, X0 + (float)(RW - 1), Y0, Y0 + 7.0f, lg_amin))
        m = (cm << 8) | rm;
    }
  }
  const unsigned hit = __ballot_sync(0xffffffffu, m != 0u);
  if (m) {
    const unsigned pos = (tail + __popc(hit & ((1u << lane) - 1u))) & (kRingItems - 1);
    float* q = ring + (pos >> 1) * kPairWords;
    const unsigned h = pos & 1u;
    q[h] = A.x;
    q[2 + h] = A.y;
    q[4 + h] = A.z;
    q[6 + h] = A.w;
    q[8 + h] = B.x;
    q[10 + h] = B.y;
    reinterpret_cast<float4*>(q + 12)[h] = make_float4(C.x, C.y, C.z, B.z);
    q[20 + h] = __uint_as_float(m);
    q[22 + h] = __int_as_float(pos0 + e);
  }
  return tail + (unsigned)__popc(hit);
}

template <int PPT>
__device__ __forceinline__ int slot_col(int i) { return PPT >= 4 ? (i & 1) : 0; }
template <int PPT>
__device__ __forceinline__ int slot_row(int i) { return PPT >= 4 ? (i >> 1) : i; }
// block columns (x offsets 0, 8) and rows (y offsets 0, 4, ...) of a thread's slots
template <int PPT>
constexpr int kSlotCols = PPT >= 4 ? 2 : 1;
template <int PPT>
constexpr int kSlotRows = PPT / kSlotCols<PPT>;

template <int TS, int PPT>
__device__ __forceinline__ TileInfo decode_tile(const BatchDev& b, int64_t id) {
  TileInfo ti;
  ti.v = view_of(b.tile_base, b.V, id);
  const ViewDev& cam = b.views[ti.v];
  // (a launch has fewer than 2^31 items, so an item's place in its view fits 32 bits)
  const uint32_t nt = (uint32_t)cam.tiles_x * (uint32_t)cam.tiles_y;
  const uint32_t rem = (uint32_t)(id - b.tile_base[ti.v]);
  ti.k = (int)(rem / nt);
  const uint32_t t = rem - (uint32_t)ti.k * nt;
  const int ty = (int)(t / (uint32_t)cam.tiles_x), tx = (int)(t - (uint32_t)ty * cam.tiles_x);
  ti.tx = tx;
  ti.ty = ty;
  const int w = (int)(threadIdx.x >> 5), l = (int)(threadIdx.x & 31);
  int rx0 = 0, ry0 = 0;
  if (PPT == 4) {  // 16 x 8 regions
    constexpr int kRegionsPerRow = TS >= 16 ? TS / 16 : 1;
    rx0 = 16 * (w % kRegionsPerRow);
    ry0 = 8 * (w / kRegionsPerRow);
  } else {  // 8 x 8 regions
    rx0 = 8 * (w % (TS / 8));
    ry0 = 8 * (w / (TS / 8));
  }
  ti.x = tx * TS + rx0 + (l & 7);
  ti.y = ty * TS + ry0 + (l >> 3);
  ti.W = cam.W;
  ti.H = cam.H;
  return ti;
}

}  // namespace

// kCount variants (eager runs only) also count the work for the roofline: thread-entries
// examined, (pixel, entry) alpha evaluations and blends / contributions.
// List entries the forward stages in shared memory per batch: one per thread.
template <int TS>
constexpr int kNBFwd = TS == 8 ? 32 : 128;
template <int TS, int PPT>
constexpr int kRingWords = TS * TS / PPT / 32 * (kRingItems / 2) * kPairWords;  // all warps' rings
// resident CTAs the backward's register limit is set for: 24 warps of 80 registers.  Six CTAs
// of four warps and 37.2 KB fit an SM's 228 KB (1 KB of it per CTA is the system's); of 8x8
// tiles' one-warp CTAs of 9.3 KB, 22 do
template <int TS>
constexpr int kMinBlocksBwd = TS == 8 ? 24 : 6;
// above this an adjoint or a colour takes the backward's careful path
constexpr float kWild = 1e18f;
// The forward of one work item.  It is bound by instruction issue (80 % of the issue slots,
// 40 % of the FMA pipe, 3 % of HBM), so everything here is there to issue fewer: a warp sees
// only the entries that can reach its region (box_reached leaves 27.7M of 36.7M
// warp-entries of the 2M-Gaussian, 4-view step), and it takes them two at a time with the
// exponents of both in packed FP32 instructions, without a branch per pixel.  Measured on
// that step (8 subsets, no skipping, 16x16 tiles): 2.89 -> 2.12 ms, 3.07e9 -> 2.06e9 warp
// instructions; 8x8 tiles 3.39 -> 1.94 ms, 32x32 4.14 -> 3.65 ms; the 10M step 58.4
// -> 55.5 ms.  Packing the colours too (channel pairs, with w moved into both halves) took
// 2.37 ms, a branch per stopping pair 2.46 ms, 10 CTAs per SM at 48 registers (spilling)
// and 7 at 72 1-2 % more than 8 at 64.
template <int TS, int PPT, bool kCount>
__device__ __forceinline__ void fwd_item(const BatchDev& b, const int64_t id, const int wave,
                                         float4* sA, float4* sB, float4* sC, float* sR) {
  constexpr int NTH = TS * TS / PPT;
  constexpr int NB = kNBFwd<TS>;
  constexpr int PER = NB > NTH ? NB / NTH : 1;  // staged entries per thread
  constexpr int NC = kSlotCols<PPT>;
  static_assert(kSlotRows<PPT> == 2, "a region is two 8 x 4 blocks high");
  const TileInfo ti = decode_tile<TS, PPT>(b, id);
  if (!in_omega(b, ti.v, ti.k, ti.tx, ti.ty)) {
    // outside the subset's visible region: no pairs; the composite never reads this tile.
    // Its transmittance is 1, which the first saturation-skipping wave must still record.
    if (kCount && threadIdx.x == 0 && b.counters) atomicAdd(b.counters + 7, 1ull);
    if (b.order && wave == 0) {
#pragma unroll
      for (int i = 0; i < PPT; ++i) {
        const int px = ti.x + 8 * slot_col<PPT>(i), py = ti.y + 4 * slot_row<PPT>(i);
        if (px < ti.W && py < ti.H) b.tpre[b.pix_off[ti.v] + (int64_t)py * ti.W + px] = 1.0f;
      }
    }
    return;
  }
  const uint2 rg = b.ranges[id];
  const uint32_t start = rg.x, len = rg.y > rg.x ? rg.y - rg.x : 0u;  // the item's list
  // the lane's pixel columns and rows, twice each for the packed evaluation of two entries
  const f32x2 pcx0 = pack2((float)ti.x + 0.5f, (float)ti.x + 0.5f),
              pcx1 = pack2((float)(ti.x + 8) + 0.5f, (float)(ti.x + 8) + 0.5f),
              pcy0 = pack2((float)ti.y + 0.5f, (float)ti.y + 0.5f),
              pcy1 = pack2((float)(ti.y + 4) + 0.5f, (float)(ti.y + 4) + 0.5f);
  const float amin = b.alpha_min, amax = b.alpha_max, epsT = b.eps_T;
  float T[PPT], c0[PPT], c1[PPT], c2[PPT], D[PPT];
  int last[PPT];
  unsigned live = 0;  // bit i: pixel i still blending
#pragma unroll
  for (int i = 0; i < PPT; ++i) {
    T[i] = 1.0f; c0[i] = c1[i] = c2[i] = D[i] = 0.0f; last[i] = -1;
    if (ti.x + 8 * slot_col<PPT>(i) < ti.W && ti.y + 4 * slot_row<PPT>(i) < ti.H) live |= 1u << i;
  }
  // (the planes' addresses are read again where they are used: nothing holds them in
  // registers across the walk)
  if ((b.order && wave > 0) || b.sat) {
    const unsigned inb = live;  // slots inside the image
    // saturation skipping: a pixel where the subsets rendered before this one took the
    // transmittance below eps_comp leaves this subset's pixel set (the composite would
    // skip this subset there anyway): it stays empty (T = 1, no contributor); a tile with
    // no open pixel is left empty as a whole.  With a stale saturation state the pixel
    // set is the one the state names (ranks below the pixel's state)
    if (b.sat) {
      const uint8_t* sp = b.sat[ti.v];
      const int rk = b.rank[ti.v * b.K + ti.k];
#pragma unroll
      for (int i = 0; i < PPT; ++i)
        if ((live >> i) & 1u &&
            !((int)sp[(int64_t)(ti.y + 4 * slot_row<PPT>(i)) * ti.W + ti.x + 8 * slot_col<PPT>(i)] >
              rk))
          live &= ~(1u << i);
    } else {
      const float* tp = b.tpre + b.pix_off[ti.v];
#pragma unroll
      for (int i = 0; i < PPT; ++i)
        if ((live >> i) & 1u &&
            !(tp[(int64_t)(ti.y + 4 * slot_row<PPT>(i)) * ti.W + ti.x + 8 * slot_col<PPT>(i)] >=
              b.eps_comp))
          live &= ~(1u << i);
    }
    if (!__syncthreads_or(live != 0)) {
      if (kCount && threadIdx.x == 0 && b.counters) {
        atomicAdd(b.counters + 6, 1ull);
        atomicAdd(b.counters + 10, (unsigned long long)len);
      }
      const ImgDev im = b.imgs[ti.v * b.K + ti.k];
      const int64_t HW = (int64_t)ti.W * ti.H;
#pragma unroll
      for (int i = 0; i < PPT; ++i) {
        if (!((inb >> i) & 1u)) continue;
        const int64_t p = (int64_t)(ti.y + 4 * slot_row<PPT>(i)) * ti.W + ti.x + 8 * slot_col<PPT>(i);
        im.rgb[p] = 0.0f;
        im.rgb[HW + p] = 0.0f;
        im.rgb[2 * HW + p] = 0.0f;
        im.T[p] = 1.0f;
        im.D[p] = 0.0f;
        im.last[p] = -1;
      }
      return;
    }
  }
  // with no selected prefix (kSelNone) the item goes straight to the full sort and its
  // second forward (a selected prefix needs nothing here: its range points into keys_alt)
  // The item's id, if its list is a selected prefix, waits in shared memory for the end of
  // the walk (no register held across it).  A second forward after a prefix (kSelResume)
  // takes the pixels' state from the planes the first one wrote and walks the whole
  // sorted list from the prefix's end: its first entries are the prefix's, in its order.
  __shared__ uint32_t s_prefix_item;
  uint32_t walk0 = 0;  // list position where the walk begins
  if (b.sel) {
    const uint32_t sv = b.sel[id];
    if (sv == kSelNone) {
      // (hand_back rewrites sel[id] and ranges[id]: not before every warp has read them, or a
      // late one would take the unsorted segment for a sorted list.  sv is the same for the
      // whole CTA, so all its threads meet here)
      __syncthreads();
      if (threadIdx.x == 0) {
        hand_back(b, (uint32_t)id, kSelNone);
        if (kCount && b.counters) atomicAdd(b.counters + 9, 1ull);
      }
      return;
    }
    if (sv & kSelResume) {
      walk0 = sv & ~kSelResume;
      const ImgDev im = b.imgs[ti.v * b.K + ti.k];
      const int64_t HW = (int64_t)ti.W * ti.H;
#pragma unroll
      for (int i = 0; i < PPT; ++i) {
        const int px = ti.x + 8 * slot_col<PPT>(i), py = ti.y + 4 * slot_row<PPT>(i);
        if (px >= ti.W || py >= ti.H) continue;
        const int64_t p = (int64_t)py * ti.W + px;
        c0[i] = im.rgb[p];
        c1[i] = im.rgb[HW + p];
        c2[i] = im.rgb[2 * HW + p];
        T[i] = im.T[p];
        D[i] = im.D[p];
        const int l = im.last[p];
        last[i] = l <= -2 ? -3 - l : l;
        if (l <= -2) live &= ~(1u << i);  // it had stopped inside the prefix
      }
    }
    if (threadIdx.x == 0) s_prefix_item = sv && !(sv & kSelResume) ? (uint32_t)id : kSelNone;
  }
  unsigned n_eval = 0, n_pix = 0, n_blend = 0;
  const int lane = (int)(threadIdx.x & 31);
  const int RX = ti.x - (lane & 7), RY = ti.y - (lane >> 3);  // the warp's region
  float* ring = sR + (threadIdx.x >> 5) * (kRingItems / 2 * kPairWords);
  unsigned tail = 0, head = 0;  // ring positions: appended, processed
  const float lg_amin = __log2f(amin);
  // (alpha is compared before its clamp: with amin above amax nothing may pass)
  const float amin_raw = amin <= amax ? amin : __int_as_float(0x7f800000);
  // a pixel's bit pair in the items' masks; kDeadPixel (which no item has) once it is done
  uint32_t pm[PPT];
#pragma unroll
  for (int i = 0; i < PPT; ++i)
    pm[i] = (live >> i) & 1u ? (1u << (8 + (lane & 7) + 8 * slot_col<PPT>(i))) |
                                   (1u << (24 + (lane >> 3) + 4 * slot_row<PPT>(i)))
                             : kDeadPixel;
  auto alive = [&]() {
    bool any = false;
#pragma unroll
    for (int i = 0; i < PPT; ++i) any |= pm[i] != kDeadPixel;
    return any;
  };
  // Blends ring entries head and head + 1.  Both entries' alphas are evaluated at every
  // pixel of the lane (packed over the two entries) and are 0 where the pixel does not take
  // the entry, which leaves T as it is bit for bit.
  auto blend_pair = [&]() {
    const float4* q = reinterpret_cast<const float4*>(ring + ((head & (kRingItems - 1)) >> 1) * kPairWords);
    const float4 P0 = q[0], P1 = q[1], P2 = q[2], CA = q[3], CB = q[4], MJ = q[5];
    const uint32_t m0 = __float_as_uint(MJ.x), m1 = __float_as_uint(MJ.y);
    const int j0 = __float_as_int(MJ.z), j1 = __float_as_int(MJ.w);
    const f32x2 u2 = pack2(P0.x, P0.y), v2 = pack2(P0.z, P0.w), qa2 = pack2(P1.x, P1.y),
                qb2 = pack2(P1.z, P1.w), qc2 = pack2(P2.x, P2.y), o2 = pack2(P2.z, P2.w);
    const f32x2 dy2[2] = {sub2(pcy0, v2), sub2(pcy1, v2)};
    head += 2;
    if (kCount && lane == 0) n_eval += 2u;
    // a column of blocks (two slots) at a time; of a 16 x 8 region's two, those that the pair's
    // rectangles meet (a small Gaussian meets one: 32x32 tiles, the 2M step 3.91 -> 3.65 ms,
    // 3M Gaussians of a pixel or less 2.15 -> 1.96; a test per slot spilled and took 5.4)
#pragma unroll
    for (int c = 0; c < NC; ++c) {
      if (NC > 1 && (((m0 | m1) >> (8 + 8 * c)) & 0xFFu) == 0u) continue;
      const f32x2 dx2 = sub2(c ? pcx1 : pcx0, u2);
      const f32x2 hx2 = mul2(mul2(qa2, dx2), dx2), bx2 = mul2(qb2, dx2);
      float al0[2], al1[2], T0[2], T1[2];
      bool ok0[2], ok1[2];
      float tmin = __int_as_float(0x7f800000);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int i = NC * r + c;
        const f32x2 dy = dy2[r];
        const f32x2 p2 = fma2(fma2(qc2, dy, bx2), dy, hx2);
        float p0, p1, r0, r1;
        unpack2(p2, p0, p1);
        unpack2(mul2(o2, pack2(ex2_approx(p0), ex2_approx(p1))), r0, r1);
        const bool in0 = (~m0 & pm[i]) == 0u, in1 = (~m1 & pm[i]) == 0u;
        ok0[r] = in0 && p0 <= 0.0f && r0 >= amin_raw;
        ok1[r] = in1 && p1 <= 0.0f && r1 >= amin_raw;
        if (kCount) n_pix += (unsigned)in0 + (unsigned)in1;
        al0[r] = ok0[r] ? fminf(r0, amax) : 0.0f;
        al1[r] = ok1[r] ? fminf(r1, amax) : 0.0f;
        T0[r] = T[i] * (1.0f - al0[r]);
        T1[r] = T0[r] * (1.0f - al1[r]);
        tmin = fminf(tmin, T1[r]);
      }
      if (__any_sync(0xffffffffu, tmin < epsT)) {
        // a pixel stops before the entry that would take it below eps_T: that entry and what
        // follows leave it as it is
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          const int i = NC * r + c;
          const bool s0 = ok0[r] && T0[r] < epsT;
          const bool s1 = s0 || (ok1[r] && T1[r] < epsT);
          ok0[r] = ok0[r] && !s0;
          ok1[r] = ok1[r] && !s1;
          T0[r] = s0 ? T[i] : T0[r];
          T1[r] = s1 ? T0[r] : T1[r];
          al0[r] = s0 ? 0.0f : al0[r];
          al1[r] = s1 ? 0.0f : al1[r];
          pm[i] = s1 ? kDeadPixel : pm[i];
        }
      }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        const int i = NC * r + c;
        const float w0 = al0[r] * T[i], w1 = al1[r] * T0[r];
        T[i] = T1[r];
        if (ok0[r]) {
          c0[i] = fmaf(CA.x, w0, c0[i]);
          c1[i] = fmaf(CA.y, w0, c1[i]);
          c2[i] = fmaf(CA.z, w0, c2[i]);
          D[i] = fmaf(CA.w, w0, D[i]);
        }
        if (ok1[r]) {
          c0[i] = fmaf(CB.x, w1, c0[i]);
          c1[i] = fmaf(CB.y, w1, c1[i]);
          c2[i] = fmaf(CB.z, w1, c2[i]);
          D[i] = fmaf(CB.w, w1, D[i]);
        }
        last[i] = ok0[r] ? j0 : last[i];
        last[i] = ok1[r] ? j1 : last[i];
        if (kCount) n_blend += (unsigned)ok0[r] + (unsigned)ok1[r];
      }
    }
  };
  bool open = alive();
  // Batches of NB entries, double-buffered: while the warps blend one, the next one's
  // records are copied behind it (cp.async; its keys were read one batch earlier still), so
  // one barrier per batch both publishes the batch and frees the other buffer.
  uint32_t nk[PER];
  auto load_keys = [&](uint32_t base) {
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const uint32_t j = base + r * NTH + threadIdx.x;
      nk[r] = j < len ? (uint32_t)b.keys[(uint64_t)start + j] : 0u;  // low half: the Gaussian
    }
  };
  auto copy_records = [&](uint32_t base, int buf) {
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const uint32_t slot = r * NTH + threadIdx.x;
      if (slot < NB && base + slot < len) {
        uint32_t g = nk[r];
        if (g >= (uint32_t)b.N) { atomicOr(b.status, ST_BOUNDS); g = 0; }
        const Rec* rp = b.rec + ((int64_t)ti.v * b.N + g);
        cp_async16(sA + buf * NB + slot, &rp->a);
        cp_async16(sB + buf * NB + slot, &rp->b);
        cp_async16(sC + buf * NB + slot, &rp->c);
      }
    }
    cp_async_commit();
  };
  if (walk0 < len) {
    load_keys(walk0);
    copy_records(walk0, 0);
    load_keys(walk0 + NB < len ? walk0 + NB : len);
  }
  int buf = 0;
  for (uint32_t base = walk0; base < len; base += NB, buf ^= 1) {
    // the thread's own records have landed: the rectangles become the tile's column and row
    // masks
    cp_async_wait<0>();
#pragma unroll
    for (int r = 0; r < PER; ++r) {
      const uint32_t slot = r * NTH + threadIdx.x;
      if (slot < NB && base + slot < len) {
        float* px = &sB[buf * NB + slot].w;
        float* py = &sC[buf * NB + slot].w;
        const uint32_t rx = __float_as_uint(*px), ry = __float_as_uint(*py);
        const int x0 = max((int)(rx & 0xFFFFu) - ti.tx * TS, 0), x1 = min((int)(rx >> 16) - ti.tx * TS, TS - 1);
        const int y0 = max((int)(ry & 0xFFFFu) - ti.ty * TS, 0), y1 = min((int)(ry >> 16) - ti.ty * TS, TS - 1);
        *px = __uint_as_float(x0 <= x1 ? ((2u << (x1 - x0)) - 1u) << x0 : 0u);
        *py = __uint_as_float(y0 <= y1 ? ((2u << (y1 - y0)) - 1u) << y0 : 0u);
      }
    }
    if (__syncthreads_count(!open) == NTH) break;
    const bool fin = len - base <= NB;
    if (!fin) {
      copy_records(base + NB, buf ^ 1);
      load_keys(len - base > 2 * NB ? base + 2 * NB : len);
    }
    const int cnt = (int)(fin ? len - base : NB);
    for (int e0 = 0; e0 < cnt; e0 += 32) {
      if (!__any_sync(0xffffffffu, open)) break;
      tail = append_group<PPT>(sA + buf * NB, sB + buf * NB, sC + buf * NB, e0, cnt, (int)base,
                               RX, RY, RX - ti.tx * TS, RY - ti.ty * TS, lane, lg_amin, ring,
                               tail);
      const bool flush = fin && e0 + 32 >= cnt;
      if (flush && ((tail - head) & 1u)) {
        // an entry of zeros that no pixel takes beside the last one
        float* q = ring + ((tail & (kRingItems - 1)) >> 1) * kPairWords;
        if (lane < 12) q[lane >= 6 && lane < 10 ? 10 + lane : 2 * lane + 1] = 0.0f;
        ++tail;
      }
      __syncwarp();
      // (fewer than half a ring stay for the next group, which so always fits)
      if (flush || tail - head >= kRingItems / 2) {
        while (tail - head >= 2u) {
          blend_pair();
          if ((head & 7u) == 0u && !__any_sync(0xffffffffu, alive())) break;
        }
        __syncwarp();
        open = alive();
      }
    }
  }
  cp_async_wait<0>();  // (a batch in flight when the walk ended early)
  live = 0;
#pragma unroll
  for (int i = 0; i < PPT; ++i) live |= pm[i] != kDeadPixel ? 1u << i : 0u;
  if (kCount) {
    flush_counter(b.counters, 0, n_eval);
    flush_counter(b.counters, 1, n_pix);
    flush_counter(b.counters, 2, n_blend);
  }
  const ImgDev im = b.imgs[ti.v * b.K + ti.k];
  const int64_t HW = (int64_t)ti.W * ti.H;
#pragma unroll
  for (int i = 0; i < PPT; ++i) {
    const int px = ti.x + 8 * slot_col<PPT>(i), py = ti.y + 4 * slot_row<PPT>(i);
    if (px >= ti.W || py >= ti.H) continue;
    const int64_t p = (int64_t)py * ti.W + px;
    im.rgb[p] = c0[i];
    im.rgb[HW + p] = c1[i];
    im.rgb[2 * HW + p] = c2[i];
    im.T[p] = T[i];
    im.D[p] = D[i];
    im.last[p] = last[i];
  }
  if (b.sel) {
    // a walk that ended inside a sorted prefix is exact unless a pixel is still blending, in
    // which case the entries after the prefix matter in their sorted order (the barrier
    // also publishes s_prefix_item)
    const bool more = __syncthreads_or(live != 0);
    const uint32_t pid = s_prefix_item;
    if (pid != kSelNone) {
      if (threadIdx.x == 0 && kCount && b.counters) atomicAdd(b.counters + 8, 1ull);
      if (more) {
        if (threadIdx.x == 0) {
          hand_back(b, pid, b.sel[pid]);
          if (kCount && b.counters) atomicAdd(b.counters + 9, 1ull);
        }
        // the planes hold the state at the prefix's end for the second forward: a pixel
        // that has stopped keeps its last index as -3 - last
#pragma unroll
        for (int i = 0; i < PPT; ++i) {
          const int px = ti.x + 8 * slot_col<PPT>(i), py = ti.y + 4 * slot_row<PPT>(i);
          if (px < ti.W && py < ti.H && !((live >> i) & 1u))
            im.last[(int64_t)py * ti.W + px] = -3 - last[i];
        }
        return;  // the second forward writes the prefix transmittance and the planes
      }
      if (threadIdx.x == 0 && kCount && b.counters) {
        uint32_t s, e;
        segment_of(b, pid, s, e);
        atomicAdd(b.counters + 11, (unsigned long long)(e - s));
      }
    }
  }
  if (b.order) {
#pragma unroll
    for (int i = 0; i < PPT; ++i) {
      const int px = ti.x + 8 * slot_col<PPT>(i), py = ti.y + 4 * slot_row<PPT>(i);
      if (px >= ti.W || py >= ti.H) continue;
      float* tp = b.tpre + b.pix_off[ti.v] + (int64_t)py * ti.W + px;
      *tp = wave == 0 ? T[i] : *tp * T[i];
    }
  }
}

// The backward's shared memory of one warp (an 8 x 8 block of pixels).
//   ring  items that can reach the block, two side by side (kBwdPair words per pair):
//         [u0 u1 v0 v1] [qa0 qa1 qb0 qb1] [qc0 qc1 o0 o1] [r0 r0 g0 g0] [b0 b0 m0 j0]
//         [r1 r1 g1 g1] [b1 b1 m1 j1]   (m: columns in bits 0-7, rows in bits 8-15 of the
//         block that the rectangle spans; j: position in the tile's list)
//   part  per item of a group of eight and lane: (ge, ge', aT, aT') of the lane's two pixels
//   qxy, qz  the composite adjoint of the block's pixels: (x, x', y, y'), (z, z') per lane
constexpr int kBwdRing = 40, kBwdPair = 28, kBwdGroup = 8, kPartStride = 36;
struct BwdShared {
  float ring[kBwdRing / 2 * kBwdPair];
  float4 raw[3][32];
  float4 part[kBwdGroup * kPartStride];
  float4 qxy[32];
  float2 qz[32];
  uint32_t gid[kBwdRing];
};

// The backward of one 8 x 8 block of a work item, one warp.  It is bound by instruction issue
// and by shared memory (69 % of the issue slots, 76 % of the shared-memory pipe, DRAM idle).
// The list's entries that can reach the block are taken back to front in groups of eight, in
// two halves: first each lane runs the recurrences of its two pixels over the eight items
// and leaves (dL/dpower / o, alpha T) per item and pixel in shared memory; then four lanes per
// item sum the item's parts over the pixels, so the nine sums take two shuffles each for
// eight items at once (18 for a group) and no atomics but three per item and block.  Before,
// one warp held a whole 16x16 tile, 8 pixels a lane, branched per 8 x 4 block and reduced
// nine sums over its 32 lanes for every entry (some 50 instructions) or let up to 20 lanes
// add their own.  2M Gaussians, 4 views, 8 subsets: 2.75 -> 2.08 ms at 16x16 tiles, 2.90 ->
// 2.12 at 8x8, 4.55 -> 2.34 at 32x32; the 10M step's 17.5 -> 13.0 ms, the city's 3.6 ->
// 2.32 ms.  Measured beside it, when it took 2.15 ms: the one-warp tile with the packed
// arithmetic and box tests alone 2.51 ms; one-warp CTAs 2.21 ms (the city 3.66: siblings share records in L1); the
// group's four pairs not unrolled 2.22 ms; one warp taking a tile's four blocks in turn,
// batch by batch, 2.41 ms (0.211 ms on 560 tiles).
// kSync: the tile's warps take the batches of 32 entries together and leave their sums per
// batch slot here; the CTA then adds them in the order of the warps, one add per tile.
struct BwdSums {
  float acc[2][4][32][9];  // two batches alternate, so that one barrier per batch is enough
  unsigned have[2][4];      // per warp, the slots it has sums for
  int maxlast;
};

template <int TS, bool kSync, bool kCount>
__device__ __forceinline__ void bwd_item(const BatchDev& b, const int64_t id, const int blk,
                                         BwdShared& sh, BwdSums* cta) {
  const TileInfo ti = decode_tile<TS, 2>(b, id);
  if (!in_omega(b, ti.v, ti.k, ti.tx, ti.ty)) return;  // nothing written there, nothing to do
  const int lane = (int)(threadIdx.x & 31);
  const uint2 rg = b.ranges[id];  // (a selected prefix's range points into keys_alt)
  const uint32_t start = rg.x;
  const int len = rg.y > rg.x ? (int)(rg.y - rg.x) : 0;
  if (len == 0) return;
  // the warp's block: RX, RY its origin on the image
  const int RX = ti.tx * TS + 8 * (blk % (TS / 8)), RY = ti.ty * TS + 8 * (blk / (TS / 8));
  const int x = RX + (lane & 7), y = RY + (lane >> 3);  // the lane's pixels: (x, y), (x, y + 4)
  // Lane l holds entry top - l of each batch of 32: its record is copied behind the batch
  // before (cp.async), its key (low half: the Gaussian) read one batch earlier still.  The
  // walk of a list of at most 32 entries starts at its end, not at the pixels' last
  // contributor (entries behind that are left out), so that its keys are on their way while
  // the pixels' state is read: a short list's time is the latency of its reads, one behind
  // the other.  500k Gaussians in 16 overlapping subsets, 2 views 1600x1064 (lists of tens):
  // 1.84 -> 1.69 ms, in 40 subsets 2.82 -> 2.51; the 2M step 2.29 -> 2.22.
  const bool whole = len <= 32;
  int top = len - 1;  // list position of the batch's first entry
  uint32_t nk = 0;
  auto load_key = [&](int j) { nk = j >= 0 ? (uint32_t)b.keys[(uint64_t)start + j] : 0u; };
  auto copy_record = [&](int j) {
    if (j >= 0) {
      if (nk >= (uint32_t)b.N) { atomicOr(b.status, ST_BOUNDS); nk = 0; }
      const Rec* rp = b.rec + ((int64_t)ti.v * b.N + nk);
      cp_async16(&sh.raw[0][lane], &rp->a);
      cp_async16(&sh.raw[1][lane], &rp->b);
      cp_async16(&sh.raw[2][lane], &rp->c);
    }
    cp_async_commit();
  };
  if (whole) load_key(top - lane);
  const float amax = b.alpha_max;
  const float amin_raw = b.alpha_min <= amax ? b.alpha_min : __int_as_float(0x7f800000);
  const float lg_amin = __log2f(b.alpha_min);
  // W = -T^m dL/dT^m - sum_ch dL/dC^m_ch B_ch: the colour suffix sums B enter the alpha
  // adjoint only through this dot product, so one scalar per pixel carries them
  f32x2 T2, W2, qx, qy, qz;
  int last0, last1;
  bool wild;  // an adjoint so large that 0 x (its products) might not be 0
  {
    const ImgDev& im = b.imgs[ti.v * b.K + ti.k];
    float Tm[2], Wm[2];
    float4 g[2];
    int last[2];
    wild = false;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      g[h] = make_float4(0.f, 0.f, 0.f, 0.f);
      Tm[h] = 1.0f;
      last[h] = -1;
      if (x < ti.W && y + 4 * h < ti.H) {
        const int64_t p = (int64_t)(y + 4 * h) * ti.W + x;
        g[h] = im.gCT[p];
        Tm[h] = im.T[p];
        last[h] = im.last[p];
        if (g[h].x == 0.0f && g[h].y == 0.0f && g[h].z == 0.0f && g[h].w == 0.0f) last[h] = -1;
      }
      Wm[h] = -Tm[h] * g[h].w;
      wild |= !(fabsf(g[h].x) <= kWild) || !(fabsf(g[h].y) <= kWild) ||
              !(fabsf(g[h].z) <= kWild) || !(fabsf(g[h].w) <= kWild);
    }
    last0 = last[0];
    last1 = last[1];
    T2 = pack2(Tm[0], Tm[1]);
    W2 = pack2(Wm[0], Wm[1]);
    qx = pack2(g[0].x, g[1].x);
    qy = pack2(g[0].y, g[1].y);
    qz = pack2(g[0].z, g[1].z);
    sh.qxy[lane] = make_float4(g[0].x, g[1].x, g[0].y, g[1].y);
    sh.qz[lane] = make_float2(g[0].z, g[1].z);
  }
  const int mylast = __reduce_max_sync(0xffffffffu, max(last0, last1));
  int maxlast = mylast;
  if (kSync) {
    if (threadIdx.x == 0) cta->maxlast = -1;
    __syncthreads();
    if (lane == 0 && mylast >= 0) atomicMax(&cta->maxlast, mylast);
    __syncthreads();
    maxlast = cta->maxlast;
  }
  if (maxlast < 0) return;
  if (!whole) {
    top = maxlast;
    load_key(top - lane);
  }
  copy_record(top - lane);
  uint32_t g = nk;
  load_key(top - 32 - lane);
  bool careful = __any_sync(0xffffffffu, wild);
  const uint32_t pm0 = (1u << (lane & 7)) | (1u << (8 + (lane >> 3))),
                 pm1 = (1u << (lane & 7)) | (1u << (12 + (lane >> 3)));
  const f32x2 pcx2 = pack2((float)x + 0.5f, (float)x + 0.5f),
              pcya = pack2((float)y + 0.5f, (float)y + 0.5f),
              pcyb = pack2((float)(y + 4) + 0.5f, (float)(y + 4) + 0.5f);
  const f32x2 one2 = pack2(1.0f, 1.0f), neg2 = pack2(-1.0f, -1.0f);
  unsigned n_evalb = 0, n_pixb = 0, n_actb = 0;

  // First half of a group: the pair of ring items at index ri, as items e and e + 1 of the
  // group, against the lane's two pixels.  The exponents are packed over the two items, the
  // recurrences of T and W over the two pixels; a pixel that does not take an item has alpha
  // 0, which leaves T and W as they are (1/1 is exact), and e^power 0.
  auto take_pair = [&](int ri, int e) {
    const float4* q = reinterpret_cast<const float4*>(sh.ring + (ri >> 1) * kBwdPair);
    const float4 P0 = q[0], P1 = q[1], P2 = q[2];
    const f32x2 dx = sub2(pcx2, pack2(P0.x, P0.y));
    const f32x2 hx = mul2(mul2(pack2(P1.x, P1.y), dx), dx), bx = mul2(pack2(P1.z, P1.w), dx);
    const f32x2 dya = sub2(pcya, pack2(P0.z, P0.w)), dyb = sub2(pcyb, pack2(P0.z, P0.w));
    const f32x2 qc2 = pack2(P2.x, P2.y), o2 = pack2(P2.z, P2.w);
    float pa[2], pb[2], ra[2], rb[2], ea[2], eb[2];  // per item: pixel a, pixel b
    unpack2(fma2(fma2(qc2, dya, bx), dya, hx), pa[0], pa[1]);
    unpack2(fma2(fma2(qc2, dyb, bx), dyb, hx), pb[0], pb[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) { ea[h] = ex2_approx(pa[h]); eb[h] = ex2_approx(pb[h]); }
    unpack2(mul2(o2, pack2(ea[0], ea[1])), ra[0], ra[1]);
    unpack2(mul2(o2, pack2(eb[0], eb[1])), rb[0], rb[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float4 K0 = q[3 + 2 * h], K1 = q[4 + 2 * h];
      const uint32_t nm = ~__float_as_uint(K1.z);
      const int j = __float_as_int(K1.w);
      const bool ina = (nm & pm0) == 0u && j <= last0, inb = (nm & pm1) == 0u && j <= last1;
      const bool oka = ina && pa[h] <= 0.0f && ra[h] >= amin_raw;
      const bool okb = inb && pb[h] <= 0.0f && rb[h] >= amin_raw;
      if (kCount) {
        n_pixb += (unsigned)ina + (unsigned)inb;
        n_actb += (unsigned)oka + (unsigned)okb;
      }
      const f32x2 al = pack2(oka ? fminf(ra[h], amax) : 0.0f, okb ? fminf(rb[h], amax) : 0.0f);
      // (dL/dpower is 0 where alpha is clamped)
      const f32x2 em = pack2(oka && ra[h] <= amax ? ea[h] : 0.0f, okb && rb[h] <= amax ? eb[h] : 0.0f);
      float oa, ob;
      unpack2(sub2(one2, al), oa, ob);
      const f32x2 rinv = pack2(rcp_approx(oa), rcp_approx(ob));
      const f32x2 Ti = mul2(T2, rinv);
      const f32x2 aT = mul2(al, Ti);
      f32x2 qc = fma2(qz, pack2(K1.x, K1.y),
                      fma2(qy, pack2(K0.z, K0.w), mul2(qx, pack2(K0.x, K0.y))));  // dL/dC^m . c_i
      f32x2 ga = fma2(Ti, qc, mul2(W2, rinv));                                    // dL/dalpha_i
      if (careful) {
        // products that may overflow: nothing of a pixel that does not take the item, no
        // dL/dpower where alpha is clamped
        float u, w;
        unpack2(qc, u, w);
        qc = pack2(oka ? u : 0.0f, okb ? w : 0.0f);
        unpack2(ga, u, w);
        ga = pack2(oka && ra[h] <= amax ? u : 0.0f, okb && rb[h] <= amax ? w : 0.0f);
      }
      W2 = fma2(mul2(qc, neg2), aT, W2);
      T2 = Ti;
      float g0, g1, t0, t1;
      unpack2(mul2(ga, em), g0, g1);
      unpack2(aT, t0, t1);
      sh.part[(e + h) * kPartStride + lane] = make_float4(g0, g1, t0, t1);
    }
  };

  // Second half: four lanes per item sum its parts over the block's pixels (16 each, two
  // columns) and add them to its 2-D gradient: the moments sum ge, ge dx, ge dy, ge dx^2,
  // ge dx dy, ge dy^2 (ge = dL/dpower / o = dL/do e^power) and dL/dcolour; the projection
  // adjoint applies the conic and the opacity.
  auto sum_group = [&](int ri, int cnt) {
    const int e = lane >> 2, qd = lane & 3;
    const float* r = sh.ring + ((ri + e) >> 1) * kBwdPair + ((ri + e) & 1);
    const float u = r[0], v = r[2];
    const float dxa = ((float)(RX + qd) + 0.5f) - u, dxb = ((float)(RX + qd + 4) + 0.5f) - u;
    const float4* part = sh.part + e * kPartStride + qd;
    f32x2 a0 = 0, a1 = 0, a2 = 0, b0 = 0, b1 = 0, b2 = 0, gr = 0, gg = 0, gb = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const f32x2 dy = sub2(pack2((float)(RY + i) + 0.5f, (float)(RY + i + 4) + 0.5f), pack2(v, v));
      const f32x2 dyy = mul2(dy, dy);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const float4 s = part[8 * i + 4 * c], q4 = sh.qxy[8 * i + 4 * c + qd];
        const float2 q2 = sh.qz[8 * i + 4 * c + qd];
        const f32x2 ge = pack2(s.x, s.y), aT = pack2(s.z, s.w);
        if (c == 0) {
          a0 = add2(a0, ge);
          a1 = fma2(ge, dy, a1);
          a2 = fma2(ge, dyy, a2);
        } else {
          b0 = add2(b0, ge);
          b1 = fma2(ge, dy, b1);
          b2 = fma2(ge, dyy, b2);
        }
        f32x2 x2 = pack2(q4.x, q4.y), y2 = pack2(q4.z, q4.w), z2 = pack2(q2.x, q2.y);
        if (careful) {
          const bool k0 = s.z != 0.0f, k1 = s.w != 0.0f;
          x2 = pack2(k0 ? q4.x : 0.0f, k1 ? q4.y : 0.0f);
          y2 = pack2(k0 ? q4.z : 0.0f, k1 ? q4.w : 0.0f);
          z2 = pack2(k0 ? q2.x : 0.0f, k1 ? q2.y : 0.0f);
        }
        gr = fma2(x2, aT, gr);
        gg = fma2(y2, aT, gg);
        gb = fma2(z2, aT, gb);
      }
    }
    auto both = [](f32x2 w) {
      float lo, hi;
      unpack2(w, lo, hi);
      return lo + hi;
    };
    const float A0 = both(a0), A1 = both(a1), B0 = both(b0), B1 = both(b1);
    float w[9] = {dxa * A0 + dxb * B0, A1 + B1, dxa * dxa * A0 + dxb * dxb * B0,
                  dxa * A1 + dxb * B1, both(a2) + both(b2), A0 + B0, both(gr), both(gg), both(gb)};
    uint32_t any = 0;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
      w[i] += __shfl_xor_sync(0xffffffffu, w[i], 1);
      w[i] += __shfl_xor_sync(0xffffffffu, w[i], 2);
      any |= __float_as_uint(w[i]);
    }
    if (kSync) {
      if (qd == 0 && e < cnt) {
        const float* c = sh.ring + ((ri + e) >> 1) * kBwdPair + 12 + 8 * ((ri + e) & 1);
        float* dst = cta->acc[(top >> 5) & 1][threadIdx.x >> 5][top - __float_as_int(c[7])];
#pragma unroll
        for (int i = 0; i < 9; ++i) dst[i] = w[i];
      }
    } else if (qd == 0 && e < cnt && (any << 1) != 0u) {  // (nothing to add where no pixel took it)
      float4* dst = b.grad2d + ((int64_t)ti.v * b.N + sh.gid[ri + e]) * 3;
      atomicAdd(dst, make_float4(w[0], w[1], w[2], w[3]));
      atomicAdd(dst + 1, make_float4(w[4], w[5], w[6], w[7]));
      atomicAdd(&dst[2].x, w[8]);
    }
  };

  int head = 0, have = 0;  // ring index of the next group, items in the ring
  for (; top >= 0; top -= 32) {
    cp_async_wait<0>();
    // append the lane's entry if it can reach a pixel of the block
    uint32_t m = 0;
    float4 A, B, C;
    if (top - lane >= 0 && top - lane <= mylast) {
      A = sh.raw[0][lane];
      B = sh.raw[1][lane];
      C = sh.raw[2][lane];
      const uint32_t rx = __float_as_uint(B.w), ry = __float_as_uint(C.w);
      const int c0 = max((int)(rx & 0xFFFFu) - RX, 0), c1 = min((int)(rx >> 16) - RX, 7);
      const int r0 = max((int)(ry & 0xFFFFu) - RY, 0), r1 = min((int)(ry >> 16) - RY, 7);
      const float X0 = ((float)RX + 0.5f) - A.x, Y0 = ((float)RY + 0.5f) - A.y;
      if (c0 <= c1 && r0 <= r1 &&
          box_reached(A.z, A.w, B.x, B.y, X0, X0 + 7.0f, Y0, Y0 + 7.0f, lg_amin))
        m = (((2u << (c1 - c0)) - 1u) << c0) | ((((2u << (r1 - r0)) - 1u) << r0) << 8);
    }
    const unsigned hit = __ballot_sync(0xffffffffu, m != 0u);
    bool big = false;
    if (m) {
      int pos = head + have + __popc(hit & ((1u << lane) - 1u));
      pos = pos >= kBwdRing ? pos - kBwdRing : pos;
      float* q = sh.ring + (pos >> 1) * kBwdPair;
      const int h = pos & 1;
      q[h] = A.x;
      q[2 + h] = A.y;
      q[4 + h] = A.z;
      q[6 + h] = A.w;
      q[8 + h] = B.x;
      q[10 + h] = B.y;
      float4* c4 = reinterpret_cast<float4*>(q + 12) + 2 * h;
      c4[0] = make_float4(C.x, C.x, C.y, C.y);
      c4[1] = make_float4(C.z, C.z, __uint_as_float(m), __int_as_float(top - lane));
      sh.gid[pos] = g;
      big = !(C.x <= kWild) || !(C.y <= kWild) || !(C.z <= kWild);
    }
    careful = __any_sync(0xffffffffu, big) || careful;
    have += __popc(hit);
    const uint32_t g_batch = g;
    copy_record(top - 32 - lane);
    g = nk;
    load_key(top - 64 - lane);
    if (kCount && lane == 0) n_evalb += (unsigned)__popc(hit);
    const bool fin = kSync || top < 32;  // take what is in the ring whole
    if (fin && (have & 1)) {
      // an item of zeros that no pixel takes beside the last one (a group starts at an even
      // index, so the last one is the first of its pair)
      int pos = head + have;
      pos = pos >= kBwdRing ? pos - kBwdRing : pos;
      float* q = sh.ring + (pos >> 1) * kBwdPair;
      if (lane < 6) q[2 * lane + 1] = 0.0f;
      else if (lane < 14) q[14 + lane] = 0.0f;
    }
    __syncwarp();
    while (have >= kBwdGroup || (fin && have > 0)) {
      const int cnt = have < kBwdGroup ? have : kBwdGroup;
#pragma unroll 4
      for (int e = 0; e < cnt; e += 2) take_pair(head + e, e);
      __syncwarp();
      sum_group(head, cnt);
      __syncwarp();
      head = head + kBwdGroup == kBwdRing ? 0 : head + kBwdGroup;
      have -= cnt;
    }
    if (kSync) {
      const int par = (top >> 5) & 1;
      if (lane == 0) cta->have[par][threadIdx.x >> 5] = hit;
      __syncthreads();
      // four threads per slot, one per part of the record
      const int slot = (int)(threadIdx.x >> 2), part = (int)(threadIdx.x & 3);
      const uint32_t gs = __shfl_sync(0xffffffffu, g_batch, slot);
      float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
      if (part < 3) {
#pragma unroll
        for (int w = 0; w < 4; ++w)
          if ((cta->have[par][w] >> slot) & 1u) {
            const float* a = cta->acc[par][w][slot] + 4 * part;
            t.x += a[0];
            if (part < 2) { t.y += a[1]; t.z += a[2]; t.w += a[3]; }
          }
        if (t.x != 0.0f || t.y != 0.0f || t.z != 0.0f || t.w != 0.0f) {
          float4* dst = b.grad2d + ((int64_t)ti.v * b.N + gs) * 3 + part;
          if (part < 2) atomicAdd(dst, t);
          else atomicAdd(&dst->x, t.x);
        }
      }
    }
  }
  cp_async_wait<0>();
  if (kCount) {
    flush_counter(b.counters, 3, n_evalb);
    flush_counter(b.counters, 4, n_pixb);
    flush_counter(b.counters, 5, n_actb);
  }
}

// One CTA per work item, or (kPersist) a grid sized to the SMs whose CTAs take work items
// in order from a device counter until none is left.
// Resident forward CTAs its register limits are set for: at 16x16 tiles 8 CTAs of 128
// threads (64 registers; the 26.6 KB of shared memory allow no more), at 32x32 3 of 256
// (80), at 8x8 28 of one warp (72).
template <int TS>
constexpr int kMinBlocksFwd = TS == 16 ? 8 : (TS == 32 ? 3 : 28);

template <int TS, int PPT, bool kCount, bool kPersist>
__global__ void __launch_bounds__(TS * TS / PPT, kMinBlocksFwd<TS>) k_raster_fwd(const BatchDev b) {
  __shared__ float4 sA[2 * kNBFwd<TS>], sB[2 * kNBFwd<TS>], sC[2 * kNBFwd<TS>];
  __shared__ __align__(16) float sR[kRingWords<TS, PPT>];
  if constexpr (!kPersist) {
    fwd_item<TS, PPT, kCount>(b, item_of(b, blockIdx.x), b.wave, sA, sB, sC, sR);
  } else {
    __shared__ long long s_id;
    for (;;) {
      __syncthreads();  // the previous item is done with shared memory and s_id
      if (threadIdx.x == 0) s_id = (long long)atomicAdd(b.work_ctr, 1ull);
      __syncthreads();
      const int64_t id = s_id;
      if (id >= items_of_launch(b)) return;
      fwd_item<TS, PPT, kCount>(b, item_of(b, id), b.wave, sA, sB, sC, sR);
    }
  }
}

// Saturation skipping without waves: a CTA per image tile of a view renders the tile's K
// subsets in the view's order, one after another; the prefix transmittance it reads is the
// one its own threads wrote.  The same items in the same order as the waves, so the same
// results; it needs every segment sorted beforehand, also those that the waves would have
// left unsorted behind saturated tiles, and no selected prefixes (a handed-back item would
// have to be finished before the next).  For scenes whose waves leave little unsorted
// (splx_batch_tune_prefix_sort): 20M Gaussians, 32 subsets, 4 views at 1080p, sorts and
// forward 3.5 ms in 128 launches of each kind, 2.5 ms in three launches.
template <int TS, int PPT, bool kCount>
__global__ void __launch_bounds__(TS * TS / PPT, kMinBlocksFwd<TS>)
    k_raster_fwd_ordered(const BatchDev b) {
  __shared__ float4 sA[2 * kNBFwd<TS>], sB[2 * kNBFwd<TS>], sC[2 * kNBFwd<TS>];
  __shared__ __align__(16) float sR[kRingWords<TS, PPT>];
  const int64_t w = blockIdx.x;
  const int v = view_of(b.tile_base, b.V, w * b.K);
  const int64_t nt = (b.tile_base[v + 1] - b.tile_base[v]) / b.K;
  const int64_t t0 = b.tile_base[v] + (w - b.tile_base[v] / b.K);
  const int32_t* order = b.order + (int64_t)v * b.K;
#pragma unroll 1
  for (int r = 0; r < b.K; ++r) {
    fwd_item<TS, PPT, kCount>(b, t0 + order[r] * nt, r, sA, sB, sC, sR);
    __syncthreads();  // shared memory is free for the next subset
  }
}

// Second forward of the items the first one handed back (b.retry, after their full sort):
// a fixed grid whose CTAs take the list's items in a grid-stride loop (few items, each a
// long walk: no register cap for occupancy).
template <int TS, int PPT, bool kCount>
__global__ void __launch_bounds__(TS * TS / PPT) k_raster_fwd_retry(const BatchDev b) {
  __shared__ float4 sA[2 * kNBFwd<TS>], sB[2 * kNBFwd<TS>], sC[2 * kNBFwd<TS>];
  __shared__ __align__(16) float sR[kRingWords<TS, PPT>];
  const unsigned n = *b.retry_count;
  for (unsigned w = blockIdx.x; w < n; w += gridDim.x) {
    __syncthreads();  // the previous item is done with shared memory
    fwd_item<TS, PPT, kCount>(b, (int64_t)b.retry[w], b.wave, sA, sB, sC, sR);
  }
}

// Backward CTAs: one warp per 8 x 8 block, up to four blocks per CTA (a 32x32 tile takes four
// CTAs); the warps walk the tile's list on their own.
template <int TS>
constexpr int kBwdWarps = TS == 8 ? 1 : 4;
template <int TS>
constexpr int kBwdSplit = TS * TS / 64 / kBwdWarps<TS>;  // CTAs per work item
template <int TS, bool kSync, bool kCount, bool kPersist>
__global__ void __launch_bounds__(32 * kBwdWarps<TS>, kSync ? 4 : kMinBlocksBwd<TS>)
    k_raster_bwd(const BatchDev b) {
  __shared__ BwdShared sh[kBwdWarps<TS>];
  BwdSums* sums = nullptr;
  if constexpr (kSync) {
    __shared__ BwdSums s_sums;
    sums = &s_sums;
  }
  const int w = (int)(threadIdx.x >> 5);
  if constexpr (!kPersist) {
    const unsigned id = blockIdx.x / kBwdSplit<TS>, part = blockIdx.x % kBwdSplit<TS>;
    bwd_item<TS, kSync, kCount>(b, id, (int)part * kBwdWarps<TS> + w, sh[w], sums);
  } else {
    __shared__ long long s_id;
    for (;;) {
      __syncthreads();
      if (threadIdx.x == 0) s_id = (long long)atomicAdd(b.work_ctr + 1, 1ull);
      __syncthreads();
      const int64_t id = s_id / kBwdSplit<TS>, part = s_id % kBwdSplit<TS>;
      if (id >= b.n_tiles) return;
      bwd_item<TS, kSync, kCount>(b, id, (int)part * kBwdWarps<TS> + w, sh[w], sums);
    }
  }
}

// Tile side -> pixels per thread of the forward: 2 (8 x 8 regions per warp) for 8x8 and 16x16
// tiles, 4 (16 x 8) for 32x32.
template <int TS>
struct PptFwd {
  static constexpr int value = TS == 32 ? 4 : 2;
};
// Launches of at most this many 16x16 items take the backward's kSync form, for the sake of
// repeatable sums: a Gaussian whose footprint lies inside one tile (or two: a sum of two adds
// does not depend on their order) gets the same 2-D gradient bit for bit in every run, so that
// small problems come out the same, as they did with a warp per tile.  It costs time: the
// tile's warps wait for each other at every batch.  Larger launches leave each warp to add on
// its own, in any order.  Measured (raster_bwd; a warp per tile | warps on their own | kSync):
// 560 tiles 0.447 | 0.084 | 0.107 ms, 3800 tiles 0.523 | 0.133 | 0.179, 34.7k tiles 1.348 |
// 0.896 | 1.219.
constexpr int64_t kSyncItems = 1024;
// Work is counted only by eager runs with a counter buffer: a captured graph launches the
// plain variants, so replays carry no counting instructions (and keep the eager counts).
static bool counting(const BatchDev& b, cudaStream_t s) {
  return b.counters && !stream_capturing(s);
}

template <int TS, bool kCount, bool kPersist>
static void launch_fwd_k(const BatchDev& b, cudaStream_t s) {
  constexpr int P = PptFwd<TS>::value;
  const int64_t items = b.order ? b.item_n : b.n_tiles;
  const unsigned grid = kPersist ? (unsigned)std::min<int64_t>(items, (int64_t)b.persist_grid)
                                 : (unsigned)items;
  k_raster_fwd<TS, P, kCount, kPersist><<<grid, TS * TS / P, 0, s>>>(b);
}
template <int TS, bool kCount, bool kPersist>
static void launch_bwd_k(const BatchDev& b, cudaStream_t s) {
  const int64_t items = b.n_tiles * kBwdSplit<TS>;
  const unsigned grid = kPersist ? (unsigned)std::min<int64_t>(items, (int64_t)b.persist_grid)
                                 : (unsigned)items;
  if constexpr (TS == 16) {
    if (b.n_tiles <= kSyncItems) {
      k_raster_bwd<TS, true, kCount, kPersist><<<grid, 32 * kBwdWarps<TS>, 0, s>>>(b);
      return;
    }
  }
  k_raster_bwd<TS, false, kCount, kPersist><<<grid, 32 * kBwdWarps<TS>, 0, s>>>(b);
}
template <int TS>
static void launch_fwd_t(const BatchDev& b, cudaStream_t s) {
  const bool c = counting(b, s), p = b.persist_grid > 0 && b.work_ctr;
  if (p) cudaMemsetAsync(b.work_ctr, 0, sizeof(unsigned long long), s);
  if (c) { if (p) launch_fwd_k<TS, true, true>(b, s); else launch_fwd_k<TS, true, false>(b, s); }
  else   { if (p) launch_fwd_k<TS, false, true>(b, s); else launch_fwd_k<TS, false, false>(b, s); }
}
template <int TS>
static void launch_bwd_t(const BatchDev& b, cudaStream_t s) {
  const bool c = counting(b, s), p = b.persist_grid > 0 && b.work_ctr;
  if (p) cudaMemsetAsync(b.work_ctr + 1, 0, sizeof(unsigned long long), s);
  if (c) { if (p) launch_bwd_k<TS, true, true>(b, s); else launch_bwd_k<TS, true, false>(b, s); }
  else   { if (p) launch_bwd_k<TS, false, true>(b, s); else launch_bwd_k<TS, false, false>(b, s); }
}

template <int TS>
static int max_ctas_t(bool bwd) {
  constexpr int PF = PptFwd<TS>::value;
  int n = 0;
  cudaError_t e =
      bwd ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_raster_bwd<TS, false, false, true>,
                                                          32 * kBwdWarps<TS>, 0)
          : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k_raster_fwd<TS, PF, false, true>,
                                                          TS * TS / PF, 0);
  return e == cudaSuccess ? n : 0;
}

int raster_max_ctas_per_sm(int tile, bool bwd) {
  switch (tile) {
    case 8: return max_ctas_t<8>(bwd);
    case 32: return max_ctas_t<32>(bwd);
    default: return max_ctas_t<16>(bwd);
  }
}

void launch_raster_fwd(const BatchDev& b, cudaStream_t s) {
  if (b.n_tiles == 0) return;
  switch (b.tile) {
    case 8: launch_fwd_t<8>(b, s); break;
    case 32: launch_fwd_t<32>(b, s); break;
    default: launch_fwd_t<16>(b, s); break;
  }
  count_launch();
}

template <int TS>
static void launch_fwd_ordered_t(const BatchDev& b, cudaStream_t s) {
  constexpr int P = PptFwd<TS>::value;
  const unsigned grid = (unsigned)(b.n_tiles / b.K);
  if (counting(b, s)) k_raster_fwd_ordered<TS, P, true><<<grid, TS * TS / P, 0, s>>>(b);
  else k_raster_fwd_ordered<TS, P, false><<<grid, TS * TS / P, 0, s>>>(b);
}

void launch_raster_fwd_ordered(const BatchDev& b, cudaStream_t s) {
  if (b.n_tiles == 0) return;
  switch (b.tile) {
    case 8: launch_fwd_ordered_t<8>(b, s); break;
    case 32: launch_fwd_ordered_t<32>(b, s); break;
    default: launch_fwd_ordered_t<16>(b, s); break;
  }
  count_launch();
}

template <int TS>
static void launch_fwd_retry_t(const BatchDev& b, cudaStream_t s) {
  constexpr int P = PptFwd<TS>::value;
  const unsigned grid = (unsigned)device_sm_count() * 2;
  if (counting(b, s)) k_raster_fwd_retry<TS, P, true><<<grid, TS * TS / P, 0, s>>>(b);
  else k_raster_fwd_retry<TS, P, false><<<grid, TS * TS / P, 0, s>>>(b);
}

void launch_raster_fwd_retry(const BatchDev& b, cudaStream_t s) {
  if (!b.sel || b.n_tiles == 0) return;
  switch (b.tile) {
    case 8: launch_fwd_retry_t<8>(b, s); break;
    case 32: launch_fwd_retry_t<32>(b, s); break;
    default: launch_fwd_retry_t<16>(b, s); break;
  }
  count_launch();
}

void launch_raster_bwd(const BatchDev& b, cudaStream_t s) {
  if (b.n_tiles == 0) return;
  switch (b.tile) {
    case 8: launch_bwd_t<8>(b, s); break;
    case 32: launch_bwd_t<32>(b, s); break;
    default: launch_bwd_t<16>(b, s); break;
  }
  count_launch();
}

}  // namespace splx
