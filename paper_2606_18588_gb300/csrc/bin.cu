// Binning and per-tile depth sort (Sec. 2 step 2 "Sorting"), bucketed by tile.
//
// The projection kernel counts the (Gaussian, tile) pairs of every image tile; an
// exclusive scan of those counts gives each tile's segment.  fill writes one key per pair
// into its tile's segment, key = FP32 depth bits << 32 | Gaussian index, taking slots by
// counting the tile's counter back down (lanes of a warp that hit the same tile take a
// block of slots with one atomic; the counters end at zero).  Keys are unique within a
// tile, so sorting each segment by the full 64-bit key yields the (depth, index) order
// exactly, whatever order fill placed them in.  With cross-boundary filtering on, a pair
// the filter removes keeps its slot with depth bits 0xFFFFFFFF, so it sorts last, and the
// tile's range ends before it.
//
// Sorting: a segment of up to 256 keys is sorted in shared memory by one warp, one of up to
// 2048 keys by one CTA of 256 threads (8 keys per thread by a transposition network, then
// merge-path merges of runs).  Longer segments are cut into 4096-key chunks, each sorted the
// same way by a CTA of 512 threads, and then merged pairwise in rounds (run width 4096, 8192,
// ...) with merge-path partitioning, one CTA per 4096 outputs, ping-ponging between the key
// buffer and its twin so that the last round ends in the key buffer.  Chunk sorts and all
// rounds are one launch (k_long_sort).  Every pair is read and written a few times instead of
// once per 8-bit pass over 50+ key bits.
#include "common.cuh"
#include "spec.cuh"
#include "walk.cuh"

namespace splx {

namespace {

constexpr int kChunk = 2048;     // a segment up to this long is sorted by one CTA
constexpr int kSortThreads = 256;
constexpr int kBig = (int)kSortChunk;  // chunk of a longer segment (sorted, then merged)
constexpr int kBigThreads = 512;

__device__ __forceinline__ int next_pow2(int n) {
  int p = 1;
  while (p < n) p <<= 1;
  return p;
}

constexpr int kItems = kChunk / kSortThreads;  // 8 keys per thread
static_assert(kBig / kBigThreads == kItems, "both sorts hold 8 keys per thread");

__device__ __forceinline__ void cas(uint64_t& a, uint64_t& b) {
  const uint64_t lo = a < b ? a : b, hi = a < b ? b : a;
  a = lo;
  b = hi;
}

// Shared buffers hold one spare slot per 8 keys, so that the 8-key runs a warp touches
// with stride 8 fall into different banks.
__device__ __forceinline__ int pad(int i) { return i + (i >> 3); }
constexpr int kPadded = kChunk + kChunk / 8;
constexpr int kBigPadded = kBig + kBig / 8;
// a segment up to this long is sorted by one warp, in its share of a CTA's buffers
constexpr int kWarpKeys = 32 * kItems;
constexpr int kWarpPadded = kWarpKeys + kWarpKeys / 8;
static_assert(kSortThreads / 32 * kWarpPadded <= kPadded, "the warps' shares fit");

// Number of elements taken from A = s[pad(a0 + i)] among the first d of merge(A, B) with
// B = s[pad(b0 + j)], in shared memory.
__device__ __forceinline__ int merge_path_smem(const uint64_t* s, int a0, int na, int b0, int nb,
                                               int d) {
  int lo = d > nb ? d - nb : 0, hi = d < na ? d : na;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (s[pad(a0 + mid)] < s[pad(b0 + d - 1 - mid)]) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// Sorts in[0, n) into out[0, n) (n <= TH * kItems; out may be in) with TH threads, t = 0 ..
// TH - 1: a CTA's, or with TH = 32 one warp.  Each thread sorts kItems keys in registers
// (odd-even transposition network), then runs of 8, 16, ... are merged pairwise through two
// shared buffers, every thread producing kItems outputs located by merge path.  The array
// is padded to a power of two P >= 8 with ~0 keys.  sa, sb: 9/8 TH kItems keys each.
template <int TH>
__device__ __forceinline__ void sort_chunk(const uint64_t* in, uint64_t* out, int n, uint64_t* sa,
                                           uint64_t* sb, const int t) {
  auto sync = [] {
    if (TH == 32) __syncwarp();
    else __syncthreads();
  };
  int P = next_pow2(n);
  if (P < kItems) P = kItems;
  for (int i = t; i < P; i += TH) sa[pad(i)] = i < n ? in[i] : ~0ull;
  sync();
  const int active = P / kItems;  // threads holding keys
  if (t < active) {
    uint64_t v[kItems];
#pragma unroll
    for (int r = 0; r < kItems; ++r) v[r] = sa[pad(t * kItems + r)];
#pragma unroll
    for (int pass = 0; pass < kItems; ++pass)
#pragma unroll
      for (int r = pass & 1; r + 1 < kItems; r += 2) cas(v[r], v[r + 1]);
#pragma unroll
    for (int r = 0; r < kItems; ++r) sa[pad(t * kItems + r)] = v[r];
  }
  sync();
  uint64_t* src = sa;
  uint64_t* dst = sb;
  for (int w = kItems; w < P; w <<= 1) {
    if (t < active) {
      const int o = t * kItems;
      const int p0 = (o / (2 * w)) * (2 * w);
      const int d = o - p0;
      int ia = merge_path_smem(src, p0, w, p0 + w, w, d);
      int ib = d - ia;
      // heads of both runs in registers (~0 past a run's end; a key is below ~0 (its index
      // is below 2^32 - 1), and the ~0 padding keys are equal, so their order does not
      // matter); each output reloads only the head it consumed
      uint64_t va = ia < w ? src[pad(p0 + ia)] : ~0ull;
      uint64_t vb = ib < w ? src[pad(p0 + w + ib)] : ~0ull;
#pragma unroll
      for (int r = 0; r < kItems; ++r) {
        const bool takeA = va < vb;
        dst[pad(o + r)] = takeA ? va : vb;
        if (r + 1 < kItems) {
          ia += takeA ? 1 : 0;
          ib += takeA ? 0 : 1;
          const bool more = takeA ? ia < w : ib < w;
          const uint64_t nv = more ? src[takeA ? pad(p0 + ia) : pad(p0 + w + ib)] : ~0ull;
          va = takeA ? nv : va;
          vb = takeA ? vb : nv;
        }
      }
    }
    sync();
    uint64_t* tmp = src;
    src = dst;
    dst = tmp;
  }
  for (int i = t; i < n; i += TH) out[i] = src[pad(i)];
}

// Merge rounds of a segment of nch chunks, and of one of n keys: ceil(log2(chunks)).
__device__ __forceinline__ int rounds_of(uint32_t nch) {
  int r = 0;
  while ((1u << r) < nch) ++r;
  return r;
}
__device__ __forceinline__ int rounds_for(uint32_t n) {
  return rounds_of(long_chunks(n));
}

// Number of elements taken from A among the first d of merge(A, B) (unique keys), found
// by one warp with 32 probes per step (a 33-ary search over global memory).
__device__ __forceinline__ uint32_t merge_path_warp(const uint64_t* A, uint32_t na,
                                                    const uint64_t* B, uint32_t nb, uint32_t d) {
  const unsigned lane = threadIdx.x & 31u;
  uint32_t lo = d > nb ? d - nb : 0, hi = d < na ? d : na;
  while (lo < hi) {
    const uint32_t span = hi - lo;
    const uint32_t m = lo + (uint32_t)(((uint64_t)span * (lane + 1)) / 33u);
    // true exactly for m below the answer (past L1: other CTAs wrote the runs)
    const bool pred = __ldcg(A + m) < __ldcg(B + (d - 1 - m));
    const unsigned bal = __ballot_sync(0xffffffffu, pred);
    const int nt = __popc(bal);
    const uint32_t m_last_true = __shfl_sync(0xffffffffu, m, nt > 0 ? nt - 1 : 0);
    const uint32_t m_first_false = __shfl_sync(0xffffffffu, m, nt < 32 ? nt : 31);
    if (nt > 0) lo = m_last_true + 1;
    if (nt < 32) hi = m_first_false;
  }
  return lo;
}

// ---- selected-prefix sort (BatchDev::sel) ----
constexpr int kHistBins = 4096;
constexpr int kHistPer = kHistBins / kSortThreads;  // bins per thread in the boundary scan

// With base + (all keys counted in hist) > cap: the bin j whose keys take the running
// count base + (keys in bins below j) from at most cap to above it.  Writes j to s_tmp[8]
// and base + (keys below j) to s_tmp[9]; s_tmp[0..7] hold the warps' totals.  Whole-CTA
// call; the results are valid after it returns.
__device__ __forceinline__ void hist_boundary(const unsigned* hist, unsigned base, unsigned cap,
                                              unsigned* s_tmp) {
  const int t = (int)threadIdx.x, lane = t & 31, w = t >> 5;
  if (t == 0) { s_tmp[8] = 0u; s_tmp[9] = base; }  // (always overwritten below)
  unsigned v[kHistPer];
  unsigned sum = 0;
#pragma unroll
  for (int r = 0; r < kHistPer; ++r) {
    v[r] = hist[t * kHistPer + r];
    sum += v[r];
  }
  unsigned inc = sum;  // inclusive prefix over the warp's threads
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) s_tmp[w] = inc;
  __syncthreads();
  unsigned before = base + inc - sum;
  for (int i = 0; i < w; ++i) before += s_tmp[i];
#pragma unroll
  for (int r = 0; r < kHistPer; ++r) {
    if (before <= cap && cap < before + v[r]) {  // true for exactly one bin
      s_tmp[8] = (unsigned)(t * kHistPer + r);
      s_tmp[9] = before;
    }
    before += v[r];
  }
  __syncthreads();
}

// Sorts the S <= kSelCap smallest keys of the segment [s, e) (n > kChunk keys) into
// keys_alt[s, s + S) and records S in sel[t] and ranges[t] = [capacity + s, capacity + s
// + S), which indexes keys_alt through keys (keys_alt = keys + capacity with sel on);
// keys[s, e) stays as the fill left it.  S is the number of keys below a threshold found
// from a histogram of key bits 62..51 (the depth's exponent and 4 mantissa bits; bit 63,
// its sign, is 0), refined by one of bits 50..39 inside the bin the threshold falls in:
// the keys below the threshold are exactly the S smallest.  If even the nearest bin holds
// more than kSelCap keys, sel[t] = kSelNone and the forward hands the item straight to
// the full sort.
__device__ __forceinline__ void select_prefix(const BatchDev& b, int64_t t, uint32_t s,
                                              uint32_t e, uint64_t* sa, uint64_t* sb,
                                              unsigned* s_tmp) {
  const uint64_t* in = b.keys + s;
  const int n = (int)(e - s);
  unsigned* hist = reinterpret_cast<unsigned*>(sa);  // 16 KB of sa's 18 KB
  for (int i = threadIdx.x; i < kHistBins; i += kSortThreads) hist[i] = 0u;
  __syncthreads();
  for (int i = threadIdx.x; i < n; i += kSortThreads)
    atomicAdd(&hist[(unsigned)(in[i] >> 51) & (kHistBins - 1)], 1u);
  __syncthreads();
  hist_boundary(hist, 0u, (unsigned)kSelCap, s_tmp);
  const unsigned b1 = s_tmp[8];
  unsigned S = s_tmp[9];
  uint64_t thr = (uint64_t)b1 << 51;
  if (8u * ((unsigned)kSelCap - S) > (unsigned)kSelCap) {
    // more than an eighth of the prefix left: refine inside bin b1
    for (int i = threadIdx.x; i < kHistBins; i += kSortThreads) hist[i] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kSortThreads) {
      const uint64_t k = in[i];
      if ((unsigned)(k >> 51) == b1) atomicAdd(&hist[(unsigned)(k >> 39) & (kHistBins - 1)], 1u);
    }
    __syncthreads();
    hist_boundary(hist, S, (unsigned)kSelCap, s_tmp);
    thr |= (uint64_t)s_tmp[8] << 39;
    S = s_tmp[9];
  }
  if (S == 0) {
    if (threadIdx.x == 0) b.sel[t] = kSelNone;
    return;
  }
  if (threadIdx.x == 0) s_tmp[10] = 0u;
  __syncthreads();
  // the keys below thr, in any order, then sorted (sort_chunk reads them before it
  // writes sb)
  for (int i = threadIdx.x; i < n; i += kSortThreads) {
    const uint64_t k = in[i];
    if (k < thr) {
      const unsigned pos = atomicAdd(&s_tmp[10], 1u);
      if (pos < S) sb[pos] = k;
    }
  }
  __syncthreads();
  if (s_tmp[10] != S) {  // not reachable for keys of positive depths; kept as a check
    if (threadIdx.x == 0) { atomicOr(b.status, ST_BOUNDS); b.sel[t] = kSelNone; }
    return;
  }
  sort_chunk<kSortThreads>(sb, b.keys_alt + s, (int)S, sa, sb, (int)threadIdx.x);
  if (threadIdx.x == 0) {
    b.sel[t] = S;
    const uint32_t off = (uint32_t)b.capacity + s;
    b.ranges[t] = make_uint2(off, off + S);
  }
}

}  // namespace

// ---------------------------------------------------------------- fill
constexpr int kFillThreads = 256;
constexpr int kFillFields = 18;  // per lane: tile test (8), rect x, rect y, tile base, width,
                                 // 1/width, tiles per row, pass bits, key (2), tiles

__global__ void __launch_bounds__(kFillThreads, 8) k_fill(const BatchDev b, int per_warp) {
  __shared__ float s_walk[kFillThreads / 32][kFillFields][32];
  __shared__ int s_own[kFillThreads / 32][32];
  const int warp = (int)(threadIdx.x >> 5);
  const unsigned lane = threadIdx.x & 31u, lt = (1u << lane) - 1u;
  const int64_t first = ((int64_t)blockIdx.x * (kFillThreads / 32) + warp) * per_warp;
  const int64_t idx = first + lane;
  if (first >= (int64_t)b.V * b.N) return;
  // lanes without a Gaussian of their own help to walk the others' tiles
  const bool own = (int)lane < per_warp && idx < (int64_t)b.V * b.N;
  const uint32_t tiles = own ? b.counts[idx] : 0u;
  const int v = (int)(idx / b.N);
  const int64_t g = idx - (int64_t)v * b.N;
  int tw = 1, tiles_x = 0, rx0 = 0, rx1 = 0, ry0 = 0, ry1 = 0;
  int64_t tbase = 0;
  uint64_t key = 0;
  TileCull tc = tile_cull_prep(0.f, 0.f, 1.f, 0.f, 1.f, -1.0f);
  uint32_t hits = 0;
  if (tiles) {
    const int k = subset_of(b, g);
    const ViewDev& cam = b.views[v];
    const Rec* r = b.rec + idx;
    const float4 rb = r->b;
    const uint32_t rx = __float_as_uint(rb.w), ry = __float_as_uint(r->c.w);
    const int B_ = b.tile;
    rx0 = (int)(rx & 0xFFFFu); rx1 = (int)(rx >> 16);
    ry0 = (int)(ry & 0xFFFFu); ry1 = (int)(ry >> 16);
    const int tx0 = rx0 / B_, ty0 = ry0 / B_;
    tw = rx1 / B_ - tx0 + 1;
    const float4 rd = r->d;  // the tile test's pass bits, or its inputs (> 32 tiles)
    if (tiles <= 32u) {
      hits = __float_as_uint(rd.w);
    } else {
      // the test centres on the specification's 2-D mean (the record holds the blend's)
      const SubsetDev S = b.subsets[k];
      const int64_t i = g - S.goff;
      const float m[3] = {__ldg(S.means + 3 * i), __ldg(S.means + 3 * i + 1),
                          __ldg(S.means + 3 * i + 2)};
      float tcam[3], terr[3], su, sv;
      spec_camera(m, cam.R, cam.t, tcam, terr);
      spec_center(tcam[0], tcam[1], tcam[2], cam.fx, cam.fy, cam.cx, cam.cy, su, sv);
      tc = tile_cull_prep(su, sv, rd.x, rd.y, rd.z, rd.w);
    }
    tiles_x = cam.tiles_x;
    tbase = b.tile_base[v] + (int64_t)k * cam.tiles_x * cam.tiles_y + (int64_t)ty0 * cam.tiles_x + tx0;
    key = ((uint64_t)__float_as_uint(rb.z) << 32) | (uint64_t)(uint32_t)g;
  }
  bool overflow = false;
  // one (tile, key) candidate per lane: aggregate per tile, take slots, write the keys
  auto place = [&](unsigned t, uint64_t k) {
    if (b.cross && t != 0xFFFFFFFFu) {
      // cross-boundary filtering: a removed pair keeps its slot with the largest depth
      const unsigned long long c = b.cross[(uint32_t)k];
      if (c) {
        const int v = view_of(b.tile_base, b.V, (int64_t)t);
        const ViewDev& cam = b.views[v];
        const int64_t nt = (int64_t)cam.tiles_x * cam.tiles_y;
        const int64_t rem = (int64_t)t - b.tile_base[v];
        const int km = (int)(rem / nt);
        const int loc = (int)(rem - (int64_t)km * nt);
        if (cross_removed(b, v, km, c, loc % cam.tiles_x, loc / cam.tiles_x,
                          (uint32_t)(k >> 32))) {
          k = (0xFFFFFFFFull << 32) | (k & 0xFFFFFFFFull);
          atomicAdd(&b.removed[t], 1u);
        }
      }
    }
    const unsigned peers = __match_any_sync(kFullWarp, t);
    const int leader = __ffs(peers) - 1;
    unsigned old = 0;
    if (t != 0xFFFFFFFFu && (int)lane == leader) old = atomicSub(&b.tile_cnt[t], (unsigned)__popc(peers));
    old = __shfl_sync(kFullWarp, old, leader);
    if (t != 0xFFFFFFFFu) {
      const uint64_t pos = (uint64_t)b.tile_start[t] + (old - 1u - (unsigned)__popc(peers & lt));
      if (pos < (uint64_t)b.capacity) b.keys[pos] = k;
      else overflow = true;
    }
  };
  // the warp's (Gaussian, tile) candidates spread evenly over its lanes (see walk.cuh;
  // here the whole list: a head walked in lockstep measured slower for this kernel)
  {
    float(*f)[32] = s_walk[warp];
    f[0][lane] = tc.u; f[1][lane] = tc.v; f[2][lane] = tc.A; f[3][lane] = tc.B;
    f[4][lane] = tc.C; f[5][lane] = tc.qmax; f[6][lane] = tc.rBC; f[7][lane] = tc.rBA;
    f[8][lane] = __uint_as_float((uint32_t)rx0 | ((uint32_t)rx1 << 16));
    f[9][lane] = __uint_as_float((uint32_t)ry0 | ((uint32_t)ry1 << 16));
    f[10][lane] = __uint_as_float((uint32_t)tbase);
    f[11][lane] = __int_as_float(tw);
    f[12][lane] = 1.0f / (float)tw;
    f[13][lane] = __int_as_float(tiles_x);
    f[14][lane] = __uint_as_float(hits);
    f[15][lane] = __uint_as_float((uint32_t)key);
    f[16][lane] = __uint_as_float((uint32_t)(key >> 32));
    f[17][lane] = __uint_as_float(tiles);
    // a rectangle of at most 32 tiles walks only the tiles its pass bits name (the test is
    // already taken); a larger one walks them all and takes the test
    const int cand = tiles <= 32u ? __popc(hits) : (int)tiles;
    const WarpWalk walk = warp_walk_begin(cand);
    for (int base = 0; base < walk.total; base += 32) {
      int j;
      const int o = warp_walk_owner(walk, base, s_own[warp], j);
      unsigned t = 0xFFFFFFFFu;
      uint64_t okey = 0;
      if (o >= 0) {
        int jx, jy;
        bool pass;
        if (__float_as_uint(f[17][o]) <= 32u) {
          // the j-th set pass bit
          unsigned m = __float_as_uint(f[14][o]);
          for (int q = 0; q < j; ++q) m &= m - 1u;
          walk_tile(__ffs(m) - 1, __float_as_int(f[11][o]), f[12][o], jx, jy);
          pass = true;
        } else {
          walk_tile(j, __float_as_int(f[11][o]), f[12][o], jx, jy);
          TileCull oc;
          oc.u = f[0][o]; oc.v = f[1][o]; oc.A = f[2][o]; oc.B = f[3][o];
          oc.C = f[4][o]; oc.qmax = f[5][o]; oc.rBC = f[6][o]; oc.rBA = f[7][o];
          const uint32_t rx = __float_as_uint(f[8][o]), ry = __float_as_uint(f[9][o]);
          const int x0 = (int)(rx & 0xFFFFu), x1 = (int)(rx >> 16);
          const int y0 = (int)(ry & 0xFFFFu), y1 = (int)(ry >> 16);
          pass = tile_hits_spec(oc, x0, x1, y0, y1, x0 / b.tile + jx, y0 / b.tile + jy, b.tile);
        }
        if (pass) {
          t = __float_as_uint(f[10][o]) + (unsigned)(jy * __float_as_int(f[13][o]) + jx);
          okey = ((uint64_t)__float_as_uint(f[16][o]) << 32) | __float_as_uint(f[15][o]);
        }
      }
      place(t, okey);
    }
  }
  if (overflow) atomicOr(b.status, ST_CAPACITY);
}

void launch_fill(const BatchDev& b, cudaStream_t s) {
  const int64_t n = (int64_t)b.V * b.N;
  if (n == 0) return;
  const int per_warp = walk_per_warp(n, device_sm_count() * 64);
  const int64_t per_block = (int64_t)(kFillThreads / 32) * per_warp;
  k_fill<<<(unsigned)((n + per_block - 1) / per_block), kFillThreads, 0, s>>>(b, per_warp);
  count_launch();
}

// ---------------------------------------------------------------- segment sorts
// Ranges and sorts of the tile segments, `group` (1 to 8) tiles per CTA.  Each of its first
// `group` warps takes a tile: a segment of up to 256 keys is sorted by its warp alone, in an
// eighth of the shared memory; a longer one by the whole CTA afterwards, if it has at most
// kChunk keys, or else as a selected prefix or registered with the long-segment sort.
//
// With one CTA per tile most tiles used one warp of eight (a 2M-Gaussian batch of 4 views
// has 180 keys a segment on average) and the others waited at its barriers: the segment
// sorts of 4 views and 32 subsets over 20M Gaussians, 20 keys a segment, 1.22 -> 0.41 ms.
// kSolo (small launches): one tile per CTA, looked up by all its warps and sorted by the
// whole CTA without the exchange (a 10k-Gaussian 256x256 render 105.6 us, 108 with it).
template <bool kSolo>
__global__ void __launch_bounds__(kSortThreads, 6) k_seg_sort(const BatchDev b, int group) {
  __shared__ uint64_t sk[2][kPadded];
  __shared__ unsigned s_base;
  __shared__ unsigned s_tmp[11];
  __shared__ uint2 s_seg[kSortThreads / 32];  // start and length of the longer segments
  const int warp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
  const int64_t first = (int64_t)blockIdx.x * group;
  uint2 longer = make_uint2(0u, 0u);
  const int mine = kSolo ? 0 : warp;
  if (mine < group && first + mine < items_of_launch(b)) {
    const int64_t t = item_of(b, first + mine);
    uint32_t s, e;
    segment_of(b, t, s, e);
    // the pairs the cross-boundary filter removed sort last and stay out of the range
    if (lane == 0 && warp == mine) {
      const uint32_t cut = b.removed ? min(b.removed[t], e - s) : 0u;
      b.ranges[t] = make_uint2(s, e - cut);
      if (b.sel) b.sel[t] = 0u;
    }
    const int n = (int)(e - s);
    // saturation-skipping waves sort only what the wave's rasteriser will walk; likewise
    // with a stale saturation state a tile pruned at every pixel stays unsorted
    if (n > 1 && !(b.order && b.wave > 0 && item_saturated(b, t)) &&
        !(b.sat && item_pruned(b, t))) {
      if (kSolo || n > kWarpKeys)
        longer = make_uint2(s, (uint32_t)n);
      else
        sort_chunk<32>(b.keys + s, b.keys + s, n, sk[0] + warp * kWarpPadded,
                       sk[1] + warp * kWarpPadded, lane);
    }
  }
  if (!kSolo) {
    if (lane == 0) s_seg[warp] = longer;
    __syncthreads();
  }
  for (int q = 0; q < (kSolo ? 1 : group); ++q) {
    const uint2 seg = kSolo ? longer : s_seg[q];
    const uint32_t s = seg.x;
    const int n = (int)seg.y;
    if (n == 0) continue;
    if (n <= kChunk) {
      sort_chunk<kSortThreads>(b.keys + s, b.keys + s, n, sk[0], sk[1], (int)threadIdx.x);
      __syncthreads();  // shared memory is free for the next segment
      continue;
    }
    const int64_t t = item_of(b, first + q);
    if (b.sel) {
      select_prefix(b, t, s, s + (uint32_t)n, sk[0], sk[1], s_tmp);
    } else {
      if (threadIdx.x == 0) s_base = register_long(b, t, (uint32_t)n);
      __syncthreads();
      const unsigned nch = long_chunks((uint32_t)n), at = s_base;
      for (unsigned c = threadIdx.x; c < nch; c += kSortThreads)
        b.chunks[at + c] = make_uint2((uint32_t)t, at);
    }
    __syncthreads();  // likewise
  }
}

// One merge item: outputs [o0, o0 + 4096) of the round that merges runs of w keys of a
// segment of n keys from src to dst (both at the segment's start).  src holds what other
// CTAs wrote earlier in the launch, so it is read past L1.
__device__ __forceinline__ void merge_item(const uint64_t* src, uint64_t* dst, uint32_t n,
                                           uint32_t w, uint32_t o0, uint64_t* sm,
                                           uint32_t* s_split) {
  constexpr int PER = kBig / kBigThreads;  // outputs per thread
  const uint32_t o1 = o0 + kBig < n ? o0 + kBig : n;
  const uint32_t p0 = (o0 / (2 * w)) * (2 * w);
  const uint32_t na = (p0 + w < n ? p0 + w : n) - p0;
  const uint32_t nb = (p0 + 2 * w < n ? p0 + 2 * w : n) - (p0 + na);
  const uint64_t* A = src + p0;
  const uint64_t* B = A + na;
  // warp 0 finds the split at the block's first output, warp 1 at its end
  if (threadIdx.x < 64) {
    const uint32_t dd = (threadIdx.x < 32 ? o0 : o1) - p0;
    const uint32_t a = merge_path_warp(A, na, B, nb, dd);
    if ((threadIdx.x & 31) == 0) {
      s_split[threadIdx.x >> 5] = a;
      s_split[2 + (threadIdx.x >> 5)] = dd - a;
    }
  }
  __syncthreads();
  const uint32_t a0 = s_split[0], a1 = s_split[1], b0 = s_split[2], b1 = s_split[3];
  const int la = (int)(a1 - a0), lb = (int)(b1 - b0);
  for (int i = threadIdx.x; i < la; i += kBigThreads) sm[pad(i)] = __ldcg(A + a0 + i);
  for (int i = threadIdx.x; i < lb; i += kBigThreads) sm[pad(la + i)] = __ldcg(B + b0 + i);
  __syncthreads();
  // each thread merges PER consecutive outputs of sm[0,la) and sm[la,la+lb)
  const int d = threadIdx.x * PER;
  if (d < la + lb) {
    int ia = merge_path_smem(sm, 0, la, la, lb, d);
    int ib = d - ia;
    const int dend = d + PER < la + lb ? d + PER : la + lb;
    uint64_t va = ia < la ? sm[pad(ia)] : ~0ull;  // run heads (~0 past the end)
    uint64_t vb = ib < lb ? sm[pad(la + ib)] : ~0ull;
    for (int o = d; o < dend; ++o) {
      const bool takeA = va < vb;
      dst[o0 + o] = takeA ? va : vb;
      ia += takeA ? 1 : 0;
      ib += takeA ? 0 : 1;
      const bool more = takeA ? ia < la : ib < lb;
      const uint64_t nv = more ? sm[takeA ? pad(ia) : pad(la + ib)] : ~0ull;
      va = takeA ? nv : va;
      vb = takeA ? vb : nv;
    }
  }
}

// The long segments' whole sort in one launch: item (0, c) sorts chunk c of the chunk list,
// item (1 + r, c) produces chunk c's 4096 outputs of merge round r (run width 4096 << r).
// CTAs take the items in that order from a counter, and an item of a round starts when its
// segment's chunk items of the round before are counted done (seg_done).  A wait longer than
// b.wait_polls polls gives up: ST_TIMEOUT, the segment stays unsorted.  The order makes
// the wait end: every earlier item was taken before and is held by a CTA that is running,
// whether or not the whole grid is resident, and the earliest unfinished one never waits.
// A segment merged in R rounds starts them in keys_alt when R is odd, so that its last round
// writes keys; waiting for the whole segment keeps a round from overwriting what the round
// before still reads.
//
// One launch instead of one per round: the rounds that the largest subset could need were
// launched unseen, and most of them found nothing to do (city-scale waves: 8 of 11 launches
// of each wave and view group; a 20M-Gaussian, 32-subset step 15.5 -> 14.1 ms, a 10k-Gaussian
// 256x256 render 123 -> 111 us).  Two 36 KB buffers, dynamic shared memory, 3 CTAs per SM.
__global__ void __launch_bounds__(kBigThreads) k_long_sort(const BatchDev b) {
  extern __shared__ uint64_t sk_dyn[];
  uint64_t* sa = sk_dyn;
  uint64_t* sb = sk_dyn + kBigPadded;
  __shared__ uint32_t s_split[4];
  __shared__ unsigned s_item;
  __shared__ int s_ok;
  const unsigned count = *b.chunk_count;
  if (count == 0) return;
  const unsigned items = count * (1u + (unsigned)rounds_of(b.big_count[1]));
  for (;;) {
    __syncthreads();  // the previous item is done with shared memory
    if (threadIdx.x == 0) s_item = atomicAdd(b.big_count, 1u);
    __syncthreads();
    const unsigned item = s_item;
    if (item >= items) return;
    const unsigned q = item / count, ci = item - q * count;
    const uint2 ch = b.chunks[ci];
    const int64_t t = ch.x;
    uint32_t s, e;
    segment_of(b, t, s, e);
    const uint32_t n = e - s, o0 = (ci - ch.y) * kBig;
    const unsigned R = (unsigned)rounds_for(n);
    if (q > R) continue;  // this segment needs no merge at this width
    if (q == 0) {
      const uint32_t c0 = s + o0, c1 = c0 + kBig < e ? c0 + kBig : e;
      uint64_t* out = ((R & 1u) ? b.keys_alt : b.keys) + c0;
      sort_chunk<kBigThreads>(b.keys + c0, out, (int)(c1 - c0), sa, sb, (int)threadIdx.x);
    } else {
      if (threadIdx.x == 0) {
        const volatile uint32_t* done = b.seg_done + t;
        const uint32_t need = q * long_chunks(n);
        int polls = 0;
        while (*done < need && polls < b.wait_polls) {
          __nanosleep(256);
          ++polls;
        }
        s_ok = *done >= need;
        if (!s_ok) atomicOr(b.status, ST_TIMEOUT);
        __threadfence();
      }
      __syncthreads();
      if (!s_ok) return;
      // the input of round r = q - 1 lies in keys_alt when R - r is odd
      const bool from_alt = ((R - (q - 1u)) & 1u) != 0u;
      merge_item((from_alt ? b.keys_alt : b.keys) + s, (from_alt ? b.keys : b.keys_alt) + s, n,
                 (uint32_t)kBig << (q - 1u), o0, sa, s_split);
    }
    if (q < R) {
      __syncthreads();  // the item's keys are written
      if (threadIdx.x == 0) {
        __threadfence();
        atomicAdd(b.seg_done + t, 1u);
      }
    }
  }
}

// Sort and merges of the segments registered in chunks (register_long).
void launch_long_sort(const BatchDev& b, cudaStream_t s) {
  // 72 KB of dynamic shared memory: opted in once per device (a refused opt-in shows as
  // the launch's error, which the callers check).  One wave of resident CTAs (3 per SM at
  // 72 KB), so that no CTA starts after the others have ended
  constexpr int kChunkSmem = 2 * kBigPadded * (int)sizeof(uint64_t);
  (void)opt_in_smem((const void*)k_long_sort, kChunkSmem, 0);
  const unsigned grid = (unsigned)device_sm_count() *
                        (unsigned)resident_ctas((const void*)k_long_sort, kBigThreads,
                                                kChunkSmem, 0);
  k_long_sort<<<grid, kBigThreads, kChunkSmem, s>>>(b);
  count_launch();
}

void launch_seg_sort(const BatchDev& b, cudaStream_t s) {
  if (b.n_tiles == 0) return;
  const int64_t items = items_of_launch(b);
  // Tiles per CTA, by the mean list: the pairs of an earlier forward where the host knows them,
  // else four fifths of the room (a batch that sizes itself leaves a quarter).  Short lists go
  // eight to a CTA, longer ones, which its tiles take in turn as whole CTAs, two: 1M lists of
  // 20 keys on average 0.42 ms at 8, 0.51 at 4, 0.74 at 2, 1.22 at 1; 165k lists of 72 0.371,
  // 0.355, 0.394, 0.490; 165k of 192 0.768, 0.709, 0.719, 0.761; 165k of 306 1.025, 0.970,
  // 0.951, 0.961.  Fewer where that would leave less than two CTAs of work for every resident
  // one.  A launch by itself (waves run beside other view groups' forwards) ends later the
  // longer its last CTAs are: 14k lists of 116 0.066 ms at one tile per CTA, 0.076 at two; 27k
  // of 680 0.193, 0.232; 42k of 249 0.242, 0.252, of 131 0.172 both; 54k of 269 0.305, 0.318,
  // of 170 0.242, 0.240
  const double mean = b.pairs > 0 ? (double)b.pairs / (double)b.n_tiles
                                  : 0.8 * (double)b.capacity / (double)b.n_tiles;
  const bool short_lists = mean < 100.0;
  int group = short_lists ? kSortThreads / 32 : 2;
  while (group > 1 && items < (int64_t)device_sm_count() * 12 * group) group /= 2;
  if (!short_lists && !b.order && !b.sat && items < (mean < 200.0 ? 1 << 14 : 1 << 16)) group = 1;
  const unsigned grid = (unsigned)((items + group - 1) / group);
  if (group == 1) k_seg_sort<true><<<grid, kSortThreads, 0, s>>>(b, 1);
  else k_seg_sort<false><<<grid, kSortThreads, 0, s>>>(b, group);
  count_launch();
  // with selected prefixes no segment is left to the long-segment sort before the forward
  if (!b.sel) launch_long_sort(b, s);
}

void launch_sort_retries(const BatchDev& b, cudaStream_t s) {
  if (b.sel && b.n_tiles != 0) launch_long_sort(b, s);
}

}  // namespace splx
