// How the 3x3 convolutions of lbm_nn.h are cut into work items, and the map from their flat positions to pixels.  Plain
// C++ (no CUDA header), so that host code can walk a plan and the map without a GPU.
#pragma once

#include <stdint.h>

#include <algorithm>

#ifdef __CUDACC__
#define LBM_NN_HD __host__ __device__ __forceinline__
#else
#define LBM_NN_HD inline
#endif

namespace lbm_nn {

LBM_NN_HD unsigned mulhi(unsigned a, unsigned b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (unsigned)(((unsigned long long)a * b) >> 32);
#endif
}

constexpr int kCvEpi = 8;                          // epilogue warps, two per TMEM lane quarter
constexpr int kCvMma = kCvEpi;                     // the warp that issues the products
constexpr int kCvProd = 12;                        // producer warps
constexpr int kCvThreads = 32 * (kCvEpi + 1 + kCvProd);
constexpr int kCvBatch = 4;                        // 8-channel groups (32 bytes) a producer thread has in flight
constexpr int kCvMaxStages = 6;
constexpr int kCvSmem = 227 * 1024;                // shared memory a CTA may use
constexpr int kCvHead = 512 + kCvEpi * 4096;       // barriers, epilogue transposition buffers

// How a convolution is cut into work items (host).
struct FwdPlan {
  int N, KC;                 // output channels per item, input channels per stage
  int Wt, pitch, strips;     // columns per item, staged columns, column strips
  int R, T;                  // rows per item, 128-position tiles per item
  int Pn;                    // staged positions allocated per channel group (Pn % 8 == 2: conflict-free stores)
  int stages, stage_bytes, smem, tmem;
  unsigned mp, mh;           // PosMap's multipliers
  int blocks, items;         // row blocks of the tall image; items = blocks * strips * (cout / N)
};

// Multiplier of the division by h + 1 for blocks of fewer than `rows` rows: 0 where a block spans fewer than h + 1 (the
// quotient is 0 or 1), else ceil(2^32 / (h + 1)) if that is exact up to the largest dividend, h + rows.  False if not.
inline bool row_multiplier(int h, long long rows, unsigned* mh) {
  const unsigned long long d = h + 1ull, m = ((1ull << 32) + d - 1) / d;
  *mh = rows <= h ? 0u : (unsigned)m;
  return rows <= h || (h + (unsigned long long)rows) * (m * d - (1ull << 32)) < (1ull << 32);
}

// Rows and columns of the flat positions of a block, by multiplication: divisions by the pitch and by the rows h + 1
// of an image of the tall image.  With m = ceil(2^32 / d) the high word of v m is v / d as long as v (m d - 2^32) < 2^32.
// By the pitch (at most 130) that holds up to 2^25 positions, by h + 1 where row_multiplier says so.
struct PosMap {
  unsigned mp, mh;           // ceil(2^32 / pitch), ceil(2^32 / (h + 1)) or 0: a block spans fewer than h + 1 rows
  int pitch, h, w;
  int img0, yy0, x0;         // image and row of the block's first row, image column of position column 0
  LBM_NN_HD void block(long long row0, int col0) {
    img0 = (int)(row0 / (h + 1LL));
    yy0 = (int)(row0 - img0 * (h + 1LL));
    x0 = col0;
  }
  // whether column c of the block's row r lies in an image: then its row yy and column xx there, and the zero rows k
  // between the block's first row and it
  LBM_NN_HD bool inside(int r, int c, unsigned& k, unsigned& yy, unsigned& xx) const {
    const unsigned v = (unsigned)yy0 + (unsigned)r;
    k = mh ? mulhi(v, mh) : (v > (unsigned)h ? 1u : 0u);
    yy = v - k * ((unsigned)h + 1u);
    xx = (unsigned)x0 + (unsigned)c;
    return yy < (unsigned)h && xx < (unsigned)w;
  }
  // pixel of a launch of fewer than 2^31, -1 outside the images
  LBM_NN_HD int pixel(int r, int c) const {
    unsigned k, yy, xx;
    return inside(r, c, k, yy, xx) ? ((img0 + (int)k) * h + (int)yy) * w + (int)xx : -1;
  }
  // the same of a launch of any number, counted from the block's first row, in a block of fewer than 2^32: origin() +
  // offset(), ~0 outside the images
  LBM_NN_HD long long origin() const { return ((long long)img0 * h + yy0) * w; }
  LBM_NN_HD unsigned offset(int r, int c) const {
    unsigned k, yy, xx;
    return inside(r, c, k, yy, xx) ? ((unsigned)r - k) * (unsigned)w + xx : ~0u;
  }
  LBM_NN_HD void split(int q, int& r, int& c) const {
    r = (int)mulhi((unsigned)q, mp);
    c = q - r * pitch;
  }
};

// Cuts the convolution into items: among the channel tiles N, the numbers of column strips (of at most 128 columns)
// and the tiles per item, the least modelled time: waves of one CTA per SM x the largest of the product time (32
// cycles per M = 128 product up to N = 64, then N / 2), the staging time and the store time (32 bytes per SM and
// cycle each), plus a fixed latency per item and stage.  Small images get many small items, so that one image of a
// deep level still reaches half of the SMs; large ones get items of up to 1024 positions, whose halo costs least.
inline FwdPlan fwd_plan(int n, int h, int w, int cin, int cout, int sms) {
  FwdPlan best{};
  double best_cost = -1.0;
  const int KC = cin % 32 == 0 ? 32 : 16;
  const int rows_all = n * (h + 1) - 1;
  for (int N = 32; N <= 128; N *= 2) {
    if (cout % N) continue;
    const int k0 = (w + 127) / 128;
    for (int k = k0; k <= k0 + 3 && k <= w; ++k) {
      const int Wt = (w + k - 1) / k, pitch = Wt + 2, strips = (w + Wt - 1) / Wt;
      for (int T = 1; T * N <= 256; ++T) {
        if (128 * T < Wt) continue;
        FwdPlan p{};
        p.N = N;
        p.KC = KC;
        p.Wt = Wt;
        p.pitch = pitch;
        p.strips = strips;
        p.T = T;
        p.R = std::min((128 * T - Wt) / pitch + 1, rows_all);
        p.blocks = (rows_all + p.R - 1) / p.R;
        p.R = (rows_all + p.blocks - 1) / p.blocks;
        p.mp = (unsigned)(((1ull << 32) + pitch - 1) / pitch);
        if (!row_multiplier(h, p.R + 2, &p.mh)) continue;         // never: R <= 342
        p.Pn = 128 * T + 2 * pitch + 2;
        p.Pn += (10 - p.Pn % 8) % 8;                              // Pn % 8 == 2
        p.stage_bytes = (KC / 8) * p.Pn * 16 + 18 * N * KC;
        p.stage_bytes = (p.stage_bytes + 511) / 512 * 512;        // the weights' swizzle pattern repeats every 512 bytes
        p.stages = std::min(kCvMaxStages, (kCvSmem - kCvHead) / p.stage_bytes);
        if (p.stages < 2) continue;
        p.smem = kCvHead + p.stages * p.stage_bytes;
        p.tmem = 32;
        while (p.tmem < 2 * T * N) p.tmem *= 2;
        p.items = p.blocks * strips * (cout / N);
        const double mma = (double)T * 9 * (cin / 16) * std::max(32, N / 2);
        const double load = ((double)(p.R + 2) * pitch * cin * 4 + 18.0 * cin * N) / 32.0;
        const double out = (double)T * N * 128 * 4 / 32.0;
        const double item = std::max(std::max(mma, load), out) + 300.0;
        const double cost = (double)((p.items + sms - 1) / sms) * item + 400.0 * (cin / KC);
        if (best_cost < 0 || cost < best_cost) best = p, best_cost = cost;
      }
    }
  }
  return best;
}

constexpr int kWgMaxSlots = 6;
constexpr int kWgHead = 512;
constexpr int kWgEpi = 4;                     // warps 0-3: products (one thread of warp 0), then the segment's epilogue
constexpr int kWgGroups = 3;                  // producer groups of four warps: group g stages steps g, g + 3, ...
constexpr int kWgGroup = 128, kWgProd = kWgGroups * kWgGroup;
constexpr int kWgThreads = 32 * kWgEpi + kWgProd;   // 16 warps: 128 registers a thread
constexpr int kWgBatch = 2;                   // 16-channel groups of each tensor a producer thread has in flight

struct WgradPlan {
  int u_dy;                    // 1: U = dy, V = x; 0: U = x, V = dy
  int mt, vt, mb;              // channels of U and V per tile; products per b (3 without folding, 2, 1)
  int utiles, vtiles;
  int Wt, pitch, strips;
  int KP;                      // positions per step
  // Steps in flight, at least kWgGroups: a group that stages step k waits for the products of step k - slots by parity,
  // which needs those of step k - 2 slots known to be done; what it knows, from its step before, is k - kWgGroups - slots
  int slots;
  int ulen, rv, vlen;          // plane lengths: U slot; V ring, V plane (ring + 16, padded)
  int u_bytes, v_bytes, smem, tmem;
  int seg_steps;               // longest segment
  unsigned mp, mh;
  long long len, steps;        // positions and steps of a strip
  long long chunks;            // partial sums
  long long bias_chunks, ws_chunks;
};

// A segment of a chunk: steps from position `first` (a multiple of KP) of a column strip on, with their map
struct WgradSegment {
  PosMap map;
  int off = 0;               // a position counted from the segment's first lies `off` past the map's row 0
  int lo = 0, hi = 0;        // the positions in [lo, hi) lie in the strip
  LBM_NN_HD WgradSegment(const WgradPlan& p, int h, int w) : map{p.mp, p.mh, p.pitch, h, w} {}
  LBM_NN_HD void start(const WgradPlan& p, long long first, int strip) {
    // the map starts at the row two above the first position's (tall-image rows shifted by two images)
    const long long row0 = first / p.pitch - 2;
    map.block(row0 + 2 * (map.h + 1LL), strip * p.Wt - 1);
    map.img0 -= 2;
    off = (int)(first - row0 * p.pitch);
    lo = (int)(-first > -(1LL << 30) ? -first : -(1LL << 30));
    hi = (int)(p.len - first < (1LL << 30) ? p.len - first : (1LL << 30));
  }
};

constexpr long long kBiasChunk = 4096;

// Tiles and chunks of the weight gradient: the orientation, channel tiles and step length with the least modelled time,
// (positions per chunk) x the larger of the staging time (12 bytes per SM and cycle, measured for the producer warps)
// and the product time (shared-memory reads: 32 cycles of U, vt / 4 of V per product).  One CTA per SM, one wave.
// The size of the workspace, which callers keep, bounds the chunks: four sets of partial sums per SM's share of channel
// tiles, 32 x 32 (up to 64 output channels) or 128 x 32 x one kernel row, the last set being the bias partials' room, and
// cout floats per 4096 pixels, which nothing uses.  It does not depend on the device: it is asked for without one.
inline WgradPlan wgrad_plan(int n, int h, int w, int cin, int cout) {
  constexpr int sms = 152;     // of a GB300
  const int ws_tiles = cout <= 64 ? ((cout + 31) / 32) * ((cin + 31) / 32) : ((cout + 127) / 128) * 3 * ((cin + 31) / 32);
  const long long most = std::max(1LL, 4LL * sms / ws_tiles - 1);
  // longest float32 chain of one accumulator: the pixels over the partial sums that fit the workspace
  const long long pixels = (long long)n * h * w;
  const long long chain = std::max(256LL, pixels * ws_tiles / (4 * sms));
  WgradPlan best{};
  double best_cost = -1.0;
  for (int u_dy = 0; u_dy < 2; ++u_dy) {
    const int cu = u_dy ? cout : cin, cv = u_dy ? cin : cout;
    for (int mt = 32; mt <= 128; mt *= 2) {
      if (mt > 32 && cu <= mt / 2) break;
      const int mb = mt / 32 > 2 ? 3 : mt / 32;
      for (int vt = 16; vt <= 128; vt += 16) {
        if (mb * 3 * vt > 512 || (vt > cv && vt > 16)) break;
        WgradPlan p{};
        p.u_dy = u_dy;
        p.mt = mt;
        p.vt = vt;
        p.mb = mb;
        p.utiles = (cu + mt - 1) / mt;
        p.vtiles = (cv + vt - 1) / vt;
        const int k = (int)((w + 127LL) / 128);
        p.Wt = (int)((w - 1LL + k) / k);
        p.pitch = p.Wt + 2;
        p.strips = (int)((w - 1LL + p.Wt) / p.Wt);
        p.len = (n * (h + 1LL) - 1) * p.pitch;
        p.tmem = 32;
        while (p.tmem < mb * 3 * vt) p.tmem *= 2;
        for (int kp : {112, 48}) {   // KP + 2 positions of U fill whole passes of a producer group
          p.KP = kp;
          // plane lengths for 16-byte stores of a warp's positions and 16-channel groups without bank conflicts
          // (two groups: 2 mod 4; more: odd)
          auto pad = [](int len, int groups) {
            const int want = groups <= 4 ? 2 : 1;   // groups of 8 channels
            return len + ((want - len) % 8 + 8) % 8;
          };
          const int ucopies = mb == 3 ? 1 : 3;
          p.ulen = pad(mb == 3 ? p.KP + 2 : p.KP, mt / 8);
          p.u_bytes = (ucopies * mt / 8 * p.ulen * 16 + 127) / 128 * 128;
          for (p.slots = kWgMaxSlots; p.slots >= kWgGroups; --p.slots) {
            p.rv = p.slots * p.KP + 2 * p.pitch;
            p.vlen = pad(p.rv + 16, vt / 8);
            p.v_bytes = vt / 8 * p.vlen * 16;
            // a product reads 16 planes of U from each block, also where fewer are staged: room for them behind
            p.smem = kWgHead + p.slots * p.u_bytes + std::max(std::max(p.v_bytes, 16 * p.ulen * 16), 64 * kWgProd);
            if (p.smem <= kCvSmem) break;
          }
          if (p.slots >= kWgGroups) break;
        }
        if (p.slots < kWgGroups) continue;
        p.steps = (p.len + p.KP - 1) / p.KP;
        const long long total = p.steps * p.strips, tiles = (long long)p.utiles * p.vtiles;
        p.chunks = std::max(1LL, std::min(std::min(total, most), sms / tiles));
        p.chunks = std::min<long long>(p.chunks, 9 * cin);         // room of the bias partials
        const double waves = (double)((tiles * p.chunks + sms - 1) / sms);
        const double load = 16.0 * 4 * (std::min(mt, cu) + std::min(vt, cv)) / 12.0;
        const double mma = mb * 3 * (32.0 + vt / 4.0);
        const double per = (double)total * p.KP / 16 / p.chunks;
        const double cost = waves * (per * std::max(load, mma) + 2.0 * p.pitch / 16 * load) + 0.5 * p.chunks * 9;
        if (best_cost < 0 || cost < best_cost) best = p, best_cost = cost;
      }
    }
  }
  WgradPlan& p = best;
  const long long per = (p.steps * p.strips + p.chunks - 1) / p.chunks * p.KP;   // positions per chunk
  const long long segs = std::max(1LL, (long long)((double)per / (1.1 * chain) + 0.999));
  p.seg_steps = (int)std::min<long long>(((per + segs - 1) / segs + p.KP - 1) / p.KP, (1 << 22) / p.KP);
  p.mp = (unsigned)(((1ull << 32) + p.pitch - 1) / p.pitch);
  // with the halo a segment touches fewer than its own positions' rows + 5.  Rows of more than 2^17 pixels: segments
  // shorter than 2^32 pixels (of the six rows that one step touches at most five are below the first: no tensor that
  // the device holds has seven rows of 2^29 pixels)
  p.seg_steps = (int)std::max(1LL, std::min<long long>(p.seg_steps, ((1LL << 32) / w - 6) * p.pitch / p.KP));
  // images of tens of thousands of rows and few
  // columns: segments shorter than an image where the division by h + 1 would not be exact over several (h > 1500 then)
  if (!row_multiplier(h, (long long)p.seg_steps * p.KP / p.pitch + 5, &p.mh)) {
    p.seg_steps = (int)((h - 5LL) * p.pitch / p.KP);
    row_multiplier(h, (long long)p.seg_steps * p.KP / p.pitch + 5, &p.mh);
  }
  p.bias_chunks = (pixels + kBiasChunk - 1) / kBiasChunk;
  p.ws_chunks = p.chunks + 1;
  return best;
}

}  // namespace lbm_nn
