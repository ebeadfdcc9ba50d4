// The tile pipeline's kernels: one launch per iteration, a block per tile of
// 48 x TH pixels, every stage of the tile in shared memory. Used for calls too
// small for the queue pipeline; detect_kernel (kernels.cuh) keeps the forms
// with map export, a given previous mask, separate launches or other shapes.
//
// A warp holds a whole row of the tile's image region (the tile and 8 columns
// each side: 64), two columns per lane, so a row of any bit map is two words:
// the even and the odd columns, as the ballots give them. A dilation is then
// shifts and ORs of two words with no neighbour word, and an aligned pair of
// pixels is one bit of the two words' OR.
//
// Stages of iteration k on a tile (sets and pruning: detect_tile's comment):
//   replace  (k >= 2) iteration k-1's replacement on the tile and 6 pixels
//            around it, only of the flagged pixels whose value can change: those
//            within 2 px of a flag that is new in M_{k-1}, and those whose
//            whole window is flagged. The pixels whose value did change are
//            kept as a bit map; no new flag lies farther than 6 px from one
//            (pipeline.cuh), so a tile without any is done, and in the others
//            S' is computed within 6 px of them only;
//   rows     column medians, L+, the bound test and med3 of the region, a warp
//            per band of rows, rows kept in registers;
//   need     the sets nsp (S' to compute) and its 5 x 5 dilation (S), as pairs;
//   S, S'    two medians per pair from one network over shared columns;
//   test     the objlim test by counting: the statistic is monotone in
//            med7(m3), so it holds at the median exactly where it holds for at
//            least 25 of the 49 values. Eight lanes per test, no 7x7 median;
//   grow     both growths from the bit maps, a lane per row.
//
// Flags live in three planes of the workspace, M_k in plane k mod 3, so a
// launch reads M_{k-1} and M_{k-2} while it writes M_k. Flags only accumulate:
// the plane still holds M_{k-3}, a subset of M_k, and is ORed into. A plane
// row is two bit streams, even and odd columns.

#pragma once

#include "kernels.cuh"

namespace crb {

constexpr int kT2W = 48;  // tile width
constexpr int kT2P = 68;  // row pitch in shared memory: rows of a column fall on different banks

// words per bit stream of a plane row
__host__ __device__ inline int tile_wps(int w) { return ((w + 1) / 2 + 31) / 32; }

// kMode as tile_kernel: iteration 1 keeps med3, the later ones the image region and the maps of S and N (whose
// place the replacement values take before), the last replacement the image region and those values.
// 53, 42 and 24 KB: 4, 5 and 6 blocks per SM, the second at 48 registers with 40 B of spills (kMany), the third at
// 40. Calls whose tiles take one round of blocks keep 64 registers and 4 blocks in mode 1.
template <int TH, int kMode>
struct TileLayout {
  static constexpr int R = TH + 16;   // rows of the image region
  static constexpr int RB = TH + 10;  // rows of med3: the tile and 5 rows each side
  static constexpr int BR = RB / 8;   // rows per warp
  static_assert(RB % 8 == 0 && R <= 64 && TH >= 8, "whole bands of rows, 6-bit rows in list entries");
  static constexpr int RS = TH + 8;   // rows of S
  static constexpr int R2 = TH + 4;   // rows of S' and N
  static constexpr int kListR = kMode == 2 ? TH * kT2W : (TH + 12) * 60;  // flagged pixels to replace at most
  static constexpr int oJ = 0;
  static constexpr int oS = oJ + R * kT2P;
  static constexpr int oN = oS + (kMode == 2 ? 0 : RS * kT2P);
  static constexpr int oM3 = oN + (kMode == 2 ? kListR : R2 * kT2P);
  static_assert(oS + kListR <= oM3, "replacement values fit in the S and N maps");
  static constexpr int nF = oM3 + (kMode == 0 ? RB * kT2P : 0);
  static constexpr int kListS = kMode == 2 ? kListR : imax(RS * 28, (kListR + 1) / 2 * 2);  // pairs of S; or the replacement list
  static constexpr int kListP = kMode == 2 ? 0 : R2 * 26;                                   // pairs of S'
  static_assert(kMode == 2 || R2 * 52 <= kListS, "the tests take the place of the pairs of S");
  static constexpr int oMask = nF * 4;  // bytes: bit maps of R rows x 2 words (mode 2: M and its new flags)
  static constexpr int oL0 = round16(oMask + (kMode == 2 ? 2 : 8) * R * 8);
  static constexpr int oL1 = oL0 + round16(kListS * 2);
  static constexpr int oCnt = oL1 + round16(kListP * 2);
  static constexpr int bytes = oCnt + 64;
};

// ---- rows of bits: x = even columns (bit i: column 2i), y = odd columns (2i + 1) ----
__device__ __forceinline__ uint2 or2(uint2 a, uint2 b) { return make_uint2(a.x | b.x, a.y | b.y); }
__device__ __forceinline__ uint2 and2(uint2 a, uint2 b) { return make_uint2(a.x & b.x, a.y & b.y); }
__device__ __forceinline__ bool any2(uint2 a) { return (a.x | a.y) != 0u; }
__device__ __forceinline__ int popc2(uint2 a) { return __popc(a.x) + __popc(a.y); }

// horizontal dilation by 1, 2 and 6 columns each way
__device__ __forceinline__ uint2 hdil1(uint2 m) { return make_uint2(m.x | m.y | (m.y << 1), m.y | m.x | (m.x >> 1)); }
__device__ __forceinline__ uint2 hdil2(uint2 m) {
  return make_uint2(m.x | (m.x << 1) | (m.x >> 1) | m.y | (m.y << 1), m.y | (m.y << 1) | (m.y >> 1) | m.x | (m.x >> 1));
}
__device__ __forceinline__ uint2 hdil6(uint2 m) { return hdil2(hdil2(hdil2(m))); }
// all of the five columns around each
__device__ __forceinline__ uint2 hero2(uint2 m) {
  return make_uint2(m.x & (m.x << 1) & (m.x >> 1) & m.y & (m.y << 1), m.y & (m.y << 1) & (m.y >> 1) & m.x & (m.x >> 1));
}
// columns [lo, hi), 0 <= lo
__device__ __forceinline__ uint2 cols2(int lo, int hi) {
  return make_uint2(bits_between((lo + 1) >> 1, (hi + 1) >> 1), bits_between(lo >> 1, hi >> 1));
}
__device__ __forceinline__ void set_bit2(uint2* row, int c) {
  atomicOr((c & 1) ? &row->y : &row->x, 1u << (c >> 1));
}

// ORs the tile's columns (8 .. 55, the low 24 bits of v >> 4) of one parity into
// its bit stream `o` of a plane row (the stream's first word).
__device__ __forceinline__ void or_plane(uint32_t* o, int x0, uint32_t v) {
  v = (v >> 4) & 0xffffffu;
  const int b = x0 / 2, sh = b & 31;
  if (v << sh) atomicOr(o + (b >> 5), v << sh);
  if (sh > 8 && (v >> (32 - sh))) atomicOr(o + (b >> 5) + 1, v >> (32 - sh));
}

// 16-byte asynchronous global -> shared copy, past L1
__device__ __forceinline__ void cp_async16(void* sdst, const void* gsrc) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(sdst)), "l"(gsrc) : "memory");
}

// A tile's place in its frame: row r, column c of the image region is pixel
// (x0 - 8 + c, y0 - 8 + r); [c0, c1) x [r0, r1) is the part inside the frame.
struct TilePos {
  int x0, y0, c0, c1, r0, r1;
  bool edge;  // part of the region within 6 px of the tile lies outside the frame
  // the columns within k px of the tile, in the frame
  __device__ __forceinline__ uint2 cols(int k) const { return cols2(max(8 - k, c0), min(8 + kT2W + k, c1)); }
  template <int TH>
  __device__ __forceinline__ bool row_in(int r, int k) const {
    return r >= max(8 - k, r0) && r < min(8 + TH + k, r1);
  }
};

// Bits of region row `gy` (clamped by the caller) of a flag plane, the columns
// outside the frame taking the flag of the frame's edge column. ahead: read before
// the wait (pdl_wait), past L1.
__device__ __forceinline__ uint2 plane_row(const uint32_t* __restrict__ plane, int wps, int gy, const TilePos& T,
                                           bool ahead) {
  const int b = T.x0 / 2 - 4, wi = b >> 5, sh = b & 31;
  uint32_t v[2], lo[2], hi[2];
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const uint32_t* p = plane + (size_t(gy) * 2 + j) * wps;
    auto word = [&](int i) { return i < 0 || i >= wps ? 0u : ahead ? __ldcg(p + i) : p[i]; };
    lo[j] = word(wi);
    hi[j] = word(wi + 1);
  }
#pragma unroll
  for (int j = 0; j < 2; ++j) v[j] = __funnelshift_r(lo[j], hi[j], sh);
  uint2 m = make_uint2(v[0], v[1]);
  if (T.c0 > 0) {  // columns left of the frame
    const uint2 out = cols2(0, T.c0);
    const bool e = (((T.c0 & 1) ? m.y : m.x) >> (T.c0 >> 1)) & 1u;
    m = e ? or2(m, out) : make_uint2(m.x & ~out.x, m.y & ~out.y);
  }
  if (T.c1 < 64) {
    const uint2 out = cols2(T.c1, 64);
    const int c = T.c1 - 1;
    const bool e = (((c & 1) ? m.y : m.x) >> (c >> 1)) & 1u;
    m = e ? or2(m, out) : make_uint2(m.x & ~out.x, m.y & ~out.y);
  }
  return m;
}

// Reserves n entries of a list for the calling lane (whole warp): its offset.
__device__ __forceinline__ int warp_reserve(int n, int* count) {
  const int lane = threadIdx.x & 31;
  int incl = n;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  int base = 0;
  if (lane == 31 && incl) base = atomicAdd(count, incl);
  return __shfl_sync(0xffffffffu, base, 31) + incl - n;
}

// Rows r-2 .. r+2 and columns c0-2 .. c0+3 (c0 even) of a map with its row 0 at `a`.
__device__ __forceinline__ void load_pair_smem(const float* a, int r, int c0, float (&v)[5][6]) {
  const float2* p = reinterpret_cast<const float2*>(a + (r - 2) * kT2P + c0 - 2);
#pragma unroll
  for (int dy = 0; dy < 5; ++dy)
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const float2 t = p[dy * (kT2P / 2) + q];
      v[dy][2 * q] = t.x;
      v[dy][2 * q + 1] = t.y;
    }
}

// The 5x5 median at (r, c), c0 = c & ~1 the pair's column, the window clamped to rows [rlo, rhi] and columns [clo,
// chi]: the network of the S and S' stages, for the rare exact path only.
__device__ __noinline__ float median25_at(const float* a, int r, int c, int rlo, int rhi, int clo, int chi) {
  const int c0 = c & ~1;
  float v[5][6], m[2];
#pragma unroll
  for (int dy = 0; dy < 5; ++dy)
#pragma unroll
    for (int dx = 0; dx < 6; ++dx)
      v[dy][dx] = a[clampi(r - 2 + dy, rlo, rhi) * kT2P + clampi(c0 - 2 + dx, clo, chi)];
  med25_row2(v, m);
  return (c & 1) ? m[1] : m[0];
}

// med3 at (r, c) of the image region.
__device__ __noinline__ float med3_at(const float* a, int r, int c) {
  const float* p = a + (r - 1) * kT2P + c - 1;
  float lo[3], mi[3], hi[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) sort3(p[d], p[d + kT2P], p[d + 2 * kT2P], lo[d], mi[d], hi[d]);
  return med3f(max3f(lo[0], lo[1], lo[2]), med3f(mi[0], mi[1], mi[2]), min3f(hi[0], hi[1], hi[2]));
}

// Scale of the objlim test of a pixel: the test holds for a value v of the 7x7
// window in the place of the median exactly where S'/max(F/N, 0.01) > objlim
// with F = m3 - v (article form: 2S for S'), that is where F < X up to
// rounding, X = N * num / objlim. The four roundings stay within 2^-22, so F
// outside X (1 -+ 2e-6) decides; num/objlim near 0.01 or below, or an X or objlim
// out of the normal range, is marked -1 (decided step by step), and num/objlim <
// 0.0099 can never pass (0: F/N is floored at 0.01).
__device__ __forceinline__ float test_scale(float num, float nn, float objlim) {
  const float q = __fdiv_rn(num, objlim), x = __fmul_rn(q, nn);
  if (q < 0.0099f) return 0.f;
  return (q > 0.0101f && x > 1e-30f && x < 1e38f && objlim > 1e-30f) ? x : -1.f;
}

__device__ __forceinline__ bool test_holds(const Params& p, float fval, float nn, float num) {
  return __fdiv_rn(num, fmaxf(__fdiv_rn(fval, nn), 0.01f)) > p.objlim;
}

// The objlim test at row rc >> 6, column rc & 63 by the stated steps for each value of the window, by a whole warp: N and S' by the
// networks again, then a value per lane (800 x 800 with objlim 500: one lane per test 105 us, this 54; 137 x 137 with
// values up to 1e38: 327, this 78). m3: med3 of the region, or nullptr where it is formed from J.
__device__ __noinline__ bool test_exact(const float* J, const float* S, const float* m3, int rc, int rlo, int rhi, int clo,
                                        int chi, float gain, float rn2, Params p) {
  const int lane = threadIdx.x & 31, r = rc >> 6, c = rc & 63;
  const float mc = m3 ? m3[r * kT2P + c] : med3_at(J, r, c);
  const float nn = noise_of(floor_m5(median25_at(J, r, c, 0, r + 2, 0, 63)), gain, rn2);
  const float s = S[r * kT2P + c];
  const float num = p.objlim_form == 1 ? __fmul_rn(2.f, s) : __fsub_rn(s, median25_at(S, r, c, rlo, rhi, clo, chi));
  int m = 0;
  for (int i = lane; i < 64; i += 32) {
    bool holds = false;
    if (i < 49) {
      const int y = clampi(r - 3 + i / 7, rlo, rhi), x = clampi(c - 3 + i % 7, clo, chi);
      holds = test_holds(p, __fsub_rn(mc, m3 ? m3[y * kT2P + x] : med3_at(J, y, x)), nn, num);
    }
    m += __popc(__ballot_sync(0xffffffffu, holds));
  }
  return m >= 25;
}

// resident blocks per SM the kernels are compiled for
constexpr int tile_blocks(int mode, bool many) { return mode == 1 && !many ? 4 : 4 + mode; }

// The frame of tile t (frame_of) by a whole warp, read past L1: each step of the search looks at 32 frames at once
// (a binary search's steps wait for memory one after another).
__device__ __forceinline__ int frame_of_ahead(const Frame* frames, int nframes, long long t) {
  const int lane = threadIdx.x & 31;
  int lo = 0;
  for (int n = nframes, step; n > 1; n = min(step, nframes - lo)) {  // the frame is one of lo .. lo + n - 1
    step = (n + 31) / 32;
    const int i = lo + lane * step;
    const bool at = lane * step < n && __ldcg(&frames[i].tile0) <= t;
    lo += (__popc(__ballot_sync(0xffffffffu, at)) - 1) * step;
  }
  return lo;
}

// What a launch does before pdl_wait depends on nothing the launch ahead of it
// writes: iteration 1 of a call of one frame (kSolo: the descriptor `one` comes
// with the launch) needs only the input until it writes its flags, so it runs
// beside the upload; later launches load M_{k-2}, iteration 2 the input, and those
// of a batch the descriptor, while the launch ahead ends (letting the next launch
// start so early: 40.6 -> 38.9 us on 137 x 137, 54.0 -> 52.8 on 800 x 800). These
// loads go past L1 (pdl_wait's comment). Only the blocks of the first round of
// resident ones (first_round of them) can start so early; the others wait first,
// which costs them nothing, and load through L1, where the descriptor is (every
// block ahead: 189 us on 2048 x 2048, and 191 on six frames of 801 x 799).
// One frame's descriptor is read as launch parameters: 185 -> 174 us on 2048 x
// 2048, 52.0 -> 51.0 on 800 x 800 against a copy in shared memory.
// kMode 0: iteration 1. 1: the replacement of iteration k-1, then iteration k.
// 2: the replacement of iteration niter (k = niter + 1) and the u8 mask.
template <int TH, int kMode, bool kMany, bool kSolo>
__global__ void __launch_bounds__(256, tile_blocks(kMode, kMany))
    tile_kernel(const Frame* __restrict__ frames, int nframes, Params p, int k, int niter, int first_round,
                const __grid_constant__ Frame one) {
  using L = TileLayout<TH, kMode>;
  constexpr int R = L::R;
  extern __shared__ __align__(128) char smem[];
  float* sJ = reinterpret_cast<float*>(smem) + L::oJ;             // rows 0 .. R-1
  float* sS = reinterpret_cast<float*>(smem) + L::oS - 4 * kT2P;  // rows 4 .. R-5
  float* sN = reinterpret_cast<float*>(smem) + L::oN - 6 * kT2P;  // rows 6 .. R-7; the test scale where tested
  float* sM3 = reinterpret_cast<float*>(smem) + L::oM3 - 3 * kT2P;  // rows 3 .. R-4
  float* val = reinterpret_cast<float*>(smem) + L::oS;            // replacement values (before S and N)
  uint2* mM = reinterpret_cast<uint2*>(smem + L::oMask);          // M_{k-1}
  uint2* mF = mM + R;                                             // new in M_{k-1}; then the pixels near a change
  uint2* mC = mF + R;                                             // changed pixels
  uint2* mHot = mC + R;
  uint2* mAct = mHot + R;
  uint2* mT = mAct + R;  // S' > sigclip
  uint2* mLow = mT + R;  // S' > sigfrac * sigclip
  uint2* mG = mLow + R;  // candidates
  uint16_t* L0 = reinterpret_cast<uint16_t*>(smem + L::oL0);
  uint16_t* L1 = reinterpret_cast<uint16_t*>(smem + L::oL1);
  int* cnt = reinterpret_cast<int*>(smem + L::oCnt);  // 0 replacement, 1 S and S', 3 tests, 4 full windows, 5.. work
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  // the bit maps and counters, and the frame's descriptor
  for (int i = tid; i < (kMode == 2 ? 0 : 6 * R); i += 256) mC[i] = make_uint2(0u, 0u);
  if (tid < 16) cnt[tid] = 0;
  __shared__ Frame sf;
  const Frame& f = [&]() -> const Frame& {
    if constexpr (kSolo) return one;
    else return sf;
  }();
  const bool ahead = int(blockIdx.x) < first_round && (kMode != 0 || kSolo);
  if (!ahead) {
    pdl_wait();
    if (kMode == 1 || (kMode == 0 && !kSolo)) pdl_launch();
  }
  if constexpr (!kSolo) {
    const uint32_t* d = reinterpret_cast<const uint32_t*>(
        frames + (ahead ? frame_of_ahead(frames, nframes, blockIdx.x) : frame_of<false>(frames, nframes, blockIdx.x)));
    for (int i = tid; i < int(sizeof(Frame) / 4); i += 256)
      reinterpret_cast<uint32_t*>(&sf)[i] = ahead ? __ldcg(d + i) : d[i];
    __syncthreads();
  }
  const int w = f.w, h = f.h, wps = f.wps;
  TilePos T;
  {
    const int tile = int((long long)blockIdx.x - f.tile0), ty = tile / f.tiles_x;
    T.x0 = (tile - ty * f.tiles_x) * kT2W;
    T.y0 = ty * TH;
    T.c0 = max(8 - T.x0, 0);
    T.c1 = min(w - T.x0 + 8, 64);
    T.r0 = max(8 - T.y0, 0);
    T.r1 = min(h - T.y0 + 8, R);
    T.edge = T.c0 > 2 || T.r0 > 2 || T.c1 < 62 || T.r1 < R - 2;
  }

  const float* src = kMode == 0 ? f.img : iter_src(f, k - 1, niter);

  // the image region (mode 2: the tile and the 2 rows around it), clamped into the frame; ahead of the wait past
  // L1, single values too (a 4-byte cp.async exists through L1 only)
  const bool early = ahead && (kMode == 0 || k == 2);
  auto load_image = [&] {
    constexpr int ra = kMode == 2 ? 6 : kMode == 0 ? 2 : 0, rb = R - ra;
    if ((w & 3) == 0 && (reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
      for (int i = tid; i < (rb - ra) * 16; i += 256) {
        const int r = ra + (i >> 4), c = (i & 15) * 4, gx = T.x0 - 8 + c;
        const float* row = src + size_t(clampi(T.y0 - 8 + r, 0, h - 1)) * w;
        float* d = sJ + r * kT2P + c;
        if (gx >= 0 && gx < w) {
          cp_async16(d, row + gx);
        } else {
          const float* e = row + (gx < 0 ? 0 : w - 1);
          if (early) {
            const float v = __ldcg(e);
            *reinterpret_cast<float4*>(d) = make_float4(v, v, v, v);
          } else {
#pragma unroll
            for (int q = 0; q < 4; ++q) cp_async4(d + q, e);
          }
        }
      }
    } else {  // a row per warp
      const int ca = clampi(T.x0 - 8 + lane, 0, w - 1), cb = clampi(T.x0 + 24 + lane, 0, w - 1);
      if (early) {
        constexpr int kRows = (rb - ra + 7) / 8;
        float va[kRows], vb[kRows];
#pragma unroll
        for (int j = 0; j < kRows; ++j) {
          const float* row = src + size_t(clampi(T.y0 - 8 + min(ra + warp + 8 * j, rb - 1), 0, h - 1)) * w;
          va[j] = __ldcg(row + ca);
          vb[j] = __ldcg(row + cb);
        }
#pragma unroll
        for (int j = 0; j < kRows; ++j) {
          const int r = ra + warp + 8 * j;
          if (r >= rb) continue;
          sJ[r * kT2P + lane] = va[j];
          sJ[r * kT2P + lane + 32] = vb[j];
        }
      } else {
        for (int r = ra + warp; r < rb; r += 8) {
          const float* row = src + size_t(clampi(T.y0 - 8 + r, 0, h - 1)) * w;
          cp_async4(sJ + r * kT2P + lane, row + ca);
          cp_async4(sJ + r * kT2P + lane + 32, row + cb);
        }
      }
    }
    cp_async_commit();
  };
  const uint2 own = T.cols(0);
  if (kMode == 0 || k == 2) load_image();

  if (kMode != 0) {
    const int kr = k - 1;  // the iteration whose replacement this is
    static_assert(R <= 256, "a thread per row");
    const int gy = clampi(T.y0 - 8 + tid, 0, h - 1);
    uint2 before = make_uint2(0u, 0u);
    if (tid < R) before = plane_row(f.mp[(kr + 2) % 3], wps, gy, T, ahead);
    if (ahead) {
      pdl_wait();
      if (kMode == 1) pdl_launch();  // the last kernel's results are the caller's: nothing starts before they are whole
    }
    if (tid < R) {
      const uint2 a = plane_row(f.mp[kr % 3], wps, gy, T, false);
      mM[tid] = a;
      mF[tid] = make_uint2(a.x & ~before.x, a.y & ~before.y);
    }
    if (k != 2) load_image();
    __syncthreads();
    // list the flagged pixels whose value can change
    constexpr int kReach = kMode == 2 ? 0 : 6;
    if (warp * 32 < R) {
      uint2 m = make_uint2(0u, 0u);
      if (tid < R && T.row_in<TH>(tid, kReach)) {
        uint2 fr = m, er = make_uint2(~0u, ~0u);
#pragma unroll
        for (int d = -2; d <= 2; ++d) {
          fr = or2(fr, mF[tid + d]);
          er = and2(er, mM[tid + d]);
        }
        m = and2(mM[tid], T.cols(kReach));
        const uint2 full = and2(hero2(er), m);
        m = and2(m, or2(hdil2(fr), full));
        if (any2(full)) {
          cnt[4] = 1;
          const int n = T.row_in<TH>(tid, 0) ? popc2(and2(full, own)) : 0;
          if (n) atomicAdd(f.counters + 2 * (kr - 1) + 1, (unsigned long long)n);
        }
      }
      int o = warp_reserve(popc2(m), &cnt[0]);
#pragma unroll
      for (int j = 0; j < 2; ++j)
        for (uint32_t v = j ? m.y : m.x; v; v &= v - 1u) L0[o++] = uint16_t((tid << 6) | (2 * (__ffs(v) - 1) + j));
    }
  }
  // I_{k-1} of the tile, by the threads from `first` on: the first write into each image buffer is whole,
  // later ones the flagged pixels
  auto write_image = [&](int first) {
    float* __restrict__ dst = iter_dst(f, k - 1, niter);
    if (k - 1 <= 2) {
      if ((w & 3) == 0 && (reinterpret_cast<uintptr_t>(dst) & 15u) == 0) {
        for (int i = tid - first; i < TH * 12; i += 256 - first) {
          const int r = 8 + i / 12, c = 8 + (i % 12) * 4;
          if (r < T.r1 && c < T.c1)
            *reinterpret_cast<float4*>(dst + size_t(T.y0 - 8 + r) * w + T.x0 - 8 + c) =
                *reinterpret_cast<const float4*>(sJ + r * kT2P + c);
        }
      } else {
        for (int r = 8 + (tid - first) / 32; r < min(8 + TH, T.r1); r += (256 - first) / 32) {  // a row per warp
          float* row = dst + size_t(T.y0 - 8 + r) * w + T.x0 - 8;
          if (8 + lane < T.c1) row[8 + lane] = sJ[r * kT2P + 8 + lane];
          if (lane < kT2W - 32 && 40 + lane < T.c1) row[40 + lane] = sJ[r * kT2P + 40 + lane];
        }
      }
    } else if (tid - first < 2 * TH) {  // a thread per row and parity
      const int r = 8 + ((tid - first) >> 1), j = (tid - first) & 1;
      if (r < T.r1) {
        const uint2 m = and2(mM[r], own);
        uint32_t v = j ? m.y : m.x;
        while (v) {
          const int c = 2 * (__ffs(v) - 1) + j;
          v &= v - 1u;
          dst[size_t(T.y0 - 8 + r) * w + T.x0 - 8 + c] = sJ[r * kT2P + c];
        }
      }
    }
  };
  cp_async_wait_all();
  __syncthreads();

  if (kMode != 0) {
    const int nR = cnt[0];
    const bool full = cnt[4] != 0;  // a fully flagged window reads replaced values: compute all, then write
    bool changed = false;
    for (int j = tid; j < nR; j += 256) {
      const int r = L0[j] >> 6, c = L0[j] & 63;
      const int i0 = (c >> 1) - 1, od = c & 1;
      // window columns c-2 .. c+2: three of c's parity from bit i0, two of the other from bit i0 + od
      uint32_t ws[5], wo[5];
      int nf = 0;
#pragma unroll
      for (int dy = 0; dy < 5; ++dy) {
        const uint2 m = mM[r - 2 + dy];
        ws[dy] = ((od ? m.y : m.x) >> i0) & 7u;
        wo[dy] = ((od ? m.x : m.y) >> (i0 + od)) & 3u;
        nf += __popc(ws[dy]) + __popc(wo[dy]);
      }
      const int n = 25 - nf;
      const int a = n > 0 ? 13 - (n + 1) / 2 : 0;  // flagged entries sent to -inf; the others to +inf
      float v[25];
      int seen = 0;
#pragma unroll
      for (int q = 0; q < 25; ++q) {
        const int dy = q / 5, dx = q % 5;
        float x = sJ[(r - 2 + dy) * kT2P + c - 2 + dx];
        const uint32_t bit = (dx & 1) ? (wo[dy] >> (dx >> 1)) & 1u : (ws[dy] >> (dx >> 1)) & 1u;
        if (bit && n > 0) {
          x = (seen < a) ? -INFINITY : INFINITY;
          ++seen;
        }
        v[q] = x;
      }
      float out = sel_med25(v);
      if (n == 0) out = floor_m5(out);
      if (kMode == 1 && __float_as_uint(out) != __float_as_uint(sJ[r * kT2P + c])) {
        changed = true;
        set_bit2(&mC[r], c);
      }
      if (full)
        val[j] = out;
      else
        sJ[r * kT2P + c] = out;
    }
    if (full) {
      __syncthreads();
      for (int j = tid; j < nR; j += 256) sJ[(L0[j] >> 6) * kT2P + (L0[j] & 63)] = val[j];
    }
    const bool any = __syncthreads_or(changed);
    if (kMode == 2) {
      write_image(0);
      uint8_t* __restrict__ om = f.out_mask;
      if (!om) return;
      if ((w & 15) == 0 && (reinterpret_cast<uintptr_t>(om) & 15u) == 0) {
        for (int i = tid; i < TH * 3; i += 256) {
          const int r = 8 + i / 3, c = 8 + (i % 3) * 16;
          if (r >= T.r1 || c >= T.c1) continue;
          const uint2 m = mM[r];
          uint32_t e = m.x >> (c >> 1), o = m.y >> (c >> 1), q[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            q[j] = (e & 1u) | (o & 1u) << 8 | (e & 2u) << 15 | (o & 2u) << 23;
            e >>= 2;
            o >>= 2;
          }
          *reinterpret_cast<uint4*>(om + size_t(T.y0 - 8 + r) * w + T.x0 - 8 + c) = make_uint4(q[0], q[1], q[2], q[3]);
        }
      } else {
        for (int r = 8 + warp; r < min(8 + TH, T.r1); r += 8) {  // a row per warp
          uint8_t* row = om + size_t(T.y0 - 8 + r) * w + T.x0 - 8;
          const uint32_t m = (lane & 1) ? mM[r].y : mM[r].x;
          if (8 + lane < T.c1) row[8 + lane] = uint8_t((m >> (4 + (lane >> 1))) & 1u);
          if (lane < kT2W - 32 && 40 + lane < T.c1) row[40 + lane] = uint8_t((m >> (20 + (lane >> 1))) & 1u);
        }
      }
      return;
    }
    if (!any) {  // J did not change within 6 px: no new flag
      write_image(0);
      if (tid < 2 * TH) {
        const int r = 8 + (tid >> 1), j = tid & 1;
        if (r < T.r1) {
          const uint2 m = and2(mM[r], own);
          or_plane(f.mp[k % 3] + (size_t(T.y0 - 8 + r) * 2 + j) * wps, T.x0, j ? m.y : m.x);
        }
      }
      return;
    }
    if (T.edge) {  // the frame's edge pixels may have changed: replicate them again
      for (int i = tid; i < (R - 4) * 64; i += 256) {
        const int r = 2 + (i >> 6), c = i & 63;
        const int rr = clampi(r, T.r0, T.r1 - 1), cc = clampi(c, T.c0, T.c1 - 1);
        if (rr != r || cc != c) sJ[r * kT2P + c] = sJ[rr * kT2P + cc];
      }
      __syncthreads();
    }
  }

  const float gain = f.gain, rn2 = __fmul_rn(f.rn, f.rn);
  // ---- rows: a warp per band
  {
    const float kl = f.bkl, kh = f.bkh;
    // iteration 1: bands of the rows of med3; later ones, with few tests, form med3 at the tests and take the
    // rows of the bound test only, warp 7 meanwhile the pixels within 6 px of a change
    constexpr int BR = kMode == 0 ? L::BR : (L::R2 + 6) / 7;
    const int ra = (kMode == 0 ? 3 : 6) + warp * BR;
    bool work = true;
    if (kMode == 1) {
      if (warp == 7) {
        for (int r = lane; r < R; r += 32) {
          uint2 z = make_uint2(0u, 0u);
#pragma unroll
          for (int d = -6; d <= 6; ++d)
            if (r + d >= 0 && r + d < R) z = or2(z, mC[r + d]);
          mF[r] = hdil6(z);
        }
        work = false;
      } else {  // a change within 8 rows
        const int rr = ra - 8 + lane;
        work = __any_sync(0xffffffffu, lane < BR + 16 && rr >= 0 && rr < R && any2(mC[rr]));
      }
    }
    if (work) {
      const uint2 cm = T.cols(2);
      float2 v[BR + 4];
#pragma unroll
      for (int j = 0; j < BR + 4; ++j) v[j] = *reinterpret_cast<const float2*>(sJ + (ra - 2 + j) * kT2P + 2 * lane);
      float me[BR], mo[BR];  // medians of the five rows around each row
#pragma unroll
      for (int j = 0; j + 1 < BR; j += 2) {
        Col4 A{v[j].x, v[j + 1].x, v[j + 2].x, v[j + 3].x}, B{v[j].y, v[j + 1].y, v[j + 2].y, v[j + 3].y};
        col_step(A, v[j + 4].x, v[j + 5].x, me[j], me[j + 1]);
        col_step(B, v[j + 4].y, v[j + 5].y, mo[j], mo[j + 1]);
      }
      if (BR & 1) {
        constexpr int j = BR - 1;
        const float a[5] = {v[j].x, v[j + 1].x, v[j + 2].x, v[j + 3].x, v[j + 4].x};
        const float b[5] = {v[j].y, v[j + 1].y, v[j + 2].y, v[j + 3].y, v[j + 4].y};
        me[j] = sel_med5(a);
        mo[j] = sel_med5(b);
      }
#pragma unroll
      for (int j = 0; j < BR; ++j) {
        const int r = ra + j;
        const float2 up = v[j + 1], ce = v[j + 2], dn = v[j + 3];
        if (kMode == 0) {  // med3 from the sorted columns, as bound_span
          float le, ne, he, lo, no, ho;
          sort3(up.x, ce.x, dn.x, le, ne, he);
          sort3(up.y, ce.y, dn.y, lo, no, ho);
          const float pl = __shfl_up_sync(0xffffffffu, lo, 1), pn = __shfl_up_sync(0xffffffffu, no, 1),
                      ph = __shfl_up_sync(0xffffffffu, ho, 1);
          const float ql = __shfl_down_sync(0xffffffffu, le, 1), qn = __shfl_down_sync(0xffffffffu, ne, 1),
                      qh = __shfl_down_sync(0xffffffffu, he, 1);
          const float mn = fminf(ne, no), mx = fmaxf(ne, no);
          float2 m3;
          m3.x = med3f(max3f(pl, le, lo), fmaxf(mn, fminf(mx, pn)), min3f(ph, he, ho));
          m3.y = med3f(max3f(le, lo, ql), fmaxf(mn, fminf(mx, qn)), min3f(he, ho, qh));
          *reinterpret_cast<float2*>(sM3 + r * kT2P + 2 * lane) = m3;
        }
        if (!T.row_in<TH>(r, 2)) continue;  // whole warp
        const float pe = __shfl_up_sync(0xffffffffu, me[j], 1), po = __shfl_up_sync(0xffffffffu, mo[j], 1);
        const float ne = __shfl_down_sync(0xffffffffu, me[j], 1), no = __shfl_down_sync(0xffffffffu, mo[j], 1);
        const float left = __shfl_up_sync(0xffffffffu, ce.y, 1), right = __shfl_down_sync(0xffffffffu, ce.x, 1);
        const float com = fminf(min3f(po, me[j], mo[j]), ne);
        const float dh = __fsub_rn(ce.y, ce.x);
        const float lpe = lplus_d(__fsub_rn(ce.x, up.x), __fsub_rn(ce.x, dn.x), __fsub_rn(ce.x, left), -dh);
        const float lpo = lplus_d(__fsub_rn(ce.y, up.y), __fsub_rn(ce.y, dn.y), dh, __fsub_rn(ce.y, right));
        bool ae, he, ao, ho;
        bound_test(lpe, fminf(com, pe), gain, rn2, kl, kh, ae, he);
        bound_test(lpo, fminf(com, no), gain, rn2, kl, kh, ao, ho);
        const unsigned be = __ballot_sync(0xffffffffu, ae), bo = __ballot_sync(0xffffffffu, ao);
        const unsigned ge = __ballot_sync(0xffffffffu, he), go = __ballot_sync(0xffffffffu, ho);
        if (lane == 0) {
          mAct[r] = make_uint2(be & cm.x, bo & cm.y);
          mHot[r] = make_uint2(ge & cm.x, go & cm.y);
        }
      }
    }
  }
  __syncthreads();

  // ---- need: nsp = dilate5(hot) & act, needS = dilate5(nsp), as lists of pairs
  if (kMode == 0 && T.edge) {  // med3 outside the frame: the value at the frame's edge
    for (int i = tid; i < L::RB * 64; i += 256) {
      const int r = 3 + (i >> 6), c = i & 63;
      const int rr = clampi(r, T.r0, T.r1 - 1), cc = clampi(c, T.c0, T.c1 - 1);
      if (rr != r || cc != c) sM3[r * kT2P + c] = sM3[rr * kT2P + cc];
    }
  }
  if (warp * 32 < 2 * L::RS) {  // two lanes per row, each listing half of its pairs
    const int r = 4 + (tid >> 1);
    const uint32_t half = (tid & 1) ? 0xffff0000u : 0x0000ffffu;
    uint2 hv[9], nsp = make_uint2(0u, 0u), need = nsp, mine = nsp;
    if (tid < 2 * L::RS) {
#pragma unroll
      for (int j = 0; j < 9; ++j)
        hv[j] = (r - 4 + j >= 6 && r - 4 + j < R - 6) ? mHot[r - 4 + j] : make_uint2(0u, 0u);
#pragma unroll
      for (int j = 0; j < 5; ++j) {
        const int q = r - 2 + j;
        if (q < 6 || q >= R - 6) continue;
        uint2 n = hdil2(or2(or2(hv[j], hv[j + 1]), or2(or2(hv[j + 2], hv[j + 3]), hv[j + 4])));
        n = and2(n, mAct[q]);
        if (kMode == 1) n = and2(n, mF[q]);
        nsp = or2(nsp, n);
        if (j == 2) mine = n;
      }
      if (T.row_in<TH>(r, 4)) need = and2(hdil2(nsp), T.cols(4));
    }
    const uint32_t ps = (need.x | need.y) & half, pp = (mine.x | mine.y) & half;
    const int o = warp_reserve(__popc(ps) | __popc(pp) << 16, &cnt[1]);  // both lists at once, 16 bits each
    int os = o & 0xffff, op = o >> 16;
    for (uint32_t v = ps; v; v &= v - 1u) L0[os++] = uint16_t((r << 6) | ((__ffs(v) - 1) << 1));
    for (uint32_t v = pp; v; v &= v - 1u) {
      const int b = __ffs(v) - 1;
      L1[op++] = uint16_t((r << 7) | (b << 2) | ((mine.x >> b) & 1u) | ((mine.y >> b) & 1u) << 1);
    }
    {
      const uint2 hm = make_uint2(half, half);
      const int n = __reduce_add_sync(0xffffffffu, unsigned(popc2(and2(need, hm))) | unsigned(popc2(and2(mine, hm))) << 16);
      if (lane == 0 && n) {
        atomicAdd(&cnt[5], n & 0xffff);
        atomicAdd(&cnt[6], n >> 16);
      }
    }
  }
  __syncthreads();

  // ---- S and N
  const int nS = cnt[1] & 0xffff, nP = cnt[1] >> 16;
  for (int j = tid; j < nS; j += 256) {
    const int r = L0[j] >> 6, c0 = L0[j] & 63;
    float v[5][6], m5[2];
    load_pair_smem(sJ, r, c0, v);
    med25_row2(v, m5);
    float s[2], nn[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const float lp = lplus(v[2][i + 2], v[1][i + 2], v[3][i + 2], v[2][i + 1], v[2][i + 3]);
      nn[i] = noise_of(floor_m5(m5[i]), gain, rn2);
      s[i] = __fdiv_rn(lp, __fmul_rn(2.f, nn[i]));
    }
    *reinterpret_cast<float2*>(sS + r * kT2P + c0) = make_float2(s[0], s[1]);
    if (r >= 6 && r < R - 6) *reinterpret_cast<float2*>(sN + r * kT2P + c0) = make_float2(nn[0], nn[1]);
  }
  __syncthreads();

  // ---- S' and the thresholds; the tests with their scale. S' takes the first warps (few pairs): the others
  // write the image meanwhile
  if (kMode == 1 && warp >= 2) write_image(64);
  const float sigclip = p.sigclip, siglow = __fmul_rn(p.sigfrac, p.sigclip);
  for (int j = tid; j < nP; j += 256) {
    const int e = L1[j], r = e >> 7, c0 = ((e >> 2) & 31) * 2;
    float v[5][6], med[2];
    if (!T.edge) {
      load_pair_smem(sS, r, c0, v);
    } else {
#pragma unroll
      for (int dy = 0; dy < 5; ++dy)
#pragma unroll
        for (int dx = 0; dx < 6; ++dx)
          v[dy][dx] = sS[clampi(r - 2 + dy, T.r0, T.r1 - 1) * kT2P + clampi(c0 - 2 + dx, T.c0, T.c1 - 1)];
    }
    med25_row2(v, med);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (!((e >> i) & 1)) continue;
      const float s = v[2][i + 2], sp = __fsub_rn(s, med[i]);
      const int c = c0 + i;
      if (sp > siglow) set_bit2(&mLow[r], c);
      if (sp > sigclip) {
        set_bit2(&mT[r], c);
        const float x = test_scale(p.objlim_form == 1 ? __fmul_rn(2.f, s) : sp, sN[r * kT2P + c], p.objlim);
        if (x != 0.f) {
          sN[r * kT2P + c] = x;
          L0[atomicAdd(&cnt[3], 1)] = uint16_t((r << 6) | c);
        }
      }
    }
  }
  __syncthreads();

  // ---- the objlim test by counting, eight lanes per test (one row of the window each)
  const int nT = cnt[3];
  for (int t0 = warp * 4; t0 < nT; t0 += 32) {
    const int t = t0 + (lane >> 3), q = lane & 7;
    const bool on = t < nT;
    const int r = on ? L0[t] >> 6 : 8, c = on ? L0[t] & 63 : 8;
    const float x = sN[r * kT2P + c];
    const float xl = x * (1.f - 2e-6f), xh = x * (1.f + 2e-6f);
    float v[7], mc;  // the window's row r-3+q of med3, and its centre
    if (kMode == 0) {
      const float* row = sM3 + (r - 3 + (q < 7 ? q : 0)) * kT2P + c - 3;
#pragma unroll
      for (int d = 0; d < 7; ++d) v[d] = row[d];
      mc = sM3[r * kT2P + c];
    } else {
      if (!T.edge) {
        const float* row = sJ + (r - 4 + (q < 7 ? q : 0)) * kT2P + c - 4;
        float lo[9], mi[9], hi[9];
#pragma unroll
        for (int d = 0; d < 9; ++d) sort3(row[d], row[d + kT2P], row[d + 2 * kT2P], lo[d], mi[d], hi[d]);
#pragma unroll
        for (int d = 0; d < 7; ++d)
          v[d] = med3f(max3f(lo[d], lo[d + 1], lo[d + 2]), med3f(mi[d], mi[d + 1], mi[d + 2]),
                       min3f(hi[d], hi[d + 1], hi[d + 2]));
      } else {
#pragma unroll
        for (int d = 0; d < 7; ++d)
          v[d] = med3_at(sJ, clampi(r - 3 + (q < 7 ? q : 0), T.r0, T.r1 - 1), clampi(c - 3 + d, T.c0, T.c1 - 1));
      }
      mc = __shfl_sync(0xffffffffu, v[3], (lane & 24) | 3);
    }
    int n = 0;  // values that pass; values that do not fail, in the upper half
    if (on && q < 7) {
#pragma unroll
      for (int d = 0; d < 7; ++d) {
        const float fv = __fsub_rn(mc, v[d]);
        n += (fv >= xl ? 0 : 1) + (fv > xh ? 0 : 65536);  // infinity less itself passes, as F/N floored at 0.01 does
      }
    }
    n += __shfl_xor_sync(0xffffffffu, n, 1);
    n += __shfl_xor_sync(0xffffffffu, n, 2);
    n += __shfl_xor_sync(0xffffffffu, n, 4);
    bool cand = (n & 0xffff) >= 25;
    const bool open = on && q == 0 && (x < 0.f || (!cand && (n >> 16) >= 25));  // the count cannot decide
    for (unsigned m = __ballot_sync(0xffffffffu, open); m; m &= m - 1u) {
      const int l = __ffs(m) - 1;
      const bool holds = test_exact(sJ, sS, kMode == 0 ? sM3 : nullptr, L0[t0 + (l >> 3)], T.r0, T.r1 - 1, T.c0,
                                    T.c1 - 1, gain, rn2, p);
      if (lane == l) cand = holds;
    }
    if (!on || q != 0) continue;
    if (open) atomicAdd(&cnt[7], 1);
    if (cand) set_bit2(&mG[r], c);
  }
  __syncthreads();

  // ---- both growths; M_k = M_{k-1} | g2
  if (kMode == 0 && kSolo) {
    pdl_wait();
    pdl_launch();
  }
  if (warp * 32 < TH) {
    const int r = 8 + tid;
    int fresh = 0;
    if (tid < TH && r < T.r1) {
      uint2 g = make_uint2(0u, 0u);
#pragma unroll
      for (int j = -1; j <= 1; ++j)
        g = or2(g, and2(hdil1(or2(or2(mG[r + j - 1], mG[r + j]), mG[r + j + 1])), mT[r + j]));
      g = and2(and2(hdil1(g), mLow[r]), own);
      const uint2 old = kMode == 0 ? make_uint2(0u, 0u) : and2(mM[r], own);
      fresh = popc2(make_uint2(g.x & ~old.x, g.y & ~old.y));
      const uint2 m = or2(g, old);
      uint32_t* o = f.mp[k % 3] + size_t(T.y0 - 8 + r) * 2 * wps;
      or_plane(o, T.x0, m.x);
      or_plane(o + wps, T.x0, m.y);
    }
    fresh = __reduce_add_sync(0xffffffffu, unsigned(fresh));
    if (lane == 0 && fresh) atomicAdd(f.counters + 2 * (k - 1), (unsigned long long)fresh);
  }
  if (tid == 255) {
    unsigned long long* wk = f.work + kWork * (k - 1);
    auto span = [&](int m) {
      return (long long)(min(8 + kT2W + m, T.c1) - max(8 - m, T.c0)) * (min(8 + TH + m, T.r1) - max(8 - m, T.r0));
    };
    if (cnt[5]) {
      atomicAdd(wk + 0, (unsigned long long)cnt[5]);
      atomicAdd(wk + 1, (unsigned long long)cnt[6]);
    }
    atomicAdd(wk + 2, (unsigned long long)(kMode == 0 ? span(5) : 49ll * nT));
    if (nT) atomicAdd(wk + 3, (unsigned long long)nT);
    if (cnt[7]) atomicAdd(wk + 4, (unsigned long long)cnt[7]);
    atomicAdd(wk + 5, (unsigned long long)span(2));
  }
}

}  // namespace crb
