// Normal-matrix sums in image space: tap sums, mask-edge sums and the chains
// that join them.
//
// Every entry of the kernel-kernel block is
//   F_m(u, u') = sum_x M(x) m(x) R(x - u) R(x - u'),   m = xt^a yt^b,
// with M the 0/1 fit mask and R the masked, sky-subtracted reference.  Moving
// both offsets by one pixel e only moves the mask against the images:
//   F(u + e, u' + e) = shift_e( F(u, u') + H(u, u') ),
//   H_m(u, u') = sum_x [M(x + e) - M(x)] m(x) R(x - u) R(x - u'),
// where shift_e substitutes xt + 2 e_x / (W - 1), yt + 2 e_y / (H - 1) in the
// monomials.  M(x + e) - M(x) is non-zero only on the mask's edges, so for
// each difference d = u - u' one sum over the image is enough (a corner of
// the offset box) and the edges give the other offsets:
//   * tap sums (k_tap_sums): per tile of 32 rows, sum_x c(x) xt^a R(x - u')
//     for the L^2 offsets u', with c = M R(. - u0) for the two upper corners
//     u0 = (+-w, w) (between them every half-plane d), and c = M S' (the
//     right-hand side) or the refinement residual; yt^b at the tile's end.
//   * edge sums (k_edge_gram): H for every pair, over the lists of mask edges
//     in x (offsets with u_y = w) and in y (all offsets below w).
//   * chains (k_edge_chain): along x at u_y = w, then down in y, in FP64.
// At 2048 x 4096, L = 11, D_K = 2 a CCD takes 221 sums over the image in place
// of 7381, and its mask has 10^4 - 10^5 edges against 8.4e6 pixels.  L <= 5
// sums every pair over the image (15 distinct u_y rows of 5 taps at L = 5):
// fewer launches, and no edges to list.
#include <algorithm>
#include <vector>

#include "common.cuh"
#include "plan.h"
#include "tap.cuh"

namespace sfft {

template <typename T>
__host__ __device__ constexpr size_t tap_smem(int wt, int tw) {
  const int pitch = (tw + 2 * wt) | 1, spitch = tw | 1;
  return sizeof(T) * ((size_t)5 * kTapScrPitch + (size_t)kTapWarps * kTapScr * kTapScrPitch + 4 * (size_t)tw +
                      (size_t)(kTapRows + 2 * wt) * pitch + (size_t)kTapRows * spitch) +
         4 * (size_t)kTapRows * (tw / 32);
}

// One CTA: a tile of 32 rows x tw columns and every nsplit-th task of the
// table, taken in order by its warps.  Partial sums go to
// part[ccd][tile][nout_tot]; k_tap_reduce adds the tiles in FP64.
// One 4096 x 2048 CCD, L = 11, D_K = 2: 502 us = 49 TFLOP/s, 0.65 of the FP32
// FMA peak (the row FFTs of the 221 products and their contraction took 6.0 ms);
// copies of the tile through registers took 638 us, R stored as
// operand pairs (two CTAs of six warps instead of three of four) 572 us.
template <typename T, int NT, int DK, int MODE>
__global__ void __launch_bounds__(kTapWarps * 32, sizeof(T) == 4 ? 3 : 2)
k_tap_sums(const T* __restrict__ Rm, const float* __restrict__ S, const unsigned* __restrict__ mfitw,
           const double* __restrict__ sky, const int4* __restrict__ tasks, int ntask,
           T* __restrict__ part, int nout_tot, double* __restrict__ mpart, char3 need, int H, int W, int w, int tw, double xs, double ys) {
  constexpr int wt = (NT - 1) / 2, RC = 2 * DK + 1, RS = DK + 1, RM = DK + 3;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned char ot[5][kTapMaxOut][2];
  __shared__ double ypd[5][32];
  __shared__ int next;
  const int pitch = (tw + 2 * wt) | 1, spitch = tw | 1, nw = tw / 32;
  T* yp = reinterpret_cast<T*>(smraw);
  T* scr = yp + 5 * kTapScrPitch;
  T* xp = scr + kTapWarps * kTapScr * kTapScrPitch;
  T* rt = xp + 4 * tw;
  T* st = rt + (kTapRows + 2 * wt) * pitch;
  unsigned* mw = reinterpret_cast<unsigned*>(st + kTapRows * spitch);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nth = kTapWarps * 32;
  const int ntx = (W + tw - 1) / tw;
  const int tile = blockIdx.x, ccd = blockIdx.z;
  const int x0 = (tile % ntx) * tw, y0 = (tile / ntx) * kTapRows;
  const int64_t img = (int64_t)ccd * H * W;
  if (tid == 0) next = 0;
  if (tid < 5) tap_outputs(tid, DK, ot[tid]);
  for (int i = tid; i < tw; i += nth) {
    const double x = (x0 + i) * xs - 1.0;
    xp[4 * i] = (T)x; xp[4 * i + 1] = (T)(x * x); xp[4 * i + 2] = (T)(x * x * x); xp[4 * i + 3] = (T)(x * x * x * x);
  }
  if (tid < kTapRows) {
    const double y = (y0 + tid) * ys - 1.0;
    double v = 1.0;
    for (int b = 0; b < 5; ++b) { yp[b * kTapScrPitch + tid] = (T)v; ypd[b][tid] = v; v *= y; }
  }
  // R with its halo, zero outside the image: copied asynchronously, every
  // element in flight at once (plain loads kept 29 % of the warps' time
  // waiting), a warp per row
  for (int row = warp; row < kTapRows + 2 * wt; row += kTapWarps) {
    const int gy = y0 - wt + row;
    const bool in = gy >= 0 && gy < H;
    const T* src = Rm + img + (int64_t)(in ? gy : 0) * W;
    for (int c = lane; c < tw + 2 * wt; c += 32) {
      const int gx = x0 - wt + c;
      const bool ok = in && gx >= 0 && gx < W;
      cp_async<sizeof(T)>(rt + row * pitch + c, src + (ok ? gx : 0), ok);
    }
  }
  // the mask's words and S, then M (S - s_S) in place
  {
    const int wpr = (W + 31) / 32;   // words per image row
    for (int i = tid; i < kTapRows * nw; i += nth) {
      const int gy = y0 + i / nw, wi = x0 / 32 + i % nw;
      mw[i] = gy < H && wi < wpr ? mfitw[((int64_t)ccd * H + gy) * wpr + wi] : 0u;
    }
  }
  for (int row = warp; row < kTapRows; row += kTapWarps) {
    const int gy = y0 + row;
    const int64_t o = img + (int64_t)gy * W;
#pragma unroll 4
    for (int c = lane; c < tw; c += 32) {
      const bool ok = gy < H && x0 + c < W;
      if constexpr (sizeof(T) == 4) cp_async<4>(st + row * spitch + c, S + (ok ? o + x0 + c : 0), ok);
      else st[row * spitch + c] = (T)(ok ? S[o + x0 + c] : 0.f);
    }
  }
  cp_async_wait_all();
  __syncthreads();
  const T sS = (T)sky[2 * ccd + 1];
  for (int row = warp; row < kTapRows; row += kTapWarps)
    for (int c = lane; c < tw; c += 32) {
      T* p = st + row * spitch + c;
      *p = (mw[row * nw + (c >> 5)] >> lane) & 1u ? *p - sS : (T)0;
    }
  __syncthreads();
  TapTile<T> t;
  t.r = rt + lane * pitch; t.s = st + lane * spitch; t.m = mw + lane * nw; t.xp = xp; t.yp = yp;
  t.scr = scr + warp * kTapScr * kTapScrPitch;
  t.pitch = pitch;
  t.n = min(tw, (W - x0 + kTapU - 1) / kTapU * kTapU);
  T* po = part + ((int64_t)ccd * gridDim.x + tile) * nout_tot;
  for (;;) {
    int k = 0;
    if (lane == 0) k = atomicAdd(&next, 1);
    k = __shfl_sync(0xffffffffu, k, 0) * gridDim.y + blockIdx.y;
    if (k >= ntask) break;
    const int4 q = tasks[k];   // type | nout << 8, u0 (x, y biased by 64), u'_y, first output
    const int type = q.x & 255, nout = q.x >> 8;
    const int u0x = (q.y & 255) - 64, u0y = (q.y >> 8) - 64;
    t.ot = ot[type];
    T* out = po + q.w;
    constexpr int KC = MODE == TAP_FIT_EDGE ? NT - 1 : NT;   // the corner (-w, w) has no d_x = 0
    if (type == TAP_CS) tap_task<T, NT, NT, RC, RS, false, 1>(t, u0x, u0y, q.z, nout, out);
    else if (type == TAP_C) tap_task<T, NT, KC, RC, 0, false, 1>(t, u0x, u0y, q.z, nout, out);
    else if (MODE == TAP_FIT_ALL && type == TAP_M) tap_task<T, NT, NT, RM, 0, true, 1>(t, 0, 0, q.z, nout, out);
    else tap_moments<T, true>(t, wt, w, ypd, need, mpart + ((int64_t)ccd * gridDim.x + tile) * kTapMom);
  }
}

// Sums of the tiles' partial sums, FP32 in fours and FP64 over them (FP64
// throughout on the FP64 path and for the moments, which follow the tap sums'
// nout outputs), to the G and moment arrays: dst = region << 28
// | offset, -1 = not needed.
struct TapDst {
  double* base[5];
  int64_t stride[5];   // per CCD
};

// Eight outputs (a 32-byte sector of a tile's partials) x 64 groups of tiles per
// CTA: the reads wait for memory, so more CTAs and eight reads in flight per
// thread (32 outputs x 16 groups: 15 us for the 747 outputs of the refinement).
constexpr int kRedOut = 8, kRedGroups = 64;

template <typename T>
__global__ void __launch_bounds__(kRedOut * kRedGroups)
k_tap_reduce(const T* __restrict__ part, const double* __restrict__ mpart, const int* __restrict__ dst, TapDst d,
             int ntile, int nout) {
  constexpr int NTH = kRedOut * kRedGroups;
  __shared__ double red[kRedGroups * (kRedOut + 1)];
  const int ccd = blockIdx.y, ntap = (nout + kRedOut - 1) / kRedOut;
  const bool mom = (int)blockIdx.x >= ntap;
  // lanes: the outputs of the CTA; groups of tiles
  const int nl = mom ? 1 : kRedOut, lane = threadIdx.x % nl, g = threadIdx.x / nl;
  const int o = mom ? nout + (int)blockIdx.x - ntap : (int)blockIdx.x * kRedOut + lane;
  const int q = o < nout || mom ? dst[o] : -1;
  if (mom && q < 0) return;
  double s = 0.0;
  if (mom) {
    // one output per CTA: FP64 additions of a CTA run one warp after another
    const double* p = mpart + (int64_t)ccd * ntile * kTapMom + o - nout;
#pragma unroll 4
    for (int t = g; t < ntile; t += NTH) s += p[(int64_t)t * kTapMom];
  } else if (o < nout) {
    const T* p = part + (int64_t)ccd * ntile * nout + o;
    int t = g * 4;
#pragma unroll 2
    for (; t + 3 < ntile; t += 4 * kRedGroups) {
      const T a = p[(int64_t)t * nout], b = p[(int64_t)(t + 1) * nout], c = p[(int64_t)(t + 2) * nout],
              e = p[(int64_t)(t + 3) * nout];
      s += (double)((a + b) + (c + e));
    }
    for (int k = t; k < min(t + 4, ntile); ++k) s += (double)p[(int64_t)k * nout];
  }
  const int pitch = mom ? 1 : kRedOut + 1;
  red[g * pitch + lane] = s;
  __syncthreads();
  for (int k = NTH / nl / 2; k > 0; k >>= 1) {
    if (g < k) red[g * pitch + lane] += red[(g + k) * pitch + lane];
    __syncthreads();
  }
  if (g == 0 && q >= 0) {
    const int r = q >> 28;
    d.base[r][ccd * d.stride[r] + (q & 0xfffffff)] = red[lane];
  }
}

// ------------------------------------------------------------------ edge sums
// H_m(u, u') over one list: a CTA stages 32 edge points at a time (the L^2
// reference values around each, signed powers of xt and powers of yt) and each
// thread keeps a tile of 2 x 2 (or 4) pairs x all monomials in registers.  The points
// of the next batch are copied (cp.async) while this one is summed, and the list
// is read two batches ahead; without it the gathers' latency took 60 % of the
// warps' time.  The list is in row order: a thread sums the powers of xt over a
// row's points and takes the result times the powers of yt at the row's end, 5
// multiply-adds per pair and point and 15 per row at D_K = 2 in place of 15 per
// point.  That, and two reads of neighbouring offsets for four pairs (five pairs
// with offsets of their own took ten), is for masks with many edges, whose rows
// are long.  Assembly of 4096 x 2048, L = 11, D_K = 2: bad pixels every 12 px
// 11.1 -> 6.4 ms, bad rows every 16 8.2 -> 4.4 ms (6.9 and 6.8 ms from spectra);
// four of 1024 x 2048, L = 7, bad pixels every 8 px 9.2 -> 2.0 ms (4.2 ms); one
// with saturated stars and two dead columns: 80 us in this kernel, 96 before.
// What bounds it are issue slots and shared-memory reads (about half of either);
// at D_K = 2 the 80 registers of sums leave spills of 68 bytes (FP64: 24), not in the
// loop over points.
// Slot g of U takes batches g, g + U, ..., at least kGramMin<T> points, and writes
// hp[ccd][slot][pair][NM]; a short list uses few slots.  The x-edge blocks, whose
// lists are the longer, come first.  The number of slots has a limit, a slot's
// share of a long list has none: an FP32 sum covers kGramRun rows (of at most 32
// points), then it is added to the slot's partials as an exact pair of floats
// (10^4 equal products one after another lose up to 1.3e-4 of their sum, 256 at
// most 4e-6).
constexpr int kGramPts = 32;
constexpr int kGramRun = 256;
constexpr int kGramThreads = 256;
constexpr int kGramOne = 122;     // L^2 <= 121 values, then (1, 0): the partner of single offsets
// offsets j of a tile: with few monomials a point's sums are few, and the copies
// of its patch in every block of tiles weigh more (assembly of four CCDs of
// 1000 x 300, L = 11, D_K = 0: 167 us with two, 160 us with four; at D_K = 1 and
// 512 x 512, L = 9, 115 with two and 121 with four)
constexpr int gram_tj(int DE) { return DE <= 1 ? 4 : 2; }
constexpr int kGramPatch = 124;   // even: two neighbouring offsets in one read
constexpr int kGramPow = 10;      // powers of a coordinate, in rows that spread over the banks
// least points of a slot: FP64 multiply-adds are 64 times slower than FP32
// ones, so there a short list spreads over more slots (a 512 x 512 pair, L = 7,
// D_K = 1: 853 us with 64 points, 819 us with 32).  FP32: more slots cost
// k_edge_reduce more than they give here (a 4096 x 2048 pair, L = 11, D_K = 2:
// 1742 us with 64 points, 1734 with 128, 1727 with 256) ...
template <typename T> constexpr int kGramMin = sizeof(T) == 4 ? 256 : kGramPts;
// ... but for the slots that give every SM a CTA: the lists of a small image are
// a few hundred points, one after another in a few CTAs (assembly of 512 x 512,
// L = 9, D_K = 1: 138 us without, 115 with; L = 11, D_K = 2: 195 and 167)
constexpr int kGramFew = 32;

struct GramArgs {
  const int* tiles;        // i | j << 8, the tile's first offsets: y tiles, then x tiles
  int nty, ntx, nbx;       // tiles and x blocks
  int npy, npx;            // pairs
  int gy, gx;              // most slots per list
  int fy, fx;              // slots that give every SM a CTA
  int64_t hp_stride;       // per CCD
  int64_t hx_off;          // x partials after the y ones
  int64_t lo_off;          // the pairs' second floats (mixed path, lists of more than kGramRun points per slot)
  double xs, ys;           // 2 / (W - 1), 2 / (H - 1)
};

template <typename T>
__device__ __forceinline__ int gram_slots(int n, int g, int fill) {
  return max(1, min(g, max((n + kGramMin<T> - 1) / kGramMin<T>, min((n + kGramFew - 1) / kGramFew, fill))));
}
// whether a slot's share of n points in U slots may be summed in more than one run
template <typename T>
__device__ __forceinline__ bool gram_runs(int n, int U) {
  return sizeof(T) == 4 && ((n + kGramPts - 1) / kGramPts + U - 1) / U * kGramPts > kGramRun;
}

// Pair numbering shared by the tiles and the chains.  y pairs: offsets
// i, j < L (L - 1) in row-major order, j <= i; then the single offsets i.
// x pairs: i in the row u_y = w with u_x < w, j <= i with u_x < w; then the
// single offsets.
__device__ __forceinline__ int ypair_id(int i, int j) { return i * (i + 1) / 2 + j; }
__host__ __device__ inline int ypair_single(int L, int i) { const int n = L * (L - 1); return n * (n + 1) / 2 + i; }
__device__ __forceinline__ int xpair_id(int L, int ix, int jy, int jx) {   // biased indices 0 .. L-1
  const int q = (L - 1) * (L - 1);
  return ix * q + ix * (ix + 1) / 2 + (jy < L - 1 ? jy * (L - 1) + jx : q + jx);
}
__host__ __device__ inline int xpair_single(int L, int ix) {
  const int q = (L - 1) * (L - 1), n = L - 1;
  return n * q + n * (n + 1) / 2 + ix;
}
// the pair of the offsets i and j (or kGramOne) of a tile; -1: not one of the list's pairs
__device__ __forceinline__ int gram_pair(int L, bool isx, int i, int j) {
  const int n = L * (L - 1);
  if (isx) {
    const int ix = i - n;
    if (ix >= L - 1) return -1;
    if (j >= kGramOne) return j == kGramOne ? xpair_single(L, ix) : -1;
    if (j >= n) return j - n <= ix ? xpair_id(L, ix, L - 1, j - n) : -1;
    return j % L < L - 1 ? xpair_id(L, ix, j / L, j % L) : -1;
  }
  if (i >= kGramOne) return i == kGramOne && j < n ? ypair_single(L, j) : -1;
  return j <= i ? ypair_id(i, j) : -1;
}

template <typename T>
__host__ __device__ constexpr size_t gram_smem() {
  // per buffer and point: the patch, xt^a and yt^a (FP32: twice, as operand pairs), the list entry; the row ends
  return 2 * (sizeof(T) * kGramPts * (kGramPatch + 2 * kGramPow * (sizeof(T) == 4 ? 2 : 1)) + sizeof(int4) * kGramPts +
              sizeof(unsigned));
}

template <typename T, int DE>
__global__ void __launch_bounds__(kGramThreads, sizeof(T) == 4 ? 2 : 1)
k_edge_gram(const T* __restrict__ Rm, const unsigned* __restrict__ lx, const unsigned* __restrict__ ly, int64_t lstride,
            const int* __restrict__ cnt, int64_t cnt_stride, GramArgs a, T* __restrict__ hp, int H, int W, int L) {
  constexpr int NM = n_mono(DE), CD = sizeof(T) == 4 ? 2 : 1, PW = kGramPow * CD, NJ = gram_tj(DE) / 2;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ int2 offs[kGramPatch];   // u as a distance in the image; u_y and u_x
  T(*px)[kGramPts][PW] = reinterpret_cast<T(*)[kGramPts][PW]>(smraw);
  T(*py)[kGramPts][PW] = px + 2;
  T(*patch)[kGramPts][kGramPatch] = reinterpret_cast<T(*)[kGramPts][kGramPatch]>(py + 2);
  int4(*ent)[kGramPts] = reinterpret_cast<int4(*)[kGramPts]>(patch + 2);   // x, y, sign, patch inside the image
  unsigned* ends = reinterpret_cast<unsigned*>(ent + 2);   // the last points of the batch's rows
  const int ccd = blockIdx.z, tid = threadIdx.x, w = (L - 1) / 2, lane = tid & 31, warp = tid >> 5;
  const bool isx = (int)blockIdx.y < a.nbx;
  const int n = cnt[ccd * cnt_stride + (isx ? 0 : H + 1) + H];
  const int U = gram_slots<T>(n, isx ? a.gx : a.gy, isx ? a.fx : a.fy), g = blockIdx.x;
  if (g >= U) return;
  const int tile = (isx ? blockIdx.y : blockIdx.y - a.nbx) * kGramThreads + tid, nt = isx ? a.ntx : a.nty;
  const unsigned* list = (isx ? lx : ly) + ccd * lstride;
  const int v = tile < nt ? a.tiles[(isx ? a.nty : 0) + tile] : 0, ti = v & 255, tj = v >> 8;
  const bool idle = tile - lane >= nt;   // a warp without tiles only copies
  if (tid < kGramPatch) {
    const int uy = tid / L - w, ux = tid % L - w;
    offs[tid] = make_int2(uy * W + ux, (uy + w) << 8 | (ux + w));
  }
  // (j, j + 1) packed, for i and i + 1 (and the same for j + 2): sums over a row, and all rows times yt^b
  v2<T> rs[2 * NJ][DE + 1], acc[2 * NJ][NM];
#pragma unroll
  for (int q = 0; q < 2 * NJ; ++q) {
#pragma unroll
    for (int k = 0; k <= DE; ++k) v2_zero(rs[q][k]);
#pragma unroll
    for (int k = 0; k < NM; ++k) v2_zero(acc[q][k]);
  }
  const T* img = Rm + (int64_t)ccd * H * W;
  if (tid < 2 * kGramPts) {
    patch[tid / kGramPts][tid % kGramPts][kGramOne] = (T)1;
    patch[tid / kGramPts][tid % kGramPts][kGramOne + 1] = (T)0;
  }
  const int nb = (n + kGramPts - 1) / kGramPts;
  // the points of batch b into buffer s
  auto stage = [&](int b, int s) {
    const int m = min(kGramPts, n - b * kGramPts);
    for (int pt = warp; pt < m; pt += kGramThreads / 32) {
      const int4 e = ent[s][pt];
      const T* src = img + ((int64_t)e.y * W + e.x);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int j = lane + 32 * k;
        if (j < L * L) {
          const int2 o = offs[j];
          bool in = true;
          if (!e.w) {
            const int yy = e.y + w - (o.y >> 8), xx = e.x + w - (o.y & 255);
            in = yy >= 0 && yy < H && xx >= 0 && xx < W;
          }
          cp_async<sizeof(T)>(&patch[s][pt][j], in ? src - o.x : img, in);
        }
      }
    }
    if (warp == kGramThreads / 32 - 1) {
      const int4 e = ent[s][lane];
      const int yn = __shfl_down_sync(0xffffffffu, e.y, 1);
      const unsigned last = __ballot_sync(0xffffffffu, lane < m && (lane == m - 1 || yn != e.y));
      if (lane == 0) ends[s] = last;
      const T xt = (T)(e.x * a.xs - 1.0), yt = (T)(e.y * a.ys - 1.0);
      T qx = (T)e.z, qy = 1;
#pragma unroll
      for (int k = 0; k <= DE; ++k) {
        st_dup(&px[s][lane][CD * k], qx);
        st_dup(&py[s][lane][CD * k], qy);
        qx *= xt;
        qy *= yt;
      }
    }
  };
  auto entry = [&](int b) { return b < nb && b * kGramPts + lane < n ? list[(int64_t)b * kGramPts + lane] : 0u; };
  auto put = [&](unsigned e, int s) {
    const int y = (int)((e >> 1) / (unsigned)W), x = (int)((e >> 1) - (unsigned)y * (unsigned)W);
    ent[s][lane] = make_int4(x, y, (e & 1u) ? -1 : 1, y >= w && y < H - w && x >= w && x < W - w);
  };
  if (warp == 0) {
    put(entry(g), 0);
    put(entry(g + U), 1);
  }
  __syncthreads();
  if (g < nb) stage(g, 0);
  T* out = hp + ccd * a.hp_stride + (isx ? a.hx_off : 0) + (int64_t)g * (isx ? a.npx : a.npy) * NM;
  const bool runs = gram_runs<T>(n, U);
  bool first = true;
  int s = 0, rows = 0;
  // an empty list takes one turn without points, for the zeros
  for (int b = g; b < max(nb, 1); b += U, s ^= 1) {
    cp_async_wait_all();
    __syncthreads();
    unsigned e2 = 0;
    if (warp == 0) e2 = entry(b + 2 * U);
    if (b + U < nb) stage(b + U, s ^ 1);
    const int m = min(kGramPts, n - b * kGramPts);
    const unsigned last = m > 0 ? ends[s] : 0u;
    for (int pt = 0; pt < m && !idle;) {
      const int c = __ffs(last >> pt);   // points of the row
      const T *pj = &patch[s][pt][tj], *pi = &patch[s][pt][ti], *pq = &px[s][pt][0];
#pragma unroll 4
      for (int i = 0; i < c; ++i, pj += kGramPatch, pi += kGramPatch, pq += PW) {
        const v2<T> ri = v2_load(pi);
        v2<T> r[2 * NJ];
#pragma unroll
        for (int h = 0; h < NJ; ++h) {
          const v2<T> rj = v2_load(pj + 2 * h);
#pragma unroll
          for (int q = 0; q < 2; ++q)
            r[2 * h + q] = v2_make(v2_get(ri, q) * v2_get(rj, 0), v2_get(ri, q) * v2_get(rj, 1));
        }
#pragma unroll
        for (int k = 0; k <= DE; k += 2) {
          v2<T> x[2];
          v2_dup2(pq + CD * k, x[0], x[1]);
#pragma unroll
          for (int h = 0; h < 2 && k + h <= DE; ++h)
#pragma unroll
            for (int q = 0; q < 2 * NJ; ++q) v2_fmav(rs[q][k + h], x[h], r[q]);
        }
      }
      pt += c;
#pragma unroll
      for (int q = 0; q <= DE; ++q) {
        const v2<T> yb = v2_dup(&py[s][pt - 1][CD * q]);
#pragma unroll
        for (int k = 0; k <= DE - q; ++k)
#pragma unroll
          for (int h = 0; h < 2 * NJ; ++h) v2_fmav(acc[h][mono_index(k, q)], yb, rs[h][k]);
      }
#pragma unroll
      for (int k = 0; k <= DE; ++k)
#pragma unroll
        for (int h = 0; h < 2 * NJ; ++h) v2_zero(rs[h][k]);
    }
    if (warp == 0) put(e2, s);
    rows += __popc(last);
    const bool end = b + U >= nb;
    if (!end && !(runs && rows > kGramRun - kGramPts)) continue;
#pragma unroll
    for (int p = 0; p < 4 * NJ; ++p) {
      const int id = tile < nt ? gram_pair(L, isx, ti + ((p >> 1) & 1), tj + 2 * (p >> 2) + (p & 1)) : -1;
      if (id >= 0)
#pragma unroll
        for (int k = 0; k < NM; ++k) {
          T* o = out + (int64_t)id * NM + k;
          T v = v2_get(acc[p >> 1][k], p & 1);
          if constexpr (sizeof(T) == 4)
            if (runs) {
              float e = 0.f;
              if (!first) v = two_sum(*o, v, e);
              o[a.lo_off] = first ? 0.f : o[a.lo_off] + e;
            }
          *o = v;
        }
    }
#pragma unroll
    for (int q = 0; q < 2 * NJ; ++q)
#pragma unroll
      for (int k = 0; k < NM; ++k) v2_zero(acc[q][k]);
    first = false;
    rows = 0;
  }
}

// the slots' partial sums: FP64, on the mixed path as pairs of floats
template <typename T>
__global__ void __launch_bounds__(256)
k_edge_reduce(const T* __restrict__ hp, GramArgs a, const int* __restrict__ cnt, int64_t cnt_stride, int H, int NM,
              double* __restrict__ hs) {
  const int ccd = blockIdx.y, ny = a.npy * NM, nx = a.npx * NM;
  const int i = blockIdx.x * 256 + threadIdx.x;
  if (i >= ny + nx) return;
  const bool isx = i >= ny;
  const int n = cnt[ccd * cnt_stride + (isx ? 0 : H + 1) + H], U = gram_slots<T>(n, isx ? a.gx : a.gy, isx ? a.fx : a.fy);
  const int64_t st = isx ? nx : ny;
  const T* p = hp + ccd * a.hp_stride + (isx ? a.hx_off + i - ny : i);
  double s = 0.0;
  if constexpr (sizeof(T) == 4) {
    const bool runs = gram_runs<T>(n, U);
    float h = 0.f, l = 0.f;
#pragma unroll 8
    for (int g = 0; g < U; ++g) {
      float e;
      h = two_sum(h, p[g * st], e);
      l += e;
      if (runs) l += p[g * st + a.lo_off];
    }
    s = (double)h + (double)l;
  } else {
#pragma unroll 8
    for (int g = 0; g < U; ++g) s += p[g * st];
  }
  hs[(int64_t)ccd * (ny + nx) + i] = s;
}

// ------------------------------------------------------------------ chains
// One CTA per (half-plane difference, CCD), and one for the kernel-background
// block (block n_hd: single offsets).  The CTA fetches the edge sums of its pairs
// into shared memory; a thread per power of yt then walks the x
// chain at u_y = w, and a thread per (u_x, power of xt) the y chains, in FP64.
// shift(h) acts within one power: new_k = sum_i binom(k, i) h^(k - i) old_i.
// The chain's FP64 additions, one after another, bound it (23 us at L = 11,
// D_K = 2; about the same for ten CCDs).
template <int DEG>
__device__ __forceinline__ void shift_poly(double (&f)[DEG + 1], int deg, double h) {
  // repeated synthetic division: f(x) coefficients' dual, highest first
#pragma unroll
  for (int s = 0; s < DEG; ++s)
#pragma unroll
    for (int k = DEG; k > s; --k)
      if (k <= deg) f[k] += h * f[k - 1];
}

__global__ void __launch_bounds__(128)
k_edge_chain(const double* __restrict__ hs, int npy, int npx, int MP, int L, int DKK, int DKB, const int2* __restrict__ dlist,
             int n_hd, double* __restrict__ gkk, int64_t kk_stride, double* __restrict__ gkb, int64_t kb_stride,
             double hx, double hy) {
  extern __shared__ double sm[];
  const int ccd = blockIdx.y, id = blockIdx.x, w = (L - 1) / 2, tid = threadIdx.x;
  const bool kb = id == n_hd;
  const int DEG = kb ? DKB : DKK, NM = n_mono(DEG);
  const int dy = kb ? 0 : dlist[id].x, dx = kb ? 0 : dlist[id].y;
  // biased ranges of u (0 .. 2w)
  const int uy_lo = kb ? 0 : max(0, dy), ux_lo = max(0, dx), ux_hi = min(L - 1, L - 1 + dx);
  const int nx = ux_hi - ux_lo + 1, ny = L - 1 - uy_lo;   // u_x count; y steps
  double* G = kb ? gkb + ccd * kb_stride : gkk + ccd * kk_stride + (int64_t)id * L * L * NM;
  double* sx = sm;                       // [nx - 1][NM]
  double* sy = sm + (L - 1) * NM;        // [ny][nx][NM]
  const double* hc = hs + (int64_t)ccd * (npy + npx) * MP;
  const int tot_x = (nx - 1) * NM, tot = tot_x + ny * nx * NM;
  for (int e = tid; e < tot; e += blockDim.x) {
    const bool isx = e < tot_x;
    const int q = isx ? e : e - tot_x;
    const int m = q % NM, k = q / NM;
    int pid;
    if (isx) {
      const int ix = ux_lo + k;
      pid = kb ? xpair_single(L, ix) : xpair_id(L, ix, L - 1 - dy, ix - dx);
    } else {
      const int iy = uy_lo + k / nx, ix = ux_lo + k % nx;
      pid = kb ? ypair_single(L, iy * L + ix) : ypair_id(iy * L + ix, (iy - dy) * L + (ix - dx));
    }
    (isx ? sx : sy)[q] = hc[(int64_t)(isx ? npy + pid : pid) * MP + m];
  }
  __syncthreads();
  // x chain at u_y = w from the corner u_x = w (d_x >= 0) or -w (d_x < 0)
  if (tid <= DEG) {
    const int b = tid, n = DEG - b;
    double f[kMaxWeightDeg + 1];
    const bool up = dx < 0;
    int ux = up ? 0 : L - 1;
    if (!up) ux = ux_hi;
#pragma unroll
    for (int k = 0; k <= kMaxWeightDeg; ++k) f[k] = k <= n ? G[((int64_t)(L - 1) * L + ux) * NM + mono_index(k, b)] : 0.0;
    for (int s = 0; s < nx - 1; ++s) {
      if (up) {
        const double* h = sx + (ux - ux_lo) * NM;
#pragma unroll
        for (int k = 0; k <= kMaxWeightDeg; ++k)
          if (k <= n) f[k] += h[mono_index(k, b)];
        shift_poly<kMaxWeightDeg>(f, n, hx);
        ++ux;
      } else {
        shift_poly<kMaxWeightDeg>(f, n, -hx);
        --ux;
        const double* h = sx + (ux - ux_lo) * NM;
#pragma unroll
        for (int k = 0; k <= kMaxWeightDeg; ++k)
          if (k <= n) f[k] -= h[mono_index(k, b)];
      }
#pragma unroll
      for (int k = 0; k <= kMaxWeightDeg; ++k)
        if (k <= n) G[((int64_t)(L - 1) * L + ux) * NM + mono_index(k, b)] = f[k];
    }
  }
  __syncthreads();
  for (int e = tid; e < nx * (DEG + 1); e += blockDim.x) {
    const int ux = ux_lo + e / (DEG + 1), av = e % (DEG + 1), n = DEG - av;
    double f[kMaxWeightDeg + 1];
#pragma unroll
    for (int k = 0; k <= kMaxWeightDeg; ++k) f[k] = k <= n ? G[((int64_t)(L - 1) * L + ux) * NM + mono_index(av, k)] : 0.0;
    for (int uy = L - 2; uy >= uy_lo; --uy) {
      shift_poly<kMaxWeightDeg>(f, n, -hy);
      const double* h = sy + ((uy - uy_lo) * nx + (ux - ux_lo)) * NM;
#pragma unroll
      for (int k = 0; k <= kMaxWeightDeg; ++k)
        if (k <= n) {
          f[k] -= h[mono_index(av, k)];
          G[((int64_t)uy * L + ux) * NM + mono_index(av, k)] = f[k];
        }
    }
  }
}

// ------------------------------------------------------------------ host: tables
// Tasks and destinations of the fit and of the right-hand side, the pair
// table of the edge sums, and the tile and slot counts.
void build_tap_plan(sfft_plan_s* p) {
  const int L = p->d.L, w = p->w, DK = p->d.DK, DB = p->d.DB, B = p->d.batch;
  const int dKK = 2 * DK, dKB = DK + DB;
  const int nkk = n_mono(dKK), nkb = n_mono(dKB), nbk = n_mono(DK);
  TapPlan& t = p->tap;
  t.nt = std::max(L, 3);
  // The line is right for the small images of small kernels and lies at L alone:
  // assembly by every pair against edge sums, in us, L = 5, D_K = 2 (L = 3) on
  // the mixed path: 160 x 192 59 / 106 (50 / 102), 512 x 512 92 / 118 (57 / 110),
  // 1024 x 1024 189 / 133 (78 / 119), 4096 x 2048 894 / 306 (259 / 235); FP64
  // 1024 x 1024 5331 / 976 (1059 / 506).  Row spectra took 2545 us where every
  // pair takes 894, and 9990 where it takes 5331.
  t.mode = L <= 5 ? TAP_FIT_ALL : TAP_FIT_EDGE;
  const int wt = (t.nt - 1) / 2;
  auto half_id = [&](int dy, int dx) {
    for (int i = 0; i < p->n_hd; ++i)
      if (p->dlist[i].x == dy && p->dlist[i].y == dx) return i;
    return -1;
  };
  auto q = [](int region, int64_t off) { return (int)((region << 28) | off); };
  auto add = [&](std::vector<int4>& tasks, std::vector<int>& dst, int type, int u0x, int u0y, int uy) {
    const int nc = type == TAP_CS || type == TAP_C ? n_mono(2 * DK) : (type == TAP_M ? n_mono(DK + 2) : 0);
    const int ns = type == TAP_CS || type == TAP_S ? nbk : 0;
    const int nout = nc + ns;
    tasks.push_back(int4{type | nout << 8, (u0x + 64) | (u0y + 64) << 8, uy, (int)dst.size()});
    const int taps = t.mode == TAP_FIT_EDGE && type == TAP_C ? t.nt - 1 : t.nt;
    for (int k = 0; k < taps; ++k) {
      const int ux = wt - k;
      const bool in = ux >= -w && ux <= w;
      const int j = (uy + w) * L + (ux + w);
      for (int m = 0; m < nc; ++m) {
        int v = -1;
        if (in && type == TAP_M) {
          if (m < nkb) v = q(1, (int64_t)j * nkb + m);
        } else if (in) {
          const int dy = u0y - uy, dx = u0x - ux;
          // the lower corner's own column repeats the upper corner's d_x = 0 entries elsewhere: not needed
          const bool want = (dy > 0 || dx >= 0) && (t.mode == TAP_FIT_ALL || u0x == w || dx < 0);
          const int id = want ? half_id(dy, dx) : -1;
          if (id >= 0) v = q(0, (((int64_t)id * L + (u0y + w)) * L + (u0x + w)) * nkk + m);
        }
        dst.push_back(v);
      }
      for (int m = 0; m < ns; ++m) dst.push_back(in ? q(2, (int64_t)j * nbk + m) : -1);
    }
  };
  auto moments = [&](std::vector<int4>& tasks, std::vector<int>& dst, bool fit) {
    // partial sums of their own; first, since its chain of FP64 sums is the longest of a small image's tasks
    // (160 x 192, L = 5: 13.4 us, 15.9 with the task last)
    tasks.insert(tasks.begin(), int4{TAP_MOM | kTapMom << 8, 0, 0, 0});
    const int64_t corner = (int64_t)(L * L - 1) * nkb;   // the single offset (w, w)
    for (int m = 0; m < 15; ++m) dst.push_back(fit && m < n_mono(2 * DB) ? q(3, m) : -1);
    for (int m = 0; m < 6; ++m) dst.push_back(m < n_mono(DB) ? q(4, m) : -1);
    for (int m = 0; m < 15; ++m) dst.push_back(fit && t.mode == TAP_FIT_EDGE && m < nkb ? q(1, corner + m) : -1);
  };
  t.tasks.clear();
  t.dst.clear();
  std::vector<int4> rhs_tasks;
  std::vector<int> rhs_dst;
  for (int uy = -w; uy <= w; ++uy) add(t.tasks, t.dst, TAP_CS, w, w, uy);
  if (t.mode == TAP_FIT_ALL) {
    for (int uy = -w; uy <= w; ++uy) add(t.tasks, t.dst, TAP_M, 0, 0, uy);
    for (int u0y = -w; u0y <= w; ++u0y)
      for (int u0x = -w; u0x <= w; ++u0x)
        if (u0x != w || u0y != w)
          for (int uy = -w; uy <= u0y; ++uy) add(t.tasks, t.dst, TAP_C, u0x, u0y, uy);
  } else {
    for (int uy = -w; uy < w; ++uy) add(t.tasks, t.dst, TAP_C, -w, w, uy);
  }
  moments(t.tasks, t.dst, true);
  for (int uy = -w; uy <= w; ++uy) add(rhs_tasks, rhs_dst, TAP_S, 0, 0, uy);
  moments(rhs_tasks, rhs_dst, false);
  t.ntask = (int)t.tasks.size();
  t.nout = (int)t.dst.size() - kTapMom;
  t.ntask_rhs = (int)rhs_tasks.size();
  t.nout_rhs = (int)rhs_dst.size() - kTapMom;
  t.tasks.insert(t.tasks.end(), rhs_tasks.begin(), rhs_tasks.end());
  t.dst.insert(t.dst.end(), rhs_dst.begin(), rhs_dst.end());
  // wide tiles amortise the halo and the fold of yt^b; a small image takes
  // narrow ones, and then splits a tile's tasks over CTAs, to reach two CTAs
  // per SM
  const int want = 2 * 152;
  auto tiles = [&](int tw) { return ((p->d.W + tw - 1) / tw) * ((p->d.H + kTapRows - 1) / kTapRows); };
  t.tw = 128;
  while (t.tw > 32 && (int64_t)tiles(t.tw) * B < want) t.tw /= 2;
  t.ntile = tiles(t.tw);
  auto split = [&](int ntask) {
    const int64_t n = (int64_t)t.ntile * B;
    return (int)std::max<int64_t>(1, std::min<int64_t>((want + n - 1) / n, (ntask + kTapWarps - 1) / kTapWarps));
  };
  t.nsplit = split(t.ntask);
  // the refinement's half tiles (kernels_apply.cu)
  t.ntile_rhs = 2 * conv_tiles(p->d.H, p->d.W, conv_half_width(p->d.H, p->d.W, B));
  // edge sums
  t.DE = std::max(dKK, dKB);
  t.MP = n_mono(t.DE);
  t.tiles.clear();
  t.npy = t.npx = t.nty = t.ntx = 0;
  if (t.mode == TAP_FIT_EDGE) {
    const int n = L * (L - 1);   // offsets below the row u_y = w, an even number
    t.npy = ypair_single(L, n);
    t.npx = xpair_single(L, L - 1);
    const int tj = gram_tj(t.DE), one = kGramOne / tj * tj;   // the tile that holds the ones
    for (int i = 0; i < n; i += 2)
      for (int j = 0; j <= i + 1; j += tj) t.tiles.push_back(i | j << 8);
    for (int j = 0; j < n; j += tj) t.tiles.push_back(kGramOne | j << 8);
    t.nty = (int)t.tiles.size();
    for (int ix = 0; ix < L - 1; ix += 2) {
      for (int j = 0; j <= n + ix + 1; j += tj) t.tiles.push_back((n + ix) | j << 8);
      t.tiles.push_back((n + ix) | one << 8);
    }
    t.ntx = (int)t.tiles.size() - t.nty;
    t.nby = (t.nty + kGramThreads - 1) / kGramThreads;
    t.nbx = (t.ntx + kGramThreads - 1) / kGramThreads;
    // a list that fills its slots gives every SM two rounds of two CTAs
    t.gy = std::max(16, 608 / (t.nby * B));
    t.gx = std::max(64, 304 / (t.nbx * B));
  }
  // M is an erosion by L x L: its zero runs are at least L wide between the borders
  t.row_cap = L == 1 ? p->d.W : std::min(p->d.W, 2 * (p->d.W / (L + 1) + 2));
  t.col_cap = L == 1 ? p->d.H : std::min(p->d.H, 2 * (p->d.H / (L + 1) + 2));
}

// ------------------------------------------------------------------ launchers
void tap_region_bytes(const sfft_plan_s* p, size_t* part, size_t* mpart, size_t* hp, size_t* hs, size_t* list, size_t* cnt) {
  const TapPlan& t = p->tap;
  const size_t B = p->d.batch;
  *part = p->elem * B * std::max((size_t)t.ntile * t.nout, (size_t)t.ntile_rhs * t.nout_rhs);
  *mpart = sizeof(double) * B * std::max(t.ntile, t.ntile_rhs) * kTapMom;
  const bool edge = t.mode == TAP_FIT_EDGE;
  *hp = edge ? sizeof(double) * B * ((size_t)t.gy * t.npy + (size_t)t.gx * t.npx) * t.MP : 0;   // FP32: pairs
  *hs = edge ? sizeof(double) * B * (size_t)(t.npy + t.npx) * t.MP : 0;
  *list = edge ? 2 * sizeof(unsigned) * B * (size_t)edge_cap(p) : 0;
  *cnt = edge ? 2 * sizeof(int) * B * (size_t)(p->d.H + 1) : 0;
}

// how many moments of M, of s and of c a fit (or its right-hand side) takes
char3 tap_moment_need(const sfft_plan_s* p, bool fit) {
  const bool edge = p->tap.mode == TAP_FIT_EDGE;
  return char3{(signed char)(fit ? n_mono(p->DM_BB) : 0), (signed char)n_mono(p->d.DB),
               (signed char)(fit && edge ? n_mono(p->DM_KB) : 0)};
}

// one pixel in xt or yt
static double step_of(int n) { return 2.0 / (double)(n > 1 ? n - 1 : 1); }

template <typename T, int NT, int DK, int MODE>
static cudaError_t tap_sums(const sfft_plan_s* p, const float* S, void* ws) {
  const TapPlan& t = p->tap;
  auto kern = k_tap_sums<T, NT, DK, MODE>;
  const size_t smem = tap_smem<T>((NT - 1) / 2, t.tw);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  dim3 grid(t.ntile, t.nsplit, p->d.batch);
  kern<<<grid, kTapWarps * 32, smem, p->stream>>>(ws_at<T>(ws, p->rm), S, ws_at<unsigned>(ws, p->mfitw),
                                                  ws_at<double>(ws, p->sky), t.d_tasks, t.ntask,
                                                  ws_at<T>(ws, p->tappart), t.nout, ws_at<double>(ws, p->mompart), tap_moment_need(p, true), p->d.H, p->d.W, p->w, t.tw,
                                                  step_of(p->d.W), step_of(p->d.H));
  p->nlaunch += 1;
  return cudaGetLastError();
}

template <typename T, int NT, int MODE>
static cudaError_t tap_sums_dk(const sfft_plan_s* p, const float* S, void* ws) {
  switch (p->d.DK) {
    case 0: return tap_sums<T, NT, 0, MODE>(p, S, ws);
    case 1: return tap_sums<T, NT, 1, MODE>(p, S, ws);
    default: return tap_sums<T, NT, 2, MODE>(p, S, ws);
  }
}

template <typename T>
static cudaError_t tap_reduce(const sfft_plan_s* p, bool rhs, void* ws) {
  const TapPlan& t = p->tap;
  const int LL = p->d.L * p->d.L, nout = rhs ? t.nout_rhs : t.nout;
  TapDst d;
  const Region* reg[5] = {&p->gkk, &p->gkb, &p->gbk, &p->mom_bb, &p->mom_b};
  const int64_t stride[5] = {(int64_t)p->n_hd * LL * n_mono(p->DM_KK), (int64_t)LL * n_mono(p->DM_KB),
                             (int64_t)LL * n_mono(p->DM_bK), n_mono(p->DM_BB), n_mono(p->d.DB)};
  for (int i = 0; i < 5; ++i) { d.base[i] = ws_at<double>(ws, *reg[i]); d.stride[i] = stride[i]; }
  k_tap_reduce<T><<<dim3((nout + kRedOut - 1) / kRedOut + kTapMom, p->d.batch), kRedOut * kRedGroups, 0, p->stream>>>(
      ws_at<T>(ws, p->tappart), ws_at<double>(ws, p->mompart), t.d_dst + (rhs ? t.nout + kTapMom : 0), d, rhs ? t.ntile_rhs : t.ntile, nout);
  p->nlaunch += 1;
  return cudaGetLastError();
}

template <typename T>
static cudaError_t tap_fit_T(const sfft_plan_s* p, const float* S, void* ws) {
  cudaError_t e = cudaErrorInvalidValue;
  switch (p->tap.nt) {
    case 3: e = tap_sums_dk<T, 3, TAP_FIT_ALL>(p, S, ws); break;
    case 5: e = tap_sums_dk<T, 5, TAP_FIT_ALL>(p, S, ws); break;
    case 7: e = tap_sums_dk<T, 7, TAP_FIT_EDGE>(p, S, ws); break;
    case 9: e = tap_sums_dk<T, 9, TAP_FIT_EDGE>(p, S, ws); break;
    case 11: e = tap_sums_dk<T, 11, TAP_FIT_EDGE>(p, S, ws); break;
  }
  return e != cudaSuccess ? e : tap_reduce<T>(p, false, ws);
}

cudaError_t launch_tap_fit(const sfft_plan_s* p, const float* S, void* ws) {
  return p->fp64 ? tap_fit_T<double>(p, S, ws) : tap_fit_T<float>(p, S, ws);
}

cudaError_t launch_tap_rhs_reduce(const sfft_plan_s* p, void* ws) {
  return p->fp64 ? tap_reduce<double>(p, true, ws) : tap_reduce<float>(p, true, ws);
}

template <typename T>
static cudaError_t edge_sums_T(const sfft_plan_s* p, void* ws) {
  const TapPlan& t = p->tap;
  const int H = p->d.H, W = p->d.W, L = p->d.L, B = p->d.batch;
  GramArgs a;
  a.tiles = t.d_tiles;
  a.nty = t.nty; a.ntx = t.ntx; a.nbx = t.nbx;
  a.npy = t.npy; a.npx = t.npx;
  a.gy = t.gy; a.gx = t.gx;
  a.fy = 152 / (t.nby * B); a.fx = 152 / (t.nbx * B);
  a.xs = step_of(W); a.ys = step_of(H);
  a.hx_off = (int64_t)t.gy * t.npy * t.MP;
  a.lo_off = a.hx_off + (int64_t)t.gx * t.npx * t.MP;
  a.hp_stride = sizeof(T) == 4 ? 2 * a.lo_off : a.lo_off;
  const unsigned* lx = ws_at<unsigned>(ws, p->elist);
  const int* cnt = ws_at<int>(ws, p->ecnt);
  const int64_t cap = edge_cap(p), cs = 2 * (int64_t)(H + 1);
  const T* rm = ws_at<T>(ws, p->rm);
  T* hp = ws_at<T>(ws, p->hpart);
  dim3 grid(std::max(t.gx, t.gy), t.nby + t.nbx, B);
  cudaError_t e = cudaSuccess;
#define SFFT_GRAM(D)                                                                                                  \
  case D:                                                                                                             \
    e = cudaFuncSetAttribute(k_edge_gram<T, D>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gram_smem<T>()); \
    if (e != cudaSuccess) return e;                                                                                   \
    k_edge_gram<T, D><<<grid, kGramThreads, gram_smem<T>(), p->stream>>>(rm, lx, lx + cap, 2 * cap, cnt, cs, a, hp, \
                                                                            H, W, L);                                 \
    break
  switch (t.DE) {
    SFFT_GRAM(0); SFFT_GRAM(1); SFFT_GRAM(2); SFFT_GRAM(3); SFFT_GRAM(4);
    default: return cudaErrorInvalidValue;
  }
#undef SFFT_GRAM
  const int LL = L * L;
  const size_t smem = sizeof(double) * (size_t)(L - 1) * (L + 1) * n_mono(t.DE);
  double* hs = ws_at<double>(ws, p->hsum);
  k_edge_reduce<T><<<dim3(((t.npy + t.npx) * t.MP + 255) / 256, B), 256, 0, p->stream>>>(hp, a, cnt, cs, H, t.MP, hs);
  k_edge_chain<<<dim3(p->n_hd + 1, B), 128, smem, p->stream>>>(
      hs, t.npy, t.npx, t.MP, L, p->DM_KK, p->DM_KB, p->d_dlist, p->n_hd, ws_at<double>(ws, p->gkk),
      (int64_t)p->n_hd * LL * n_mono(p->DM_KK), ws_at<double>(ws, p->gkb), (int64_t)LL * n_mono(p->DM_KB),
      a.xs, a.ys);
  p->nlaunch += 3;
  return cudaGetLastError();
}

cudaError_t launch_edge_sums(const sfft_plan_s* p, void* ws) {
  if (p->tap.mode != TAP_FIT_EDGE) return cudaSuccess;
  return p->fp64 ? edge_sums_T<double>(p, ws) : edge_sums_T<float>(p, ws);
}

}  // namespace sfft
