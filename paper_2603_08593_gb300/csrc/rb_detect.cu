// Candidate detection on difference images and the plain SNR/shape cuts.
//
// Per CCD: four passes of clipped statistics over the interior (pass 0
// unclipped, passes 1-3 clipped at 3 RMS about the previous pass's mean), then
// one tile kernel for the separable FP32 Gaussian matched filter (rows, then
// columns with the 1 / (sigma_D ||G||) scale folded in) and the 5 x 5
// local-maximum test, whose result is one bit per pixel and a count per row;
// an exclusive scan over rows, an ordered compaction that writes the candidates
// in row-major order, and a stamp gather.  Masks travel as bits.  Block
// partials of the statistics are reduced in a fixed order, so results are
// deterministic.
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <string>
#include <type_traits>

#include "common.cuh"
#include "plan.h"
#include "rb.h"

namespace {

constexpr int kMargin = 15, kHalf = 15, kNms = 2, kMaxR = 15;
constexpr int kStatBlocks = 608, kStatPasses = 4;   // four CTAs per SM
constexpr int kClipWords = 8;   // words of a row in flight per warp of a pass
constexpr double kClipNsig = 3.0, kClipVarShare = 0.97334;

struct Taps {
  float g[2 * kMaxR + 1];
  int r;
};

size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

// What one statistics pass hands to the next, and the last one to the filter
struct PassStats {
  float shift, lo, hi;   // the next pass sums about shift the pixels in [lo, hi]
  int about0;            // ... with the loop's sums about zero, and no value that float arithmetic could lose
  float scale;           // 1 / (sigma_D ||G||)
};

struct DetectLayout {
  size_t snr, good, bad, guard, cand, part, stats, zero, rowcnt, rowoff, total;
  size_t zero_bytes;
  int words;   // mask words per row
  DetectLayout(int H, int W, int B) {
    words = (W + 31) / 32;
    const size_t bits = align256((size_t)B * H * words * sizeof(unsigned));
    snr = 0;   // first: callers view the SNR map here
    good = snr + align256((size_t)B * H * W * sizeof(float));
    bad = good + bits;
    guard = bad + bits;
    cand = guard + bits;
    part = cand + bits;
    stats = part + align256((size_t)B * kStatBlocks * 3 * sizeof(double));
    zero = stats + align256((size_t)B * sizeof(PassStats));   // counters and row counts, cleared together
    rowcnt = zero + (size_t)B * kStatPasses * sizeof(int);
    zero_bytes = (size_t)B * (kStatPasses + H) * sizeof(int);
    rowoff = zero + align256(zero_bytes);
    total = rowoff + align256((size_t)B * H * sizeof(int));
  }
};

using sfft::two_sum;

// (s, e, f) += x, and e and f alone for an x below s's last place
__device__ __forceinline__ void add_low(float& e, float& f, float x) {
  float u;
  e = two_sum(e, x, u);
  f += u;
}
__device__ __forceinline__ void add_triple(float& s, float& e, float& f, float x) {
  float r;
  s = two_sum(s, x, r);
  add_low(e, f, r);
}
// two_sum of both halves, in packed instructions
__device__ __forceinline__ float2 two_sum2(float2 x, float2 y, float2& e) {
  const float2 m1 = make_float2(-1.f, -1.f), s = __fadd2_rn(x, y), t = __ffma2_rn(x, m1, s);   // products by -1 are exact
  e = __fadd2_rn(__ffma2_rn(__ffma2_rn(t, m1, s), m1, x), __ffma2_rn(t, m1, y));
  return s;
}

// the clipping rule of a pass
__device__ __forceinline__ bool kept(float x, double mean, double thr) { return fabs((double)x - mean) <= thr; }

// floats in order as integers
__device__ __forceinline__ unsigned float_key(float x) {
  const unsigned b = __float_as_uint(x);
  return b ^ (b >> 31 ? 0xffffffffu : 0x80000000u);
}
__device__ __forceinline__ float key_float(unsigned k) { return __uint_as_float(k ^ (k >> 31 ? 0x80000000u : 0xffffffffu)); }

// One statistics pass over the rows blockIdx.x, blockIdx.x + gridDim.x, ...
// Sums n, sum d, sum d^2 of d = x - shift in triples of floats: d as an exact
// pair, its square with every term down to 2^-48, and both sums with their
// rounding errors summed exactly once more, so that what is left is below an
// FP64 sum's error (1e-16 of a thread's sum; FP64 additions, at 1/64 of the FP32
// rate, left 7e-16 and took 70 us per pass of 2048 x 4096, pairs of floats 5e-15
// and 25 us, these 28 us).  FP64 from the thread's end on.  Where the mean lies
// within three times the scatter, as it does in a difference image, the loop sums
// about zero, where d is one float (11 us for the four passes), and the thread's
// triples are moved to the shift at its end: they hold some 70 bits, of which
// that takes a few.
// The loop is without branches but for values whose square leaves the range of a
// float, which wait for the word group's end.  What bounds a pass is the wait for
// its pixels between the arithmetic of two word groups (more of them in flight
// cost a CTA per SM: 207 against 204 us for the detector) and, of a small image,
// the chain of FP64 operations at the end: a CTA converts its sums once, the last
// one takes a warp per sum, warp 0 tests the candidates of both interval ends at
// once, and a pass forms only what the next kernel reads (the whole detector,
// conversions and FP64 additions in every warp -> one per CTA: 128 x 128
// 66 -> 59 us, 1024 x 1024 95 -> 78 us, 4096 x 2048 197 -> 191 us).
// The last CTA to finish adds the partials in index order and prepares the next
// pass: its clipping rule |x - mean| <= 3 sqrt(var), evaluated in FP64, becomes
// the float interval of the pixels that satisfy it (the rule is monotone on
// either side of the mean).  Pass 0 keeps every good pixel, about 0, and packs
// the masks of all rows.
template <bool FIRST>
__global__ void __launch_bounds__(256)
k_clip_pass(int H, int W, const float* __restrict__ D, const uint8_t* __restrict__ bad, unsigned* __restrict__ goodw,
            unsigned* __restrict__ badw, double* __restrict__ part, PassStats* __restrict__ stats,
            int* __restrict__ counter, int pass, Taps taps) {
  const int b = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = (W + 31) / 32;
  const float* Db = D + (int64_t)b * H * W;
  const uint8_t* bb = bad ? bad + (int64_t)b * H * W : nullptr;
  unsigned* gw = goodw + (int64_t)b * H * nw;
  unsigned* bw = badw + (int64_t)b * H * nw;
  double* pb = part + (int64_t)b * kStatBlocks * 3;
  float shift = 0.f, lo = 0.f, hi = 0.f;
  bool about0 = true;
  if (!FIRST) { shift = stats[b].shift; lo = stats[b].lo; hi = stats[b].hi; about0 = stats[b].about0 != 0; }
  int n = 0, n_wide = 0;   // pixels, and those among them in b1 and b2
  const float2 zero = make_float2(0.f, 0.f);
  float2 s = zero, e = zero, f = zero;   // sum d in .x, sum d^2 in .y
  double b1 = 0.0, b2 = 0.0;
  constexpr int U = kClipWords;
  const int ng = (nw + U - 1) / U, nit = ((H - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x) * ng;
  for (int it = warp; it < nit; it += 8) {   // the CTA's (row, word group) pairs
    const int y = blockIdx.x + it / ng * gridDim.x, w0 = it % ng * U;
    const bool row_in = y >= kMargin && y < H - kMargin;
    if (!FIRST && !row_in) continue;
    float v[U];
    unsigned m[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int x = (w0 + k) * 32 + lane;
      const bool in = x < W;
      v[k] = in ? Db[(int64_t)y * W + x] : 0.f;
      if (FIRST) m[k] = in && bb ? bb[(int64_t)y * W + x] : 0u;
      else m[k] = w0 + k < nw ? gw[(int64_t)y * nw + w0 + k] : 0u;
    }
    unsigned wide = 0;   // words whose square or its error leaves the range of a float
    auto group = [&](auto about0) {   // about0: the shift is zero, and d the pixel's value
      constexpr bool ABOUT0 = decltype(about0)::value;
#pragma unroll
      for (int k = 0; k < U; ++k) {
        const int x = (w0 + k) * 32 + lane;
        bool ok;
        if (FIRST) {
          const bool isbad = m[k] != 0u;
          ok = x < W && !isbad && isfinite(v[k]);
          const unsigned g = __ballot_sync(0xffffffffu, ok), q = __ballot_sync(0xffffffffu, isbad);
          if (lane == 0 && w0 + k < nw) {
            gw[(int64_t)y * nw + w0 + k] = g;
            if (bb) bw[(int64_t)y * nw + w0 + k] = q;
          }
        } else {
          ok = ((m[k] >> lane) & 1u) && v[k] >= lo && v[k] <= hi;
        }
        ok = ok && row_in && x >= kMargin && x < W - kMargin;
        n += ok;
        // a pixel that does not count adds zeros, which change no sum
        float dl = 0.f;
        float d = ABOUT0 ? v[k] : two_sum(v[k], -shift, dl);
        if (FIRST || !ABOUT0) {
          const float ad = fabsf(d);
          if (ok && (ad > 1e17f || (ad < 1e-12f && ad > 0.f))) wide |= 1u << k;
          ok = ok && !(wide >> k & 1u);
        }
        d = ok ? d : 0.f;
        dl = ok ? dl : 0.f;
        const float p = __fmul_rn(d, d), pe = __fmaf_rn(d, d, -p);
        float2 r, u;
        s = two_sum2(s, make_float2(d, p), r);
        e = two_sum2(e, r, u);
        f = __fadd2_rn(f, u);
        add_low(e.y, f.y, pe);
        if (!ABOUT0) {   // d's second float, and the square's terms in it
          add_low(e.x, f.x, dl);
          const float q = __fmul_rn(2.f * d, dl);
          add_low(e.y, f.y, q);
          f.y += __fmaf_rn(dl, dl, __fmaf_rn(2.f * d, dl, -q));
        }
      }
    };
    if (about0) group(std::true_type{});
    else group(std::false_type{});
    if (wide) {
#pragma unroll
      for (int k = 0; k < U; ++k)
        if (wide >> k & 1u) {
          ++n_wide;
          float dl = 0.f;
          const float d = two_sum(v[k], -shift, dl);
          const double dd = (double)d + (double)dl;
          b1 += dd;
          b2 += dd * dd;
        }
    }
  }
  if (!FIRST && about0) {
    // sum (x - c) = S1 - n c and sum (x - c)^2 = S2 - c (S1 + (S1 - n c)), c the shift
    const float c = shift, nf = (float)(n - n_wide), p = __fmul_rn(nf, c);
    float3 o = make_float3(s.x, e.x, f.x);
    add_triple(s.x, e.x, f.x, -p);
    add_low(e.x, f.x, -__fmaf_rn(nf, c, -p));
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const float q = __fmul_rn(c, o.x), ql = __fmul_rn(c, o.y);
      add_triple(s.y, e.y, f.y, -q);
      add_low(e.y, f.y, -__fmaf_rn(c, o.x, -q));
      add_low(e.y, f.y, -ql);
      f.y -= __fmaf_rn(c, o.y, -ql) + c * o.z;
      o = make_float3(s.x, e.x, f.x);
    }
  }
  // The threads' triples are joined as triples, four at a time in shared memory,
  // and the CTA's goes to FP64: an FP64 instruction occupies its pipe for 16
  // cycles, and conversions and shuffled additions in every warp took 5 us of a pass.
  __shared__ float tr[6][256];
  __shared__ double rb[2][8], red[3];
  __shared__ int rn[8], any_wide;
  __shared__ bool last;
  const int tid = threadIdx.x;
  n = __reduce_add_sync(0xffffffffu, n);
  if (lane == 0) rn[warp] = n;
  if (tid == 0) any_wide = 0;
  tr[0][tid] = s.x; tr[1][tid] = s.y; tr[2][tid] = e.x; tr[3][tid] = e.y; tr[4][tid] = f.x; tr[5][tid] = f.y;
  __syncthreads();
  if (n_wide) any_wide = 1;
  for (int m = 64; m > 0; m >>= 2) {
    if (tid < m) {
#pragma unroll
      for (int k = m; k < 4 * m; k += m) {
        float2 r, u;
        s = two_sum2(s, make_float2(tr[0][tid + k], tr[1][tid + k]), r);
        e = two_sum2(e, r, u);
        f = __fadd2_rn(f, u);
        e = two_sum2(e, make_float2(tr[2][tid + k], tr[3][tid + k]), u);
        f = __fadd2_rn(__fadd2_rn(f, u), make_float2(tr[4][tid + k], tr[5][tid + k]));
      }
      tr[0][tid] = s.x; tr[1][tid] = s.y; tr[2][tid] = e.x; tr[3][tid] = e.y; tr[4][tid] = f.x; tr[5][tid] = f.y;
    }
    __syncthreads();
  }
  if (any_wide) {
    b1 = sfft::warp_sum(b1);
    b2 = sfft::warp_sum(b2);
    if (lane == 0) { rb[0][warp] = b1; rb[1][warp] = b2; }
    __syncthreads();
  }
  if (tid == 0) {
    double v1 = (double)s.x + ((double)e.x + (double)f.x), v2 = (double)s.y + ((double)e.y + (double)f.y);
    int c = 0;
    for (int w = 0; w < 8; ++w) c += rn[w];
    if (any_wide)
      for (int w = 0; w < 8; ++w) { v1 += rb[0][w]; v2 += rb[1][w]; }
    pb[blockIdx.x * 3] = (double)c;
    pb[blockIdx.x * 3 + 1] = v1;
    pb[blockIdx.x * 3 + 2] = v2;
    __threadfence();
    last = atomicAdd(&counter[b * kStatPasses + pass], 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  // a warp per sum: an FP64 addition occupies its pipe for 16 cycles whatever the lanes hold
  if (warp < 3) {
    double a = 0.0;
#pragma unroll 4
    for (int i = lane; i < (int)gridDim.x; i += 32) a += __ldcg(pb + i * 3 + warp);
    a = sfft::warp_sum(a);
    if (lane == 0) red[warp] = a;
  }
  __syncthreads();
  if (warp != 0) return;
  const double t[3] = {red[0], red[1], red[2]};
  const double m1 = t[1] / t[0];
  const double mean = (double)shift + m1, var = t[2] / t[0] - m1 * m1;
  if (pass == kStatPasses - 1) {   // only the matched filter's scale is left to form
    float norm = 0.f;
    for (int k = 0; k <= 2 * taps.r; ++k) norm += taps.g[k] * taps.g[k];
    const double sigma = sqrt(var / kClipVarShare);
    if (lane == 0) stats[b].scale = (float)(1.0 / (sigma * (double)norm));
    return;
  }
  // the outermost floats that the rule keeps (none: an empty interval), among the
  // four on either side of the rounded ends: a lane per candidate
  const double thr = kClipNsig * sqrt(var);
  const int up = lane >> 4, j = (lane & 15) - 4;
  const float x = key_float(float_key((float)(up ? mean + thr : mean - thr)) + (unsigned)j);
  const unsigned in = __ballot_sync(0xffffffffu, (lane & 15) <= 8 && kept(x, mean, thr));
  const unsigned inl = in & 0xffffu, inh = in >> 16;
  const float lo_x = __shfl_sync(0xffffffffu, x, inl ? __ffs(inl) - 1 : 0);
  const float hi_x = __shfl_sync(0xffffffffu, x, inh ? 47 - __clz(inh) : 0);
  const bool any = inl != 0u && inh != 0u;
  if (lane == 0) {
    stats[b].shift = (float)mean;
    stats[b].about0 = fabs(mean) <= thr && thr <= 1e16 && thr >= 1e-9;
    stats[b].lo = any ? lo_x : INFINITY;
    stats[b].hi = any ? hi_x : -INFINITY;
  }
}

// bad pixels within Chebyshev distance g, a thread per 32-pixel word
__global__ void __launch_bounds__(256)
k_guard(int H, int nw, const unsigned* __restrict__ badw, int g, unsigned* __restrict__ out) {
  const int64_t base = (int64_t)blockIdx.y * H * nw;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < (int64_t)H * nw; e += (int64_t)gridDim.x * blockDim.x) {
    const int wi = (int)(e % nw), y = (int)(e / nw);
    unsigned l = 0, c = 0, r = 0;
    for (int yy = max(0, y - g); yy <= min(H - 1, y + g); ++yy) {
      const unsigned* p = badw + base + (int64_t)yy * nw + wi;
      if (wi > 0) l |= p[-1];
      c |= p[0];
      if (wi + 1 < nw) r |= p[1];
    }
    unsigned v = c;
    for (int k = 1; k <= g; ++k) v |= __funnelshift_l(l, c, k) | __funnelshift_r(c, r, k);
    out[base + e] = v;
  }
}

// Matched filter and candidate test of one 64 x 32 tile.  The tile of D^ (zero
// at bad and non-finite pixels and outside the image) carries a halo of R + 2;
// the row sums, the column sums (taps ascending in both) and the SNR of the
// 68 x 36 pixels that the 5 x 5 test reads stay in shared memory.  Four outputs
// per thread slide over a register window, so a staged value is read (2 R + 4) /
// 4 times per pass instead of 2 R + 1; only the SNR map and one bit per pixel
// are written.
constexpr int kMtX = 64, kMtY = 32;

template <int R>
__global__ void __launch_bounds__(256)
k_match(int H, int W, const float* __restrict__ D, const unsigned* __restrict__ goodw,
        const unsigned* __restrict__ guardw, Taps taps, const PassStats* __restrict__ stats, float thresh,
        float* __restrict__ snr, unsigned* __restrict__ cand, int* __restrict__ rowcnt) {
  constexpr int OX = kMtX + 2 * kNms, OY = kMtY + 2 * kNms;       // SNR pixels of the tile
  constexpr int NV = (4 + 2 * R + 3) / 4, PD = OX - 4 + 4 * NV;   // staged columns, read in groups of four
  constexpr int RY = OY + 2 * R, PS = OX + 1;
  __shared__ __align__(16) float dt[RY * PD > OY * PS ? RY * PD : OY * PS];
  __shared__ __align__(16) float tt[RY * OX];
  const int b = blockIdx.y, nw = (W + 31) / 32, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ntx = (W + kMtX - 1) / kMtX, x0 = (int)(blockIdx.x % ntx) * kMtX, y0 = (int)(blockIdx.x / ntx) * kMtY;
  const float* Db = D + (int64_t)b * H * W;
  const unsigned* gw = goodw + (int64_t)b * H * nw;
  const float scale = stats[b].scale;
  for (int j = warp; j < RY; j += 8) {
    const int y = y0 - kNms - R + j;
    const bool iny = y >= 0 && y < H;
#pragma unroll
    for (int i0 = 0; i0 < PD; i0 += 32) {
      const int i = i0 + lane, x = x0 - kNms - R + i;
      float v = 0.f;
      if (iny && x >= 0 && x < W && i < PD) {
        const float d = Db[(int64_t)y * W + x];
        v = (gw[(int64_t)y * nw + (x >> 5)] >> (x & 31)) & 1u ? d : 0.f;
      }
      if (i < PD) dt[j * PD + i] = v;
    }
  }
  __syncthreads();
  for (int e = tid; e < RY * (OX / 4); e += 256) {
    const int j = e / (OX / 4), i = 4 * (e % (OX / 4));
    float w[4 * NV], s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const float4 q = *reinterpret_cast<const float4*>(&dt[j * PD + i + 4 * k]);
      w[4 * k] = q.x; w[4 * k + 1] = q.y; w[4 * k + 2] = q.z; w[4 * k + 3] = q.w;
    }
#pragma unroll
    for (int k = 0; k <= 2 * R; ++k)
#pragma unroll
      for (int o = 0; o < 4; ++o) s[o] = fmaf(taps.g[k], w[k + o], s[o]);
    *reinterpret_cast<float4*>(&tt[j * OX + i]) = make_float4(s[0], s[1], s[2], s[3]);
  }
  __syncthreads();
  float* sn = dt;
  for (int e = tid; e < (OY / 4) * OX; e += 256) {
    const int i = e % OX, j = 4 * (e / OX);
    float w[4 + 2 * R], s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int k = 0; k < 4 + 2 * R; ++k) w[k] = tt[(j + k) * OX + i];
#pragma unroll
    for (int k = 0; k <= 2 * R; ++k)
#pragma unroll
      for (int o = 0; o < 4; ++o) s[o] = fmaf(taps.g[k], w[k + o], s[o]);
#pragma unroll
    for (int o = 0; o < 4; ++o) sn[(j + o) * PS + i] = s[o] * scale;
  }
  __syncthreads();
  for (int j = warp; j < kMtY; j += 8) {
    const int y = y0 + j;
    if (y >= H) break;
    int c = 0;
#pragma unroll
    for (int h = 0; h < kMtX / 32; ++h) {
      const int x = x0 + 32 * h + lane, wi = x0 / 32 + h;
      if (wi >= nw) break;
      const float* p = sn + (j + kNms) * PS + 32 * h + lane + kNms;
      const float v = *p;
      if (x < W) snr[((int64_t)b * H + y) * W + x] = v;
      bool ok = y >= kMargin && y < H - kMargin && x >= kMargin && x < W - kMargin && isfinite(v) && v >= thresh;
      if (ok && guardw) ok = !((guardw[((int64_t)b * H + y) * nw + wi] >> lane) & 1u);
      if (ok)
        for (int dy = -kNms; dy <= kNms; ++dy)
          for (int dx = -kNms; dx <= kNms; ++dx) {
            const float q = p[dy * PS + dx];
            if (isfinite(q) && q > v) ok = false;
          }
      const unsigned word = __ballot_sync(0xffffffffu, ok);
      if (lane == 0) cand[((int64_t)b * H + y) * nw + wi] = word;
      c += __popc(word);
    }
    if (lane == 0 && c) atomicAdd(&rowcnt[(int64_t)b * H + y], c);
  }
}

template <int R>
void run_match(int r, dim3 grid, cudaStream_t s, int H, int W, const float* D, const unsigned* goodw,
               const unsigned* guardw, const Taps& taps, const PassStats* stats, float thresh, float* snr,
               unsigned* cand, int* rowcnt) {
  if constexpr (R <= kMaxR) {
    if (r == R)
      k_match<R><<<grid, 256, 0, s>>>(H, W, D, goodw, guardw, taps, stats, thresh, snr, cand, rowcnt);
    else
      run_match<R + 1>(r, grid, s, H, W, D, goodw, guardw, taps, stats, thresh, snr, cand, rowcnt);
  }
}

// exclusive scan of the row counts of one CCD; count[b] = total
__global__ void __launch_bounds__(1024)
k_cand_scan(int H, const int* __restrict__ rowcnt, int* __restrict__ rowoff, int32_t* __restrict__ count) {
  __shared__ int part[1024];
  const int b = blockIdx.x, t = threadIdx.x;
  const int per = (H + 1023) / 1024;
  const int y0 = t * per;
  int s = 0;
  for (int k = 0; k < per; ++k)
    if (y0 + k < H) s += rowcnt[(int64_t)b * H + y0 + k];
  part[t] = s;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const int v = t >= off ? part[t - off] : 0;
    __syncthreads();
    part[t] += v;
    __syncthreads();
  }
  int run = part[t] - s;
  for (int k = 0; k < per; ++k)
    if (y0 + k < H) {
      rowoff[(int64_t)b * H + y0 + k] = run;
      run += rowcnt[(int64_t)b * H + y0 + k];
    }
  if (t == 1023) count[b] = part[1023];
}

// candidates of a row from its bits, in order: a warp per row, a lane per word
__global__ void __launch_bounds__(256)
k_cand_write(int H, int W, const float* __restrict__ snr, const unsigned* __restrict__ cand,
             const int* __restrict__ rowcnt, const int* __restrict__ rowoff, int max_cand, int32_t* __restrict__ xy,
             float* __restrict__ osnr) {
  const int b = blockIdx.y, y = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, nw = (W + 31) / 32;
  if (y >= H || rowcnt[(int64_t)b * H + y] == 0) return;
  const unsigned* cw = cand + ((int64_t)b * H + y) * nw;
  const float* sr = snr + ((int64_t)b * H + y) * W;
  int base = rowoff[(int64_t)b * H + y];
  for (int w0 = 0; w0 < nw; w0 += 32) {
    unsigned m = w0 + lane < nw ? cw[w0 + lane] : 0u;
    int off = __popc(m);
    const int mine = off;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, off, o);
      if (lane >= o) off += t;
    }
    const int total = __shfl_sync(0xffffffffu, off, 31);
    int idx = base + off - mine;
    for (; m; m &= m - 1u, ++idx) {
      const int x = (w0 + lane) * 32 + __ffs(m) - 1;
      if (idx < max_cand) {
        xy[((int64_t)b * max_cand + idx) * 2 + 0] = x;
        xy[((int64_t)b * max_cand + idx) * 2 + 1] = y;
        osnr[(int64_t)b * max_cand + idx] = sr[x];
      }
    }
    base += total;
  }
}

__global__ void __launch_bounds__(256)
k_stamps(int H, int W, const float* __restrict__ S, const float* __restrict__ R, const float* __restrict__ D,
         const int32_t* __restrict__ count, const int32_t* __restrict__ xy, int max_cand, float* __restrict__ stamps) {
  const int b = blockIdx.y, i = blockIdx.x;
  const int n = min(count[b], max_cand);
  if (i >= n) return;
  const int x = xy[((int64_t)b * max_cand + i) * 2], y = xy[((int64_t)b * max_cand + i) * 2 + 1];
  const int64_t img = (int64_t)H * W;
  const int side = 2 * kHalf + 1, pix = side * side;
  float* out = stamps + ((int64_t)b * max_cand + i) * 3 * pix;
  for (int e = threadIdx.x; e < 3 * pix; e += blockDim.x) {
    const int ch = e / pix, p = e % pix;
    const int yy = y - kHalf + p / side, xx = x - kHalf + p % side;
    const float* src = ch == 0 ? S : (ch == 1 ? R : D);
    const float v = src[b * img + (int64_t)yy * W + xx];
    out[e] = isfinite(v) ? v : 0.f;
  }
}

// one thread per stamp; FP64 moments of the difference channel
__global__ void k_shape_cuts(const float* __restrict__ stamps, const float* __restrict__ snr, int64_t n,
                             double psf_fwhm, double snr_min, int32_t* __restrict__ pass) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int side = 2 * kHalf + 1;
  const float* d = stamps + (i * 3 + 2) * side * side;
  const int c = kHalf;
  double tot = 0.0, sx = 0.0, sy = 0.0;
  for (int yy = -4; yy <= 4; ++yy)
    for (int xx = -4; xx <= 4; ++xx) {
      const double p = fmax((double)d[(c + yy) * side + c + xx], 0.0);
      tot += p;
      sx += p * xx;
      sy += p * yy;
    }
  if (!((double)snr[i] >= snr_min) || !(tot > 0.0)) {
    pass[i] = 0;
    return;
  }
  const double mx = sx / tot, my = sy / tot;
  double sxx = 0.0, syy = 0.0, sxy = 0.0;
  for (int yy = -4; yy <= 4; ++yy)
    for (int xx = -4; xx <= 4; ++xx) {
      const double p = fmax((double)d[(c + yy) * side + c + xx], 0.0);
      sxx += p * (xx - mx) * (xx - mx);
      syy += p * (yy - my) * (yy - my);
      sxy += p * (xx - mx) * (yy - my);
    }
  sxx /= tot;
  syy /= tot;
  sxy /= tot;
  const double tr = sxx + syy, det = sxx * syy - sxy * sxy;
  const double disc = sqrt(fmax(tr * tr / 4.0 - det, 0.0));
  const double l1 = tr / 2.0 + disc, l2 = fmax(tr / 2.0 - disc, 1e-12);
  const double fwhm = 2.0 * sqrt(2.0 * log(2.0)) * sqrt(fmax(0.5 * (l1 + l2), 0.0));
  double neg = 0.0, absum = 0.0;
  for (int yy = -3; yy <= 3; ++yy)
    for (int xx = -3; xx <= 3; ++xx) {
      const double v = (double)d[(c + yy) * side + c + xx];
      neg += fabs(fmin(v, 0.0));
      absum += fabs(v);
    }
  const double neg_frac = neg / fmax(absum, 1e-12);
  const double ratio = sqrt(l1 / l2);
  pass[i] = (0.5 * psf_fwhm <= fwhm && fwhm <= 2.0 * psf_fwhm && neg_frac < 0.3 && ratio < 2.5) ? 1 : 0;
}

// The same cuts with the size and axis ratio from Gaussian-weighted adaptive
// moments of the difference channel over the central 15 x 15: from a round
// weight of the PSF's width at the centre, 40 times w = exp(-(r - mu)^T M^-1
// (r - mu) / 2), mu = sum w I r / sum w I, M = 2 sum w I (r - mu)(r - mu)^T /
// sum w I (a Gaussian source of covariance C is the fixed point M = C); a
// candidate whose weighted flux is not positive, whose M is not positive
// definite, whose centroid moves more than 3 px or whose M grows past
// 25 px^2 fails.  One thread per stamp, FP64.
constexpr int kAmHalf = 7, kAmIters = 40;

__global__ void k_shape_cuts_adaptive(const float* __restrict__ stamps, const float* __restrict__ snr, int64_t n,
                                      double psf_fwhm, double snr_min, int32_t* __restrict__ pass) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int side = 2 * kHalf + 1;
  const float* d = stamps + (i * 3 + 2) * side * side;
  const int c = kHalf;
  const double fw2s = 2.0 * sqrt(2.0 * log(2.0));
  const double s0w = psf_fwhm / fw2s;
  double mxx = s0w * s0w, myy = s0w * s0w, mxy = 0.0, mx = 0.0, my = 0.0;
  bool ok = (double)snr[i] >= snr_min;
  for (int it = 0; ok && it < kAmIters; ++it) {
    const double det = mxx * myy - mxy * mxy;
    if (!(det > 0.0 && mxx > 0.0 && myy > 0.0)) { ok = false; break; }
    const double ia = myy / det, ib = -mxy / det, ic = mxx / det;   // M^-1 = [[ia, ib], [ib, ic]]
    double s0 = 0.0, sx = 0.0, sy = 0.0, sxx = 0.0, syy = 0.0, sxy = 0.0;
    for (int yy = -kAmHalf; yy <= kAmHalf; ++yy)
      for (int xx = -kAmHalf; xx <= kAmHalf; ++xx) {
        const double dx = xx - mx, dy = yy - my;
        const double wv = exp(-0.5 * (ia * dx * dx + 2.0 * ib * dx * dy + ic * dy * dy)) *
                          (double)d[(c + yy) * side + c + xx];
        s0 += wv;
        sx += wv * xx;
        sy += wv * yy;
        sxx += wv * xx * xx;
        syy += wv * yy * yy;
        sxy += wv * xx * yy;
      }
    if (!(s0 > 0.0)) { ok = false; break; }
    mx = sx / s0;
    my = sy / s0;
    // central moments about the new centroid from the raw sums
    mxx = 2.0 * (sxx / s0 - mx * mx);
    myy = 2.0 * (syy / s0 - my * my);
    mxy = 2.0 * (sxy / s0 - mx * my);
    if (fabs(mx) > 3.0 || fabs(my) > 3.0 || mxx > 25.0 || myy > 25.0) ok = false;
  }
  if (ok && !(mxx * myy - mxy * mxy > 0.0 && mxx > 0.0 && myy > 0.0)) ok = false;
  if (!ok) {
    pass[i] = 0;
    return;
  }
  const double tr = mxx + myy, det = mxx * myy - mxy * mxy;
  const double disc = sqrt(fmax(tr * tr / 4.0 - det, 0.0));
  const double l1 = tr / 2.0 + disc, l2 = fmax(tr / 2.0 - disc, 1e-12);
  const double fwhm = fw2s * sqrt(0.5 * (l1 + l2));
  double neg = 0.0, absum = 0.0;
  for (int yy = -3; yy <= 3; ++yy)
    for (int xx = -3; xx <= 3; ++xx) {
      const double v = (double)d[(c + yy) * side + c + xx];
      neg += fabs(fmin(v, 0.0));
      absum += fabs(v);
    }
  const double neg_frac = neg / fmax(absum, 1e-12);
  const double ratio = sqrt(l1 / l2);
  pass[i] = (0.5 * psf_fwhm <= fwhm && fwhm <= 2.0 * psf_fwhm && neg_frac < 0.3 && ratio < 2.5) ? 1 : 0;
}

sfft_status_t fail(cudaError_t e, const char* where) {
  sfft::set_last_error((std::string(where) + ": " + cudaGetErrorString(e)).c_str());
  return SFFT_ERR_CUDA;
}

}  // namespace

extern "C" size_t rb_detect_workspace_bytes(int32_t H, int32_t W, int32_t batch, int32_t max_cand) {
  (void)max_cand;
  if (H < 1 || W < 1 || batch < 1) return 0;
  return DetectLayout(H, W, batch).total;
}

extern "C" sfft_status_t rb_detect(int32_t H, int32_t W, int32_t batch, const float* D, const float* S,
                                   const float* R, const uint8_t* bad, float psf_sigma, float thresh,
                                   int32_t guard, int32_t max_cand, int32_t* xy, float* snr, int32_t* count, float* stamps, void* ws,
                                   void* stream) {
  if (H < 2 * kHalf + 1 || W < 2 * kHalf + 1 || batch < 1 || max_cand < 0 || !D || !S || !R || !count || !ws ||
      (max_cand > 0 && (!xy || !snr || !stamps)) || !(psf_sigma > 0.f) || !(psf_sigma <= 5.f) || guard < 0 ||
      guard > kMargin ||
      (reinterpret_cast<uintptr_t>(ws) & 255))
    return SFFT_ERR_ARG;
  if (batch > 65535 || sizeof(float) * (W + 2 * kMaxR) > 48 * 1024) return SFFT_ERR_UNSUPPORTED;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const DetectLayout L(H, W, batch);
  char* base = static_cast<char*>(ws);
  float* snr_map = reinterpret_cast<float*>(base + L.snr);
  unsigned* goodw = reinterpret_cast<unsigned*>(base + L.good);
  unsigned* badw = reinterpret_cast<unsigned*>(base + L.bad);
  unsigned* cand = reinterpret_cast<unsigned*>(base + L.cand);
  double* part = reinterpret_cast<double*>(base + L.part);
  PassStats* stats = reinterpret_cast<PassStats*>(base + L.stats);
  int* counter = reinterpret_cast<int*>(base + L.zero);
  int* rowcnt = reinterpret_cast<int*>(base + L.rowcnt);
  int* rowoff = reinterpret_cast<int*>(base + L.rowoff);

  Taps taps{};
  taps.r = (int)ceil(3.0 * (double)psf_sigma);
  for (int k = 0; k <= 2 * taps.r; ++k) {
    const double t = k - taps.r;
    taps.g[k] = (float)exp(-t * t / (2.0 * (double)psf_sigma * (double)psf_sigma));
  }
  cudaError_t z = cudaMemsetAsync(counter, 0, L.zero_bytes, s);
  if (z != cudaSuccess) return fail(z, "rb_detect");
  // eight words of a row per warp at least: a narrow image's rows share CTAs
  // (with a CTA per row, one of its eight warps had work at 200 columns)
  const int groups = (L.words + kClipWords - 1) / kClipWords;
  const dim3 gs((int)std::min<int64_t>(std::min(kStatBlocks, H), ((int64_t)H * groups + 7) / 8), batch);
  k_clip_pass<true><<<gs, 256, 0, s>>>(H, W, D, bad, goodw, badw, part, stats, counter, 0, taps);
  for (int p = 1; p < kStatPasses; ++p)
    k_clip_pass<false><<<gs, 256, 0, s>>>(H, W, D, bad, goodw, badw, part, stats, counter, p, taps);
  const unsigned* guardw = bad ? badw : nullptr;   // the mask the candidate test reads
  if (bad && guard > 0) {
    unsigned* gm = reinterpret_cast<unsigned*>(base + L.guard);
    const int gx = (int)std::min<int64_t>(((int64_t)H * L.words + 255) / 256, 2048);
    k_guard<<<dim3(gx, batch), 256, 0, s>>>(H, L.words, badw, guard, gm);
    guardw = gm;
  }
  run_match<1>(taps.r, dim3((unsigned)(((W + kMtX - 1) / kMtX) * ((H + kMtY - 1) / kMtY)), batch), s, H, W, D, goodw, guardw, taps,
               stats, thresh, snr_map, cand, rowcnt);
  k_cand_scan<<<batch, 1024, 0, s>>>(H, rowcnt, rowoff, count);
  if (max_cand > 0) {
    k_cand_write<<<dim3((H + 7) / 8, batch), 256, 0, s>>>(H, W, snr_map, cand, rowcnt, rowoff, max_cand, xy, snr);
    k_stamps<<<dim3(max_cand, batch), 256, 0, s>>>(H, W, S, R, D, count, xy, max_cand, stamps);
  }
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SFFT_OK : fail(e, "rb_detect");
}

extern "C" sfft_status_t rb_shape_cuts(const float* stamps, const float* snr, int64_t n, float psf_fwhm,
                                       float snr_min, int32_t* pass, void* stream) {
  if (n < 0 || (n > 0 && (!stamps || !snr || !pass)) || !(psf_fwhm > 0.f)) return SFFT_ERR_ARG;
  if (n == 0) return SFFT_OK;
  k_shape_cuts<<<(unsigned)((n + 127) / 128), 128, 0, static_cast<cudaStream_t>(stream)>>>(stamps, snr, n, psf_fwhm,
                                                                                             snr_min, pass);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SFFT_OK : fail(e, "rb_shape_cuts");
}

extern "C" sfft_status_t rb_shape_cuts_adaptive(const float* stamps, const float* snr, int64_t n, float psf_fwhm,
                                                float snr_min, int32_t* pass, void* stream) {
  if (n < 0 || (n > 0 && (!stamps || !snr || !pass)) || !(psf_fwhm > 0.f)) return SFFT_ERR_ARG;
  if (n == 0) return SFFT_OK;
  k_shape_cuts_adaptive<<<(unsigned)((n + 127) / 128), 128, 0, static_cast<cudaStream_t>(stream)>>>(
      stamps, snr, n, psf_fwhm, snr_min, pass);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? SFFT_OK : fail(e, "rb_shape_cuts_adaptive");
}
