// Mask and sky-offset preparation, fit-mask erosion and the background
// moments.
//   good(x)  = bad(x) == 0 && finite(R(x)) && finite(S(x))
//   R_m(x)   = good ? R - s_R : 0
//   M_fit(x) = x at least w from every edge and good on the whole L x L
//              footprint (separable erosion: a row pass, then a column pass)
//   moments  sum_x M_fit xt^a yt^b (a + b <= 2 D_B)  and
//            sum_x M_fit xt^a yt^b v(x) (a + b <= D_B), v = S - s_S or the
//            refinement residual e; FP32 per-thread partials, FP64 block and
//            global accumulation.
// The image-space assembly keeps the masks as bits, a 32-bit word per 32 pixels
// of a row, and lists the edges of M_fit (below).
// The sky constants, when not given, are the mean of the good pixels rounded
// to an integer, so R - s_R and S - s_S are exact in FP32 for |R|, |S| < 2^24.
#include "common.cuh"
#include "plan.h"

namespace sfft {

// Sums of R, S and the count over the good pixels, per CCD.  Where a CCD's
// images start on 16-byte boundaries the pixels go in groups of four (float4
// and uchar4 loads); the launch gives each thread at most 64 groups, so a
// thread's FP32 partial sums cover at most 256 pixels before the FP64 block
// sums.
__global__ void __launch_bounds__(256)
k_sky_sum(const float* __restrict__ R, const float* __restrict__ S, const uint8_t* __restrict__ bad, int64_t npx,
          double* __restrict__ acc, double* __restrict__ sky) {
  __shared__ double red[2][8];
  __shared__ int redn[8];
  const int ccd = blockIdx.y;
  const float* r = R + ccd * npx;
  const float* s = S + ccd * npx;
  const uint8_t* b = bad ? bad + ccd * npx : nullptr;
  float sr = 0.f, ss = 0.f;
  int cnt = 0;
  const int64_t t0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, nt = (int64_t)gridDim.x * blockDim.x;
  const bool vec = ((reinterpret_cast<uintptr_t>(r) | reinterpret_cast<uintptr_t>(s)) & 15) == 0 &&
                   (reinterpret_cast<uintptr_t>(b) & 3) == 0;
  int64_t i0 = 0;
  if (vec) {
    const int64_t n4 = npx / 4;
    const float4* r4 = reinterpret_cast<const float4*>(r);
    const float4* s4 = reinterpret_cast<const float4*>(s);
    const uchar4* b4 = reinterpret_cast<const uchar4*>(b);
#pragma unroll 4
    for (int64_t q = t0; q < n4; q += nt) {
      const float4 rv = r4[q], sv = s4[q];
      const uchar4 bv = b ? b4[q] : make_uchar4(0, 0, 0, 0);
      const float ra[4] = {rv.x, rv.y, rv.z, rv.w}, sa[4] = {sv.x, sv.y, sv.z, sv.w};
      const unsigned char ba[4] = {bv.x, bv.y, bv.z, bv.w};
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (ba[k] == 0 && isfinite(ra[k]) && isfinite(sa[k])) { sr += ra[k]; ss += sa[k]; ++cnt; }
    }
    i0 = n4 * 4;
  }
  for (int64_t i = i0 + t0; i < npx; i += nt) {
    const float rv = r[i], sv = s[i];
    if ((!b || b[i] == 0) && isfinite(rv) && isfinite(sv)) { sr += rv; ss += sv; ++cnt; }
  }
  // the lower half warp reduces R, the upper S: one FP64 addition per step for
  // both (they run at 1/64 of the FP32 rate: 20 -> 16 us at 2048 x 4096 with
  // the count in integers)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double give = (double)(lane < 16 ? ss : sr);
  double v = (double)(lane < 16 ? sr : ss) + __shfl_xor_sync(0xffffffffu, give, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  cnt = __reduce_add_sync(0xffffffffu, cnt);
  if ((lane & 15) == 0) red[lane >> 4][warp] = v;
  if (lane == 0) redn[warp] = cnt;
  __syncthreads();
  if (threadIdx.x < 3) {
    double t = 0.0;
    for (int k = 0; k < 8; ++k) t += threadIdx.x < 2 ? red[threadIdx.x][k] : (double)redn[k];
    atomicAdd(&acc[4 * ccd + threadIdx.x], t);
    __threadfence();
  }
  __syncthreads();
  // the CCD's last CTA (the count is the fourth, cleared word of its sums)
  if (threadIdx.x == 0) {
    unsigned* done = reinterpret_cast<unsigned*>(&acc[4 * ccd + 3]);
    if (atomicAdd(done, 1u) == gridDim.x - 1) {
      __threadfence();
      const double m = __ldcg(&acc[4 * ccd + 2]);
      for (int k = 0; k < 2; ++k) sky[2 * ccd + k] = m > 0 ? rint(__ldcg(&acc[4 * ccd + k]) / m) : 0.0;
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256)
k_prep(const float* __restrict__ R, const float* __restrict__ S, const uint8_t* __restrict__ bad,
       const double* __restrict__ sky, int64_t npx, uint8_t* __restrict__ good, T* __restrict__ Rm) {
  const int ccd = blockIdx.y;
  const T sR = (T)sky[2 * ccd];
  const int64_t base = ccd * npx;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < npx; i += (int64_t)gridDim.x * blockDim.x) {
    const float rv = R[base + i], sv = S[base + i];
    const bool g = (!bad || bad[base + i] == 0) && isfinite(rv) && isfinite(sv);
    good[base + i] = g ? 1 : 0;
    Rm[base + i] = g ? (T)rv - sR : (T)0;
  }
}

// row pass: gh(y, x) = w <= x < W - w and good on [x - w, x + w]
__global__ void __launch_bounds__(256)
k_erode_rows(const uint8_t* __restrict__ good, uint8_t* __restrict__ gh, int H, int W, int w) {
  const int y = blockIdx.x, ccd = blockIdx.y;
  const uint8_t* g = good + ((int64_t)ccd * H + y) * W;
  uint8_t* o = gh + ((int64_t)ccd * H + y) * W;
  for (int x = threadIdx.x; x < W; x += blockDim.x) {
    uint8_t v = 0;
    if (x >= w && x < W - w) {
      v = 1;
      for (int dx = -w; dx <= w; ++dx) v &= g[x + dx];
    }
    o[x] = v;
  }
}

// column pass: M(y, x) = w <= y < H - w and gh on [y - w, y + w]
__global__ void __launch_bounds__(256)
k_erode_cols(const uint8_t* __restrict__ gh, uint8_t* __restrict__ mfit, int H, int W, int w) {
  const int y = blockIdx.x, ccd = blockIdx.y;
  const uint8_t* g = gh + (int64_t)ccd * H * W;
  uint8_t* o = mfit + ((int64_t)ccd * H + y) * W;
  const bool inside = (y >= w && y < H - w);
  for (int x = threadIdx.x; x < W; x += blockDim.x) {
    uint8_t v = 0;
    if (inside) {
      v = 1;
      for (int dy = -w; dy <= w; ++dy) v &= g[(int64_t)(y + dy) * W + x];
    }
    o[x] = v;
  }
}

// one block per (row, ccd).  mom_bb[mono(a,b)] for a+b <= DBB, mom_v[mono(a,b)] for a+b <= DV.
// Per CCD the background moments sum_x M_fit xt^a yt^b (a + b <= DBB) and
// sum_x M_fit xt^a yt^b v(x) (a + b <= DV), with yt^b factored out of each
// row.  A CTA takes kMomRows consecutive rows, a warp per row at a time.  A
// lane sums its pixels in groups of four (float4 / uchar4 loads where the row
// is 16-byte aligned): each group's sum in T, added to the lane's T sums, then
// a warp tree in T gives the row's sums.  The row's FP64 contributions are
// added over the CTA's rows (fixed order) and then atomically to the CCD's
// moments, so each moment takes H / kMomRows atomic adds per CCD instead of H.
constexpr int kMomRows = 8;

template <typename T>
__device__ __forceinline__ void load4(const T* p, T (&v)[4]);
template <>
__device__ __forceinline__ void load4<float>(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
template <>
__device__ __forceinline__ void load4<double>(const double* p, double (&v)[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

template <typename T>
__global__ void __launch_bounds__(256)
k_moments(const uint8_t* __restrict__ mfit, const float* __restrict__ S, const double* __restrict__ sky,
          const T* __restrict__ E, int H, int W, int DBB, int DV, double* __restrict__ mom_bb, int64_t bb_stride,
          double* __restrict__ mom_v, int64_t v_stride, int* __restrict__ rowflag, int rf_stride) {
  constexpr int NBB = n_mono(kMaxWeightDeg), NV = n_mono(kMaxD);
  __shared__ double part[8][NBB + NV];
  const int ccd = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const T sS = S ? (T)sky[2 * ccd + 1] : (T)0;
  const T xs = (T)2 / (T)(W > 1 ? W - 1 : 1);
  const double ysc = 2.0 / (double)(H > 1 ? H - 1 : 1);
  // part[w]: warp w's rows, FP64, added to by its lane 0
  for (int i = threadIdx.x; i < 8 * (NBB + NV); i += blockDim.x) (&part[0][0])[i] = 0.0;
  __syncthreads();
  const int y_end = min(H, ((int)blockIdx.x + 1) * kMomRows);
  for (int y = (int)blockIdx.x * kMomRows + warp; y < y_end; y += 8) {
    const int64_t row = ((int64_t)ccd * H + y) * W;
    const uint8_t* mr = mfit + row;
    const float* sr = S ? S + row : nullptr;
    const T* er = E ? E + row : nullptr;
    T pm[kMaxWeightDeg + 1] = {0, 0, 0, 0, 0};
    T pv[kMaxD + 1] = {0, 0, 0};
    int cnt = 0;
    // adds the pixels of one group (mk: in the fit mask, vk: S - s_S or e)
    auto add_group = [&](const int x0, const bool (&mk)[4], const T (&vk)[4], int n) {
      T gm[kMaxWeightDeg + 1] = {0, 0, 0, 0, 0};
      T gv[kMaxD + 1] = {0, 0, 0};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        if (k >= n || !mk[k]) continue;
        ++cnt;
        const T xt = (T)(x0 + k) * xs - (T)1;
        T pw = 1;
#pragma unroll
        for (int a = 0; a <= kMaxWeightDeg; ++a) {
          gm[a] += pw;
          if (a <= kMaxD) gv[a] += pw * vk[k];
          pw *= xt;
        }
      }
#pragma unroll
      for (int a = 0; a <= kMaxWeightDeg; ++a) pm[a] += gm[a];
#pragma unroll
      for (int a = 0; a <= kMaxD; ++a) pv[a] += gv[a];
    };
    const bool vec = (W & 3) == 0 && (reinterpret_cast<uintptr_t>(mr) & 3) == 0 &&
                     (reinterpret_cast<uintptr_t>(sr) & 15) == 0 && (reinterpret_cast<uintptr_t>(er) & 15) == 0;
    if (vec) {
#pragma unroll 4
      for (int x0 = 4 * lane; x0 < W; x0 += 128) {
        const uchar4 m4 = *reinterpret_cast<const uchar4*>(mr + x0);
        const bool mk[4] = {m4.x != 0, m4.y != 0, m4.z != 0, m4.w != 0};
        T vk[4] = {0, 0, 0, 0};
        if (sr) {
          float f[4];
          load4<float>(sr + x0, f);
#pragma unroll
          for (int k = 0; k < 4; ++k) vk[k] = (T)f[k] - sS;
        } else if (er) {
          load4<T>(er + x0, vk);
        }
        add_group(x0, mk, vk, 4);
      }
    } else {
      for (int x0 = 4 * lane; x0 < W; x0 += 128) {
        const int n = min(4, W - x0);
        bool mk[4];
        T vk[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          mk[k] = k < n && mr[x0 + k] != 0;
          vk[k] = k < n ? (sr ? (T)sr[x0 + k] - sS : (er ? er[x0 + k] : (T)0)) : (T)0;
        }
        add_group(x0, mk, vk, n);
      }
    }
    cnt = warp_sum(cnt);
#pragma unroll
    for (int a = 0; a <= kMaxWeightDeg; ++a) pm[a] = warp_sum(pm[a]);
#pragma unroll
    for (int a = 0; a <= kMaxD; ++a) pv[a] = warp_sum(pv[a]);
    if (lane == 0) {
      if (rowflag) rowflag[(int64_t)ccd * rf_stride + y] = cnt > 0 ? 1 : 0;
      const double yt = (double)y * ysc - 1.0;
#pragma unroll
      for (int a = 0; a <= kMaxWeightDeg; ++a) {
        double yp = 1.0;
#pragma unroll
        for (int b = 0; a + b <= kMaxWeightDeg; ++b) {
          if (a + b <= DBB) part[warp][mono_index(a, b)] += (double)pm[a] * yp;
          yp *= yt;
        }
      }
#pragma unroll
      for (int a = 0; a <= kMaxD; ++a) {
        double yp = 1.0;
#pragma unroll
        for (int b = 0; a + b <= kMaxD; ++b) {
          if (a + b <= DV) part[warp][NBB + mono_index(a, b)] += (double)pv[a] * yp;
          yp *= yt;
        }
      }
    }
  }
  __syncthreads();
  const int nbb = mom_bb ? n_mono(DBB) : 0, nv = n_mono(DV);
  if (threadIdx.x < nbb + nv) {
    const int i = threadIdx.x < nbb ? threadIdx.x : NBB + (threadIdx.x - nbb);
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += part[w][i];
    if (threadIdx.x < nbb) atomicAdd(&mom_bb[ccd * bb_stride + threadIdx.x], s);
    else atomicAdd(&mom_v[ccd * v_stride + (threadIdx.x - nbb)], s);
  }
}

// ------------------------------------------------------------------ masks as bits, mask edges
// R_m and the good pixels as bits: a warp per run of words, four in flight.
// 9 bytes in (R, S, bad) and 4 (FP64: 8) out per pixel; the byte masks it replaces cost two
// more passes over the image (k_prep, k_erode_rows and k_erode_cols: 94 us per
// 2048 x 4096 CCD).
template <typename T>
__global__ void __launch_bounds__(256)
k_prep_bits(const float* __restrict__ R, const float* __restrict__ S, const uint8_t* __restrict__ bad,
            const double* __restrict__ sky, int H, int W, unsigned* __restrict__ goodw, T* __restrict__ Rm) {
  constexpr int U = 4;
  const int ccd = blockIdx.y, lane = threadIdx.x & 31, nw = (W + 31) / 32;
  const T sR = (T)sky[2 * ccd];
  const int64_t base = (int64_t)ccd * H * W;
  unsigned* gw = goodw + (int64_t)ccd * H * nw;
  const int runs = (nw + U - 1) / U;
  const int64_t total = (int64_t)H * runs;
  for (int64_t i = blockIdx.x * 8ll + (threadIdx.x >> 5); i < total; i += gridDim.x * 8ll) {
    const int y = (int)(i / runs), w0 = (int)(i % runs) * U;
    const int64_t row = base + (int64_t)y * W;
    float r[U], s[U];
    uint8_t b[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int x = (w0 + k) * 32 + lane;
      const bool in = x < W;
      r[k] = in ? R[row + x] : INFINITY;
      s[k] = in ? S[row + x] : 0.f;
      b[k] = in && bad ? bad[row + x] : 0;
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int x = (w0 + k) * 32 + lane;
      const bool g = b[k] == 0 && isfinite(r[k]) && isfinite(s[k]);
      if (x < W) Rm[row + x] = g ? (T)r[k] - sR : (T)0;
      const unsigned word = __ballot_sync(0xffffffffu, g);
      if (lane == 0 && w0 + k < nw) gw[(int64_t)y * nw + w0 + k] = word;
    }
  }
}

// M_fit words: 1 where the pixel is at least w from every edge and good on its
// whole L x L footprint.  The footprint's rows are ANDed word by word, then the
// word with its neighbours is eroded by w on either side.
__device__ __forceinline__ unsigned fit_word(const unsigned* g, int H, int W, int nw, int w, int y, int wi) {
  if (y < w || y >= H - w || wi >= nw) return 0u;
  unsigned l = ~0u, c = ~0u, r = ~0u;
  for (int d = -w; d <= w; ++d) {
    const unsigned* p = g + (int64_t)(y + d) * nw + wi;
    l &= wi > 0 ? p[-1] : 0u;
    c &= p[0];
    r &= wi + 1 < nw ? p[1] : 0u;
  }
  unsigned m = c;
  for (int k = 1; k <= w; ++k) m &= __funnelshift_l(l, c, k) & __funnelshift_r(c, r, k);
  // columns [w, W - w)
  const int lo = max(0, w - 32 * wi), hi = min(32, W - w - 32 * wi);
  if (lo >= 32 || hi <= 0) return 0u;
  const unsigned cut = (hi == 32 ? ~0u : (1u << hi) - 1u) & (~0u << lo);
  return m & cut;
}

// Eight rows per CTA.  With EDGES also the numbers of x edges (M differs from
// its right neighbour) and y edges (from the pixel above it in y) per row, for
// which the CTA forms one more row.
constexpr int kFmRows = 8;

template <bool EDGES>
__global__ void __launch_bounds__(256)
k_fit_mask(const unsigned* __restrict__ goodw, int H, int W, int w, unsigned* __restrict__ mfitw,
           int* __restrict__ cnt, int64_t cnt_stride) {
  __shared__ unsigned m[kFmRows + 1][65];   // W <= 2048: at most 64 words, and a zero
  const int ccd = blockIdx.y, y0 = blockIdx.x * kFmRows, nw = (W + 31) / 32;
  const unsigned* g = goodw + (int64_t)ccd * H * nw;
  constexpr int rows = EDGES ? kFmRows + 1 : kFmRows;
  for (int i = threadIdx.x; i < rows * nw; i += 256) {
    const int j = i / nw, wi = i % nw, y = y0 + j;
    const unsigned v = y < H ? fit_word(g, H, W, nw, w, y, wi) : 0u;
    m[j][wi] = v;
    if (j < kFmRows && y < H) mfitw[((int64_t)ccd * H + y) * nw + wi] = v;
  }
  if (!EDGES) return;
  if (threadIdx.x <= kFmRows) m[threadIdx.x][nw] = 0u;
  __syncthreads();
  const int j = threadIdx.x >> 5, lane = threadIdx.x & 31, y = y0 + j;
  if (y >= H) return;
  int nx = 0, ny = 0;
  for (int wi = lane; wi < nw; wi += 32) {
    const unsigned c = m[j][wi];
    nx += __popc(c ^ __funnelshift_r(c, m[j][wi + 1], 1));
    if (y + 1 < H) ny += __popc(c ^ m[j + 1][wi]);
  }
  nx = __reduce_add_sync(0xffffffffu, nx);
  ny = __reduce_add_sync(0xffffffffu, ny);
  if (lane == 0) {
    cnt[ccd * cnt_stride + y] = nx;
    cnt[ccd * cnt_stride + H + 1 + y] = ny;
  }
}

// exclusive scan of the row counts; entry H is the total
__global__ void __launch_bounds__(1024)
k_edge_scan(int* __restrict__ cnt, int64_t cnt_stride, int H) {
  __shared__ int wsum[32];
  __shared__ int carry;
  int* c = cnt + blockIdx.x * cnt_stride + blockIdx.y * (H + 1);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < H; base += 1024) {
    const int i = base + tid;
    const int v = i < H ? c[i] : 0;
    int s = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    if (lane == 31) wsum[warp] = s;
    __syncthreads();
    int off = carry;
    for (int k = 0; k < warp; ++k) off += wsum[k];
    if (i < H) c[i] = off + s - v;
    __syncthreads();
    if (tid == 1023) carry = off + s;
    __syncthreads();
  }
  if (tid == 0) c[H] = carry;
}

// The edge lists in row order, entry (y W + x) << 1 | (M falls): a warp per row,
// a lane per word.
__global__ void __launch_bounds__(256)
k_edge_list(const unsigned* __restrict__ mfitw, int H, int W, const int* __restrict__ cnt, int64_t cnt_stride,
            unsigned* __restrict__ lx, unsigned* __restrict__ ly, int64_t lstride) {
  const int y = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31, ccd = blockIdx.y, nw = (W + 31) / 32;
  if (y >= H) return;
  const unsigned* m = mfitw + ((int64_t)ccd * H + y) * nw;
  const int* c = cnt + ccd * cnt_stride;
  int base[2] = {c[y], c[H + 1 + y]};
  unsigned* out[2] = {lx + ccd * lstride, ly + ccd * lstride};
  for (int w0 = 0; w0 < nw; w0 += 32) {
    const int wi = w0 + lane;
    const unsigned v = wi < nw ? m[wi] : 0u, nx = wi + 1 < nw ? m[wi + 1] : 0u;
    const unsigned dn = wi < nw && y + 1 < H ? m[nw + wi] : v;
    unsigned e[2] = {v ^ __funnelshift_r(v, nx, 1), v ^ dn};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int n = __popc(e[q]);
      int off = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, off, o);
        if (lane >= o) off += t;
      }
      const int total = __shfl_sync(0xffffffffu, off, 31);
      unsigned* p = out[q] + base[q] + off - n;
      for (unsigned b = e[q]; b; b &= b - 1u) {
        const int k = __ffs(b) - 1;
        *p++ = ((unsigned)y * (unsigned)W + (unsigned)(32 * wi + k)) << 1 | ((v >> k) & 1u);
      }
      base[q] += total;
    }
  }
}

static int grid_for(int64_t n, int threads, int cap) {
  int64_t g = (n + threads - 1) / threads;
  return (int)(g < cap ? (g < 1 ? 1 : g) : cap);
}

cudaError_t launch_sky(const sfft_plan_s* p, const float* R, const float* S, const uint8_t* bad,
                       const double* sky_in, void* ws) {
  double* sky = ws_at<double>(ws, p->sky);
  const int B = p->d.batch;
  // the status words, the sky constants and their sums follow each other
  const size_t clear = sky_in ? p->status.bytes : p->skyacc.off + p->skyacc.bytes - p->status.off;
  cudaError_t e = cudaMemsetAsync(ws_at<char>(ws, p->status), 0, clear, p->stream);
  if (e != cudaSuccess) return e;
  if (sky_in) {
    return cudaMemcpyAsync(sky, sky_in, sizeof(double) * 2 * B, cudaMemcpyDeviceToDevice, p->stream);
  }
  double* acc = ws_at<double>(ws, p->skyacc);
  const int64_t npx = (int64_t)p->d.H * p->d.W;
  // at least four CTAs per SM, and at most 64 groups of four pixels per thread
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t per_cta = 256 * 64 * 4;
  const int gx = (int)std::min<int64_t>(std::max<int64_t>(4 * (int64_t)std::max(sms, 1), (npx + per_cta - 1) / per_cta),
                                        1 << 20);
  k_sky_sum<<<dim3(gx, B), 256, 0, p->stream>>>(R, S, bad, npx, acc, sky);
  p->nlaunch += 1;
  return cudaGetLastError();
}

template <typename T>
static cudaError_t prep_T(const sfft_plan_s* p, const float* R, const float* S, const uint8_t* bad, void* ws) {
  const int H = p->d.H, W = p->d.W, B = p->d.batch;
  const int64_t npx = (int64_t)H * W;
  uint8_t* good = ws_at<uint8_t>(ws, p->good);
  uint8_t* gh = ws_at<uint8_t>(ws, p->gh);
  uint8_t* mfit = ws_at<uint8_t>(ws, p->mfit);
  T* Rm = ws_at<T>(ws, p->rm);
  dim3 g1(grid_for(npx, 256 * 8, 1184), B);
  k_prep<T><<<g1, 256, 0, p->stream>>>(R, S, bad, ws_at<double>(ws, p->sky), npx, good, Rm);
  dim3 g2(H, B);
  k_erode_rows<<<g2, 256, 0, p->stream>>>(good, gh, H, W, p->w);
  k_erode_cols<<<g2, 256, 0, p->stream>>>(gh, mfit, H, W, p->w);
  p->nlaunch += 3;
  return cudaGetLastError();
}

cudaError_t launch_prep(const sfft_plan_s* p, const float* R, const float* S, const uint8_t* bad, void* ws) {
  return p->fp64 ? prep_T<double>(p, R, S, bad, ws) : prep_T<float>(p, R, S, bad, ws);
}

int64_t edge_cap(const sfft_plan_s* p) {
  return std::max((int64_t)p->d.H * p->tap.row_cap, (int64_t)p->d.W * p->tap.col_cap);
}

cudaError_t launch_prep_bits(const sfft_plan_s* p, const float* R, const float* S, const uint8_t* bad, bool edges,
                             void* ws) {
  const int H = p->d.H, W = p->d.W, B = p->d.batch, nw = (W + 31) / 32;
  unsigned* goodw = ws_at<unsigned>(ws, p->goodw);
  unsigned* mfitw = ws_at<unsigned>(ws, p->mfitw);
  const double* sky = ws_at<double>(ws, p->sky);
  const int64_t runs = (int64_t)H * ((nw + 3) / 4);
  const dim3 g1((unsigned)std::min<int64_t>((runs + 7) / 8, 152 * 8), B);
  if (p->fp64) k_prep_bits<double><<<g1, 256, 0, p->stream>>>(R, S, bad, sky, H, W, goodw, ws_at<double>(ws, p->rm));
  else k_prep_bits<float><<<g1, 256, 0, p->stream>>>(R, S, bad, sky, H, W, goodw, ws_at<float>(ws, p->rm));
  const dim3 g2((H + kFmRows - 1) / kFmRows, B);
  p->nlaunch += 2;
  if (!edges) {
    k_fit_mask<false><<<g2, 256, 0, p->stream>>>(goodw, H, W, p->w, mfitw, nullptr, 0);
    return cudaGetLastError();
  }
  int* cnt = ws_at<int>(ws, p->ecnt);
  unsigned* lx = ws_at<unsigned>(ws, p->elist);
  const int64_t cap = edge_cap(p), cs = 2 * (int64_t)(H + 1);
  k_fit_mask<true><<<g2, 256, 0, p->stream>>>(goodw, H, W, p->w, mfitw, cnt, cs);
  k_edge_scan<<<dim3(B, 2), 1024, 0, p->stream>>>(cnt, cs, H);
  k_edge_list<<<dim3((H + 7) / 8, B), 256, 0, p->stream>>>(mfitw, H, W, cnt, cs, lx, lx + cap, 2 * cap);
  p->nlaunch += 2;
  return cudaGetLastError();
}

// resid == false: BB moments, b_B (from S) and row flags;  resid == true: b_B-part of the
// refinement right-hand side from the residual image (written into vec slot 0 tail).
template <typename T>
static cudaError_t moments_T(const sfft_plan_s* p, const float* S, const void* eimg, bool resid, void* ws) {
  const int H = p->d.H, W = p->d.W, B = p->d.batch;
  const uint8_t* mfit = ws_at<uint8_t>(ws, p->mfit);
  const double* sky = ws_at<double>(ws, p->sky);
  dim3 g((H + kMomRows - 1) / kMomRows, B);
  if (!resid) {
    double* bb = ws_at<double>(ws, p->mom_bb);
    double* bv = ws_at<double>(ws, p->mom_b);
    const int nbb = n_mono(p->DM_BB), nb = n_mono(p->d.DB);
    cudaMemsetAsync(bb, 0, sizeof(double) * nbb * B, p->stream);
    cudaMemsetAsync(bv, 0, sizeof(double) * nb * B, p->stream);
    k_moments<T><<<g, 256, 0, p->stream>>>(mfit, S, sky, (const T*)nullptr, H, W, p->DM_BB, p->d.DB, bb, nbb, bv,
                                           nb, ws_at<int>(ws, p->rowflag), p->rf_stride);
  } else {
    double* bv = ws_at<double>(ws, p->mom_b);
    const int nb = n_mono(p->d.DB);
    cudaMemsetAsync(bv, 0, sizeof(double) * nb * B, p->stream);
    k_moments<T><<<g, 256, 0, p->stream>>>(mfit, nullptr, sky, (const T*)eimg, H, W, 0, p->d.DB, nullptr, 0, bv,
                                           nb, nullptr, 0);
  }
  p->nlaunch += 1;
  return cudaGetLastError();
}

cudaError_t launch_moments(const sfft_plan_s* p, const float* S, const void* eimg, bool resid, void* ws) {
  return p->fp64 ? moments_T<double>(p, S, eimg, resid, ws) : moments_T<float>(p, S, eimg, resid, ws);
}

}  // namespace sfft
