// Spatially varying convolution and subtraction, and the refinement residual.
//
//   model(x) = sum_p phi_p(x) sum_j theta[j, p] R~(x - u_j) + B'(x),
//   R~ = finite(R) ? R - s_R : 0, zero outside the image;
//   D(x) = S(x) - s_S - model(x)                       (apply)
//   e(x) = M_fit(x) ? S(x) - s_S - model(x) : 0        (refinement residual)
//
// Along a row the kernel is a polynomial in xt alone,
//   sum_p theta[j, p] phi_p = sum_a xt^a c_{j,a}(y),  c_{j,a}(y) = sum_b theta[j, (a, b)] yt^b,
// so a tile forms its rows' D_K + 1 coefficients per tap once and a pixel takes
// (D_K + 1) L^2 multiply-adds instead of N_K L^2 (363 against 726 at L = 11,
// D_K = 2).  A CTA covers 16 rows x 2 half tiles of up to 128 columns: a warp's
// lanes are the rows of both halves, each with 16 neighbouring pixels, whose
// D_K + 1 sums stay in registers while the taps of one u_y slide over a
// register window.  A tap's coefficients are read once for 16 pixels.  R is kept
// in shared memory twice per pixel (FP32), as the operand pair of the packed
// multiply-adds: duplicating it in registers at each use took a quarter of the
// issued instructions.  The sums start from -S' and take the taps from the
// centre outwards, with the polynomials about the tile's centre, so that at a
// bright star the partial sums shrink with the first taps instead of carrying
// the star's full value through all 121: the refinement's theta came out three
// times nearer to the 64-bit fit.  Odd row pitches keep the reads free of bank conflicts.
// What bounds it is the FMA pipe and the issue slots (50 % each, two CTAs per
// SM): 4096 x 2048, L = 11, D_K = 2 takes 170 us per pass, 0.48 of the FP32 FMA
// peak (all N_K L^2 products per pixel: 310 us); 330 us with the sums below.
//
// The refinement needs e only for its sums against R(x - u'): in the
// image-space assembly the CTA keeps e in shared memory and runs the tap-sum
// tasks of the right-hand side on it (tap.cuh) with the R tile that it already
// holds, so the residual image is neither written nor read.
#include <algorithm>

#include "common.cuh"
#include "plan.h"
#include "tap.cuh"

namespace sfft {

constexpr int kCvRows = 16;
constexpr int kCvPx = 16;       // pixels per lane
constexpr int kCvWarps = 8;
enum { CV_D = 0, CV_E = 1, CV_SUMS = 2 };

constexpr int kCvHalo = 8;      // staged columns on each side (w <= 5, in whole groups of four)
// stored copies of a pixel of R
template <typename T> constexpr int kCvDup = sizeof(T) == 4 ? 2 : 1;
__host__ __device__ constexpr int cv_pitch(int hw) { return hw + 2 * kCvHalo + 1; }   // pixels, odd
__host__ __device__ constexpr int cv_half(int wt, int hw) { return (kCvRows + 2 * wt) * cv_pitch(hw); }
__host__ __device__ constexpr int cv_shalf(int hw) { return (kCvRows * (hw | 1) + 15) / 32 * 32 + 16; }

// scratch of the right-hand side's tasks: x powers, y powers and the warps' fold rows
template <typename T>
__host__ __device__ constexpr size_t cv_rhs_words(int hw) {
  return 4 * 2 * (size_t)hw + 5 * kTapScrPitch + (size_t)kCvWarps * kTapScr * kTapScrPitch;
}

// words of the rows' coefficients; the right-hand side's tasks use the space again
template <typename T>
__host__ __device__ constexpr size_t cv_coef_words(int nt, int na, int hw, int mode) {
  size_t n = (size_t)(nt * nt * na + 3) * kCvRows;
  if (mode == CV_SUMS && cv_rhs_words<T>(hw) > n) n = cv_rhs_words<T>(hw);
  return (n + 3) / 4 * 4;
}
template <typename T>
__host__ __device__ constexpr size_t cv_smem(int nt, int na, int hw, int mode) {
  const int wt = (nt - 1) / 2;
  return sizeof(T) * (cv_coef_words<T>(nt, na, hw, mode) + 2 * (size_t)hw + nt * nt * na * (na + 1) / 2 + 6 +
                      1 + kCvDup<T> * 2 * (size_t)cv_half(wt, hw) + 2 * (size_t)cv_shalf(hw)) +
         4 * (size_t)kCvRows * 2 * ((hw + 31) / 32);
}

template <typename T>
struct ConvArgs {
  const float *R, *S;
  const T* Rm;
  const double *theta, *sky;
  const uint8_t* mfit;      // CV_E: M_fit as bytes
  const unsigned* mfitw;    // CV_SUMS: M_fit as bits
  float* D;
  T* E;
  const int4* tasks;
  T* part;
  double* mpart;
  char3 need;              // moments taken
  int ntask, nout_tot;
  int H, W, L, DB, hw;
  double xsc, ysc;         // 2 / (W - 1), 2 / (H - 1): an FP64 division per thread cost a tenth of the kernel
  int vec;                 // rows start on 16-byte boundaries: groups of four pixels
  unsigned magic;          // ceil(2^20 / groups per staged row)
};

// Two CTAs per SM; FP64 only where window and sums fit 128 registers (L = 7,
// D_K = 1, one 512 x 512 pair: 64.8 us, 121.5 us at one CTA) or miss them by a few
// spilled values (L = 3, D_K = 2: 44 bytes, 102 us per 1024 x 1024 against 105 at one
// CTA; the residual image at L = 11, D_K = 0: 16 bytes)
template <typename T, int NT, int DK, int MODE>
__global__ void __launch_bounds__(kCvWarps * 32, sizeof(T) == 4 || NT * (DK + 1) <= 14 ? 2 : 1)
k_conv(const ConvArgs<T> a) {
  constexpr int wt = (NT - 1) / 2, NA = DK + 1, NK = n_mono(DK);
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ unsigned char ot[2][kTapMaxOut][2];
  __shared__ double ypd[MODE == CV_SUMS ? 5 : 1][32];
  __shared__ int next;
  const int H = a.H, W = a.W, hw = a.hw, L = a.L, w = (L - 1) / 2;
  constexpr int CD = kCvDup<T>;
  const int pitch = cv_pitch(hw), HB = cv_half(wt, hw), sp = hw | 1, SB = cv_shalf(hw), nw = (hw + 31) / 32;
  T* coef = reinterpret_cast<T*>(smraw);            // [NT^2][NA][16], then the background's [3][16]
  T* beta = coef + NT * NT * NA * kCvRows;
  T* rt = coef + cv_coef_words<T>(NT, NA, hw, MODE);   // [half][16 + 2 wt][pitch][copies], column 0 = x0 - 8
  T* xt1 = rt + CD * 2 * HB;                           // [2 hw]
  T* tht = xt1 + 2 * hw;                               // theta in T, a box of NT x NT offsets
  T* st = tht + NT * NT * NK + 6;
  unsigned* mw = reinterpret_cast<unsigned*>(st + 2 * SB);   // [half][16][nw]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ntx = (W + 2 * hw - 1) / (2 * hw);
  const int tile = blockIdx.x, ccd = blockIdx.z;
  const int x0 = (tile % ntx) * 2 * hw, y0 = (tile / ntx) * kCvRows;
  const int64_t img = (int64_t)ccd * H * W;
  const T sR = (T)a.sky[2 * ccd], sS = (T)a.sky[2 * ccd + 1];
  // theta and the columns' xt, converted once per CTA (FP64 arithmetic and
  // conversions run at 1/64 of the FP32 rate)
  const double ysc = a.ysc, xsc = a.xsc;
  const int row = lane & 15, half = lane >> 4, NB = n_mono(a.DB);
  {
    const double* th = a.theta + (int64_t)ccd * (L * L * NK + NB);
#pragma unroll 3
    for (int i = tid; i < NT * NT * NK; i += kCvWarps * 32) {
      if (L == NT) {
        tht[i] = (T)th[i];
      } else {   // L = 1 in the box of three
        const int j = i / NK, jy = j / NT - wt + w, jx = j % NT - wt + w;
        tht[i] = jy >= 0 && jy < L && jx >= 0 && jx < L ? (T)th[(jy * L + jx) * NK + i % NK] : (T)0;
      }
    }
    if (tid < NB) tht[NT * NT * NK + tid] = (T)th[L * L * NK + tid];
    for (int i = tid; i < 2 * hw; i += kCvWarps * 32) xt1[i] = (T)((x0 + i) * xsc - 1.0);
  }
  // the mask's words (hw < 32: the low bits of one)
  if constexpr (MODE == CV_SUMS) {
    const int wpr = (W + 31) / 32;
    for (int i = tid; i < 2 * kCvRows * nw; i += kCvWarps * 32) {
      const int r = i / nw, gy = y0 + r % kCvRows, gx = x0 + r / kCvRows * hw + 32 * (i % nw);
      mw[i] = gy < H && gx < W ? a.mfitw[((int64_t)ccd * H + gy) * wpr + (gx >> 5)] >> (gx & 31) : 0u;
    }
  } else if constexpr (MODE == CV_E) {
    for (int r = warp; r < 2 * kCvRows; r += kCvWarps) {
      const int gy = y0 + r % kCvRows, gx0 = x0 + r / kCvRows * hw;
      for (int k = 0; k < nw; ++k) {
        const int cc = 32 * k + lane;
        const bool on = cc < hw && gy < H && gx0 + cc < W && a.mfit[img + (int64_t)gy * W + gx0 + cc] != 0;
        const unsigned word = __ballot_sync(0xffffffffu, on);
        if (lane == 0) mw[r * nw + k] = word;
      }
    }
  }
  // R - s_R at finite pixels (R_m: as it is), zero elsewhere and outside the
  // image, and S - s_S: four pixels of a row at a time, every group of the CTA
  // in flight before the first is stored (one memory round trip per CTA)
  {
    const int ng = (hw + 2 * kCvHalo) / 4, total = 2 * (kCvRows + 2 * wt) * ng;
    auto put = [&](int i, const T (&v)[4]) {
      const int r = (int)(((unsigned)i * a.magic) >> 20), g = i - r * ng;
      T* dst = rt + CD * (r * pitch + 4 * g);          // rows of both halves follow each other
#pragma unroll
      for (int k = 0; k < 4; ++k) st_dup(dst + CD * k, MODE == CV_SUMS ? v[k] : (isfinite(v[k]) ? v[k] - sR : (T)0));
    };
    auto get = [&](int i, T (&v)[4]) {
      const int r = (int)(((unsigned)i * a.magic) >> 20), g = i - r * ng;
      const int half = r >= kCvRows + 2 * wt, row = r - half * (kCvRows + 2 * wt);
      const int gy = y0 - wt + row, gx = x0 + half * hw - kCvHalo + 4 * g;
      const bool in = gy >= 0 && gy < H;
      const int64_t o = img + (int64_t)gy * W + gx;
      bool ok[4];
      if (a.vec) {
        const bool all = in && gx >= 0 && gx < W;
#pragma unroll
        for (int k = 0; k < 4; ++k) ok[k] = all;
        if constexpr (MODE == CV_SUMS) {
          if (all) ld4(a.Rm + o, v);
        } else {
          float f[4] = {0.f, 0.f, 0.f, 0.f};
          if (all) ld4(a.R + o, f);
#pragma unroll
          for (int k = 0; k < 4; ++k) v[k] = (T)f[k];
        }
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          ok[k] = in && gx + k >= 0 && gx + k < W;
          if constexpr (MODE == CV_SUMS) v[k] = ok[k] ? a.Rm[o + k] : (T)0;
          else v[k] = (T)(ok[k] ? a.R[o + k] : 0.f);
        }
      }
      // outside the image: not finite, so that put() stores zero
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (!ok[k]) v[k] = MODE == CV_SUMS ? (T)0 : (T)INFINITY;
    };
    constexpr int NTH = kCvWarps * 32, NRV = (2 * (kCvRows + 2 * wt) * (128 + 2 * kCvHalo) / 4 + NTH - 1) / NTH;
    constexpr int NSV = 2 * kCvRows * 128 / 4 / NTH;
    const int sg = hw / 4, lg = 31 - __clz(sg), stotal = 2 * kCvRows * sg;   // a power of two
    T rv[NRV][4];
    float sv[NSV][4];
#pragma unroll
    for (int k = 0; k < NRV; ++k)
      if (tid + k * NTH < total) get(tid + k * NTH, rv[k]);
#pragma unroll
    for (int k = 0; k < NSV; ++k) {
      const int i = tid + k * NTH, r = i >> lg, g = i & (sg - 1);
      const int gy = y0 + r % kCvRows, gx = x0 + r / kCvRows * hw + 4 * g;
      const int64_t o = img + (int64_t)gy * W + gx;
#pragma unroll
      for (int q = 0; q < 4; ++q) sv[k][q] = 0.f;
      if (i < stotal && gy < H) {
        if (a.vec) {
          if (gx < W) ld4(a.S + o, sv[k]);
        } else {
#pragma unroll
          for (int q = 0; q < 4; ++q)
            if (gx + q < W) sv[k][q] = a.S[o + q];
        }
      }
    }
#pragma unroll
    for (int k = 0; k < NRV; ++k)
      if (tid + k * NTH < total) put(tid + k * NTH, rv[k]);
#pragma unroll
    for (int k = 0; k < NSV; ++k) {
      const int i = tid + k * NTH, r = i >> lg, g = i & (sg - 1);
      if (i < stotal) {
        T* dst = st + r / kCvRows * SB + r % kCvRows * sp + 4 * g;
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[q] = (T)sv[k][q] - sS;
      }
    }
  }
  __syncthreads();
  // the rows' coefficients: a half warp per tap, lane = row
  {
    const T yt = (T)((y0 + row) * ysc - 1.0), xc = xt1[hw];
#pragma unroll 2
    for (int i = 2 * warp + half; i < NT * NT; i += 2 * kCvWarps) {
      const int iy = i / NT;                                   // table: u_y ascending, u_x descending
      const T* q = tht + (2 * iy * NT + NT - 1 - i) * NK;      // (iy NT + NT - 1 - (i - iy NT)) N_K
      // about (xc, y): the value at the tile's centre is theta_0 plus small terms
      T* o = coef + i * NA * kCvRows + row;
      if constexpr (DK == 0) {
        o[0] = q[0];
      } else if constexpr (DK == 1) {
        o[0] = q[0] + (xc * q[1] + yt * q[2]);
        o[kCvRows] = q[1];
      } else {
        o[0] = q[0] + (xc * (q[1] + xc * q[3] + yt * q[4]) + yt * (q[2] + yt * q[5]));
        o[kCvRows] = q[1] + ((T)2 * xc * q[3] + yt * q[4]);
        o[2 * kCvRows] = q[3];
      }
    }
    if (warp == 0) {
      const T* q = tht + NT * NT * NK;
      for (int ap = half; ap < 3; ap += 2) {
        T c = 0;
        for (int b = a.DB; b >= 0; --b)
          if (ap + b <= a.DB) c = c * yt + q[mono_index(ap, b)];
        beta[ap * kCvRows + row] = c;
      }
    }
  }
  if (MODE == CV_SUMS && tid < 2) tap_outputs(tid == 0 ? TAP_S : TAP_MOM, DK, ot[tid]);
  if (tid == 0) next = 0;
  __syncthreads();
  for (int sg = warp; sg < hw / kCvPx; sg += kCvWarps) {
    const int xl = sg * kCvPx;
    // sums over the taps of each power: the first two packed, the third alone
    v2<T> acc[kCvPx];
    T last[kCvPx];
#pragma unroll
    for (int i = 0; i < kCvPx; ++i) {
      const T s0 = -st[half * SB + row * sp + xl + i];
      acc[i] = v2_make(s0, (T)0);
      last[i] = NA == 1 ? s0 : (T)0;
    }
    const T* base = rt + CD * (half * HB + row * pitch + xl + kCvHalo - wt);
#pragma unroll 1
    for (int r = 0; r < NT; ++r) {
      const int uy = (r & 1) ? -(r + 1) / 2 : r / 2;   // 0, -1, 1, -2, ...
      v2<T> win[NT - 1 + kCvPx];
      const T* p = base + CD * (wt - uy) * pitch;
#pragma unroll
      for (int i = 0; i < NT - 1 + kCvPx; ++i) win[i] = v2_dup(p + CD * i);
      const T* cp = coef + (uy + wt) * NT * NA * kCvRows + row;
#pragma unroll
      for (int kk = 0; kk < NT; ++kk) {
        const int k = wt + ((kk & 1) ? -(kk + 1) / 2 : kk / 2);
        T c[NA];
#pragma unroll
        for (int q = 0; q < NA; ++q) c[q] = cp[(k * NA + q) * kCvRows];
        const v2<T> c01 = v2_make(c[0], c[NA > 1 ? 1 : 0]);
#pragma unroll
        for (int i = 0; i < kCvPx; ++i) {
          if (NA > 1) v2_fmav(acc[i], c01, win[i + k]);
          if (NA != 2) last[i] = fma(c[NA - 1], v2_get(win[i + k], 0), last[i]);
        }
      }
    }
    T* so = st + half * SB + row * sp + xl;
    unsigned bits = 0;
    if (MODE != CV_D) bits = mw[(half * kCvRows + row) * nw + (xl >> 5)] >> (xl & 31);
    const T b0 = beta[row], b1 = beta[kCvRows + row], b2 = beta[2 * kCvRows + row], xc = xt1[hw];
#pragma unroll
    for (int i = 0; i < kCvPx; ++i) {
      const T xt = xt1[half * hw + xl + i], dx = xt - xc;
      T m = NA > 1 ? v2_get(acc[i], 0) : last[i];                    // model - S' at the tile's centre ...
      if (NA > 1) m += dx * (v2_get(acc[i], 1) + (NA > 2 ? dx * last[i] : (T)0));   // ... and here
      const T d = -(m + (b0 + xt * (b1 + xt * b2)));
      so[i] = MODE == CV_D ? d : (((bits >> i) & 1u) ? d : (T)0);
    }
  }
  __syncthreads();
  if constexpr (MODE != CV_SUMS) {
    const int ng = hw / 4, lg = 31 - __clz(ng);
#pragma unroll 2
    for (int i = tid; i < 2 * kCvRows * ng; i += kCvWarps * 32) {
      const int r = i >> lg, g = i & (ng - 1), h = r / kCvRows, rr = r % kCvRows;
      const int gy = y0 + rr, gx = x0 + h * hw + 4 * g;
      if (gy >= H || gx >= W) continue;
      const T* src = st + h * SB + rr * sp + 4 * g;
      const int64_t o = img + (int64_t)gy * W + gx;
      if (MODE == CV_D && a.vec) {
        *reinterpret_cast<float4*>(a.D + o) =
            make_float4((float)src[0], (float)src[1], (float)src[2], (float)src[3]);
      } else {
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (gx + k >= W) break;
          if constexpr (MODE == CV_D) a.D[o + k] = (float)src[k];
          else a.E[o + k] = src[k];
        }
      }
    }
  } else {
    // the right-hand side's sums of e, in the coefficients' space
    T* xp = coef;                          // [2 hw][4]
    T* yp = xp + 8 * hw;
    T* scr = yp + 5 * kTapScrPitch;
    for (int i = tid; i < 2 * hw; i += kCvWarps * 32) {
      const T x = xt1[i];
      xp[4 * i] = x; xp[4 * i + 1] = x * x; xp[4 * i + 2] = x * x * x; xp[4 * i + 3] = x * x * x * x;
    }
    if (warp == 0) {
      const double y = (y0 + row) * ysc - 1.0;
      double v = 1.0;
      for (int b = 0; b < 5; ++b) { yp[b * kTapScrPitch + lane] = (T)v; ypd[b][lane] = v; v *= y; }
    }
    __syncthreads();
    // a task takes half of the lanes' columns: 22 taps tasks and 2 of moments at
    // L = 11 are three rounds of eight warps (whole runs are one and a half)
    const int hn = hw / 2;
    for (;;) {
      int k = 0;
      if (lane == 0) k = atomicAdd(&next, 1);
      k = __shfl_sync(0xffffffffu, k, 0);
      if (k >= 2 * a.ntask) break;
      const int4 q = a.tasks[k >> 1];
      const int type = q.x & 255, nout = q.x >> 8, c0 = (k & 1) * hn;
      TapTile<T> t;
      t.r = rt + CD * (half * HB + row * pitch + kCvHalo - wt + c0);
      t.s = st + half * SB + row * sp + c0;
      t.m = nullptr;
      t.xp = xp + 4 * (half * hw + c0);
      t.pitch = pitch;
      t.n = hn;
      t.yp = yp;
      t.scr = scr + warp * kTapScr * kTapScrPitch;
      t.ot = ot[type == TAP_S ? 0 : 1];
      const int64_t half_tile = ((int64_t)ccd * gridDim.x + tile) * 2 + (k & 1);
      if (type == TAP_S) tap_task<T, NT, NT, 0, NA, false, CD>(t, 0, 0, q.z, nout, a.part + half_tile * a.nout_tot + q.w);
      else tap_moments<T, false>(t, wt, w, ypd, a.need, a.mpart + half_tile * kTapMom);
    }
  }
}

// half-tile width: 128 columns amortise the halo and the rows' coefficients; a
// small image takes narrower tiles until every SM has one
int conv_half_width(int H, int W, int batch) {
  int hw = 128;
  while (hw > kCvPx && (int64_t)conv_tiles(H, W, hw) * batch < 152) hw /= 2;
  return hw;
}
int conv_tiles(int H, int W, int hw) { return ((W + 2 * hw - 1) / (2 * hw)) * ((H + kCvRows - 1) / kCvRows); }

template <typename T, int NT, int DK, int MODE>
static cudaError_t conv_run(cudaStream_t s, const ConvArgs<T>& a, int batch) {
  auto kern = k_conv<T, NT, DK, MODE>;
  const size_t smem = cv_smem<T>(NT, DK + 1, a.hw, MODE);
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kern<<<dim3(conv_tiles(a.H, a.W, a.hw), 1, batch), kCvWarps * 32, smem, s>>>(a);
  return cudaGetLastError();
}

template <typename T, int NT, int MODE>
static cudaError_t conv_dk(cudaStream_t s, const ConvArgs<T>& a, int DK, int batch) {
  switch (DK) {
    case 0: return conv_run<T, NT, 0, MODE>(s, a, batch);
    case 1: return conv_run<T, NT, 1, MODE>(s, a, batch);
    case 2: return conv_run<T, NT, 2, MODE>(s, a, batch);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T, int MODE>
static cudaError_t conv(cudaStream_t s, ConvArgs<T> a, int DK, int batch) {
  a.hw = conv_half_width(a.H, a.W, batch);
  const uintptr_t bits = (uintptr_t)a.R | (uintptr_t)a.S | (uintptr_t)a.D | (uintptr_t)a.Rm;
  a.vec = a.W % 4 == 0 && bits % 16 == 0;   // images of a batch are H W pixels apart
  const unsigned ng = (a.hw + 2 * kCvHalo) / 4;
  a.magic = ((1u << 20) + ng - 1) / ng;
  switch (std::max(a.L, 3)) {
    case 3: return conv_dk<T, 3, MODE>(s, a, DK, batch);
    case 5: return conv_dk<T, 5, MODE>(s, a, DK, batch);
    case 7: return conv_dk<T, 7, MODE>(s, a, DK, batch);
    case 9: return conv_dk<T, 9, MODE>(s, a, DK, batch);
    case 11: return conv_dk<T, 11, MODE>(s, a, DK, batch);
    default: return cudaErrorInvalidValue;
  }
}

template <typename T>
static ConvArgs<T> conv_args(const float* R, const float* S, const double* theta_off, const double* sky, int H, int W,
                             int L, int DB) {
  ConvArgs<T> a{};
  a.R = R; a.S = S; a.theta = theta_off; a.sky = sky;
  a.H = H; a.W = W; a.L = L; a.DB = DB;
  a.xsc = 2.0 / (double)(W > 1 ? W - 1 : 1);
  a.ysc = 2.0 / (double)(H > 1 ? H - 1 : 1);
  return a;
}

cudaError_t launch_apply_raw(cudaStream_t s, bool fp64, const float* R, const float* S, const double* theta_off,
                             const double* sky, float* D, int H, int W, int L, int DK, int DB, int batch) {
  if (fp64) {
    ConvArgs<double> a = conv_args<double>(R, S, theta_off, sky, H, W, L, DB);
    a.D = D;
    return conv<double, CV_D>(s, a, DK, batch);
  }
  ConvArgs<float> a = conv_args<float>(R, S, theta_off, sky, H, W, L, DB);
  a.D = D;
  return conv<float, CV_D>(s, a, DK, batch);
}

cudaError_t launch_apply(const sfft_plan_s* p, const float* R, const float* S, const double* theta_off,
                         const double* sky, float* D, void* ws) {
  p->nlaunch += 1;
  return launch_apply_raw(p->stream, p->fp64, R, S, theta_off, sky ? sky : ws_at<double>(ws, p->sky), D, p->d.H,
                          p->d.W, p->d.L, p->d.DK, p->d.DB, p->d.batch);
}

template <typename T>
static cudaError_t residual_image_T(const sfft_plan_s* p, const float* R, const float* S, const double* theta_off,
                                    void* eimg, void* ws) {
  ConvArgs<T> a = conv_args<T>(R, S, theta_off, ws_at<double>(ws, p->sky), p->d.H, p->d.W, p->d.L, p->d.DB);
  a.mfit = ws_at<uint8_t>(ws, p->mfit);
  a.E = (T*)eimg;
  p->nlaunch += 1;
  return conv<T, CV_E>(p->stream, a, p->d.DK, p->d.batch);
}

cudaError_t launch_residual_image(const sfft_plan_s* p, const float* R, const float* S, const double* theta_off,
                                  void* eimg, void* ws) {
  return p->fp64 ? residual_image_T<double>(p, R, S, theta_off, eimg, ws)
                 : residual_image_T<float>(p, R, S, theta_off, eimg, ws);
}

template <typename T>
static cudaError_t residual_sums_T(const sfft_plan_s* p, const float* S, const double* theta_off, void* ws) {
  ConvArgs<T> a = conv_args<T>(nullptr, S, theta_off, ws_at<double>(ws, p->sky), p->d.H, p->d.W, p->d.L, p->d.DB);
  a.Rm = ws_at<T>(ws, p->rm);
  a.mfitw = ws_at<unsigned>(ws, p->mfitw);
  a.tasks = p->tap.d_tasks + p->tap.ntask;
  a.ntask = p->tap.ntask_rhs;
  a.nout_tot = p->tap.nout_rhs;
  a.part = ws_at<T>(ws, p->tappart);
  a.mpart = ws_at<double>(ws, p->mompart);
  a.need = tap_moment_need(p, false);
  p->nlaunch += 1;
  return conv<T, CV_SUMS>(p->stream, a, p->d.DK, p->d.batch);
}

cudaError_t launch_residual_sums(const sfft_plan_s* p, const float* S, const double* theta_off, void* ws) {
  return p->fp64 ? residual_sums_T<double>(p, S, theta_off, ws) : residual_sums_T<float>(p, S, theta_off, ws);
}

}  // namespace sfft
