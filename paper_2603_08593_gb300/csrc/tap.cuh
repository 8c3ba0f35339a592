// Device pieces of the image-space sums shared by kernels_tap.cu and
// kernels_apply.cu: packed multiply-adds, asynchronous copies and the tap-sum
// tasks of one warp.
#pragma once
#include "common.cuh"

namespace sfft {

// ------------------------------------------------------------------ packed pairs
template <typename T> struct v2 { T x, y; };
template <> struct v2<float> { float2 p; };

__device__ __forceinline__ void v2_zero(v2<float>& a) { a.p = make_float2(0.f, 0.f); }
__device__ __forceinline__ void v2_zero(v2<double>& a) { a.x = 0.0; a.y = 0.0; }
// acc += (q0, q1) r
__device__ __forceinline__ void v2_fma(v2<float>& a, float q0, float q1, float r) {
  a.p = __ffma2_rn(make_float2(q0, q1), make_float2(r, r), a.p);
}
__device__ __forceinline__ void v2_fma(v2<double>& a, double q0, double q1, double r) {
  a.x = fma(q0, r, a.x);
  a.y = fma(q1, r, a.y);
}
// acc += c w, element by element; pairs, and a value twice
__device__ __forceinline__ void v2_fmav(v2<float>& a, const v2<float>& c, const v2<float>& w) {
  a.p = __ffma2_rn(c.p, w.p, a.p);
}
__device__ __forceinline__ void v2_fmav(v2<double>& a, const v2<double>& c, const v2<double>& w) {
  a.x = fma(c.x, w.x, a.x);
  a.y = fma(c.y, w.y, a.y);
}
__device__ __forceinline__ v2<float> v2_make(float x, float y) { v2<float> r; r.p = make_float2(x, y); return r; }
__device__ __forceinline__ v2<double> v2_make(double x, double y) { v2<double> r; r.x = x; r.y = y; return r; }
// (p[0], p[0]): FP32 values are stored twice and loaded as a pair
__device__ __forceinline__ v2<float> v2_dup(const float* p) {
  v2<float> r;
  r.p = *reinterpret_cast<const float2*>(p);
  return r;
}
__device__ __forceinline__ v2<double> v2_dup(const double* p) { return v2_make(*p, *p); }
// the dups of two neighbouring values, 16-byte aligned
__device__ __forceinline__ void v2_dup2(const float* p, v2<float>& a, v2<float>& b) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  a.p = make_float2(q.x, q.y);
  b.p = make_float2(q.z, q.w);
}
__device__ __forceinline__ void v2_dup2(const double* p, v2<double>& a, v2<double>& b) {
  const double2 q = *reinterpret_cast<const double2*>(p);
  a = v2_make(q.x, q.x);
  b = v2_make(q.y, q.y);
}
// (p[0], p[1]) of an even element of an aligned row
__device__ __forceinline__ v2<float> v2_load(const float* p) {
  v2<float> r;
  r.p = *reinterpret_cast<const float2*>(p);
  return r;
}
__device__ __forceinline__ v2<double> v2_load(const double* p) {
  const double2 q = *reinterpret_cast<const double2*>(p);
  return v2_make(q.x, q.y);
}
__device__ __forceinline__ void st_dup(float* p, float v) { *reinterpret_cast<float2*>(p) = make_float2(v, v); }
__device__ __forceinline__ void st_dup(double* p, double v) { *p = v; }
__device__ __forceinline__ float v2_get(const v2<float>& a, int i) { return i ? a.p.y : a.p.x; }
__device__ __forceinline__ double v2_get(const v2<double>& a, int i) { return i ? a.y : a.x; }

__device__ __forceinline__ void ld4(const float* p, float (&v)[4]) {
  const float4 q = *reinterpret_cast<const float4*>(p);
  v[0] = q.x; v[1] = q.y; v[2] = q.z; v[3] = q.w;
}
__device__ __forceinline__ void ld4(const double* p, double (&v)[4]) {
  const double2 a = reinterpret_cast<const double2*>(p)[0], b = reinterpret_cast<const double2*>(p)[1];
  v[0] = a.x; v[1] = a.y; v[2] = b.x; v[3] = b.y;
}

template <int BYTES>
__device__ __forceinline__ void cp_async(void* dst, const void* src, bool valid) {
  const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(d), "l"(src), "n"(BYTES), "r"(valid ? BYTES : 0)
               : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ------------------------------------------------------------------ tap sums
// A task is one row u'_y of taps against one centre image c: a warp's lanes
// are the tile's 32 rows, each lane walks its row with the NT taps in a
// sliding register window and keeps (rows of powers) x (taps) sums in
// registers, so a shared-memory value read once feeds 2 x NT multiply-adds
// per row of powers.  What bounds it is the FP32 FMA pipe (55 multiply-adds per
// pixel, centre and tap row at D_K = 2, packed in pairs); lanes as rows need no
// reduction until the row's end, and the odd pitch keeps their reads free of
// bank conflicts.
enum { TAP_CS = 0, TAP_C = 1, TAP_S = 2, TAP_M = 3, TAP_MOM = 4 };
enum { TAP_FIT_EDGE = 0, TAP_FIT_ALL = 1 };

constexpr int kTapRows = 32;
constexpr int kTapWarps = 4;
constexpr int kTapU = 8;          // pixels per unrolled step
constexpr int kTapScr = 16;       // staged rows of the y fold per warp
constexpr int kTapScrPitch = 36;
constexpr int kTapMaxOut = 40;
constexpr int kTapMomS = 15, kTapMomC = 21, kTapMom = 36;   // moments: of M, of s from kTapMomS, of c from kTapMomC

// outputs of each task type: (row of powers, power of yt), in monomial order
__device__ __forceinline__ void tap_outputs(int type, int DK, unsigned char (*ot)[2]) {
  const int RC = 2 * DK + 1;
  int n = 0;
  auto put = [&](int deg, int row0) {
    for (int g = 0; g <= deg; ++g)
      for (int b = 0; b <= g; ++b, ++n) { ot[n][0] = (unsigned char)(row0 + g - b); ot[n][1] = (unsigned char)b; }
  };
  if (type == TAP_CS) { put(2 * DK, 0); put(DK, RC); }
  if (type == TAP_C) put(2 * DK, 0);
  if (type == TAP_S) put(DK, 0);
  if (type == TAP_M) put(DK + 2, 0);
  if (type == TAP_MOM) { put(4, 0); put(2, 5); put(4, 8); }
}

template <typename T>
struct TapTile {
  // this lane's run of pixels
  const T* r;              // R, wt rows above and wt columns left of the run's first pixel
  const T* s;              // M S' or the residual
  const unsigned* m;       // mask bits
  const T* xp;             // [n][4] xt .. xt^4
  int pitch, n;            // of r; n: pixels to walk (a multiple of kTapU)
  const T* yp;             // [5][kTapScrPitch] yt^b of the 32 lanes' rows
  T* scr;                  // this warp's [kTapScr][kTapScrPitch]
  const unsigned char (*ot)[2];   // this type's outputs: (row of powers, b)
};

// A value of the sliding window: R kept once per pixel, or twice (FP32) as
// the operand pair of the packed multiply-adds
template <typename T, int DUP>
struct TapWin {
  T v;
  __device__ __forceinline__ void load(const T* p) { v = *p; }
  __device__ __forceinline__ void fma2(v2<T>& a, T q0, T q1) const { v2_fma(a, q0, q1, v); }
  __device__ __forceinline__ T get() const { return v; }
};
template <typename T>
struct TapWin<T, 2> {
  v2<T> v;
  __device__ __forceinline__ void load(const T* p) { v = v2_dup(p); }
  __device__ __forceinline__ void fma2(v2<T>& a, T q0, T q1) const { v2_fmav(a, v2_make(q0, q1), v); }
  __device__ __forceinline__ T get() const { return v2_get(v, 0); }
};

// sum over the 32 staged values of row `row` times yt^b
template <typename T>
__device__ __forceinline__ T fold_row(const TapTile<T>& t, int row, int b) {
  const T* v = t.scr + row * kTapScrPitch;
  const T* y = t.yp + b * kTapScrPitch;
  T s[4] = {0, 0, 0, 0};
#pragma unroll
  for (int i = 0; i < 32; i += 4) {
    T a[4], c[4];
    ld4(v + i, a);
    ld4(y + i, c);
#pragma unroll
    for (int k = 0; k < 4; ++k) s[k] += a[k] * c[k];
  }
  return (s[0] + s[1]) + (s[2] + s[3]);
}

// RC rows of powers of the centre c (MB: the mask itself), RS rows of s, against
// the first K of the NT taps.  Rows go in packed pairs (two cycles of the FMA
// pipe), an odd last row alone (one cycle).  DUP: copies of each value of R.
template <typename T, int NT, int K, int RC, int RS, bool MB, int DUP>
__device__ __forceinline__ void tap_task(const TapTile<T>& t, int u0x, int u0y, int uy, int nout, T* __restrict__ out) {
  constexpr int NR = RC + RS, NP = NR / 2, ODD = NR & 1, wt = (NT - 1) / 2;
  const int lane = threadIdx.x & 31;
  const T* rr = t.r + DUP * ((wt - uy) * t.pitch);
  const T* cr = t.r + DUP * ((wt - u0y) * t.pitch + (wt - u0x));
  const T* sr = t.s;
  const unsigned* mr = t.m;
  v2<T> acc[K][NP > 0 ? NP : 1];
  T last[K];
#pragma unroll
  for (int k = 0; k < K; ++k) {
    last[k] = 0;
#pragma unroll
    for (int p = 0; p < NP; ++p) v2_zero(acc[k][p]);
  }
  TapWin<T, DUP> win[K - 1 + kTapU];
#pragma unroll
  for (int k = 0; k < K - 1; ++k) win[k].load(rr + DUP * k);
  for (int xb = 0; xb < t.n; xb += kTapU) {
#pragma unroll
    for (int i = 0; i < kTapU; ++i) win[K - 1 + i].load(rr + DUP * (xb + K - 1 + i));
    const unsigned bits = RC > 0 ? mr[xb >> 5] >> (xb & 31) : 0u;
#pragma unroll
    for (int i = 0; i < kTapU; ++i) {
      T q[NR];
      T xp[4];
      if (RC > 1 || RS > 1) ld4(t.xp + 4 * (xb + i), xp);
      if constexpr (RC > 0) {
        const bool on = (bits >> i) & 1u;
        const T c = MB ? (on ? (T)1 : (T)0) : (on ? cr[DUP * (xb + i)] : (T)0);
        q[0] = c;
#pragma unroll
        for (int a = 1; a < RC; ++a) q[a] = c * xp[a - 1];
      }
      if constexpr (RS > 0) {
        const T s = sr[xb + i];
        q[RC] = s;
#pragma unroll
        for (int a = 1; a < RS; ++a) q[RC + a] = s * xp[a - 1];
      }
#pragma unroll
      for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int p = 0; p < NP; ++p) win[i + k].fma2(acc[k][p], q[2 * p], q[2 * p + 1]);
        if (ODD) last[k] = fma(q[NR - 1], win[i + k].get(), last[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < K - 1; ++k) win[k] = win[k + kTapU];
  }
  // yt^b over the tile's rows, KT taps at a time
  constexpr int KT = kTapScr / NR;
#pragma unroll
  for (int k0 = 0; k0 < K; k0 += KT) {
    __syncwarp();
#pragma unroll
    for (int k = 0; k < KT; ++k)
#pragma unroll
      for (int a = 0; a < NR; ++a)
        if (k0 + k < K) {
          const int kk = k0 + k < K ? k0 + k : 0;
          t.scr[(k * NR + a) * kTapScrPitch + lane] = a < 2 * NP ? v2_get(acc[kk][a < 2 * NP ? a / 2 : 0], a & 1) : last[kk];
        }
    __syncwarp();
    const int nk = K - k0 < KT ? K - k0 : KT;
    for (int o = lane; o < nk * nout; o += 32) {
      const int k = o / nout, j = o % nout;
      out[(k0 + k) * nout + j] = fold_row(t, k * NR + t.ot[j][0], t.ot[j][1]);
    }
  }
}

// Moments without taps (FIT; else those of s alone): M xt^a (a <= 4), s xt^a (a <= 2), c xt^a (a <= 4),
// c = M R(. - (w, w)).  The background block of A, b_B and the corner of the kernel-background block come from
// these alone, so only a row's sums over the run are in T, in groups of kTapU; yt^b and the sums over rows are
// FP64 (ypd: [5][32]; with FP32 powers and sums over the rows A's block was off by 1.2e-7, now by 2e-8).
template <typename T, bool FIT>
__device__ __forceinline__ void tap_moments(const TapTile<T>& t, int wt, int w, const double (*ypd)[32], char3 need,
                                            double* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const T* cr = t.r + (wt - w) * t.pitch + (wt - w);
  const T* sr = t.s;
  const unsigned* mr = t.m;
  T acc[13];
#pragma unroll
  for (int a = 0; a < 13; ++a) acc[a] = 0;
  for (int x0 = 0; x0 < t.n; x0 += kTapU) {
    T g[13];
#pragma unroll
    for (int a = 0; a < 13; ++a) g[a] = 0;
#pragma unroll
    for (int x = x0; x < x0 + kTapU; ++x) {
      const bool on = FIT && ((mr[x >> 5] >> (x & 31)) & 1u);
      const T m = on ? (T)1 : (T)0, c = on ? cr[x] : (T)0, s = sr[x];
      const T* xp = t.xp + 4 * x;
      g[5] += s;
      g[6] += s * xp[0];
      g[7] += s * xp[1];
      if (FIT) {
        g[0] += m;
        g[8] += c;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
          g[1 + a] += m * xp[a];
          g[9 + a] += c * xp[a];
        }
      }
    }
#pragma unroll
    for (int a = 0; a < 13; ++a) acc[a] += g[a];
  }
  __syncwarp();
#pragma unroll
  for (int a = 0; a < 13; ++a) t.scr[a * kTapScrPitch + lane] = acc[a];
  __syncwarp();
  // the first need.x outputs of M, need.y of s and need.z of c; a quarter of the rows per lane: an FP64
  // instruction occupies its pipe for 16 cycles whatever its lanes do
  const int n = need.x + need.y + need.z;
#pragma unroll 1
  for (int k0 = 0; k0 < 4 * n; k0 += 32) {
    int o = min((k0 + lane) / 4, n - 1);
    const int r0 = 8 * (lane & 3);
    o = o < need.x ? o : (o - need.x < need.y ? o - need.x + kTapMomS : o - need.x - need.y + kTapMomC);
    const T* v = t.scr + t.ot[o][0] * kTapScrPitch + r0;
    const double* y = ypd[t.ot[o][1]] + r0;
    double s = 0.0;
#pragma unroll
    for (int i = 0; i < 8; ++i) s = fma((double)v[i], y[i], s);
    s += __shfl_xor_sync(0xffffffffu, s, 1);
    s += __shfl_xor_sync(0xffffffffu, s, 2);
    if ((lane & 3) == 0) out[o] = s;
  }
}

}  // namespace sfft
