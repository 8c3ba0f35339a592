// Inference stack of the rotation-invariant classifier (rb_ri.cu): conv1 + pool,
// res1, conv2 + pool in one kernel and res2 + pool in another, a persistent CTA
// per SM.  The weights stay in shared memory for the whole launch and an image's
// activations never leave it: each convolution reads its A fragments with
// ldmatrix from the zero-bordered image at the tap's offset (records of 80 or
// 144 bytes, so that eight neighbouring pixels fall into different banks), so no
// im2col matrix, FP32 pre-activation or separate ReLU, skip and pool pass exists.
// The products are the m16n8k16 steps of rb_gemm.cuh in the same order of k, so
// the logits are the same bit for bit.  Rows of the pooled layers are 2 x 2
// windows (four neighbouring rows), pooled by two shuffles.  1000 stamps (4000
// rotated images, 102 GFLOP): 1.5 ms as seventeen launches of the implicit GEMM
// and elementwise kernels.
#pragma once
#include "rb_layers.cuh"

namespace {

constexpr int RiP1 = 40, RiP2 = 72;              // record pitch (values) of 32 and 64 channels
constexpr int RiImRows = 57 * 16;                // 225 windows x 4, padded to whole tiles
constexpr size_t kRiFrontSmem =
    sizeof(bf16) * (32 * RiP1 + 2 * KA_RI * RiP1 + K2 * RiP2 + RiImRows * RiP1 + 2 * 289 * RiP1 + 3272);
constexpr size_t kRiBackSmem = sizeof(bf16) * (2 * K3 * RiP2 + 4 * 81 * RiP2);

// [rows][n] weights (row stride n) into rows of `pitch`
__device__ __forceinline__ void ri_weights(bf16* dst, int pitch, const bf16* src, int rows, int n) {
  const int v = n / 8;
  for (int e = threadIdx.x; e < rows * v; e += blockDim.x)
    *reinterpret_cast<uint4*>(dst + e / v * pitch + e % v * 8) = *reinterpret_cast<const uint4*>(src + (int64_t)e * 8);
}

// acc += A B over the nine taps of C channels: base[i] is this lane's record (and
// k half) of tile i's A rows in an image of row width RW records, w the weights
// at the warp's 32 columns
template <int C, int RW>
__device__ __forceinline__ void ri_conv(float (&acc)[2][4][4], const bf16* const (&base)[2], bool two, const bf16* w,
                                        int wpitch) {
  constexpr int AP = C == 32 ? RiP1 : RiP2;
  const int lane = threadIdx.x & 31;
  const bf16* wl = w + ((lane & 7) + ((lane >> 3) & 1) * 8) * wpitch + (lane >> 4) * 8;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
#pragma unroll 3
  for (int tap = 0; tap < 9; ++tap) {   // three taps of fragments ahead of their products
    const int off = (tap / 3 * RW + tap % 3) * AP;
#pragma unroll
    for (int h = 0; h < C / 16; ++h) {
      unsigned af[2][4], bf[2][4];
      rbg::ldm_x4(af[0], base[0] + off + 16 * h);
      if (two) rbg::ldm_x4(af[1], base[1] + off + 16 * h);
#pragma unroll
      for (int j = 0; j < 2; ++j) rbg::ldm_x4_t(bf[j], wl + (tap * C + 16 * h) * wpitch + 16 * j);
#pragma unroll
      for (int j = 0; j < 4; ++j) rbg::mma16816(acc[0][j], af[0], bf[j >> 1][(j & 1) * 2], bf[j >> 1][(j & 1) * 2 + 1]);
      if (two)
#pragma unroll
        for (int j = 0; j < 4; ++j) rbg::mma16816(acc[1][j], af[1], bf[j >> 1][(j & 1) * 2], bf[j >> 1][(j & 1) * 2 + 1]);
    }
  }
}

__device__ __forceinline__ void ri_store2(bf16* p, float a, float b) {
  *reinterpret_cast<__nv_bfloat162*>(p) = __floats2bfloat162_rn(a, b);
}
__device__ __forceinline__ float2 ri_load2(const bf16* p) {
  return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(p));
}
// the maximum over a 2 x 2 window: rows 4 q .. 4 q + 3 of a tile sit in lanes 4 apart
__device__ __forceinline__ float ri_pool(float v) {
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
}

// conv1 + pool, res1, conv2 + pool: a2 [image][7][7][64]; image r n + i is the
// r-th quarter turn of stamp i
__global__ void __launch_bounds__(256, 1)
k_ri_front(const bf16* __restrict__ xn, int n, const bf16* __restrict__ W1, const bf16* __restrict__ WA,
           const bf16* __restrict__ WB, const bf16* __restrict__ W2, const float* __restrict__ b1,
           const float* __restrict__ ba, const float* __restrict__ bb, const float* __restrict__ b2,
           bf16* __restrict__ a2) {
  extern __shared__ __align__(16) bf16 ri_smem[];
  bf16* w1 = ri_smem;
  bf16* wa = w1 + 32 * RiP1;
  bf16* wb = wa + KA_RI * RiP1;
  bf16* w2 = wb + KA_RI * RiP1;
  bf16* im = w2 + K2 * RiP2;            // conv1 rows [900][27 + 5]
  bf16* p1 = im + RiImRows * RiP1;      // [17][17] records, zero border
  bf16* ra = p1 + 289 * RiP1;
  bf16* sx = ra + 289 * RiP1;           // the rotated stamp, [33][33][3], zero border
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int lrow = (lane & 7) + ((lane >> 3) & 1) * 8, lk = (lane >> 4) * 8;
  ri_weights(w1, RiP1, W1, 32, 32);
  ri_weights(wa, RiP1, WA, KA_RI, 32);
  ri_weights(wb, RiP1, WB, KA_RI, 32);
  ri_weights(w2, RiP2, W2, K2, 64);
  const uint4 z = rbg::zero4();
  for (int e = tid; e < (RiImRows * RiP1 + 2 * 289 * RiP1 + 3272) / 8; e += 256) reinterpret_cast<uint4*>(im)[e] = z;
  __syncthreads();
  unsigned w1f[2][2][4];
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int j = 0; j < 2; ++j) rbg::ldm_x4_t(w1f[h][j], w1 + (16 * h + lrow) * RiP1 + 16 * j + lk);
  // this lane's records: pixels of conv a and b (tiles 2 warp, 2 warp + 1 of 225 rows)
  int pa[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int p = min((2 * warp + i) * 16 + lrow, PIX2 - 1);
    pa[i] = (p / 15 * 17 + p % 15) * RiP1 + lk;
  }
  float acc[2][4][4];
  constexpr int NS = (3 * PIX1 + 255) / 256;
  bf16 next[NS];   // the next image's values, fetched while this one is convolved
  auto fetch = [&](int img) {
    const bf16* src = xn + (int64_t)(img % n) * 3 * PIX1;
#pragma unroll
    for (int k = 0; k < NS; ++k)
      if (tid + 256 * k < 3 * PIX1) next[k] = src[tid + 256 * k];
  };
  fetch(blockIdx.x);
  for (int img = blockIdx.x; img < NROT_RI * n; img += gridDim.x) {
    const int rot = img / n;
#pragma unroll
    for (int k = 0; k < NS; ++k) {
      const int e = tid + 256 * k;
      if (e >= 3 * PIX1) break;
      const int p = e / 3, sy = p / S31, sxx = p - sy * S31;
      int y = sy, x = sxx;
      if (rot == 1) { y = S31 - 1 - sxx; x = sy; }
      else if (rot == 2) { y = S31 - 1 - sy; x = S31 - 1 - sxx; }
      else if (rot == 3) { y = sxx; x = S31 - 1 - sy; }
      sx[((y + 1) * 33 + x + 1) * 3 + e - 3 * p] = next[k];
    }
    __syncthreads();
    if (img + gridDim.x < NROT_RI * n) fetch(img + gridDim.x);
    for (int m = tid; m < 900; m += 256) {
      const int win = m >> 2, y = 2 * (win / 15) + ((m >> 1) & 1), x = 2 * (win % 15) + (m & 1);
      const unsigned short* s = reinterpret_cast<const unsigned short*>(sx) + (y * 33 + x) * 3;
      unsigned v[28];
#pragma unroll
      for (int k = 0; k < 27; ++k) v[k] = s[k / 9 * 99 + k % 9];
      v[27] = 0;
      unsigned* d = reinterpret_cast<unsigned*>(im + m * RiP1);
#pragma unroll
      for (int k = 0; k < 14; ++k) d[k] = v[2 * k] | v[2 * k + 1] << 16;
    }
    __syncthreads();
    // conv1 + ReLU + pool
    for (int mt = warp; mt < RiImRows / 16; mt += 8) {
#pragma unroll
      for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[0][j][q] = 0.f;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        unsigned af[4];
        rbg::ldm_x4(af, im + (mt * 16 + lrow) * RiP1 + 16 * h + lk);
#pragma unroll
        for (int j = 0; j < 4; ++j) rbg::mma16816(acc[0][j], af, w1f[h][j >> 1][(j & 1) * 2], w1f[h][j >> 1][(j & 1) * 2 + 1]);
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 8 * j + 2 * t;
        const float2 b = *reinterpret_cast<const float2*>(b1 + c);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const float v0 = ri_pool(fmaxf(acc[0][j][2 * q] + b.x, 0.f)), v1 = ri_pool(fmaxf(acc[0][j][2 * q + 1] + b.y, 0.f));
          const int win = mt * 4 + 2 * q + (g >> 2);
          if ((g & 3) == 0 && win < PIX2) ri_store2(p1 + ((win / 15 + 1) * 17 + win % 15 + 1) * RiP1 + c, v0, v1);
        }
      }
    }
    __syncthreads();
    // res1: ra = relu(conv_a(p1)), then p1 = relu(conv_b(ra) + p1)
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      const bf16* in = half == 0 ? p1 : ra;
      const bf16* const base[2] = {in + pa[0], in + pa[1]};
      ri_conv<32, 17>(acc, base, true, half == 0 ? wa : wb, RiP1);
      const float* bias = half == 0 ? ba : bb;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 8 * j + 2 * t;
        const float2 b = *reinterpret_cast<const float2*>(bias + c);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const int p = (2 * warp + i) * 16 + g + 8 * q;
            if (p >= PIX2) continue;
            const int o = ((p / 15 + 1) * 17 + p % 15 + 1) * RiP1 + c;
            float v0 = acc[i][j][2 * q] + b.x, v1 = acc[i][j][2 * q + 1] + b.y;
            if (half == 0) {
              ri_store2(ra + o, fmaxf(v0, 0.f), fmaxf(v1, 0.f));
            } else {
              const float2 s = ri_load2(p1 + o);
              v0 += s.x;
              v1 += s.y;
              ri_store2(p1 + o, fmaxf(v0, 0.f), fmaxf(v1, 0.f));
            }
          }
      }
      __syncthreads();
    }
    // conv2 + ReLU + pool: 13 tiles of window rows in pairs, 32 of the 64 columns per warp
    for (int pr = warp >> 1; pr < 7; pr += 4) {
      const int n0 = (warp & 1) * 32;
      const bf16* base[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const int m = min((2 * pr + i) * 16 + lrow, 4 * PIX3 - 1), win = m >> 2;
        base[i] = p1 + ((2 * (win / 7) + ((m >> 1) & 1)) * 17 + 2 * (win % 7) + (m & 1)) * RiP1 + lk;
      }
      const bf16* const bc[2] = {base[0], base[1]};
      ri_conv<32, 17>(acc, bc, pr < 6, w2 + n0, RiP2);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int c = n0 + 8 * j + 2 * t;
          const float2 b = *reinterpret_cast<const float2*>(b2 + c);
#pragma unroll
          for (int q = 0; q < 2; ++q) {
            const float v0 = ri_pool(fmaxf(acc[i][j][2 * q] + b.x, 0.f)), v1 = ri_pool(fmaxf(acc[i][j][2 * q + 1] + b.y, 0.f));
            const int win = (2 * pr + i) * 4 + 2 * q + (g >> 2);
            if ((g & 3) == 0 && win < PIX3) ri_store2(a2 + ((int64_t)img * PIX3 + win) * C2 + c, v0, v1);
          }
        }
    }
  }
}

// res2 + pool of two images at a time: a3 [image][3][3][64]
__global__ void __launch_bounds__(256, 1)
k_ri_back(const bf16* __restrict__ a2, int nimg, const bf16* __restrict__ WC, const bf16* __restrict__ WD,
          const float* __restrict__ bc, const float* __restrict__ bd, bf16* __restrict__ a3) {
  extern __shared__ __align__(16) bf16 ri_smem[];
  bf16* wc = ri_smem;
  bf16* wd = wc + K3 * RiP2;
  bf16* p2 = wd + K3 * RiP2;            // two images of [9][9] records, zero border
  bf16* rc = p2 + 2 * 81 * RiP2;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, t = lane & 3;
  const int lrow = (lane & 7) + ((lane >> 3) & 1) * 8, lk = (lane >> 4) * 8, n0 = (warp & 1) * 32, t0 = warp >> 1;
  ri_weights(wc, RiP2, WC, K3, 64);
  ri_weights(wd, RiP2, WD, K3, 64);
  const uint4 z = rbg::zero4();
  for (int e = tid; e < 4 * 81 * RiP2 / 8; e += 256) reinterpret_cast<uint4*>(p2)[e] = z;
  __syncthreads();
  // conv c: 98 pixel rows, tiles t0 and t0 + 4; conv d: 72 window rows, tiles t0 and (t0 = 0) 4
  const bf16 *bcr[2], *bdr[2];
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int m = min((t0 + 4 * i) * 16 + lrow, 2 * PIX3 - 1), im = m / PIX3, p = m % PIX3;
    bcr[i] = p2 + (im * 81 + p / 7 * 9 + p % 7) * RiP2 + lk;
    const int w = min((t0 + 4 * i) * 16 + lrow, 8 * PIX4 - 1), iw = w / (4 * PIX4), win = (w >> 2) % PIX4;
    bdr[i] = rc + (iw * 81 + (2 * (win / 3) + ((w >> 1) & 1)) * 9 + 2 * (win % 3) + (w & 1)) * RiP2 + lk;
  }
  const bf16* const cb[2] = {bcr[0], bcr[1]};
  const bf16* const db[2] = {bdr[0], bdr[1]};
  float acc[2][4][4];
  for (int i0 = 2 * blockIdx.x; i0 < nimg; i0 += 2 * gridDim.x) {
    const int ni = min(2, nimg - i0);
    for (int e = tid; e < ni * PIX3 * 8; e += 256) {
      const int r = e >> 3, im = r / PIX3, p = r % PIX3;
      *reinterpret_cast<uint4*>(p2 + (im * 81 + (p / 7 + 1) * 9 + p % 7 + 1) * RiP2 + (e & 7) * 8) =
          *reinterpret_cast<const uint4*>(a2 + ((int64_t)i0 * PIX3 + r) * C2 + (e & 7) * 8);
    }
    __syncthreads();
    ri_conv<64, 9>(acc, cb, t0 < 3, wc + n0, RiP2);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = n0 + 8 * j + 2 * t;
        const float2 b = *reinterpret_cast<const float2*>(bc + c);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int m = (t0 + 4 * i) * 16 + g + 8 * q, im = m / PIX3, p = m % PIX3;
          if (m < 2 * PIX3)
            ri_store2(rc + (im * 81 + (p / 7 + 1) * 9 + p % 7 + 1) * RiP2 + c, fmaxf(acc[i][j][2 * q] + b.x, 0.f),
                      fmaxf(acc[i][j][2 * q + 1] + b.y, 0.f));
        }
      }
    __syncthreads();
    ri_conv<64, 9>(acc, db, t0 == 0, wd + n0, RiP2);
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = n0 + 8 * j + 2 * t;
        const float2 b = *reinterpret_cast<const float2*>(bd + c);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
          const int m = min((t0 + 4 * i) * 16 + g + 8 * q, 8 * PIX4 - 1), im = m / (4 * PIX4), win = (m >> 2) % PIX4;
          const int y = 2 * (win / 3) + ((m >> 1) & 1), x = 2 * (win % 3) + (m & 1);
          const float2 s = ri_load2(p2 + (im * 81 + (y + 1) * 9 + x + 1) * RiP2 + c);
          const float z0 = acc[i][j][2 * q] + b.x, z1 = acc[i][j][2 * q + 1] + b.y;
          const float v0 = ri_pool(fmaxf(z0 + s.x, 0.f)), v1 = ri_pool(fmaxf(z1 + s.y, 0.f));
          const int row = (t0 + 4 * i) * 16 + g + 8 * q;
          if ((g & 3) == 0 && row < 8 * PIX4 && im < ni) ri_store2(a3 + ((int64_t)(i0 + im) * PIX4 + win) * C2 + c, v0, v1);
        }
      }
    __syncthreads();
  }
}

}  // namespace
