// Learned refinement predictor: a 3-layer convolutional network on 16 x 16
// downsampled patch features, BF16 operands on the tensor cores (warp-level
// mma m16n8k16) with FP32 accumulation, its backward pass and an Adam step.
//
// Network (per patch): x0 = features on an 18 x 18 grid, the 16 x 16 patch
// pixels and a one-pixel ring from beyond its edges ([324 px][16 ch]);
// a_1 = relu(conv3x3_valid(x0; W_1) + b_1) on the 16 x 16 pixels, a_l =
// relu(conv3x3(a_{l-1}; W_l) + b_l) with zero padding for l = 2, 3, 16
// channels each; v = mean over pixels of a_3; logit = wh . v + bh.
// Layouts: features [patch][324][16] BF16 (pixel-major, pixel = y*18 + x);
// conv weights [16 co][144 k] with k = tap*16 + ci and tap = (dy+1)*3 +
// (dx+1).  Every conv is an implicit GEMM with M = 256 pixels, N = 16,
// K = 144; the weight gradient is a GEMM with M = 16, N = 144 and K =
// pixels x patches.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cstdint>

namespace {

using bf16 = __nv_bfloat16;
constexpr int NPIX = 256, NCH = 16, KK = 144, PADW = 18, NPAD = PADW * PADW;

__device__ __forceinline__ unsigned saddr(const void* p) {
  return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void ldsm_x4(unsigned (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(saddr(p)));
}

__device__ __forceinline__ void ldsm_x4_t(unsigned (&r)[4], const void* p) {
  asm volatile(
      "ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
      : "r"(saddr(p)));
}

// D = A (16x16 bf16, row) * B (16x8 bf16, col) + D (f32)
__device__ __forceinline__ void mma16816(float (&d)[4], const unsigned (&a)[4],
                                         unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
      "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// A patch's activations in shared memory: 18 x 18 pixels of 16 channels, two
// 16-byte pieces a pixel.  The pieces of a pixel change places with bit 2 of
// the pixel's index, so that the eight rows of an ldmatrix (eight pixels in a
// row, one piece each) fall into eight different bank groups.
constexpr int TILE = NPAD * 2;  // 16-byte pieces
constexpr int WROW = KK + 8;    // weight row in shared memory (conflict-free)

__device__ __forceinline__ int piece(int pix, int half) {
  return pix * 2 + (half ^ ((pix >> 2) & 1));
}

// Pixel (y, x) of the 16 x 16 in the padded tile, moved by (dy, dx).
__device__ __forceinline__ int padded(int y, int x, int dy = 0, int dx = 0) {
  return (y + dy + 1) * PADW + x + dx + 1;
}

// 3 x 3 convolution of a tile by warps 0..7, 32 pixels each (M = 256, N = 16,
// K = 144); done(pixel, channel pair's half, word, value, value) gets every
// output.
template <typename F>
__device__ __forceinline__ void conv(const uint4* in, const bf16* w, int warp, int lane, F done) {
  float acc[2][2][4] = {};
  const bf16* wl = w + ((lane & 7) + 8 * (lane >> 4)) * WROW + 8 * ((lane >> 3) & 1);
  const int x = (lane & 7) + 8 * ((lane >> 3) & 1);
#pragma unroll 3
  for (int tap = 0; tap < 9; ++tap) {
    unsigned b[4];
    ldsm_x4(b, wl + tap * 16);
#pragma unroll
    for (int mt = 0; mt < 2; ++mt) {
      unsigned a[4];
      ldsm_x4(a, in + piece(padded(warp * 2 + mt, x, tap / 3 - 1, tap % 3 - 1), lane >> 4));
      mma16816(acc[mt][0], a, b[0], b[1]);
      mma16816(acc[mt][1], a, b[2], b[3]);
    }
  }
#pragma unroll
  for (int mt = 0; mt < 2; ++mt)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int pix = padded(warp * 2 + mt, (lane >> 2) + 8 * h);
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
        done(piece(pix, nt) * 4 + (lane & 3), nt * 8 + (lane & 3) * 2, acc[mt][nt][2 * h],
             acc[mt][nt][2 * h + 1]);
    }
}

__device__ __forceinline__ __nv_bfloat162 pair_bf16(float a, float b) {
  __nv_bfloat162 r;
  r.x = __float2bfloat16_rn(a);
  r.y = __float2bfloat16_rn(b);
  return r;
}

// One patch's part of a weight gradient, dW[co][tap*16+ci] += sum_p dY[p][co]
// in[p + tap][ci] (M = 16, N = 144, K = 256), one warp per tap, and of the
// bias gradient, each thread over its own pixels of two channels.
__device__ __forceinline__ void conv_dw(const uint4* dy, const uint4* in, int tap, int lane,
                                        float (&acc)[2][4], float2& db) {
  const int xa = (lane & 7) + 8 * (lane >> 4), xb = (lane & 7) + 8 * ((lane >> 3) & 1);
  const int ty = tap / 3 - 1, tx = tap % 3 - 1;
#pragma unroll 2
  for (int y = 0; y < 16; ++y) {
    unsigned a[4], b[4];
    ldsm_x4_t(a, dy + piece(padded(y, xa), (lane >> 3) & 1));
    ldsm_x4_t(b, in + piece(padded(y, xb, ty, tx), lane >> 4));
    mma16816(acc[0], a, b[0], b[1]);
    mma16816(acc[1], a, b[2], b[3]);
  }
  const unsigned* w = reinterpret_cast<const unsigned*>(dy);
  for (int px = threadIdx.x >> 3; px < NPIX; px += 36) {
    const unsigned v =
        w[piece(padded(px >> 4, px & 15), (threadIdx.x >> 2) & 1) * 4 + (threadIdx.x & 3)];
    db.x += __uint_as_float(v << 16);
    db.y += __uint_as_float(v & 0xffff0000u);
  }
}

// The network on whole patches: every layer of a patch in one CTA, the
// activations in shared memory, the weights staged once per CTA, the patches
// p, p + gridDim.x, ... one after another.  GRAD adds the backward pass of
// the weighted cross-entropy: weight gradients stay in registers over the
// CTA's patches and are added to grad once at its end.  What bounds it is a
// patch's chain of eight phases between barriers, so as many CTAs share an SM
// as shared memory and registers allow (74 KB: three; forward alone 45 KB: four).
// 1024 samples' loss and gradient on the device: nine launches with the
// activations written and read between them about 120 us, this one 51; the
// whole call 268 -> 175 us.
//
// Head: v = mean_p a3[p][:], logit = wh . v + bh.  Backward: dlogit =
// w_y (sigmoid(z) - y) / n; dwh += dlogit v; dbh += dlogit;
// da3[p][c] = dlogit wh[c] / 256; each d through its layer's relu.
template <bool GRAD>
struct Net {
  static constexpr int NT = GRAD ? 288 : 256;  // a warp per tap | 32 pixels per warp
  static constexpr int NTILE = GRAD ? 5 : 3;
  static constexpr int NW = GRAD ? 5 : 3;
  static constexpr int PER_SM = GRAD ? 3 : 4;
  static constexpr size_t smem() { return (size_t)NTILE * TILE * 16 + (size_t)NW * NCH * WROW * 2; }
};

template <bool GRAD>
__global__ void __launch_bounds__(Net<GRAD>::NT, Net<GRAD>::PER_SM)
    k_net(const bf16* __restrict__ x0, const int* __restrict__ idx, const bf16* __restrict__ wb,
          const bf16* __restrict__ wf, const float* __restrict__ prm,
          const float* __restrict__ label, float pos_weight, float inv_n,
          float* __restrict__ logit, float* __restrict__ grad, float* __restrict__ loss,
          int npatch) {
  constexpr int NT = Net<GRAD>::NT, LAYER = NCH * KK + NCH;
  extern __shared__ __align__(16) uint4 smem[];
  __shared__ float sprm[3 * NCH + NCH + 1];  // biases, head weights, head bias
  __shared__ float shead[NCH + 2];           // sums of dwh, dbh, loss
  __shared__ float sdz;
  uint4* X = smem;
  uint4* A1 = X + TILE;
  uint4* A2 = A1 + TILE;
  uint4* A3 = GRAD ? A2 + TILE : A1;      // then d3, then d1
  uint4* D2 = A2 + 2 * TILE;              // GRAD only
  bf16* w = reinterpret_cast<bf16*>(smem + Net<GRAD>::NTILE * TILE);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  for (int k = threadIdx.x; k < (Net<GRAD>::NTILE - 1) * TILE; k += NT)
    A1[k] = make_uint4(0u, 0u, 0u, 0u);  // the borders stay zero
  constexpr int ROWP = KK / 8;  // 16-byte pieces of a weight row
  for (int k = threadIdx.x; k < Net<GRAD>::NW * NCH * ROWP; k += NT) {
    const int row = k / ROWP, c = k % ROWP;
    // the flipped weights of layers 2 and 3 after the three layers'
    const bf16* src = row < 3 * NCH ? wb + row * KK : wf + (row - 2 * NCH) * KK;
    *reinterpret_cast<uint4*>(w + row * WROW + c * 8) = reinterpret_cast<const uint4*>(src)[c];
  }
  for (int k = threadIdx.x; k < 3 * NCH + NCH + 1; k += NT)
    sprm[k] = k < 3 * NCH ? prm[(k >> 4) * LAYER + NCH * KK + (k & 15)]
                          : prm[3 * LAYER + k - 3 * NCH];
  if (GRAD && threadIdx.x < NCH + 2) shead[threadIdx.x] = 0.f;
  float dw[3][2][4] = {};
  float2 db[3] = {};

  for (int p = blockIdx.x; p < npatch; p += gridDim.x) {
    const int src = idx ? idx[p] : p;
    const uint4* s4 = reinterpret_cast<const uint4*>(x0 + (size_t)src * NPAD * NCH);
    if (p != (int)blockIdx.x) __syncthreads();  // the last patch's tiles are done with
    for (int k = threadIdx.x; k < TILE; k += NT) X[piece(k >> 1, k & 1)] = s4[k];
    __syncthreads();
    auto layer = [&](const uint4* in, uint4* out, int l) {
      unsigned* o = reinterpret_cast<unsigned*>(out);
      if (warp < 8)
        conv(in, w + l * NCH * WROW, warp, lane, [&](int at, int co, float v0, float v1) {
          const float* b = sprm + l * NCH + co;
          *reinterpret_cast<__nv_bfloat162*>(o + at) =
              pair_bf16(fmaxf(v0 + b[0], 0.f), fmaxf(v1 + b[1], 0.f));
        });
      __syncthreads();
    };
    layer(X, A1, 0);
    layer(A1, A2, 1);
    layer(A2, A3, 2);
    if (warp == 0) {
      // a lane takes the same eight channels of every sixteenth pixel
      float s[8] = {};
      const int half = lane & 1;
#pragma unroll 4
      for (int r = 0; r < 16; ++r) {
        const uint4 v = A3[piece(padded(r, lane >> 1), half)];
        const unsigned q4[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          s[2 * q] += __uint_as_float(q4[q] << 16);
          s[2 * q + 1] += __uint_as_float(q4[q] & 0xffff0000u);
        }
      }
#pragma unroll
      for (int o = 2; o < 32; o <<= 1)
#pragma unroll
        for (int q = 0; q < 8; ++q) s[q] += __shfl_xor_sync(0xffffffffu, s[q], o);
      const float* wh = sprm + 3 * NCH + 8 * half;
      float z = 0.f;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        s[q] *= 1.0f / NPIX;
        z += wh[q] * s[q];
      }
      z += __shfl_xor_sync(0xffffffffu, z, 1);
      z += sprm[4 * NCH];
      if (lane == 0) logit[p] = z;
      if (GRAD && lane < 2) {
        const float y = label[src];
        const float sg = 1.f / (1.f + expf(-z));
        const float wy = y > 0.5f ? pos_weight : 1.f;
        const float dz = wy * (sg - y) * inv_n;
#pragma unroll
        for (int q = 0; q < 8; ++q) shead[8 * half + q] += dz * s[q];
        if (lane == 0) {
          sdz = dz;
          shead[NCH] += dz;
          // softplus form of the cross-entropy
          const float l = fmaxf(z, 0.f) - z * y + log1pf(expf(-fabsf(z)));
          shead[NCH + 1] += wy * l * inv_n;
        }
      }
    }
    if constexpr (GRAD) {
      __syncthreads();
      {  // d3 in place of a3
        const float dz = sdz;
        const float* wh = sprm + 3 * NCH + 8 * (threadIdx.x & 1);
        __nv_bfloat162 g[4];
#pragma unroll
        for (int q = 0; q < 4; ++q)
          g[q] = pair_bf16(dz * wh[2 * q] * (1.0f / NPIX), dz * wh[2 * q + 1] * (1.0f / NPIX));
        for (int k = threadIdx.x; k < NPIX * 2; k += NT) {
          uint4* c = A3 + piece(padded(k >> 5, (k >> 1) & 15), k & 1);
          uint4 v = *c;
          unsigned* q4 = &v.x;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const unsigned gq = *reinterpret_cast<const unsigned*>(&g[q]);
            const unsigned lo = __uint_as_float(q4[q] << 16) > 0.f ? gq & 0xffffu : 0u;
            const unsigned hi = __uint_as_float(q4[q] & 0xffff0000u) > 0.f ? gq & 0xffff0000u : 0u;
            q4[q] = lo | hi;
          }
          *c = v;
        }
      }
      __syncthreads();
      // weight gradient of a layer, and the gradient of its input through the
      // relu that made it (act), which both only read d
      auto back = [&](const uint4* d, const uint4* act, uint4* out, int l) {
        conv_dw(d, act, warp, lane, dw[l], db[l]);
        if (warp < 8) {
          const unsigned* m = reinterpret_cast<const unsigned*>(act);
          unsigned* o = reinterpret_cast<unsigned*>(out);
          conv(d, w + (2 + l) * NCH * WROW, warp, lane, [&](int at, int, float v0, float v1) {
            const unsigned a = m[at];
            if (!(__uint_as_float(a << 16) > 0.f)) v0 = 0.f;
            if (!(__uint_as_float(a & 0xffff0000u) > 0.f)) v1 = 0.f;
            *reinterpret_cast<__nv_bfloat162*>(o + at) = pair_bf16(v0, v1);
          });
        }
        __syncthreads();
      };
      back(A3, A2, D2, 2);
      back(D2, A1, A3, 1);
      conv_dw(A3, X, warp, lane, dw[0], db[0]);
    }
  }
  if constexpr (GRAD) {
    // the CTA's sums to the gradient: channel pairs are neighbours in dW
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
      for (int nt = 0; nt < 2; ++nt)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int co = (lane >> 2) + 8 * h, ci = nt * 8 + (lane & 3) * 2;
          atomicAdd(reinterpret_cast<float2*>(grad + l * LAYER + co * KK + warp * 16 + ci),
                    make_float2(dw[l][nt][2 * h], dw[l][nt][2 * h + 1]));
        }
    __syncthreads();
    float2* sdb = reinterpret_cast<float2*>(X);  // [3][36 pixels][8 channel pairs]
#pragma unroll
    for (int l = 0; l < 3; ++l) sdb[l * 288 + threadIdx.x] = db[l];
    __syncthreads();
    if (threadIdx.x < 3 * NCH) {
      const int l = threadIdx.x >> 4, c = threadIdx.x & 15;
      const float* f = reinterpret_cast<const float*>(sdb + l * 288) + c;
      float t = 0.f;
      for (int k = 0; k < 36; ++k) t += f[k * 16];
      atomicAdd(&grad[l * LAYER + NCH * KK + c], t);
    } else if (threadIdx.x >= 64 && threadIdx.x < 64 + NCH + 2) {
      const int k = threadIdx.x - 64;
      atomicAdd(k <= NCH ? &grad[3 * LAYER + k] : loss, shead[k]);
    }
  }
}

// Adam on the FP32 master parameters, then the BF16 copies of the conv
// weights and of their flipped transposes (the input-gradient pass):
// Wf[ci][(8 - tap)*16 + co] = W[co][tap*16 + ci].
__global__ void k_adam(float* __restrict__ prm, const float* __restrict__ grad,
                       float* __restrict__ m, float* __restrict__ v, int n,
                       float lr, float b1, float b2, float eps, float c1,
                       float c2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const float g = grad[k];
  const float mk = b1 * m[k] + (1.f - b1) * g;
  const float vk = b2 * v[k] + (1.f - b2) * g * g;
  m[k] = mk;
  v[k] = vk;
  prm[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

__global__ void k_cast_weights(const float* __restrict__ prm, int layer_stride,
                               bf16* __restrict__ wb, bf16* __restrict__ wf) {
  const int l = blockIdx.y;
  const float* W = prm + (size_t)l * layer_stride;
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= NCH * KK) return;
  const int co = k / KK, kk = k % KK, tap = kk / 16, ci = kk % 16;
  const bf16 w = __float2bfloat16_rn(W[k]);
  wb[(size_t)l * NCH * KK + k] = w;
  wf[(size_t)l * NCH * KK + ci * KK + (8 - tap) * 16 + co] = w;
}

__global__ void k_to_bf16(const float* __restrict__ x, bf16* __restrict__ y,
                          size_t n) {
  const size_t k = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) y[k] = __float2bfloat16_rn(x[k]);
}

template <bool GRAD>
int launch_net(const void* x0, const int* idx, const void* wb, const void* wf, const float* prm,
               const float* label, float pos_weight, float* logit, float* grad, float* loss,
               int npatch, cudaStream_t st) {
  constexpr size_t bytes = Net<GRAD>::smem();
  if (cudaFuncSetAttribute(k_net<GRAD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)bytes) != cudaSuccess)
    return -2;
  const int fit = 152 * Net<GRAD>::PER_SM;
  k_net<GRAD><<<npatch < fit ? npatch : fit, Net<GRAD>::NT, bytes, st>>>(
      static_cast<const bf16*>(x0), idx, static_cast<const bf16*>(wb),
      static_cast<const bf16*>(wf), prm, label, pos_weight, 1.0f / npatch, logit, grad, loss,
      npatch);
  return cudaGetLastError() == cudaSuccess ? 0 : -2;
}

inline int ok() { return cudaGetLastError() == cudaSuccess ? 0 : -2; }

}  // namespace

namespace gf {

// Parameter block (FP32): W1, b1, W2, b2, W3, b3 (stride 144*16 + 16 each),
// then wh[16], bh[1].
constexpr int CNN_LAYER = NCH * KK + NCH;
constexpr int CNN_NPARAM = 3 * CNN_LAYER + NCH + 1;

int cnn_nparam() { return CNN_NPARAM; }

// Logits of npatch feature tiles x0 (BF16) with the BF16 weights wb.
int cnn_forward(const void* x0, const void* wb, const float* prm, float* logit, int npatch,
                void* stream) {
  if (npatch <= 0) return 0;
  return launch_net<false>(x0, nullptr, wb, nullptr, prm, nullptr, 1.f, logit, nullptr, nullptr,
                           npatch, static_cast<cudaStream_t>(stream));
}

// Forward and backward pass: logits, the gradient of the mean weighted
// cross-entropy added to grad (FP32, same layout as the parameters) and the
// loss to *loss.  Sample p is row idx[p] of x0 and label (idx null: row p).
int cnn_grad(const void* x0, const int* idx, const void* wb, const void* wf, const float* prm,
             const float* label, float pos_weight, float* logit, float* grad, float* loss,
             int npatch, void* stream) {
  if (npatch <= 0) return 0;
  return launch_net<true>(x0, idx, wb, wf, prm, label, pos_weight, logit, grad, loss, npatch,
                          static_cast<cudaStream_t>(stream));
}

int cnn_adam(float* prm, const float* grad, float* m, float* v, float lr,
             int t, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const float b1 = 0.9f, b2 = 0.999f;
  float c1 = 1.f, c2 = 1.f;
  for (int k = 0; k < t; ++k) { c1 *= b1; c2 *= b2; }
  k_adam<<<(CNN_NPARAM + 255) / 256, 256, 0, st>>>(prm, grad, m, v, CNN_NPARAM, lr,
                                                   b1, b2, 1e-8f, 1.f - c1, 1.f - c2);
  return ok();
}

int cnn_cast(const float* prm, void* wb, void* wf, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  k_cast_weights<<<dim3((NCH * KK + 255) / 256, 3), 256, 0, st>>>(
      prm, CNN_LAYER, static_cast<bf16*>(wb), static_cast<bf16*>(wf));
  return ok();
}

int cnn_to_bf16(const float* x, void* y, size_t n, void* stream) {
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (n == 0) return 0;
  k_to_bf16<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(x, static_cast<bf16*>(y), n);
  return ok();
}

}  // namespace gf
