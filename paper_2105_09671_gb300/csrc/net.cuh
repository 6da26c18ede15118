// Learned 16-step jump network: shapes, parameter layout and index helpers
// shared by its kernels (k_net.cu) and its C-ABI layer (ac_net.cu).
//
// Network (2D; 3D replaces 3x3 by 3x3x3, T = 3^d taps):
//   z1 = conv(phi, W1) + b1, a1 = gelu(z1)               1 -> 32 channels
//   zl = conv(a_{l-1}, Wl) + bl, al = gelu(zl)            32 -> 32, l = 2..5
//   z6 = conv(a5, W6) + b6                                32 -> 1
//   phi_hat = phi + s * z6
// conv uses replicate padding (the zero-Neumann ghost of Section 2); gelu is
// the tanh form.  Parameters (FP32, flat): for each layer W[t][ci][co] then
// b[co]; tap t enumerates offsets (-1, 0, 1)^d with the last axis (x)
// fastest.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace ac {

constexpr int kNetC = 32;       // hidden channels
constexpr int kNetLayers = 6;

__host__ __device__ constexpr int net_taps(int ndim) { return ndim == 3 ? 27 : 9; }

struct NetShape {
  int ndim;
  int batch;
  int nx, ny, nz;  // nz = 1 in 2D
  // padded extents: +2 on every spatial axis of the grid's dimension
  __host__ __device__ int px() const { return nx + 2; }
  __host__ __device__ int py() const { return ny + 2; }
  __host__ __device__ int pz() const { return ndim == 3 ? nz + 2 : 1; }
  __host__ __device__ int64_t cells() const { return (int64_t)batch * nz * ny * nx; }
  __host__ __device__ int64_t padded_cells() const { return (int64_t)batch * pz() * py() * px(); }
  // linear index of cell (b, z, y, x) and of padded cell (b, zp, yp, xp)
  __host__ __device__ int64_t u(int b, int z, int y, int x) const {
    return (((int64_t)b * nz + z) * ny + y) * nx + x;
  }
  __host__ __device__ int64_t p(int b, int zp, int yp, int xp) const {
    return (((int64_t)b * pz() + zp) * py() + yp) * px() + xp;
  }
  // padded index of the cell (b, z, y, x) shifted by (oz, oy, ox)
  __host__ __device__ int64_t ps(int b, int z, int y, int x, int oz, int oy, int ox) const {
    return p(b, ndim == 3 ? z + 1 + oz : 0, y + 1 + oy, x + 1 + ox);
  }
};

// Tap t -> offsets, x fastest: 2D t = (oy+1)*3 + (ox+1); 3D adds (oz+1)*9.
__host__ __device__ inline void net_tap(int ndim, int t, int &oz, int &oy, int &ox) {
  ox = t % 3 - 1;
  oy = (t / 3) % 3 - 1;
  oz = ndim == 3 ? t / 9 - 1 : 0;
}

// Parameter offsets (in floats) inside the flat vector.
struct NetLayout {
  int ndim, T;
  int64_t w[kNetLayers], b[kNetLayers], total;
  __host__ __device__ static int cin(int l) { return l == 0 ? 1 : kNetC; }
  __host__ __device__ static int cout(int l) { return l == kNetLayers - 1 ? 1 : kNetC; }
};

inline NetLayout net_layout(int ndim) {
  NetLayout L;
  L.ndim = ndim;
  L.T = net_taps(ndim);
  int64_t off = 0;
  for (int l = 0; l < kNetLayers; ++l) {
    L.w[l] = off;
    off += (int64_t)L.T * NetLayout::cin(l) * NetLayout::cout(l);
    L.b[l] = off;
    off += NetLayout::cout(l);
  }
  L.total = off;
  return L;
}

typedef __nv_bfloat16 bf16;

// Device buffers of one network (parameters, optimiser state, packed BF16
// weights) and of one batch shape (activations, pre-activations, gradients).
struct NetBuffers {
  NetLayout layout;
  float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
  bf16 *wf = nullptr, *wd = nullptr;  // B operands of layers 1..4 (forward, data gradient)
  bf16 *a[5] = {};                    // padded activations (inference uses a[0], a[1])
  bf16 *z[5] = {};                    // pre-activations (training)
  bf16 *gz[5] = {};                   // padded gradients wrt z (zero ghost ring)
  float *raw = nullptr;               // [cells][32] FP32 scratch: the data gradient of face cells
  float *g6 = nullptr;                // [cells] gradient wrt the last pre-activation
  double *loss = nullptr;             // sum of squared scaled errors
  int *status = nullptr;
};

cudaError_t net_forward(const NetBuffers &nb, const NetShape &sh, const float *phi, float scale,
                        float *phihat, const float *target, bool train, int num_sms, cudaStream_t s);
cudaError_t net_backward(const NetBuffers &nb, const NetShape &sh, const float *phi, int num_sms,
                         cudaStream_t s);
cudaError_t net_pack(const NetBuffers &nb, cudaStream_t s);
// One 32 -> 32 tensor-core convolution over padded activations `in` (mode 0:
// forward epilogue into zout / outpad; mode 1, data gradient: x gelu'(zin)
// into outpad inside the grid, raw FP32 into outraw for the face cells).
cudaError_t net_conv_rows(int mode, const bf16 *in, const bf16 *Wx, const float *bias,
                          const NetShape &sh, bf16 *zout, bf16 *outpad, float *outraw, const bf16 *zin,
                          int *status, int num_sms, cudaStream_t s);
// Weight and bias gradients of one 32 -> 32 layer, added to gw / gb, from its
// padded input activations and the padded gradient of its pre-activations
// (zero ghost ring).
cudaError_t net_wgrad(const bf16 *apad, const bf16 *gpad, const NetShape &sh, float *gw, float *gb, int *status,
                      int num_sms, cudaStream_t s);
cudaError_t net_adam(const NetBuffers &nb, float lr, float b1, float b2, float eps, int step,
                     cudaStream_t s);

// BF16 packing of 8 FP32 values into one 16-byte word and back.
__device__ __forceinline__ uint4 pack8_bf16(const float *v) {
  uint4 u;
  __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) h[i] = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
  return u;
}
__device__ __forceinline__ void unpack8_bf16(const uint4 &u, float *v) {
  const __nv_bfloat162 *h = reinterpret_cast<const __nv_bfloat162 *>(&u);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float2 f = __bfloat1622float2(h[i]);
    v[2 * i] = f.x;
    v[2 * i + 1] = f.y;
  }
}

// 32 bytes of one lane in one access: a cell's 64 bytes of activations then
// take two accesses of whole sectors instead of four of half sectors.
__device__ __forceinline__ void st_global32(void *p, const uint4 &a, const uint4 &b) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y),
               "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}
__device__ __forceinline__ void ld_global32(const void *p, uint4 &a, uint4 &b) {
  asm volatile("ld.global.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(a.x), "=r"(a.y), "=r"(a.z), "=r"(a.w), "=r"(b.x), "=r"(b.y), "=r"(b.z), "=r"(b.w)
               : "l"(p)
               : "memory");
}

// Store one cell's 32 activations at its padded position and at the ghost
// copies it stands for (replicate padding: a boundary cell is also its
// outside neighbour).
template <int NDIM>
__device__ __forceinline__ void store_replicated(bf16 *outpad, const NetShape &sh, int b, int z,
                                                 int y, int x, const float *a) {
  uint4 w[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) w[c] = pack8_bf16(a + 8 * c);
  int xs[3], ys[3], zs[3];
  int nxs = 0, nys = 0, nzs = 0;
  xs[nxs++] = x + 1;
  if (x == 0) xs[nxs++] = 0;
  if (x == sh.nx - 1) xs[nxs++] = sh.nx + 1;
  ys[nys++] = y + 1;
  if (y == 0) ys[nys++] = 0;
  if (y == sh.ny - 1) ys[nys++] = sh.ny + 1;
  if (NDIM == 3) {
    zs[nzs++] = z + 1;
    if (z == 0) zs[nzs++] = 0;
    if (z == sh.nz - 1) zs[nzs++] = sh.nz + 1;
  } else {
    zs[nzs++] = 0;
  }
  for (int iz = 0; iz < nzs; ++iz)
    for (int iy = 0; iy < nys; ++iy)
      for (int ix = 0; ix < nxs; ++ix) {
        bf16 *dst = outpad + sh.p(b, zs[iz], ys[iy], xs[ix]) * kNetC;
        st_global32(dst, w[0], w[1]);
        st_global32(dst + 16, w[2], w[3]);
      }
}

// Two FP32 values as an operand of packed arithmetic (fma/mul/add.rn.f32x2: half
// the issue slots).
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float &a, float &b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t mul2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// The forward passes' GELU (tanh form) of two values, with the hardware tanh
// approximation (tanh.approx.f32, relative error about 2^-11, below the BF16
// rounding of the stored activation).
__device__ __forceinline__ uint64_t net_gelu_fast2(uint64_t x) {
  const float k = 0.7978845608028654f;
  const uint64_t u = mul2(x, fma2(pack2(k * 0.044715f, k * 0.044715f), mul2(x, x), pack2(k, k)));
  float a, b;
  unpack2(u, a, b);
  asm("tanh.approx.f32 %0, %0;" : "+f"(a));
  asm("tanh.approx.f32 %0, %0;" : "+f"(b));
  const uint64_t h = mul2(x, pack2(0.5f, 0.5f));
  return fma2(h, pack2(a, b), h);
}

// Its derivative for the backward passes, to FP32 accuracy.  With e = exp(-2u)
// and s = 1 / (1 + e), tanh u = 2 s - 1 and 1 - tanh^2 u = 4 s (e s), so
//   gelu'(x) = (1 + t) / 2 + x/2 (1 - t^2) u' = s + 2 x u' s (e s),
// in which nothing cancels: against FP64 over [-10, 10] its error is at most
// 2.1e-7 (2.9e-8 rms), that of the form with tanhf 5.6e-7 (1.1e-7 rms).  e is
// 2^y with the factor -2 log2(e) in u's coefficients.  Beyond, it is 0 and 1: the
// exponent's bound keeps e s finite while s, 2^-127, is flushed to 0, and x^2's
// (from |x| = 20 on) the factor 2 x u' up to 1e36.
__device__ __forceinline__ float net_exp2(float y) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fminf(y, 127.0f)));
  return r;
}
__device__ __forceinline__ float net_rcp(float y) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(y));
  return r;
}
__device__ __forceinline__ float net_gelu_grad(float x) {
  const float k = 0.7978845608028654f, l2e = 1.4426950408889634f, c = 0.044715f;
  const float x2 = fminf(x * x, 400.0f);
  const float e = net_exp2(x * fmaf(-2.0f * k * l2e * c, x2, -2.0f * k * l2e));
  const float s = net_rcp(1.0f + e);
  return fmaf(x * fmaf(6.0f * k * c, x2, 2.0f * k), s * (e * s), s);
}
// The same on two values, packed: the data gradient's kernel takes 87 us with
// it, 115 with the scalar form (32 x 256^2 pixels).
__device__ __forceinline__ uint64_t net_gelu_grad2(uint64_t x) {
  const float k = 0.7978845608028654f, l2e = 1.4426950408889634f, c = 0.044715f;
  const float a1 = -2.0f * k * l2e * c, a0 = -2.0f * k * l2e, b1 = 6.0f * k * c, b0 = 2.0f * k;
  float qa, qb;
  unpack2(mul2(x, x), qa, qb);
  const uint64_t x2 = pack2(fminf(qa, 400.0f), fminf(qb, 400.0f));
  float ya, yb;
  unpack2(mul2(x, fma2(pack2(a1, a1), x2, pack2(a0, a0))), ya, yb);
  const uint64_t e = pack2(net_exp2(ya), net_exp2(yb));
  float da, db;
  unpack2(add2(e, pack2(1.0f, 1.0f)), da, db);
  const uint64_t s = pack2(net_rcp(da), net_rcp(db));
  return fma2(mul2(x, fma2(pack2(b1, b1), x2, pack2(b0, b0))), mul2(s, mul2(e, s)), s);
}

}  // namespace ac
