// Device pieces of the closure's network (5 -> 64 -> 64 -> 6, GELU) for the MLP
// kernels (ps_mlp.cu): the BF16 tensor-core fragments, the activations, and the
// forward pass of a 16-sample tile held in the registers of one warp.
//
// Parameter vector (FP32): W1 [5][64] | b1 [64] | W2 [64][64] | b2 [64] |
// W3 [64][6] | b3 [6]   (row-major, y = x W + b).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace ps {
namespace mlp {

constexpr int H = 64, NI = 5, NO = 6;
constexpr int OFF_W1 = 0, OFF_B1 = OFF_W1 + NI * H, OFF_W2 = OFF_B1 + H, OFF_B2 = OFF_W2 + H * H,
              OFF_W3 = OFF_B2 + H, OFF_B3 = OFF_W3 + H * NO, NPARAM = OFF_B3 + NO;

// Two FP32 values rounded to BF16, lo in the lower half.
__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}
__device__ __forceinline__ float lo_of(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float hi_of(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// D += A (16x16, bf16) * B (16x8, bf16), FP32 accumulate.  Fragments (lane l,
// q = l % 4, g = l / 4): A rows g and g + 8, columns 2q + {0, 1} (+ 8); B column
// g, rows 2q + {0, 1} (+ 8); D rows g and g + 8, columns 2q + {0, 1}.
__device__ __forceinline__ void mma16(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                      uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// The same with a k extent of 8 (A columns 2q + {0, 1}, B rows 2q + {0, 1}):
// the layers whose inner dimension is 5 or 6.
__device__ __forceinline__ void mma8(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Packed FP32 operations (two lanes per instruction).
union F2 {
  float2 f;
  unsigned long long u;
};
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  F2 x{a}, y{b}, r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.u) : "l"(x.u), "l"(y.u));
  return r.f;
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  F2 x{a}, y{b}, z{c}, r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.u) : "l"(x.u), "l"(y.u), "l"(z.u));
  return r.f;
}
__device__ __forceinline__ float2 both(float a) { return make_float2(a, a); }
// max(z, lo) that keeps a NaN
__device__ __forceinline__ float clamp_low(float z, float lo) {
  float y;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(y) : "f"(z), "f"(lo));
  return y;
}

// GELU (tanh form) and its derivative from one tanh, as training uses them.  (The
// sigmoid form of gelu4 takes 538 us per 2.1 M samples instead of 692, but rounds
// some activations to the neighbouring BF16 number, which moves the loss and the
// gradients.)
__device__ __forceinline__ void gelu_with_grad(float x, float& h, float& g) {
  constexpr float C = 0.7978845608028654f;  // sqrt(2/pi)
  const float t = tanhf(C * (x + 0.044715f * x * x * x));
  h = 0.5f * x * (1.f + t);
  g = 0.5f * (1.f + t) + 0.5f * x * (1.f - t * t) * C * (1.f + 3.f * 0.044715f * x * x);
}

// GELU (tanh form) of four values, two of one sample (z[0], z[1]) and two of
// another, for inference: 0.5 z (1 + tanh u) = z s with s = 1/(1 + exp(-2u)),
// u = sqrt(2/pi) (z + 0.044715 z^3).  The sigmoid takes one ex2 each; the two
// values of a sample share one rcp of their product, each refined by one Newton
// step, and the rest runs two values per instruction, since issue bounds the
// kernel.  A NaN thus stays within its own sample (one rcp for all four values
// took it to the other one, and ten 64^3 closure steps 2744 instead of 2721 us).
// z is clamped at -7.5 so that the product of two and its reciprocal stay normal
// numbers: there and below the result is -4.0e-18 (1 + tanhf: up to 7.7e-8 off
// by cancellation).
__device__ __forceinline__ void gelu4(const float (&z)[4], float (&h)[4]) {
  constexpr float A = -2.f * 0.7978845608028654f * 1.4426950408889634f;  // -2 sqrt(2/pi) log2(e)
  constexpr float B = A * 0.044715f;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float2 x = make_float2(clamp_low(z[2 * i], -7.5f), clamp_low(z[2 * i + 1], -7.5f));
    const float2 v = mul2(x, fma2(mul2(x, x), both(B), both(A)));
    const float d0 = 1.f + ex2(v.x), d1 = 1.f + ex2(v.y);
    const float r = rcp(d0 * d1);
    float2 s = make_float2(r * d1, r * d0);
    s = fma2(s, fma2(make_float2(-d0, -d1), s, both(1.f)), s);
    const float2 y = mul2(x, s);
    h[2 * i] = y.x;
    h[2 * i + 1] = y.y;
  }
}

// BF16 weight fragments and biases of the whole network, held by every warp.
struct Net {
  uint32_t w1[H / 8], w2[H / 16][H / 8][2], w3[H / 16][2];
  float b1[H / 8][2], b2[H / 8][2], b3[2];
  __device__ __forceinline__ void load(const float* __restrict__ p) {
    const int lane = threadIdx.x & 31, q = lane & 3, g = lane >> 2;
#pragma unroll
    for (int nt = 0; nt < H / 8; ++nt) {
      const int n = 8 * nt + g, k = 2 * q;
      w1[nt] = pack2(k < NI ? p[OFF_W1 + k * H + n] : 0.f, k + 1 < NI ? p[OFF_W1 + (k + 1) * H + n] : 0.f);
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        b1[nt][j] = p[OFF_B1 + 8 * nt + 2 * q + j];
        b2[nt][j] = p[OFF_B2 + 8 * nt + 2 * q + j];
      }
    }
#pragma unroll
    for (int kt = 0; kt < H / 16; ++kt)
#pragma unroll
      for (int hf = 0; hf < 2; ++hf) {
        const int k = 16 * kt + 8 * hf + 2 * q;
#pragma unroll
        for (int nt = 0; nt < H / 8; ++nt)
          w2[kt][nt][hf] = pack2(p[OFF_W2 + k * H + 8 * nt + g], p[OFF_W2 + (k + 1) * H + 8 * nt + g]);
        w3[kt][hf] = pack2(g < NO ? p[OFF_W3 + k * NO + g] : 0.f, g < NO ? p[OFF_W3 + (k + 1) * NO + g] : 0.f);
      }
#pragma unroll
    for (int j = 0; j < 2; ++j) b3[j] = 2 * q + j < NO ? p[OFF_B3 + 2 * q + j] : 0.f;
  }
  // y (D fragment: rows g and g + 8, outputs 2q + {0, 1}) of the tile whose
  // layer-1 A fragment (inputs 2q + {0, 1} of rows g and g + 8) is a0, a1.  The
  // m16n8 accumulators of two neighbouring 8-column tiles of one layer are,
  // after bias, GELU and BF16 packing, exactly the A fragment of the next
  // layer's 16-column k tile, so activations never leave the registers.
  __device__ __forceinline__ void forward(uint32_t a0, uint32_t a1, float (&y)[4]) const {
    uint32_t h[H / 16][4];
    float o[4];
#pragma unroll
    for (int nt = 0; nt < H / 8; ++nt) {
      float d[4] = {0.f, 0.f, 0.f, 0.f};
      mma8(d, a0, a1, w1[nt]);
      const float z[4] = {d[0] + b1[nt][0], d[1] + b1[nt][1], d[2] + b1[nt][0], d[3] + b1[nt][1]};
      gelu4(z, o);
      h[nt >> 1][(nt & 1) * 2 + 0] = pack2(o[0], o[1]);
      h[nt >> 1][(nt & 1) * 2 + 1] = pack2(o[2], o[3]);
    }
    float acc[H / 8][4];
#pragma unroll
    for (int nt = 0; nt < H / 8; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
#pragma unroll
    for (int kt = 0; kt < H / 16; ++kt)
#pragma unroll
      for (int nt = 0; nt < H / 8; ++nt)
        mma16(acc[nt], h[kt][0], h[kt][1], h[kt][2], h[kt][3], w2[kt][nt][0], w2[kt][nt][1]);
#pragma unroll
    for (int nt = 0; nt < H / 8; ++nt) {
      const float z[4] = {acc[nt][0] + b2[nt][0], acc[nt][1] + b2[nt][1], acc[nt][2] + b2[nt][0],
                          acc[nt][3] + b2[nt][1]};
      gelu4(z, o);
      h[nt >> 1][(nt & 1) * 2 + 0] = pack2(o[0], o[1]);
      h[nt >> 1][(nt & 1) * 2 + 1] = pack2(o[2], o[3]);
    }
    y[0] = y[1] = y[2] = y[3] = 0.f;
#pragma unroll
    for (int kt = 0; kt < H / 16; ++kt) mma16(y, h[kt][0], h[kt][1], h[kt][2], h[kt][3], w3[kt][0], w3[kt][1]);
    y[0] += b3[0];
    y[1] += b3[1];
    y[2] += b3[0];
    y[3] += b3[1];
  }
};

}  // namespace mlp
}  // namespace ps
