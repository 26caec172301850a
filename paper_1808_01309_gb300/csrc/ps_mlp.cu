// Pointwise MLP of the learned LES closure (5 -> 64 -> 64 -> 6, GELU) on the
// BF16 tensor cores with FP32 accumulation (mma.sync), forward, backward and
// the Adam update.  See include/ps.h (ps_mlp_*).
//
// Operands are rounded to BF16 where they enter a tensor-core product; biases,
// pre-activations, GELU and all accumulations stay FP32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>
#include <string>

#include "ps.h"
#include "ps_mlp.cuh"
#include "ps_tb.cuh"

namespace ps {
void set_last_error(const std::string& msg);
}

namespace {

using namespace ps::mlp;
static_assert(NPARAM == PS_MLP_NPARAM, "parameter layout");
constexpr int CH = 128;  // samples per chunk of the training kernel
typedef __nv_bfloat16 bf;

// Inference: each warp keeps the whole network in registers and runs 16-sample
// tiles through it.
__global__ void __launch_bounds__(128) k_mlp_forward(const float* __restrict__ p, const float* __restrict__ X,
                                                     float* __restrict__ Y, long long B) {
  const int lane = threadIdx.x & 31, q = lane & 3, g = lane >> 2;
  Net net;
  net.load(p);
  const long long ntiles = (B + 15) / 16;
  const long long wstride = (long long)gridDim.x * (blockDim.x >> 5);
  for (long long tile = (long long)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); tile < ntiles;
       tile += wstride) {
    const long long r0 = tile * 16 + g, r1 = r0 + 8;
    auto xin = [&](long long r, int c) { return r < B && c < NI ? X[r * NI + c] : 0.f; };
    float y[4];
    net.forward(pack2(xin(r0, 2 * q), xin(r0, 2 * q + 1)), pack2(xin(r1, 2 * q), xin(r1, 2 * q + 1)), y);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = 2 * q + j;
      if (c < NO) {
        if (r0 < B) Y[r0 * NO + c] = y[j];
        if (r1 < B) Y[r1 * NO + c] = y[2 + j];
      }
    }
  }
}

// ---- training ------------------------------------------------------------------
// One CTA (4 warps) processes chunks of 128 samples.  Warp w takes samples
// 32w..32w+31 as two 16-sample tiles: forward and backward stay in registers
// (activations and deltas go from accumulator to operand fragment as in
// Net::forward; the derivative of the activation is kept in FP32), and the BF16
// operands of the weight gradients (h1, h2, dz1, dz2, x, dy) are left in shared
// memory.  Then warp w forms rows 16w..16w+15 of dW2 and dW3 and columns
// 16w..16w+15 of dW1 over the chunk's 128 samples.  Rows are 128 bytes with
// their 16-byte pieces permuted by the row (piece ^ (row & 7)), so that fragment
// stores, ldmatrix rows and the bias sums are free of bank conflicts.
//
// Bound: instruction issue (128 activations with their derivatives a sample);
// 2.1 M samples in 692 us (4050 us with activations exchanged through
// shared memory in 2-byte accesses with eight-way bank conflicts, tanhf twice
// per activation and the loss summed by FP64 conversions).
struct Smem {
  bf w2[H * H];
  bf h1[CH * H], h2[CH * H], dz1[CH * H], dz2[CH * H];
  bf x[CH * 8], dy[CH * 8];       // inputs (5) and output deltas (6), padded with zeros
  float b1[H], b2[H];
  float yf[4][16 * 8];            // network outputs of a warp's tile (tensor-basis fit)
  float tb[CH * 37];              // tensor basis of the chunk's samples (36 values, odd stride)
};

// Byte offset of 16-byte piece c of row r in a permuted [rows][64] BF16 array.
__device__ __forceinline__ uint32_t sw(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }
__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void ldm4(uint32_t (&v)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void ldm4t(uint32_t (&v)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void ldm2t(uint32_t (&v)[2], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(v[0]), "=r"(v[1])
               : "r"(a)
               : "memory");
}

// Sum of squares as an unevaluated FP32 pair (about 48 bits): the FP64 pipe
// takes 1/64 of the FP32 rate, and one conversion, product and sum per residual
// there cost more than the residual.  Residuals whose squares leave the FP32
// range are summed in FP64.
struct SquareSum {
  float hi = 0.f, lo = 0.f;
  double big = 0.0;
  __device__ __forceinline__ void add(float e) {
    const float ae = fabsf(e);
    if (ae < 1e15f && (ae > 1e-15f || ae == 0.f)) {
      const float p = e * e, pe = fmaf(e, e, -p);
      const float s = hi + p, b = s - hi;
      lo += ((hi - (s - b)) + (p - b)) + pe;
      hi = s;
    } else {
      big += (double)e * e;
    }
  }
  __device__ __forceinline__ double total() const { return ((double)hi + (double)lo) + big; }
};

// Forward + backward over B samples; parameter gradients accumulate
// (atomically) into grad[NPARAM] and the loss into *loss.
//   MODE_PLAIN: mean-squared error of y against T
//   MODE_TB   : mean-squared error of the model stress sum_n y_n T_n(A/s_A)
//               (T_n the tensor basis of the gradient rows Ag[B][9]) against T/s_tau
//   MODE_DY   : no loss; T holds dL/dy per sample (backpropagation only)
enum { MODE_PLAIN = 0, MODE_TB = 1, MODE_DY = 2 };
template <int MODE>
__global__ void __launch_bounds__(128, 2) k_mlp_grad(const float* __restrict__ p, const float* __restrict__ X,
                                                     const float* __restrict__ Ag, const float* __restrict__ T,
                                                     long long B, float inv_sA, float inv_stau, float* grad,
                                                     double* loss) {
  extern __shared__ __align__(128) unsigned char raw[];
  Smem& s = *reinterpret_cast<Smem*>(raw);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31, q = lane & 3, g = lane >> 2;
  const int mi = lane >> 3, mr = lane & 7;  // ldmatrix: matrix and row this lane addresses
  for (int i = threadIdx.x; i < H * H / 2; i += blockDim.x) {
    const int r = i / (H / 2), c = (i % (H / 2)) * 2;  // row, even column
    *reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(s.w2) + sw(r, c >> 3) + (c & 7) * 2) =
        pack2(p[OFF_W2 + r * H + c], p[OFF_W2 + r * H + c + 1]);
  }
  for (int i = threadIdx.x; i < H; i += blockDim.x) {
    s.b1[i] = p[OFF_B1 + i];
    s.b2[i] = p[OFF_B2 + i];
  }
  // fragments of the small layers: W1 (k = 5), W3 (n = 6) and W3^T (k = 6)
  uint32_t w1[H / 8], w3[H / 16][2], w3t[H / 8];
  float b3[2];
#pragma unroll
  for (int nt = 0; nt < H / 8; ++nt) {
    const int n = 8 * nt + g, k = 2 * q;
    w1[nt] = pack2(k < NI ? p[OFF_W1 + k * H + n] : 0.f, k + 1 < NI ? p[OFF_W1 + (k + 1) * H + n] : 0.f);
    w3t[nt] = pack2(k < NO ? p[OFF_W3 + n * NO + k] : 0.f, k + 1 < NO ? p[OFF_W3 + n * NO + k + 1] : 0.f);
  }
#pragma unroll
  for (int kt = 0; kt < H / 16; ++kt)
#pragma unroll
    for (int hf = 0; hf < 2; ++hf) {
      const int k = 16 * kt + 8 * hf + 2 * q;
      w3[kt][hf] = pack2(g < NO ? p[OFF_W3 + k * NO + g] : 0.f, g < NO ? p[OFF_W3 + (k + 1) * NO + g] : 0.f);
    }
#pragma unroll
  for (int j = 0; j < 2; ++j) b3[j] = 2 * q + j < NO ? p[OFF_B3 + 2 * q + j] : 0.f;
  const float scale = 2.f / (float)(B * NO);
  SquareSum lsum;
  // gradients of this CTA, flushed once: rows 16w.. of dW2 (a2) and dW3 (a3),
  // columns 16w.. of dW1 (a1); sums of the deltas over 64 of the chunk's rows
  // for two columns of dz1 (warps 0, 1) or dz2 (warps 2, 3), and of dy
  float a1[2][4], a2[H / 8][4], a3[4], bs[2] = {0.f, 0.f}, bs3[3] = {0.f, 0.f, 0.f};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
#pragma unroll
    for (int nt = 0; nt < H / 8; ++nt) a2[nt][i] = 0.f;
    a1[0][i] = a1[1][i] = a3[i] = 0.f;
  }
  const uint32_t aw2 = saddr(s.w2), ah1 = saddr(s.h1), ah2 = saddr(s.h2), az1 = saddr(s.dz1), az2 = saddr(s.dz2),
                 ax = saddr(s.x), ady = saddr(s.dy);
  for (long long c0 = (long long)blockIdx.x * CH; c0 < B; c0 += (long long)gridDim.x * CH) {
    const int count = (int)(B - c0 < CH ? B - c0 : CH);
    __syncthreads();  // the previous chunk's weight gradients have read the arrays
    if constexpr (MODE == MODE_TB) {
      const int r = 32 * w + lane;
      if (r < count) {
        float a[3][3], Tb[6][6];
        const float* ar = Ag + (c0 + r) * 9;
#pragma unroll
        for (int i = 0; i < 9; ++i) a[i / 3][i % 3] = __ldg(ar + i);
        ps::tensor_basis(a, inv_sA, Tb);
#pragma unroll
        for (int i = 0; i < 36; ++i) s.tb[r * 37 + i] = Tb[i / 6][i % 6];
      }
    }
#pragma unroll 1
    for (int t = 0; t < 2; ++t) {
      const int r0 = 32 * w + 16 * t, ra = r0 + g, rb = ra + 8;  // this lane's rows
      uint32_t h[H / 16][4];
      float g1[H / 8][4], g2[H / 8][4];
      // inputs
      uint32_t xa, xb;
      {
        auto xin = [&](int r, int c) { return r < count && c < NI ? __ldg(X + (c0 + r) * NI + c) : 0.f; };
        xa = pack2(xin(ra, 2 * q), xin(ra, 2 * q + 1));
        xb = pack2(xin(rb, 2 * q), xin(rb, 2 * q + 1));
        uint32_t* xs = reinterpret_cast<uint32_t*>(s.x);
        xs[ra * 4 + q] = xa;
        xs[rb * 4 + q] = xb;
      }
      auto put = [&](bf* arr, int nt, uint32_t lo, uint32_t hi) {
        *reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(arr) + sw(ra, nt) + 4 * q) = lo;
        *reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(arr) + sw(rb, nt) + 4 * q) = hi;
      };
      __syncwarp();
      // layer 1
#pragma unroll
      for (int nt = 0; nt < H / 8; ++nt) {
        const float2 b = *reinterpret_cast<const float2*>(s.b1 + 8 * nt + 2 * q);
        float z[4] = {0.f, 0.f, 0.f, 0.f}, o[4];
        mma8(z, xa, xb, w1[nt]);
        z[0] += b.x;
        z[1] += b.y;
        z[2] += b.x;
        z[3] += b.y;
#pragma unroll
        for (int i = 0; i < 4; ++i) gelu_with_grad(z[i], o[i], g1[nt][i]);
        const uint32_t lo = pack2(o[0], o[1]), hi = pack2(o[2], o[3]);
        h[nt >> 1][(nt & 1) * 2 + 0] = lo;
        h[nt >> 1][(nt & 1) * 2 + 1] = hi;
        put(s.h1, nt, lo, hi);
      }
      // layer 2
      float acc[H / 8][4];
#pragma unroll
      for (int nt = 0; nt < H / 8; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
#pragma unroll
      for (int kt = 0; kt < H / 16; ++kt)
#pragma unroll
        for (int np = 0; np < H / 16; ++np) {
          uint32_t b[4];
          ldm4t(b, aw2 + sw(16 * kt + 8 * (mi & 1) + mr, 2 * np + (mi >> 1)));
          mma16(acc[2 * np], h[kt][0], h[kt][1], h[kt][2], h[kt][3], b[0], b[1]);
          mma16(acc[2 * np + 1], h[kt][0], h[kt][1], h[kt][2], h[kt][3], b[2], b[3]);
        }
#pragma unroll
      for (int nt = 0; nt < H / 8; ++nt) {
        const float2 b = *reinterpret_cast<const float2*>(s.b2 + 8 * nt + 2 * q);
        const float z[4] = {acc[nt][0] + b.x, acc[nt][1] + b.y, acc[nt][2] + b.x, acc[nt][3] + b.y};
        float o[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) gelu_with_grad(z[i], o[i], g2[nt][i]);
        const uint32_t lo = pack2(o[0], o[1]), hi = pack2(o[2], o[3]);
        h[nt >> 1][(nt & 1) * 2 + 0] = lo;
        h[nt >> 1][(nt & 1) * 2 + 1] = hi;
        put(s.h2, nt, lo, hi);
      }
      // layer 3
      float y[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int kt = 0; kt < H / 16; ++kt) mma16(y, h[kt][0], h[kt][1], h[kt][2], h[kt][3], w3[kt][0], w3[kt][1]);
      y[0] += b3[0];
      y[1] += b3[1];
      y[2] += b3[0];
      y[3] += b3[1];
      // output deltas (BF16, outputs 2q + {0, 1} of rows ra and rb)
      uint32_t da, db;
      if constexpr (MODE == MODE_TB) {
        // lane (sample i, half m): residuals of three stress components, then
        // three outputs' deltas 2/(6B) sum_m T_n,m e_m
        float* yf = s.yf[w];
        *reinterpret_cast<float2*>(yf + g * 8 + 2 * q) = make_float2(y[0], y[1]);
        *reinterpret_cast<float2*>(yf + (g + 8) * 8 + 2 * q) = make_float2(y[2], y[3]);
        __syncwarp();
        const int i = lane & 15, hf = lane >> 4, r = r0 + i;
        float dy[3] = {0.f, 0.f, 0.f};
        float e[6];
        const float* tb = s.tb + r * 37;
        if (r < count) {
#pragma unroll
          for (int m = 0; m < 3; ++m) {
            float mv = 0.f;
#pragma unroll
            for (int n = 0; n < NO; ++n) mv += tb[n * 6 + 3 * hf + m] * yf[i * 8 + n];
            e[m] = mv - __ldg(T + (c0 + r) * NO + 3 * hf + m) * inv_stau;
            lsum.add(e[m]);
          }
        } else {
          e[0] = e[1] = e[2] = 0.f;
        }
#pragma unroll
        for (int m = 0; m < 3; ++m) e[3 + m] = __shfl_xor_sync(0xffffffffu, e[m], 16);
        if (r < count) {
#pragma unroll
          for (int m = 0; m < 6; ++m) {
            const float em = (m < 3) == (hf == 0) ? e[m % 3] : e[3 + m % 3];
#pragma unroll
            for (int n = 0; n < 3; ++n) dy[n] += scale * tb[(3 * hf + n) * 6 + m] * em;
          }
        }
#pragma unroll
        for (int n = 0; n < 3; ++n) {
          const bf v = __float2bfloat16(dy[n]);
          bs3[n] += __bfloat162float(v);
          s.dy[r * 8 + 3 * hf + n] = v;
        }
        s.dy[r * 8 + 6 + hf] = __float2bfloat16(0.f);
        __syncwarp();
        const uint32_t* ds = reinterpret_cast<const uint32_t*>(s.dy);
        da = ds[ra * 4 + q];
        db = ds[rb * 4 + q];
      } else {
        float dv[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int r = i < 2 ? ra : rb, c = 2 * q + (i & 1);
          dv[i] = 0.f;
          if (c < NO && r < count) {
            const float tv = __ldg(T + (c0 + r) * NO + c);
            if constexpr (MODE == MODE_DY) {
              dv[i] = tv;
            } else {
              const float e = y[i] - tv;
              lsum.add(e);
              dv[i] = scale * e;
            }
          }
        }
        da = pack2(dv[0], dv[1]);
        db = pack2(dv[2], dv[3]);
        bs3[0] += lo_of(da) + lo_of(db);
        bs3[1] += hi_of(da) + hi_of(db);
        uint32_t* ds = reinterpret_cast<uint32_t*>(s.dy);
        ds[ra * 4 + q] = da;
        ds[rb * 4 + q] = db;
      }
      // dh2 = dy W3^T, dz2 = dh2 * gelu'(z2)
#pragma unroll
      for (int nt = 0; nt < H / 8; ++nt) {
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        mma8(d, da, db, w3t[nt]);
        const uint32_t lo = pack2(d[0] * g2[nt][0], d[1] * g2[nt][1]), hi = pack2(d[2] * g2[nt][2], d[3] * g2[nt][3]);
        h[nt >> 1][(nt & 1) * 2 + 0] = lo;
        h[nt >> 1][(nt & 1) * 2 + 1] = hi;
        put(s.dz2, nt, lo, hi);
      }
      // dh1 = dz2 W2^T, dz1 = dh1 * gelu'(z1)
#pragma unroll
      for (int nt = 0; nt < H / 8; ++nt) acc[nt][0] = acc[nt][1] = acc[nt][2] = acc[nt][3] = 0.f;
#pragma unroll
      for (int kt = 0; kt < H / 16; ++kt)
#pragma unroll
        for (int np = 0; np < H / 16; ++np) {
          uint32_t b[4];
          ldm4(b, aw2 + sw(16 * np + 8 * (mi >> 1) + mr, 2 * kt + (mi & 1)));
          mma16(acc[2 * np], h[kt][0], h[kt][1], h[kt][2], h[kt][3], b[0], b[1]);
          mma16(acc[2 * np + 1], h[kt][0], h[kt][1], h[kt][2], h[kt][3], b[2], b[3]);
        }
#pragma unroll
      for (int nt = 0; nt < H / 8; ++nt)
        put(s.dz1, nt, pack2(acc[nt][0] * g1[nt][0], acc[nt][1] * g1[nt][1]),
            pack2(acc[nt][2] * g1[nt][2], acc[nt][3] * g1[nt][3]));
    }
    __syncthreads();
    // weight gradients over the chunk's samples (padded rows have zero deltas):
    // dW2 = h1^T dz2, dW3 = h2^T dy, dW1 = x^T dz1
#pragma unroll 2
    for (int kt = 0; kt < CH / 16; ++kt) {
      uint32_t a[4], b[4];
      ldm4t(a, ah1 + sw(16 * kt + 8 * (mi >> 1) + mr, 2 * w + (mi & 1)));
#pragma unroll
      for (int np = 0; np < H / 16; ++np) {
        ldm4t(b, az2 + sw(16 * kt + 8 * (mi & 1) + mr, 2 * np + (mi >> 1)));
        mma16(a2[2 * np], a[0], a[1], a[2], a[3], b[0], b[1]);
        mma16(a2[2 * np + 1], a[0], a[1], a[2], a[3], b[2], b[3]);
      }
      uint32_t v[2];
      ldm4t(a, ah2 + sw(16 * kt + 8 * (mi >> 1) + mr, 2 * w + (mi & 1)));
      ldm2t(v, ady + (16 * kt + 8 * (mi & 1) + mr) * 16);
      mma16(a3, a[0], a[1], a[2], a[3], v[0], v[1]);
      ldm2t(v, ax + (16 * kt + 8 * (mi & 1) + mr) * 16);
      ldm4t(b, az1 + sw(16 * kt + 8 * (mi & 1) + mr, 2 * w + (mi >> 1)));
      mma16(a1[0], v[0], 0u, v[1], 0u, b[0], b[1]);
      mma16(a1[1], v[0], 0u, v[1], 0u, b[2], b[3]);
    }
    // bias gradients: column sums of the deltas as stored (BF16), like the
    // weight gradients that use them
    {
      const char* arr = reinterpret_cast<const char*>(w < 2 ? s.dz1 : s.dz2);
#pragma unroll 8
      for (int i = 0; i < CH / 2; ++i) {
        const int r = (w & 1) * (CH / 2) + i;
        const uint32_t v = *reinterpret_cast<const uint32_t*>(arr + sw(r, lane >> 2) + 4 * (lane & 3));
        bs[0] += lo_of(v);
        bs[1] += hi_of(v);
      }
    }
  }
  // flush this CTA's gradients
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = g + 8 * (i >> 1), c = 2 * q + (i & 1);
#pragma unroll
    for (int nt = 0; nt < H / 8; ++nt) atomicAdd(grad + OFF_W2 + (16 * w + r) * H + 8 * nt + c, a2[nt][i]);
    if (c < NO) atomicAdd(grad + OFF_W3 + (16 * w + r) * NO + c, a3[i]);
    if (r < NI) {
      atomicAdd(grad + OFF_W1 + r * H + 16 * w + c, a1[0][i]);
      atomicAdd(grad + OFF_W1 + r * H + 16 * w + 8 + c, a1[1][i]);
    }
  }
  atomicAdd(grad + (w < 2 ? OFF_B1 : OFF_B2) + 2 * lane, bs[0]);
  atomicAdd(grad + (w < 2 ? OFF_B1 : OFF_B2) + 2 * lane + 1, bs[1]);
  if constexpr (MODE == MODE_TB) {
    // lanes of one half hold outputs 3 hf + {0, 1, 2}
#pragma unroll
    for (int n = 0; n < 3; ++n) {
      float v = bs3[n];
#pragma unroll
      for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if ((lane & 15) == 0) atomicAdd(grad + OFF_B3 + 3 * (lane >> 4) + n, v);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      float v = bs3[j];
#pragma unroll
      for (int o = 16; o > 2; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (g == 0 && 2 * q + j < NO) atomicAdd(grad + OFF_B3 + 2 * q + j, v);
    }
  }
  // loss
  if constexpr (MODE != MODE_DY) {
    double l = lsum.total();
    for (int o = 16; o > 0; o >>= 1) l += __shfl_xor_sync(0xffffffffu, l, o);
    if (lane == 0) atomicAdd(loss, l / (double)(B * NO));
  }
}

__global__ void k_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int n, float lr, float b1, float b2, float eps, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

int grid_for(long long B) {
  int dev = 0, nsm = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const long long chunks = (B + CH - 1) / CH;
  const long long g = 2LL * nsm;
  return (int)(chunks < g ? chunks : g);
}

ps_status cuerr(cudaError_t e, const char* what) {
  if (e == cudaSuccess) return PS_OK;
  ps::set_last_error(std::string(what) + ": " + cudaGetErrorString(e));
  return PS_ERR_CUDA;
}

}  // namespace

extern "C" {

ps_status ps_mlp_forward(const float* params, const float* X, float* Y, long long count, void* stream) {
  if (!params || !X || !Y || count < 0) {
    ps::set_last_error("ps_mlp_forward: NULL buffer or negative count");
    return PS_ERR_INVALID_ARG;
  }
  if (count == 0) return PS_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  k_mlp_forward<<<grid_for(count), 128, 0, s>>>(params, X, Y, count);
  return cuerr(cudaGetLastError(), "ps_mlp_forward");
}

ps_status ps_mlp_grad(const float* params, const float* X, const float* T, long long count, float* grad,
                      double* loss, void* stream) {
  if (!params || !X || !T || !grad || !loss || count <= 0) {
    ps::set_last_error("ps_mlp_grad: NULL buffer or non-positive count");
    return PS_ERR_INVALID_ARG;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemsetAsync(grad, 0, sizeof(float) * NPARAM, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(loss, 0, sizeof(double), s);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mlp_grad<MODE_PLAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
  if (e != cudaSuccess) return cuerr(e, "ps_mlp_grad");
  k_mlp_grad<MODE_PLAIN><<<grid_for(count), 128, sizeof(Smem), s>>>(params, X, nullptr, T, count, 1.f, 1.f, grad, loss);
  return cuerr(cudaGetLastError(), "ps_mlp_grad");
}

ps_status ps_mlp_grad_tb(const float* params, const float* X, const float* A, const float* T, long long count,
                         double s_A, double s_tau, float* grad, double* loss, void* stream) {
  if (!params || !X || !A || !T || !grad || !loss || count <= 0) {
    ps::set_last_error("ps_mlp_grad_tb: NULL buffer or non-positive count");
    return PS_ERR_INVALID_ARG;
  }
  if (!(s_A > 0) || !(s_tau > 0) || !std::isfinite(s_A) || !std::isfinite(s_tau)) {
    ps::set_last_error("ps_mlp_grad_tb: scales must be positive and finite");
    return PS_ERR_INVALID_ARG;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaMemsetAsync(grad, 0, sizeof(float) * NPARAM, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(loss, 0, sizeof(double), s);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_mlp_grad<MODE_TB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
  if (e != cudaSuccess) return cuerr(e, "ps_mlp_grad_tb");
  k_mlp_grad<MODE_TB><<<grid_for(count), 128, sizeof(Smem), s>>>(params, X, A, T, count, (float)(1.0 / s_A),
                                                              (float)(1.0 / s_tau), grad, loss);
  return cuerr(cudaGetLastError(), "ps_mlp_grad_tb");
}

ps_status ps_mlp_backward(const float* params, const float* X, const float* dY, long long count, float* grad,
                          void* stream) {
  if (!params || !X || !dY || !grad || count < 0) {
    ps::set_last_error("ps_mlp_backward: NULL buffer or negative count");
    return PS_ERR_INVALID_ARG;
  }
  if (count == 0) return PS_OK;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e =
      cudaFuncSetAttribute(k_mlp_grad<MODE_DY>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
  if (e != cudaSuccess) return cuerr(e, "ps_mlp_backward");
  k_mlp_grad<MODE_DY><<<grid_for(count), 128, sizeof(Smem), s>>>(params, X, nullptr, dY, count, 1.f, 1.f, grad,
                                                                 nullptr);
  return cuerr(cudaGetLastError(), "ps_mlp_backward");
}

ps_status ps_mlp_adam(float* params, const float* grad, float* m, float* v, int step, float lr, float beta1,
                      float beta2, float eps, void* stream) {
  if (!params || !grad || !m || !v || step < 1) {
    ps::set_last_error("ps_mlp_adam: NULL buffer or step < 1");
    return PS_ERR_INVALID_ARG;
  }
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  k_adam<<<(NPARAM + 255) / 256, 256, 0, static_cast<cudaStream_t>(stream)>>>(params, grad, m, v, NPARAM, lr,
                                                                             beta1, beta2, eps, c1, c2);
  return cuerr(cudaGetLastError(), "ps_mlp_adam");
}

}  // extern "C"
