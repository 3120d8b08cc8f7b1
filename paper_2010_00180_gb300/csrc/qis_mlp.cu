// qis_mlp.cu -- learned warm start: a per-site MLP that proposes initial states.
//
// The QI search starts every search from a random state (rand_between of Alg. 4). Here a
// small network maps features of each site (h_i and statistics of row i of J) to a logit
// z_i of P(s_i = +1); the R initial states of an instance are its argmax (search 0) and
// Bernoulli draws from sigmoid(z) (searches 1..R-1). The network is trained on the GPU by
// the kernels below on states the search itself found; random initial states remain the
// default and the reference for comparison.
//
// Network: F = 8 features -> H -> H -> H -> 1, ReLU, BF16 weights (rounded from an FP32
// master copy after every update), FP32 activations and accumulation, BCE loss, Adam.
// Features (FP64, then FP32): h_i, sum_j J_ij / sqrt n, sum_j |J_ij| / n,
// sqrt(sum_j J_ij^2 / n), max_{j!=i} J_ij, min_{j!=i} J_ij, sum_j J_ij h_j / sqrt n,
// sum_j J_ij sign(h_j) / sqrt n.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <string>
#include <vector>

#include "qis_common.cuh"

namespace qis {

constexpr int kF = 8;   // features per site

// ---------------------------------------------------------------- features
// J row i at J + i * stride (n valid entries), h[0..n). A warp per row, its lanes over the columns
// (a thread per row read them uncoalesced, a chain of n FP64 additions: 148 us at n = 300, now 16).
// |v|, the signs of h and the extrema are integer operations on the bits (FP64 has two lanes per SM).
__global__ void __launch_bounds__(256) k_mlp_features(const double* J, long long stride, const double* h, int n, float* X) {
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (i >= n) return;   // warp-uniform
  const double* row = J + (long long)i * stride;
  double s = 0, a = 0, q = 0, jh = 0, js = 0;
  unsigned long long mx = 0, mn = ~0ull;   // order keys of the extrema over j != i
#pragma unroll 4
  for (int j = lane; j < n; j += 32) {
    const double v = row[j], hj = h[j];
    s += v;
    a += fabs(v);
    q = fma(v, v, q);
    jh = fma(v, hj, jh);
    const long long hb = __double_as_longlong(hj);
    if (hb << 1) js += hb < 0 ? -v : v;   // h_j != 0
    const unsigned long long k = dkey(v);
    if (j != i) {
      mx = max(mx, k);
      mn = min(mn, k);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s += __shfl_xor_sync(0xffffffffu, s, o);
    a += __shfl_xor_sync(0xffffffffu, a, o);
    q += __shfl_xor_sync(0xffffffffu, q, o);
    jh += __shfl_xor_sync(0xffffffffu, jh, o);
    js += __shfl_xor_sync(0xffffffffu, js, o);
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    mn = min(mn, __shfl_xor_sync(0xffffffffu, mn, o));
  }
  if (lane) return;
  const double rn = sqrt((double)n);
  float* x = X + (long long)i * kF;
  x[0] = (float)h[i];
  x[1] = (float)(s / rn);
  x[2] = (float)(a / n);
  x[3] = (float)sqrt(q / n);
  x[4] = (float)dkey_inv(mx);
  x[5] = (float)dkey_inv(mn);
  x[6] = (float)(jh / rn);
  x[7] = (float)(js / rn);
}

__global__ void k_mlp_labels(const uint64_t* bits, int n, float* y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) y[i] = ((bits[i >> 6] >> (i & 63)) & 1ull) ? 0.f : 1.f;   // y = 1 <=> s_i = +1
}

// ---------------------------------------------------------------- network
// out = in W for TM rows of activations in shared memory (in: TM x K, row-major) and BF16 weights W
// (K x H, row-major). A warp takes RT rows x 128 columns, a lane 4 adjacent columns: one weight
// load per k serves RT rows, the activations are broadcast reads, and every sum is one chain of
// FP32 fused multiply-adds over k ascending (the logits' bits do not depend on the tile). The
// next D rows of W are loaded while the current D are used. put(row, column, the sums of
// 4 columns) receives the results; in and the results must not share memory.
constexpr int kCT = 4;   // columns of a lane
template <int RT, int D, typename Put>
static __device__ __forceinline__ void mlp_layer(const float* in, int K, const __nv_bfloat16* __restrict__ W, int H, int TM,
                                                 Put put) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int CG = (H + 32 * kCT - 1) / (32 * kCT);
  for (int u = warp; u < TM / RT * CG; u += 8) {
    const int r0 = u / CG * RT, c = (u % CG) * 32 * kCT + lane * kCT;
    if (c >= H) continue;   // H is a multiple of 16: a lane's columns are all in or all out
    float acc[RT][kCT];
#pragma unroll
    for (int r = 0; r < RT; ++r)
#pragma unroll
      for (int x = 0; x < kCT; ++x) acc[r][x] = 0.f;
    uint2 w[D];
#pragma unroll
    for (int k = 0; k < D; ++k)
      if (k < K) w[k] = *reinterpret_cast<const uint2*>(W + (long long)k * H + c);
#pragma unroll 1
    for (int k0 = 0; k0 < K; k0 += D) {
      uint2 v[D];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        v[k] = w[k];
        if (k0 + D + (k & ~7) < K) w[k] = *reinterpret_cast<const uint2*>(W + (long long)(k0 + D + k) * H + c);
      }
#pragma unroll
      for (int k4 = 0; k4 < D; k4 += 4) {
        if (D > 8 && k0 + k4 >= K) break;   // (K is a multiple of 8)
        float4 a[RT];
#pragma unroll
        for (int r = 0; r < RT; ++r) a[r] = *reinterpret_cast<const float4*>(in + (r0 + r) * K + k0 + k4);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const uint32_t* p = reinterpret_cast<const uint32_t*>(&v[k4 + k]);
          float b[kCT];
#pragma unroll
          for (int x = 0; x < kCT; x += 2) {
            b[x] = __uint_as_float(p[x / 2] << 16);
            b[x + 1] = __uint_as_float(p[x / 2] & 0xffff0000u);
          }
#pragma unroll
          for (int r = 0; r < RT; ++r) {
            const float ar = k == 0 ? a[r].x : k == 1 ? a[r].y : k == 2 ? a[r].z : a[r].w;
#pragma unroll
            for (int x = 0; x < kCT; ++x) acc[r][x] = fmaf(ar, b[x], acc[r][x]);
          }
        }
      }
    }
#pragma unroll
    for (int r = 0; r < RT; ++r) put(r0 + r, c, acc[r]);
  }
}

// Everything of a pass but the weight gradients, for TM rows per block: the three layers, the logits,
// and with labels y the loss (added to *loss) and the gradients of the pre-activations d3, d2, d1
// (d_l = (d_{l+1} W_{l+1}^T) where h_l > 0, with the transposed weights W2t, W3t), all from one
// block's shared memory; h1, h2, h3 and d1, d2, d3 are written for the weight gradients. G (grads
// values, or NULL) is cleared for them.
// FP32 issue bounds it (M (4 H^2 + ..) multiply-adds); it replaces eleven launches whose tiles of
// 64 x 64 fed four accumulators per shared-memory read. Loss and gradients of 4096 rows at H = 256
// from host memory, with the weight gradients' kernel below (which took 3 x 90 us): 542 -> 195 us;
// warm start of 120 instances of n = 300 and their searches: 44.1 -> 14.7 ms with the search kernel of
// that time.
struct MlpNet {
  const float* P;                   // master parameters (biases are read from it)
  const __nv_bfloat16 *Pb, *W2t, *W3t;
  int H, oW1, ob1, oW2, ob2, oW3, ob3, ow4, ob4;
};

template <int TM, int RT, int D>
__global__ void __launch_bounds__(256) k_mlp_pass(MlpNet N, int M, const float* X, const float* y, float* z, float* dz,
                                                  double* loss, float inv_m, float* h1, float* h2, float* h3, float* d1,
                                                  float* d2, float* d3, float* G, int grads) {
  extern __shared__ __align__(16) float act[];
  const int H = N.H, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  float* A = act;              // [TM][H]
  float* B = act + TM * H;     // [TM][H]
  __shared__ float sdz[TM];
  __shared__ double sl[TM];
  const int m0 = blockIdx.x * TM, rows = min(TM, M - m0);
  if (G)
    for (int e = blockIdx.x * 256 + tid; e < grads; e += gridDim.x * 256) G[e] = 0.f;
  for (int e = tid; e < TM * kF; e += 256) B[e] = e < rows * kF ? X[(long long)m0 * kF + e] : 0.f;
  __syncthreads();
  // h = relu(in W + b) into `out`, and to global memory for a pass with labels
  auto forward = [&](const float* in, int K, int oW, int ob, float* out, float* h) {
    mlp_layer<RT, D>(in, K, N.Pb + oW, H, TM, [&](int r, int c, const float* s) {
#pragma unroll
      for (int x = 0; x < kCT; x += 4) {
        const float4 b = *reinterpret_cast<const float4*>(N.P + ob + c + x);
        const float4 v = make_float4(fmaxf(s[x] + b.x, 0.f), fmaxf(s[x + 1] + b.y, 0.f), fmaxf(s[x + 2] + b.z, 0.f),
                                     fmaxf(s[x + 3] + b.w, 0.f));
        *reinterpret_cast<float4*>(out + r * H + c + x) = v;
        if (y && r < rows) *reinterpret_cast<float4*>(h + (long long)(m0 + r) * H + c + x) = v;
      }
    });
    __syncthreads();
  };
  forward(B, kF, N.oW1, N.ob1, A, h1);
  forward(A, H, N.oW2, N.ob2, B, h2);
  forward(B, H, N.oW3, N.ob3, A, h3);
  // z = h3 w4 + b4, loss and dz = (sigmoid(z) - y) / M: a warp per row
  const __nv_bfloat16* w4 = N.Pb + N.ow4;
  for (int r = warp; r < TM; r += 8) {
    float s = 0.f;
    for (int k = lane; k < H; k += 32) s = fmaf(A[r * H + k], __bfloat162float(w4[k]), s);
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      const float zz = s + N.P[N.ob4];
      float g = 0.f;
      double l = 0.0;
      if (r < rows) {
        z[m0 + r] = zz;
        if (y) {
          const float yy = y[m0 + r];
          const float sp = fmaxf(zz, 0.f) + log1pf(expf(-fabsf(zz)));   // softplus
          l = (double)(sp - yy * zz) * inv_m;
          g = (1.f / (1.f + expf(-zz)) - yy) * inv_m;
          dz[m0 + r] = g;
        }
      }
      sdz[r] = g;
      sl[r] = l;
    }
  }
  if (!y) return;
  __syncthreads();
  if (tid == 0) {
    double l = 0.0;
    for (int r = 0; r < rows; ++r) l += sl[r];
    atomicAdd(loss, l);
  }
  // d3 = outer(dz, w4) where h3 > 0, in the place of h3
  for (int e = tid; e < TM * H; e += 256) {
    const int r = e / H, k = e - r * H;
    const float v = A[e] > 0.f ? sdz[r] * __bfloat162float(w4[k]) : 0.f;
    A[e] = v;
    if (r < rows) d3[(long long)m0 * H + e] = v;
  }
  __syncthreads();
  auto backward = [&](const float* in, const __nv_bfloat16* Wt, const float* h, float* out, float* d) {
    mlp_layer<RT, D>(in, H, Wt, H, TM, [&](int r, int c, const float* s) {
#pragma unroll
      for (int x = 0; x < kCT; x += 4) {
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < rows) {
          const long long at = (long long)(m0 + r) * H + c + x;
          const float4 g = *reinterpret_cast<const float4*>(h + at);   // (this block's own rows)
          v = make_float4(g.x > 0.f ? s[x] : 0.f, g.y > 0.f ? s[x + 1] : 0.f, g.z > 0.f ? s[x + 2] : 0.f,
                          g.w > 0.f ? s[x + 3] : 0.f);
          *reinterpret_cast<float4*>(d + at) = v;
        }
        *reinterpret_cast<float4*>(out + r * H + c + x) = v;
      }
    });
    __syncthreads();
  };
  backward(A, N.W3t, h2, B, d2);
  backward(B, N.W2t, h1, A, d1);
}

// ---------------------------------------------------------------- weight gradients
// dW3 = h2^T d3, dW2 = h1^T d2 (128 x 64 tiles, the rows of the batch split over blockIdx.y, the
// parts added with vector atomics), db3, db2 (the column sums of the staged d tiles, by the blocks
// of the first tile row), and in the blocks past those tiles dW1 = X^T d1, db1, dw4 = h3^T dz, db4
// (128 rows each, a thread per column). G is zero on entry.
constexpr int kWM = 128, kWN = 64, kWK = 16;
__global__ void __launch_bounds__(256) k_mlp_wgrad(MlpNet N, int M, int rows_per, const float* X, const float* h1,
                                                   const float* h2, const float* h3, const float* d1, const float* d2,
                                                   const float* d3, const float* dz, float* G) {
  const int H = N.H, tid = threadIdx.x;
  const int tm = (H + kWM - 1) / kWM, tn = (H + kWN - 1) / kWN, tiles = 2 * tm * tn;
  __shared__ __align__(16) float As[2][kWK][kWM], Bs[2][kWK][kWN];
  if ((int)blockIdx.x >= tiles) {
    // the thin gradients: column c of 128 rows
    const int x = blockIdx.x - tiles, cgs = (H + 255) / 256;
    const int c = (x % cgs) * 256 + tid;
    const int r0 = ((x / cgs) * gridDim.y + blockIdx.y) * 128, r1 = min(M, r0 + 128);
    if (r0 >= M) return;   // block-uniform
    float* xs = &As[0][0][0];   // [128][8] features, then [128] dz
    float* zs = xs + 128 * kF;
    for (int e = tid; e < (r1 - r0) * kF; e += 256) xs[e] = X[(long long)r0 * kF + e];
    for (int e = tid; e < r1 - r0; e += 256) zs[e] = dz[r0 + e];
    __syncthreads();
    if (c < H) {
      float g[kF] = {}, gb = 0.f, g4 = 0.f;
#pragma unroll 4
      for (int r = r0; r < r1; ++r) {
        const float d = d1[(long long)r * H + c], hh = h3[(long long)r * H + c];
        gb += d;
        g4 = fmaf(hh, zs[r - r0], g4);
#pragma unroll
        for (int f = 0; f < kF; ++f) g[f] = fmaf(xs[(r - r0) * kF + f], d, g[f]);
      }
#pragma unroll
      for (int f = 0; f < kF; ++f) atomicAdd(&G[N.oW1 + f * H + c], g[f]);
      atomicAdd(&G[N.ob1 + c], gb);
      atomicAdd(&G[N.ow4 + c], g4);
    }
    if (x % cgs == 0 && tid < 32) {
      float s = 0.f;
      for (int r = tid; r < r1 - r0; r += 32) s += zs[r];
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
      if (tid == 0) atomicAdd(&G[N.ob4], s);
    }
    return;
  }
  const int layer = blockIdx.x / (tm * tn), t = blockIdx.x % (tm * tn);
  const int m0 = t / tn * kWM, n0 = t % tn * kWN;
  const float* A = layer ? h1 : h2;
  const float* D = layer ? d2 : d3;
  const int r0 = blockIdx.y * rows_per, r1 = min(M, r0 + rows_per);
  if (r0 >= M) return;   // block-uniform
  const int tx = tid & 15, ty = tid >> 4;
  float4 ra[2], rb;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
  auto fetch = [&](int k0) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = tid + 256 * u, r = k0 + (e >> 5), c = m0 + (e & 31) * 4;
      ra[u] = r < r1 && c < H ? *reinterpret_cast<const float4*>(A + (long long)r * H + c) : zero;
    }
    const int r = k0 + (tid >> 4), c = n0 + (tid & 15) * 4;
    rb = r < r1 && c < H ? *reinterpret_cast<const float4*>(D + (long long)r * H + c) : zero;
  };
  float acc[8][4] = {};
  float gb = 0.f;
  fetch(r0);
  int buf = 0;
  for (int k0 = r0; k0 < r1; k0 += kWK, buf ^= 1) {
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int e = tid + 256 * u;
      *reinterpret_cast<float4*>(&As[buf][e >> 5][(e & 31) * 4]) = ra[u];
    }
    *reinterpret_cast<float4*>(&Bs[buf][tid >> 4][(tid & 15) * 4]) = rb;
    __syncthreads();   // (two buffers: the writes of the next step follow this step's reads)
    if (k0 + kWK < r1) fetch(k0 + kWK);
#pragma unroll
    for (int k = 0; k < kWK; ++k) {
      const float4 b = *reinterpret_cast<const float4*>(&Bs[buf][k][tx * 4]);
      const float4 a0 = *reinterpret_cast<const float4*>(&As[buf][k][ty * 8]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[buf][k][ty * 8 + 4]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        acc[u][0] = fmaf(a[u], b.x, acc[u][0]);
        acc[u][1] = fmaf(a[u], b.y, acc[u][1]);
        acc[u][2] = fmaf(a[u], b.z, acc[u][2]);
        acc[u][3] = fmaf(a[u], b.w, acc[u][3]);
      }
    }
    if (m0 == 0 && tid < kWN)
#pragma unroll
      for (int k = 0; k < kWK; ++k) gb += Bs[buf][k][tid];
  }
  float* g = G + (layer ? N.oW2 : N.oW3);
  if (n0 + tx * 4 < H)
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int m = m0 + ty * 8 + u;
      if (m < H)
        atomicAdd(reinterpret_cast<float4*>(g + (long long)m * H + n0 + tx * 4),
                  make_float4(acc[u][0], acc[u][1], acc[u][2], acc[u][3]));
    }
  if (m0 == 0 && tid < kWN && n0 + tid < H) atomicAdd(&G[(layer ? N.ob2 : N.ob3) + n0 + tid], gb);
}

// BF16 copies of parameter e of value p: the flat copy, and the transposed ones of W2 and W3.
__device__ __forceinline__ void mlp_copy_bf16(const MlpNet& N, int e, float p, __nv_bfloat16* Pb, __nv_bfloat16* W2t,
                                              __nv_bfloat16* W3t) {
  const __nv_bfloat16 q = __float2bfloat16_rn(p);
  Pb[e] = q;
  const int H = N.H, a = e - N.oW2, b = e - N.oW3;
  if (a >= 0 && a < H * H) W2t[a % H * H + a / H] = q;
  if (b >= 0 && b < H * H) W3t[b % H * H + b / H] = q;
}

__global__ void k_adam(MlpNet N, int count, float* p, const float* g, float* m, float* v, float lr, float b1, float b2,
                       float eps, float c1, float c2, __nv_bfloat16* Pb, __nv_bfloat16* W2t, __nv_bfloat16* W3t) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= count) return;
  const float gg = g[e];
  const float mm = b1 * m[e] + (1.f - b1) * gg;
  const float vv = b2 * v[e] + (1.f - b2) * gg * gg;
  m[e] = mm;
  v[e] = vv;
  const float x = p[e] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
  p[e] = x;
  mlp_copy_bf16(N, e, x, Pb, W2t, W3t);
}

__global__ void k_to_bf16(MlpNet N, int count, const float* p, __nv_bfloat16* Pb, __nv_bfloat16* W2t, __nv_bfloat16* W3t) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < count) mlp_copy_bf16(N, e, p[e], Pb, W2t, W3t);
}

// Initial states from logits: search 0 takes s_i = sign(z_i) (s_i = +1 when z_i >= 0), search
// r >= 1 draws s_i = +1 with probability sigmoid(z_i) using value (r n + i) of the SplitMix64
// stream keyed by `key` (the top 53 bits as a uniform in [0, 1)).
// A warp per 32 sites and 8 searches: a lane forms its site's probability once, the ballot of the
// lanes is half a word (a thread per word drew 64 sites in a row: 62 us at n = 300, R = 32, now 4).
constexpr int kSampleR = 8;
__global__ void __launch_bounds__(32) k_mlp_sample(const float* z, int n, int R, uint64_t key, uint64_t* bits, int Wstride) {
  const int half = blockIdx.x, i = half * 32 + (int)threadIdx.x;
  const float zi = i < n ? z[i] : 0.f;
  const double p = 1.0 / (1.0 + exp(-(double)zi));
  for (int r = blockIdx.y * kSampleR; r < min(R, (int)(blockIdx.y + 1) * kSampleR); ++r) {
    bool sigma;
    if (r == 0) {
      sigma = zi < 0.f;
    } else {
      const double u = (double)(splitmix64(key, (uint64_t)r * n + i) >> 11) * 0x1.0p-53;
      sigma = !(u < p);
    }
    const unsigned m = __ballot_sync(0xffffffffu, sigma && i < n);
    if (threadIdx.x == 0) reinterpret_cast<uint32_t*>(bits + (long long)r * Wstride)[half] = m;   // little-endian halves
  }
}

}  // namespace qis

using namespace qis;

struct qis_mlp {
  qis_mlp_config cfg{};
  int H = 256, F = kF, cap = 0, batch = 0, max_n = 0;
  int n_params = 0;
  cudaStream_t stream = nullptr;
  std::vector<void*> allocs;
  float* P = nullptr;          // master parameters, flattened W1 b1 W2 b2 W3 b3 w4 b4
  float* G = nullptr;          // gradients
  float* Mm = nullptr;         // Adam first moment
  float* Vv = nullptr;         // Adam second moment
  __nv_bfloat16* Pb = nullptr; // BF16 copy of all parameters (biases read from P)
  __nv_bfloat16 *W2t = nullptr, *W3t = nullptr;   // BF16 copies of W2 and W3, transposed
  float* X = nullptr;          // training features [cap x F]
  float* Y = nullptr;          // labels [cap]
  int n_examples = 0;          // rows of X / Y in use
  float *h1 = nullptr, *h2 = nullptr, *h3 = nullptr, *d1 = nullptr, *d2 = nullptr, *d3 = nullptr, *zb = nullptr, *dzb = nullptr;
  double* loss = nullptr;
  double* Jst = nullptr;       // staging of one instance's couplings [max_n^2]
  double* hst = nullptr;
  uint64_t* bst = nullptr;
  float* Xq = nullptr;         // query features [max_n x F]
  float* Yq = nullptr;         // labels of a query
  cudaEvent_t busy = nullptr;  // the last use of the network's buffers on a context's stream
  int sms = 0;
  int adam_t = 0;
  std::string err = "no error";
  // offsets into the flattened parameter vector
  int oW1, ob1, oW2, ob2, oW3, ob3, ow4, ob4;
};

namespace {
int mfail(qis_mlp* m, int code, const std::string& msg) {
  if (m) m->err = msg;
  else set_global_error(msg.c_str());
  return code;
}
#define MCK(call)                                                                            \
  do {                                                                                       \
    cudaError_t e_ = (call);                                                                 \
    if (e_ != cudaSuccess) {                                                                 \
      cudaGetLastError(); /* consume it: a later call must not see this error */              \
      return mfail(m, QIS_ERR_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_));     \
    }                                                                                        \
  } while (0)

template <typename T>
int malloc_m(qis_mlp* m, T** p, size_t count) {
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), (count ? count : 1) * sizeof(T));
  if (e != cudaSuccess) {
    cudaGetLastError();
    return mfail(m, QIS_ERR_OOM, "cudaMalloc failed");
  }
  m->allocs.push_back(*p);
  cudaMemset(*p, 0, (count ? count : 1) * sizeof(T));
  return 0;
}
#define MALLOC(ptr, count)                      \
  do {                                          \
    int rc_ = malloc_m(m, &(ptr), (count));     \
    if (rc_) return rc_;                        \
  } while (0)

MlpNet net_of(const qis_mlp* m) {
  return MlpNet{m->P, m->Pb, m->W2t, m->W3t, m->H, m->oW1, m->ob1, m->oW2, m->ob2, m->oW3, m->ob3, m->ow4, m->ob4};
}

template <int TM, int RT, int D>
cudaError_t pass_tm(qis_mlp* m, int M, const float* X, const float* y, cudaStream_t s) {
  const size_t sm = (size_t)2 * TM * m->H * sizeof(float);
  // (a launch without the attribute gets 48 KiB with the kernel's static arrays, not beside them)
  const cudaError_t e = allow_smem((const void*)k_mlp_pass<TM, RT, D>, sm);
  if (e != cudaSuccess) return e;
  k_mlp_pass<TM, RT, D><<<(M + TM - 1) / TM, 256, sm, s>>>(net_of(m), M, X, y, m->zb, m->dzb, m->loss, 1.f / (float)M, m->h1,
                                                            m->h2, m->h3, m->d1, m->d2, m->d3, y ? m->G : nullptr,
                                                            m->n_params);
  return cudaGetLastError();
}

// Rows X[0..M): the logits, and with labels the loss and the gradients of the pre-activations (G
// cleared). Rows per block: few for small batches, whose latency is the blocks' own work, more
// where a weight load then serves more rows and the SMs are still full. Measured, call of
// qis_mlp_forward at H = 256 with 4 / 8 / 16 / 32 (8 columns a lane) rows: M = 300 45 / 47 / 58 /
// 72 us, M = 2000 72 / 60 / 60 / 73, M = 4096 104 / 92 / 72 / 81; of qis_mlp_loss_grad M = 700 111 /
// 114 / 135 / 172, M = 2000 160 / 127 / 142 / 176, M = 4096 232 / 207 / 180 / 194.
// With one block of 4 rows per SM at most, its loads from L2 bound it and 32 rows of W are in flight
// (163 registers); beyond that two blocks per SM have to fit (56 registers with 8). 32 / 8 at M = 300:
// qis_mlp_loss_grad H = 256 97 / 110 us, H = 512 220 / 267, qis_mlp_forward H = 512 82 / 107; at M = 700
// qis_mlp_loss_grad H = 256 135 / 112. Warm starts of 120 instances of n = 300 and their searches
// 12.4 / 13.0 ms.
// Widths above 512 have more than four groups of columns, so a warp that takes one or two rows of a block
// reads the weights once for each of several units of work; it takes all of the block's rows there.
// Calls of qis_mlp_forward / qis_mlp_loss_grad in us, with the forms of narrow networks and so (in
// brackets the layers as launches of their own, which both replaced): H = 1024 M = 1 242 / 814 and 118 / 552
// (209 / 630), M = 700 345 / 966 and 181 / 581 (326 / 1158), M = 4096 944 / 2503 and 539 / 1615 (938 / 3194);
// H = 768 M = 700 207 / 539 and 143 / 402 (192 / 703), M = 4096 378 / 1079 and 399 / 1079 (639 / 2104); H = 640
// M = 300 120 / 330 and 81 / 252 (163 / 570), M = 2000 213 / 566 and 160 / 451 (288 / 1028).
cudaError_t mlp_pass(qis_mlp* m, int M, const float* X, const float* y, cudaStream_t s) {
  if (m->H > 512) return M <= 4 * m->sms ? pass_tm<4, 4, 16>(m, M, X, y, s) : pass_tm<8, 8, 8>(m, M, X, y, s);
  if (M <= 4 * m->sms) return pass_tm<4, 1, 32>(m, M, X, y, s);
  if (M <= 8 * m->sms) return pass_tm<4, 1, 8>(m, M, X, y, s);
  if (M <= 18 * m->sms) return pass_tm<8, 2, 8>(m, M, X, y, s);
  return pass_tm<16, 4, 8>(m, M, X, y, s);
}

// Gradients of the mean loss over the rows of the last mlp_pass with labels, into G.
cudaError_t mlp_weight_grads(qis_mlp* m, int M, const float* X, cudaStream_t s) {
  const int H = m->H, tiles = 2 * ((H + kWM - 1) / kWM) * ((H + kWN - 1) / kWN);
  // the batch split so that two blocks share an SM, 32 rows at least
  const int parts = std::max(1, std::min(std::min(2 * m->sms / tiles, (M + 31) / 32), 64));
  const int per = ((M + parts - 1) / parts + kWK - 1) / kWK * kWK;
  const int thin = ((M + 127) / 128 + parts - 1) / parts * ((H + 255) / 256);
  k_mlp_wgrad<<<dim3(tiles + thin, parts), 256, 0, s>>>(net_of(m), M, per, X, m->h1, m->h2, m->h3, m->d1, m->d2, m->d3,
                                                        m->dzb, m->G);
  return cudaGetLastError();
}

void refresh_bf16(qis_mlp* m, cudaStream_t s) {
  k_to_bf16<<<(m->n_params + 255) / 256, 256, 0, s>>>(net_of(m), m->n_params, m->P, m->Pb, m->W2t, m->W3t);
}

// The network's stream waits for the last use of its buffers on a context's stream.
cudaError_t wait_idle(qis_mlp* m) { return cudaStreamWaitEvent(m->stream, m->busy, 0); }
}  // namespace

extern "C" {

int qis_mlp_create(const qis_mlp_config* cfg, qis_mlp** out) {
  qis_mlp* m = nullptr;
  if (!cfg || !out) return mfail(nullptr, QIS_ERR_INVALID_ARG, "NULL argument");
  *out = nullptr;
  if (cfg->hidden < 16 || cfg->hidden > 1024 || cfg->hidden % 16) return mfail(nullptr, QIS_ERR_INVALID_ARG, "hidden must be a multiple of 16 in [16, 1024]");
  if (cfg->max_sites < 1 || cfg->batch < 1 || cfg->max_n < 2 || cfg->max_n > kMaxN)
    return mfail(nullptr, QIS_ERR_INVALID_ARG, "bad max_sites / batch / max_n");
  if (cudaSetDevice(cfg->device) != cudaSuccess) return mfail(nullptr, QIS_ERR_CUDA, "cudaSetDevice failed");
  m = new qis_mlp();
  m->cfg = *cfg;
  m->H = cfg->hidden;
  m->cap = cfg->max_sites;
  m->batch = cfg->batch;
  m->max_n = cfg->max_n;
  const int H = m->H, F = m->F;
  m->oW1 = 0;
  m->ob1 = m->oW1 + F * H;
  m->oW2 = m->ob1 + H;
  m->ob2 = m->oW2 + H * H;
  m->oW3 = m->ob2 + H;
  m->ob3 = m->oW3 + H * H;
  m->ow4 = m->ob3 + H;
  m->ob4 = m->ow4 + H;
  m->n_params = m->ob4 + 1;
  auto run = [&]() -> int {
    MCK(cudaStreamCreateWithFlags(&m->stream, cudaStreamNonBlocking));
    MALLOC(m->P, m->n_params);
    MALLOC(m->G, m->n_params);
    MALLOC(m->Mm, m->n_params);
    MALLOC(m->Vv, m->n_params);
    MALLOC(m->Pb, m->n_params);
    MALLOC(m->W2t, (size_t)H * H);
    MALLOC(m->W3t, (size_t)H * H);
    MCK(cudaEventCreateWithFlags(&m->busy, cudaEventDisableTiming));
    MCK(cudaDeviceGetAttribute(&m->sms, cudaDevAttrMultiProcessorCount, cfg->device));
    MALLOC(m->X, (size_t)m->cap * F);
    MALLOC(m->Y, m->cap);
    const size_t rows = (size_t)std::max(m->batch, m->max_n);
    MALLOC(m->h1, rows * H);
    MALLOC(m->h2, rows * H);
    MALLOC(m->h3, rows * H);
    MALLOC(m->d1, rows * H);
    MALLOC(m->d2, rows * H);
    MALLOC(m->d3, rows * H);
    MALLOC(m->Yq, rows);
    MALLOC(m->zb, rows);
    MALLOC(m->dzb, rows);
    MALLOC(m->loss, 1);
    MALLOC(m->Jst, (size_t)m->max_n * m->max_n);
    MALLOC(m->hst, m->max_n);
    MALLOC(m->bst, (m->max_n + 63) / 64);
    MALLOC(m->Xq, rows * F);
    // He initialisation from the SplitMix64 stream keyed by the seed (Box-Muller pairs)
    std::vector<float> p(m->n_params, 0.f);
    uint64_t key = splitmix64(cfg->seed ^ 0x4D4C50ull, 0);
    uint64_t c = 0;
    auto gauss = [&]() {
      const double u1 = ((double)(splitmix64(key, c++) >> 11) + 1.0) * 0x1.0p-53;
      const double u2 = (double)(splitmix64(key, c++) >> 11) * 0x1.0p-53;
      return sqrt(-2.0 * log(u1)) * cos(6.283185307179586 * u2);
    };
    for (int e = 0; e < F * H; ++e) p[m->oW1 + e] = (float)(gauss() * sqrt(2.0 / F));
    for (int e = 0; e < H * H; ++e) p[m->oW2 + e] = (float)(gauss() * sqrt(2.0 / H));
    for (int e = 0; e < H * H; ++e) p[m->oW3 + e] = (float)(gauss() * sqrt(2.0 / H));
    for (int e = 0; e < H; ++e) p[m->ow4 + e] = (float)(gauss() * sqrt(1.0 / H));
    MCK(cudaMemcpy(m->P, p.data(), sizeof(float) * m->n_params, cudaMemcpyHostToDevice));
    refresh_bf16(m, m->stream);
    MCK(cudaStreamSynchronize(m->stream));
    return 0;
  };
  const int rc = run();
  if (rc) {
    set_global_error(m->err.c_str());
    qis_mlp_destroy(m);
    return rc;
  }
  *out = m;
  return 0;
}

void qis_mlp_destroy(qis_mlp* m) {
  if (!m) return;
  cudaSetDevice(m->cfg.device);
  if (m->stream) cudaStreamSynchronize(m->stream);
  if (m->busy) {
    cudaEventSynchronize(m->busy);
    cudaEventDestroy(m->busy);
  }
  for (void* p : m->allocs) cudaFree(p);
  if (m->stream) cudaStreamDestroy(m->stream);
  delete m;
}

const char* qis_mlp_last_error(const qis_mlp* m) { return m ? m->err.c_str() : "NULL network"; }

int qis_mlp_num_params(qis_mlp* m, int* count) {
  if (!m || !count) return mfail(m, QIS_ERR_INVALID_ARG, "NULL argument");
  *count = m->n_params;
  return 0;
}

int qis_mlp_get_params(qis_mlp* m, float* flat) {
  if (!m || !flat) return mfail(m, QIS_ERR_INVALID_ARG, "NULL argument");
  MCK(cudaSetDevice(m->cfg.device));
  MCK(cudaStreamSynchronize(m->stream));
  MCK(cudaMemcpy(flat, m->P, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost));
  return 0;
}

int qis_mlp_set_params(qis_mlp* m, const float* flat) {
  if (!m || !flat) return mfail(m, QIS_ERR_INVALID_ARG, "NULL argument");
  MCK(cudaSetDevice(m->cfg.device));
  MCK(wait_idle(m));
  MCK(cudaStreamSynchronize(m->stream));
  MCK(cudaMemcpy(m->P, flat, sizeof(float) * m->n_params, cudaMemcpyHostToDevice));
  MCK(cudaMemset(m->Mm, 0, sizeof(float) * m->n_params));
  MCK(cudaMemset(m->Vv, 0, sizeof(float) * m->n_params));
  m->adam_t = 0;
  refresh_bf16(m, m->stream);
  MCK(cudaStreamSynchronize(m->stream));
  return 0;
}

int qis_mlp_features(qis_mlp* m, int n, const double* J, const double* h, float* X_out) {
  if (!m || !J || !h || !X_out) return mfail(m, QIS_ERR_INVALID_ARG, "NULL argument");
  if (n < 2 || n > m->max_n) return mfail(m, QIS_ERR_INVALID_ARG, "n must be in [2, max_n]");
  MCK(cudaSetDevice(m->cfg.device));
  cudaStream_t s = m->stream;
  MCK(wait_idle(m));
  MCK(cudaMemcpyAsync(m->Jst, J, sizeof(double) * n * n, cudaMemcpyHostToDevice, s));
  MCK(cudaMemcpyAsync(m->hst, h, sizeof(double) * n, cudaMemcpyHostToDevice, s));
  k_mlp_features<<<(n + 7) / 8, 256, 0, s>>>(m->Jst, n, m->hst, n, m->Xq);
  MCK(cudaGetLastError());
  MCK(cudaMemcpyAsync(X_out, m->Xq, sizeof(float) * n * kF, cudaMemcpyDeviceToHost, s));
  MCK(cudaStreamSynchronize(s));
  return 0;
}

int qis_mlp_clear_examples(qis_mlp* m) {
  if (!m) return mfail(m, QIS_ERR_INVALID_ARG, "NULL argument");
  m->n_examples = 0;
  return 0;
}

int qis_mlp_add_example(qis_mlp* m, int n, const double* J, const double* h, const uint64_t* bits) {
  if (!m || !J || !h || !bits) return mfail(m, QIS_ERR_INVALID_ARG, "NULL argument");
  if (n < 2 || n > m->max_n) return mfail(m, QIS_ERR_INVALID_ARG, "n must be in [2, max_n]");
  if (m->n_examples + n > m->cap) return mfail(m, QIS_ERR_CAPACITY, "training set full (max_sites)");
  MCK(cudaSetDevice(m->cfg.device));
  cudaStream_t s = m->stream;
  MCK(wait_idle(m));
  MCK(cudaMemcpyAsync(m->Jst, J, sizeof(double) * n * n, cudaMemcpyHostToDevice, s));
  MCK(cudaMemcpyAsync(m->hst, h, sizeof(double) * n, cudaMemcpyHostToDevice, s));
  MCK(cudaMemcpyAsync(m->bst, bits, sizeof(uint64_t) * ((n + 63) / 64), cudaMemcpyHostToDevice, s));
  k_mlp_features<<<(n + 7) / 8, 256, 0, s>>>(m->Jst, n, m->hst, n, m->X + (size_t)m->n_examples * kF);
  k_mlp_labels<<<(n + 127) / 128, 128, 0, s>>>(m->bst, n, m->Y + m->n_examples);
  MCK(cudaGetLastError());
  MCK(cudaStreamSynchronize(s));   // staging buffers are reused by the next call
  m->n_examples += n;
  return 0;
}

int qis_mlp_forward(qis_mlp* m, int M, const float* X, float* z_out) {
  if (!m || !X || !z_out || M < 1) return mfail(m, QIS_ERR_INVALID_ARG, "bad argument");
  if (M > std::max(m->batch, m->max_n)) return mfail(m, QIS_ERR_INVALID_ARG, "M exceeds the activation buffers");
  MCK(cudaSetDevice(m->cfg.device));
  cudaStream_t s = m->stream;
  MCK(wait_idle(m));
  MCK(cudaMemcpyAsync(m->Xq, X, sizeof(float) * M * kF, cudaMemcpyHostToDevice, s));
  MCK(mlp_pass(m, M, m->Xq, nullptr, s));
  MCK(cudaMemcpyAsync(z_out, m->zb, sizeof(float) * M, cudaMemcpyDeviceToHost, s));
  MCK(cudaStreamSynchronize(s));
  return 0;
}

int qis_mlp_loss_grad(qis_mlp* m, int M, const float* X, const float* y, double* loss, float* grad_out) {
  if (!m || !X || !y || M < 1) return mfail(m, QIS_ERR_INVALID_ARG, "bad argument");
  if (M > std::max(m->batch, m->max_n)) return mfail(m, QIS_ERR_INVALID_ARG, "M exceeds the activation buffers");
  MCK(cudaSetDevice(m->cfg.device));
  cudaStream_t s = m->stream;
  MCK(wait_idle(m));
  MCK(cudaMemcpyAsync(m->Xq, X, sizeof(float) * M * kF, cudaMemcpyHostToDevice, s));
  MCK(cudaMemcpyAsync(m->Yq, y, sizeof(float) * M, cudaMemcpyHostToDevice, s));
  MCK(cudaMemsetAsync(m->loss, 0, sizeof(double), s));
  MCK(mlp_pass(m, M, m->Xq, m->Yq, s));
  MCK(mlp_weight_grads(m, M, m->Xq, s));
  if (loss) MCK(cudaMemcpyAsync(loss, m->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
  if (grad_out) MCK(cudaMemcpyAsync(grad_out, m->G, sizeof(float) * m->n_params, cudaMemcpyDeviceToHost, s));
  MCK(cudaStreamSynchronize(s));
  return 0;
}

int qis_mlp_train(qis_mlp* m, int epochs, float lr, double* final_loss) {
  if (!m || epochs < 0 || !(lr > 0)) return mfail(m, QIS_ERR_INVALID_ARG, "bad argument");
  if (m->n_examples < 1) return mfail(m, QIS_ERR_STATE, "no training examples");
  MCK(cudaSetDevice(m->cfg.device));
  cudaStream_t s = m->stream;
  MCK(wait_idle(m));
  const int N = m->n_examples, Bt = m->batch;
  double last = 0.0;
  for (int ep = 0; ep < epochs; ++ep) {
    MCK(cudaMemsetAsync(m->loss, 0, sizeof(double), s));
    int nb = 0;
    for (int r0 = 0; r0 < N; r0 += Bt, ++nb) {
      const int M = std::min(Bt, N - r0);
      const float* X = m->X + (size_t)r0 * kF;
      MCK(mlp_pass(m, M, X, m->Y + r0, s));
      MCK(mlp_weight_grads(m, M, X, s));
      ++m->adam_t;
      const float b1 = 0.9f, b2 = 0.999f;
      const float c1 = 1.f - powf(b1, (float)m->adam_t), c2 = 1.f - powf(b2, (float)m->adam_t);
      k_adam<<<(m->n_params + 255) / 256, 256, 0, s>>>(net_of(m), m->n_params, m->P, m->G, m->Mm, m->Vv, lr, b1, b2, 1e-8f,
                                                       c1, c2, m->Pb, m->W2t, m->W3t);
    }
    MCK(cudaGetLastError());
    double sum = 0.0;
    MCK(cudaMemcpyAsync(&sum, m->loss, sizeof(double), cudaMemcpyDeviceToHost, s));
    MCK(cudaStreamSynchronize(s));
    last = sum / nb;   // mean of the batch losses of this epoch
  }
  if (final_loss) *final_loss = last;
  return 0;
}

}  // extern "C"

// ---------------------------------------------------------------- warm start of a context
namespace qis {
cudaError_t mlp_propose_states(qis_mlp* m, const double* J64, long long stride, const double* h64, int n, int R,
                               uint64_t key, uint64_t* init_bits, int Wstride, cudaStream_t s) {
  // the network runs on the context's stream: after its own stream's work (idle once a call has
  // returned) and after an earlier use on any other context's
  cudaError_t e = cudaStreamSynchronize(m->stream);
  if (e == cudaSuccess) e = cudaStreamWaitEvent(s, m->busy, 0);
  if (e != cudaSuccess) return e;
  k_mlp_features<<<(n + 7) / 8, 256, 0, s>>>(J64, stride, h64, n, m->Xq);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = mlp_pass(m, n, m->Xq, nullptr, s);
  if (e != cudaSuccess) return e;
  k_mlp_sample<<<dim3((n + 31) / 32, (R + kSampleR - 1) / kSampleR), 32, 0, s>>>(m->zb, n, R, key, init_bits, Wstride);
  e = cudaGetLastError();
  return e == cudaSuccess ? cudaEventRecord(m->busy, s) : e;
}
int mlp_max_n(const qis_mlp* m) { return m->max_n; }
}  // namespace qis
