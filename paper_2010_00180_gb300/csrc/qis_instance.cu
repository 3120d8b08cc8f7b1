// qis_instance.cu -- per-instance preparation and search initialisation.
//
// Instance data (H0 of Eq. (1)) lives in padded n_pad x n_pad planes:
//   J64  FP64 couplings as given (zero padding)
//   Jq   fixed-point couplings Jq = J * 2^q (int64, exact on the 2^-q grid)
//   J4   fl32(4 * Jq * 2^-q): the candidate filter's coupling term
//   D16  Jq written in balanced base-4096 digits, Jq = sum_d 4096^d D_d, D_d in [-2048, 2047],
//        one FP16 plane per digit (every digit is an exact FP16 integer)
#include <algorithm>

#include "qis_common.cuh"

namespace qis {

constexpr int kMaxGridY = 65535;   // a grid's second dimension: instances per launch of the batch kernels

// ---------------------------------------------------------------- validation
// stats layout (doubles): [0] bad flags (as bits of an int), [1] max frac bits, [2] max|J| bits,
// [3] max|h| bits, [4 .. 4+n) row sums sum_{j>i} |J_ij|; the host adds [4+n] = sum_i |h_i|.
// Fraction bits of x: the smallest f >= 0 with x 2^f an integer, from the bit pattern
// (|x| = M 2^(e - 1075) with the 53-bit significand M for a normal x, m 2^-1074 for a
// subnormal one; the lowest set bit of the significand decides).
__device__ inline int frac_bits(double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
  if (u == 0) return 0;
  const int e = (int)(u >> 52);
  const unsigned long long m = u & 0xfffffffffffffull;
  const int fb = (e == 0) ? 1074 - (__ffsll((long long)m) - 1)
                          : 1075 - e - (__ffsll((long long)(m | (1ull << 52))) - 1);
  return fb > 0 ? fb : 0;
}

// One warp per row i (its lanes over the columns, coalesced): finiteness, zero diagonal,
// bitwise symmetry, fraction bits and max |J_ij| (as the bit patterns of non-negative
// doubles, which order as integers), and the row sum of |J_ij|, j > i, reduced in a fixed
// shuffle order (deterministic). Sum of |h| is formed on the host.
__device__ __forceinline__ void validate_row(const double* J64, const double* h64, int n, int n_pad, double* stats, int i) {
  int* bad = reinterpret_cast<int*>(stats);
  int* maxfrac = reinterpret_cast<int*>(stats + 1);
  unsigned long long* maxJ = reinterpret_cast<unsigned long long*>(stats + 2);
  unsigned long long* maxh = reinterpret_cast<unsigned long long*>(stats + 3);
  const int lane = threadIdx.x & 31;
  const double* row = J64 + (long long)i * n_pad;
  double rs = 0.0;
  int fb = 0, b = 0;
  unsigned long long mj = 0;
  for (int j = lane; j < n; j += 32) {
    const double x = row[j];
    const unsigned long long ax = (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
    if (ax >= 0x7ff0000000000000ull) b |= 1;   // Inf or NaN
    if (j == i) {
      if (ax != 0) b |= 2;
      continue;
    }
    if (__double_as_longlong(x) != __double_as_longlong(J64[(long long)j * n_pad + i])) b |= 4;
    fb = max(fb, frac_bits(x));
    mj = max(mj, ax);
    if (j > i) rs += fabs(x);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    rs += __shfl_xor_sync(0xffffffffu, rs, o);
    fb = max(fb, __shfl_xor_sync(0xffffffffu, fb, o));
    mj = max(mj, __shfl_xor_sync(0xffffffffu, mj, o));
    b |= __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane == 0) {
    const double hv = h64[i];
    const unsigned long long ah = (unsigned long long)__double_as_longlong(hv) & 0x7fffffffffffffffull;
    if (ah >= 0x7ff0000000000000ull) b |= 8;
    fb = max(fb, frac_bits(hv));
    stats[4 + i] = rs;
    if (b) atomicOr(bad, b);
    atomicMax(maxfrac, fb);
    atomicMax(maxJ, mj);
    atomicMax(maxh, ah);
  }
}

// A batch of instances at once: blockIdx.y is the instance of the batch (its layout item).
__global__ void __launch_bounds__(256) k_validate_batch(const LayoutItem* items, const double* J64, const double* h64) {
  const LayoutItem L = items[blockIdx.y];
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= L.n) return;   // warp-uniform
  validate_row(J64 + L.off_mat, h64 + L.off_vec, L.n, L.n_pad, L.stats, i);
}

// ---------------------------------------------------------------- padded layout
// J (n x n, contiguous, as given by the host) into the padded n_pad x n_pad plane; zeros past n.
// Rows i = blockIdx.x, blockIdx.x + gridDim.x, ... of every instance (blockIdx.y), the threads
// over the columns: coalesced reads of the caller's rows (page-locked host memory read in place
// where it is), no index division.
__global__ void k_restride_batch(const LayoutItem* items, double* J64) {
  const LayoutItem L = items[blockIdx.y];
  double* dst = J64 + L.off_mat;
  for (int i = blockIdx.x; i < L.n_pad; i += gridDim.x) {
    const double* src = L.src + (long long)i * L.n;
    double* row = dst + (long long)i * L.n_pad;
    for (int j = threadIdx.x; j < L.n_pad; j += blockDim.x) row[j] = (i < L.n && j < L.n) ? src[j] : 0.0;
  }
}

// Layout and validation of `count` staged instances (items on the device), two launches per kMaxGridY.
cudaError_t launch_layout_batch(const DevPtrs& P, const LayoutItem* items, int count, int max_n_pad, double* J64,
                                cudaStream_t s) {
  for (int y = 0; y < count; y += kMaxGridY) {
    const int c = std::min(count - y, kMaxGridY);
    k_restride_batch<<<dim3(max_n_pad, c), 256, 0, s>>>(items + y, J64);
    k_validate_batch<<<dim3((max_n_pad + 7) / 8, c), 256, 0, s>>>(items + y, P.J64, P.h64);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------- fixed point + digits
// D16 holds, per digit and instance, an NP x NP plane in the tiled layout of d16_offset.
// Instances first .. first+count-1 at once (blockIdx.y), descriptors read on the device; rows
// i = blockIdx.x, blockIdx.x + gridDim.x, ..., the threads over the columns (no index division).
// Jq = rn(J 2^q), J4 = fl32(4 Jq 2^-q) (= fl32(Jq) 2^(2-q): scaling by a power of two commutes
// with rounding), the balanced base-2^dbits digits of Jq.
__global__ void k_quantize_batch(DevPtrs P, int first, __half* D16, long long* Jq, float* J4, long long* hq) {
  const int inst = first + blockIdx.y;
  const InstDesc d = P.inst[inst];
  const double* J64 = P.J64 + d.off_mat;
  __half* D = D16 + (long long)inst * P.NP * P.NP;
  const long long base = 1ll << d.dbits;
  const bool wide_q = d.q > 120;   // 2^(2-q) below the normal floats (tiny couplings): FP64 path
  const float s4 = wide_q ? 0.f : __int_as_float((127 + 2 - d.q) << 23);   // 2^(2-q)
  for (int i = blockIdx.x; i < d.n_pad; i += gridDim.x) {
    for (int j = threadIdx.x; j < d.n_pad; j += blockDim.x) {
      const long long e = (long long)i * d.n_pad + j;
      long long v = 0;
      if (i < d.n && j < d.n) v = fixed_point_rn(J64[e], d.q);
      Jq[d.off_mat + e] = v;
      J4[d.off_mat + e] = wide_q ? (float)(4.0 * ldexp((double)v, -d.q)) : __ll2float_rn(v) * s4;
      long long x = v;
      for (int dg = 0; dg < d.digits; ++dg) {
        long long r = x & (base - 1);           // x mod base
        if (r >= base / 2) r -= base;           // balanced digit in [-base/2, base/2)
        D[dg * P.pool_mat + d16_offset(i, j, P.NP)] = __float2half_rn((float)(int)r);
        x = (x - r) >> d.dbits;                 // exact
      }
    }
  }
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < d.n_pad; e += gridDim.x * blockDim.x)
    hq[d.off_vec + e] = (e < d.n) ? __double2ll_rn(ldexp(P.h64[d.off_vec + e], d.q)) : 0;
}

__global__ void __launch_bounds__(256) k_rowmax4_batch(DevPtrs P, int first) {
  const InstDesc d = P.inst[first + blockIdx.y];
  const int lane = threadIdx.x & 31;
  const int i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= d.n_pad) return;   // warp-uniform
  const float* J4 = P.J4 + d.off_mat;
  float m = 0.f;
  if (i < d.n)
    for (int j = lane; j < d.n; j += 32) m = fmaxf(m, fabsf(J4[(long long)i * d.n_pad + j]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) P.rm4[d.off_vec + i] = m;
}

// Fixed-point planes, digits and row maxima of instances first .. first+count-1, two launches per kMaxGridY.
cudaError_t launch_prepare_batch(const DevPtrs& P, int first, int count, int max_n_pad, __half* D16, long long* Jq,
                                 float* J4, long long* hq, cudaStream_t s) {
  for (int y = 0; y < count; y += kMaxGridY) {
    const int c = std::min(count - y, kMaxGridY);
    k_quantize_batch<<<dim3(max_n_pad, c), 256, 0, s>>>(P, first + y, D16, Jq, J4, hq);
    k_rowmax4_batch<<<dim3((max_n_pad + 7) / 8, c), 256, 0, s>>>(P, first + y);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------- search initialisation
// FP64 mode: E(psi0) of the initial states of instances inst0, inst0 + 1, ... into init_E, the pair
// terms added i-major, j ascending, then the field terms. A lane per search, 32 searches of an
// instance per block: the lanes share every coupling's load, and the chain of n^2 / 2 dependent
// additions is what it costs (one search per block took as long for each: 1.5 ms for 3840 searches
// of n = 100).
__global__ void __launch_bounds__(32) k_init_energy_f64(DevPtrs P, int inst0) {
  const int inst = inst0 + blockIdx.y, r = blockIdx.x * 32 + (int)threadIdx.x;
  const InstDesc d = P.inst[inst];
  const int n = d.n;
  const long long b = (long long)d.first_search + min(r, P.R - 1);
  const uint64_t* bits = P.init_bits + b * P.Wmax;
  const double* J = P.J64 + d.off_mat;
  double Pp = 0.0, F = 0.0;
  for (int i = 0; i < n; ++i) {
    const uint64_t si = 0ull - (uint64_t)sigma_of(bits, i);   // all ones where s_i = -1
    const double* row = J + (long long)i * d.n_pad;
    for (int j0 = (i + 1) & ~63; j0 < n; j0 += 64) {
      const uint64_t w = bits[j0 >> 6] ^ si;
      const int u1 = min(64, n - j0);
#pragma unroll 8
      for (int u = max(0, i + 1 - j0); u < u1; ++u)
        Pp = __dadd_rn(Pp, __longlong_as_double(__double_as_longlong(row[j0 + u]) ^ (long long)((w >> u) << 63)));
    }
  }
  for (int i = 0; i < n; ++i) F = __dadd_rn(F, P.h64[d.off_vec + i] * (sigma_of(bits, i) ? -1.0 : 1.0));
  if (r < P.R) P.init_E[b] = __dadd_rn(Pp, F);
}

cudaError_t launch_init_energy_f64(const DevPtrs& P, int inst0, int n_inst, cudaStream_t s) {
  for (int y = 0; y < n_inst; y += kMaxGridY)
    k_init_energy_f64<<<dim3((P.R + 31) / 32, std::min(n_inst - y, kMaxGridY)), 32, 0, s>>>(P, inst0 + y);
  return cudaGetLastError();
}

// Alg. 3 initial list: [psi0, K placeholders], E(psi0) from Eq. (1), nothing used. E(psi0) is taken
// from init_E / init_q, written by launch_init_energy (split modes: exact int64 E 2^q),
// launch_init_energy_f64 or an earlier start from the same initial states; or (deferred, split
// modes) it is left to the first iteration of the fused search kernel, which forms it from the
// exact fields of psi0 that the iteration computes anyway: the entry holds 0 until then and
// e0_pend marks the search.
__global__ void __launch_bounds__(256) k_init_search(DevPtrs P, int b0, int deferred) {
  const int b = b0 + blockIdx.x;
  const InstDesc d = P.inst[b / P.R];
  const int n = d.n, W = d.W;
  __shared__ uint64_t bits[kMaxN / 64];
  for (int w = threadIdx.x; w < W; w += blockDim.x) bits[w] = P.init_bits[(long long)b * P.Wmax + w];
  __syncthreads();
  const double E0 = deferred ? 0.0 : P.init_E[b];
  const long long q0 = deferred || P.mode == QIS_FP64 ? 0 : P.init_q[b];
  // Zobrist hash of psi0: XOR over the threads' sites, then over the warps
  __shared__ uint64_t s_h[8];
  uint64_t hsh = 0;
  for (int i = threadIdx.x; i < n; i += blockDim.x)
    if (sigma_of(bits, i)) hsh ^= P.zob[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) hsh ^= __shfl_xor_sync(0xffffffffu, hsh, o);
  if ((threadIdx.x & 31) == 0) s_h[threadIdx.x >> 5] = hsh;
  const long long base = (long long)b * P.K1;
  for (int w = threadIdx.x; w < W; w += blockDim.x) P.lst_bits[base * P.Wmax + w] = bits[w];
  for (int k = threadIdx.x; k < P.K1; k += blockDim.x) {
    P.lst_used[base + k] = 0;
    P.lst_ord[base + k] = (k == 0) ? 0 : -1;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) hsh ^= s_h[w];
    P.init_E[b] = E0;
    P.init_q[b] = q0;
    P.lst_E[base] = E0;
    if (P.mode != QIS_FP64) P.lst_q[base] = q0;
    P.lst_key[base] = (P.mode != QIS_FP64) ? qkey(q0) : dkey(E0);
    P.lst_stamp[base] = 0;
    P.lst_hash[base] = hsh;
    P.lst_count[b] = 1;
    P.active[b] = 1;
    P.iter_t[b] = 0;
    if (P.ring_t0) P.ring_t0[b] = 0;
    P.surv_cnt[b] = 0;
    P.e0_pend[b] = deferred;
  }
}

cudaError_t launch_init_search(const DevPtrs& P, int b0, int nb, cudaStream_t s, bool deferred) {
  if (nb <= 0) return cudaSuccess;
  k_init_search<<<nb, 256, 0, s>>>(P, b0, deferred ? 1 : 0);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- merged-list gather
__global__ void k_gather_merged(DevPtrs P, int inst, int k, int Wn, uint64_t* out) {
  const int r = blockIdx.x;
  if (r >= k) return;
  const int ref = P.mrg_ref[inst * P.K1 + r];
  const int b = ref / P.K1, slot = ref % P.K1;
  for (int w = threadIdx.x; w < Wn; w += blockDim.x)
    out[(long long)r * Wn + w] = P.lst_bits[((long long)b * P.K1 + slot) * P.Wmax + w];
}

cudaError_t launch_gather_merged(const DevPtrs& P, int inst, const InstDesc& d, int k, uint64_t* bits_out,
                                 cudaStream_t s) {
  if (k <= 0) return cudaSuccess;
  k_gather_merged<<<k, 32, 0, s>>>(P, inst, k, d.W, bits_out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- imported lists
// Zobrist hash of the first `count` slots of search b's list (the bits were copied in by the
// host): the same key the merge and the dedup use for states generated on the device.
__global__ void k_hash_list(DevPtrs P, int b, int count) {
  const InstDesc d = P.inst[b / P.R];
  const long long base = (long long)b * P.K1;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < count; k += gridDim.x * blockDim.x) {
    const uint64_t* bits = P.lst_bits + (base + k) * P.Wmax;
    uint64_t h = 0;
    for (int i = 0; i < d.n; ++i)
      if ((bits[i >> 6] >> (i & 63)) & 1ull) h ^= P.zob[i];
    P.lst_hash[base + k] = h;
  }
}

cudaError_t launch_hash_list(const DevPtrs& P, int b, int count, cudaStream_t s) {
  if (count <= 0) return cudaSuccess;
  k_hash_list<<<(count + 127) / 128, 128, 0, s>>>(P, b, count);
  return cudaGetLastError();
}

// The instances are removed: their candidates are added to those of earlier ones, their counts and the
// device flags cleared. One block per instance, one launch: the same by copies to the host and memsets
// were five blocking calls (a pipeline on one instance of n = 16, 4 searches, 8 iterations: 232 us with
// them, 215 us with this launch).
__global__ void __launch_bounds__(128) k_retire(DevPtrs P) {
  const int n = P.inst[blockIdx.x].n;   // (up to date wherever a search has run)
  unsigned long long pairs = 0, singles = 0;
  for (int r = threadIdx.x; r < P.R; r += 128) {
    const int b = blockIdx.x * P.R + r;
    pairs += P.npair[b];
    singles += (unsigned long long)P.nprod[b] * (unsigned)n;
    P.npair[b] = 0;
    P.nprod[b] = 0;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    pairs += __shfl_xor_sync(0xffffffffu, pairs, o);
    singles += __shfl_xor_sync(0xffffffffu, singles, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (pairs) atomicAdd(P.cand_acc, pairs);
    if (singles && P.flips != QIS_FLIPS_EXCHANGE) atomicAdd(P.cand_acc + 1, singles);
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) P.status[0] = 0;
}

cudaError_t launch_retire(const DevPtrs& P, cudaStream_t s) {
  k_retire<<<P.n_inst, 128, 0, s>>>(P);
  return cudaGetLastError();
}

}  // namespace qis
