// qis_search.cu -- every iteration of one search in one thread block (the fused, persistent
// form of the iteration of Alg. 3; single flips alone: qis_single.cu).
//
// The R searches of an instance, and the instances, share nothing until the Alg. 4 merge, so
// one block can take one search through all the iterations of a qis_iterate call without ever
// waiting for another block. Per iteration t the block runs, back to back:
//   pick    the first unused kept state in key order becomes the parent (Alg. 3)
//   fields  its exact integer fields from its generating parent's, held in the aq ring, minus
//           the flipped sites' coupling columns (the Sec. III energy algebra; a parent whose
//           generator is no longer in the ring gets them from a full row sum instead);
//           a_i = -2 s_i f_i. The sites with a_i up to a cut, guessed from the last iteration, are
//           listed on the way: only they can be flipped by a candidate that enters the list, and
//           what follows works on this list (a fifth of the sites at n = 600) in a bucket order of a_i
//   near    the kept states one or two flips from the parent (the only possible duplicates), from
//           the flips of its own generation and from the hashes of the others (near_sites)
//   bound   filter threshold: the last kept energy and an order-statistic bound from the flips of
//           the lowest listed sites; a list that does not reach what the threshold needs is
//           taken again. In a kept list that has settled the last kept energy alone leaves few
//           enough, and the order-statistic bound (a fifth of such an iteration) is not formed
//   scan    pair flips dE_ij = a_i + a_j + 4 s_i s_j J_ij decided by the output-sensitive scan: a
//           live row's partners are the sites after it in the order, up to the bucket of its bound
//   merge   exact integer keys of the survivors, duplicates dropped, the new states ranked by
//           a counting sort over buckets of their keys (no sort), first K+1 of the old list and
//           the new states by (E, stamp)
// The kept list's order, keys, flips, hashes and used flags and the parent's spins stay in shared
// memory across the iterations; a new state is kept as (iteration, flips), its words being its
// parent's (stored per iteration) with at most two bits flipped, and the words are written into
// the list once, at the end of the launch. The aq ring and the survivors past 512 are in global
// memory (written and read by this block only, within the L2 cache).
// Split modes: the first iteration's parent is picked, and its fields computed (update, or the
// tensor-core GEMM for a parent without a stored generator), by the kernels launched before this one;
// not for instances of at most 128 spins, whose row sums here cost less than those launches (4 searches
// of n = 16, 8 iterations: 82 us with them, 70 without).
// FP64 mode: the same filter, the survivors' energies in the defining FP64 arithmetic.
// Every decision is that of the per-kernel form (k_bound, k_scan_sparse, k_merge), so the kept
// lists are identical bit for bit.
//
// What bounds it: the latency and issue of many short dependent steps (32 warps per SM at 64
// registers, about 2 instructions per SM cycle); no phase takes more than a sixth of the time. 7680
// searches of n = 600, 120 iterations: 31.9 ms with passes over all sites for each of histogram,
// selection, rows, bucket counts and order, with the near states found by comparing words, and with
// every new state's words written in every iteration; 26.6 ms with the listed sites, hashes and
// words at the end; 21.6 ms with the own generation's near states from their flips alone (3840 searches
// of n = 64: 6.2 ms with the order-statistic bound in every iteration, 5.1 without it in settled lists;
// of n = 200 8.2 and 7.9).
#include "qis_block.cuh"

namespace qis {

constexpr int kSSV = 512;   // survivors held in shared memory (more go to the global buffer)

__host__ __device__ inline int search_pcs(int cap, int merge_cand) {
  const int pc = next_pow2(cap > 256 ? cap : 256);
  return pc < merge_cand ? pc : merge_cand;
}

// Byte offsets of the dynamic shared memory of a search block of `warps` warps.
struct SearchLayout {
  int pb, okey0, okey1, oflip, ohash, oslot0, oslot1, htab, ssv, oused, ogen, ad, scratch, total;
  // the scratch region while candidates are found (later the merge's): the low sites as taken and in
  // order, the rows' list offsets (the bound's histogram before), the buckets
  int oa, orm, os, ua, us, pc, bs, bcur;
};

__host__ __device__ inline SearchLayout search_layout(int NP, int Wmax, int K1, int cap, int merge_cand, int warps, bool f64) {
  SearchLayout L;
  int o = 0;
  auto take = [&](int bytes) {
    o = align_up(o, 16);
    const int r = o;
    o += bytes;
    return r;
  };
  L.pb = take(Wmax * 8);
  L.okey0 = take(K1 * 8);
  L.okey1 = take(K1 * 8);
  L.ohash = take(K1 * 8);
  L.oflip = take(K1 * 4);
  L.oslot0 = take(K1 * 4);
  L.oslot1 = take(K1 * 4);
  L.htab = take(next_pow2(2 * K1) * 4);
  L.ssv = take(kSSV * 8);
  L.oused = take(K1);
  L.ogen = take(K1);
  L.ad = take(f64 ? NP * 8 : 0);
  o = align_up(o, 16);
  L.scratch = o;
  L.oa = take(NP * 4);
  L.orm = take(NP * 4);
  L.os = take(NP * 2);
  L.ua = take(NP * 4);
  L.us = take(NP * 2);
  L.pc = take(NP * 4 > 2048 ? NP * 4 : 2048);
  L.bs = take((kSparseNB + 1) * 4);
  L.bcur = take(kSparseNB * 4);
  // (keep_lowest's 256 bins lie 2 kMB past the bucket sizes: within the starts of three or more warps)
  const int merge = search_pcs(cap, merge_cand) * 16 + (512 + kMB + warps * (kMB + 4)) * 4;
  L.total = align_up(o - L.scratch > merge ? o : L.scratch + merge, 16);
  return L;
}

// Orderable unsigned key of a float (ascending floats -> ascending keys) and its inverse.
__device__ __forceinline__ unsigned fkey(float x) {
  const unsigned u = __float_as_uint(x + 0.f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float fkey_inv(unsigned k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7fffffffu) : ~k);
}

// Fields of a parent without a stored generator, from scratch: fq_k = hq_k + sum_j s_j Jq_jk
// (columns coalesced), aq_k = -2 s_k fq_k. Rarely taken (out of line: the hot loop stays small).
static __device__ __noinline__ void fields_full(const DevPtrs& P, const InstDesc& d, const uint64_t* pb,
                                                long long* ax) {
  const long long* Jq = P.Jq + d.off_mat;
  for (int k = threadIdx.x; k < d.n; k += blockDim.x) {
    long long acc = P.hq[d.off_vec + k];
    for (int jj = 0; jj < d.n; ++jj) {
      const long long v = Jq[(long long)jj * d.n_pad + k];
      acc += sigma_of(pb, jj) ? -v : v;
    }
    ax[k] = sigma_of(pb, k) ? 2 * acc : -2 * acc;
  }
}

// The k-th lowest dE of the m survivors held (radix select, the values formed anew in each pass). More
// survivors than the buffer holds are rare: out of line.
static __device__ __noinline__ float kth_survivor(const unsigned long long* ssv, const unsigned long long* surv, int m, int k,
                                                  const long long* ax, float scale_q, const float* J4, int n_pad,
                                                  const uint64_t* pb, int* hist) {
  unsigned prefix = 0u;
  int rank = k - 1;
  for (int shift = 24; shift >= 0; shift -= 8) {
    for (int x = threadIdx.x; x < 256; x += blockDim.x) hist[x] = 0;
    __syncthreads();
    for (int e = threadIdx.x; e < m; e += blockDim.x) {
      int i, j;
      surv_sites((e < kSSV) ? ssv[e] : surv[e], i, j);
      float v = __ll2float_rn(ax[i]) * scale_q;
      if (j >= 0) {
        const float j4 = J4[(long long)i * n_pad + j];
        v += fmaf(sigma_of(pb, i) != sigma_of(pb, j) ? -1.f : 1.f, j4, __ll2float_rn(ax[j]) * scale_q);
      }
      const unsigned key = fkey(v);
      if (shift == 24 || key >> (shift + 8) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1);
    }
    __syncthreads();
    int bin;
    find_bin(hist, rank, bin, rank);   // every warp alike
    prefix = (prefix << 8) | (unsigned)bin;
    __syncthreads();
  }
  return fkey_inv(prefix);
}

// FP64 mode: a_i = -2 s_i f_i with f_i = (sum_{j != i} s_j J_ij, j ascending from +0.0) + h_i (the
// order of k_fields_fp64) of the m sites of `list`, ascending. A chain of n additions per site, on
// two FP64 lanes per SM, is what bounds the FP64 search, so only the sites of the survivors pay it
// (the filter works on the fixed-point fields): 120 iterations of 3840 searches of n = 100 take
// 9.7 ms, 12.4 with the sites of the duplicates too, and 86 ms in the per-kernel form (every pair in
// FP64). An instance exactly on its grid needs no
// chain: every partial sum is exact, so the fixed-point field is the same double.
template <int U = 8>
static __device__ __forceinline__ void fields_f64(const DevPtrs& P, const InstDesc& d, const uint64_t* pb,
                                                  const long long* aq, const unsigned short* list, int m, double* ad) {
  const int n = d.n;
  for (int q = threadIdx.x; q < m; q += blockDim.x) {
    const int i = list[q];
    if (!d.rounded) {   // block-uniform
      ad[i] = (double)aq[i] * d.inv_scale;
      continue;
    }
    const double* J = P.J64 + d.off_mat + i;   // J_ji = J_ij
    double acc = 0.0;
    for (int j0 = 0; j0 < n; j0 += 64) {
      const uint64_t w = pb[j0 >> 6];
      const int e = min(64, n - j0);
#pragma unroll U
      for (int u = 0; u < e; ++u) {
        const double v = J[(long long)(j0 + u) * d.n_pad];
        const double x = __longlong_as_double(__double_as_longlong(v) ^ (long long)((w >> u) << 63));
        if (j0 + u != i) acc = __dadd_rn(acc, x);
      }
    }
    const double f = __dadd_rn(acc, P.h64[d.off_vec + i]);
    ad[i] = sigma_of(pb, i) ? 2.0 * f : -2.0 * f;
  }
}

// FP64 mode, more survivors than the buffer holds and none to be told apart by the FP32 band (equal or
// nearly equal changes of energy): the survivors taken again by their defining energies, as the per-kernel
// form takes them, E' < T and E' at or below the k-th lowest of such candidates (radix select of the
// order keys, the energies formed anew in each pass). Returns their number, of which the first cap are
// held. Rare: out of line, every candidate nine times; it takes little from the caller, whose registers
// are full, and finds the block's arrays again.
static __device__ __noinline__ int exact_survivors(const DevPtrs& P, const long long* aq, double Ep, double T, int k, int* s_cnt) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int b = blockIdx.x;
  const InstDesc& d = P.inst[b / P.R];
  const bool ex = P.flips == QIS_FLIPS_EXCHANGE;
  const SearchLayout L = search_layout(P.NP, P.Wmax, P.K1, P.cap, P.merge_cand, blockDim.x >> 5, true);
  const uint64_t* pb = reinterpret_cast<const uint64_t*>(smem + L.pb);
  unsigned long long* ssv = reinterpret_cast<unsigned long long*>(smem + L.ssv);
  double* ad = reinterpret_cast<double*>(smem + L.ad);
  unsigned short* list = reinterpret_cast<unsigned short*>(smem + L.us);
  int* hist = reinterpret_cast<int*>(smem + L.pc);
#pragma unroll 1
  for (int i = threadIdx.x; i < d.n; i += blockDim.x) list[i] = (unsigned short)i;
  if (threadIdx.x == 0) *s_cnt = 0;
  __syncthreads();
  fields_f64<1>(P, d, pb, aq, list, d.n, ad);
  unsigned long long prefix = 0;
  int rank = k - 1;
  // passes over the candidates below T: eight bits of the k-th lowest key each (all ones where there are
  // fewer than k: find_bin gives the last bin then), then the taking
#pragma unroll 1
  for (int shift = 56; shift >= -8; shift -= 8) {
#pragma unroll 1
    for (int x = threadIdx.x; x < 256; x += blockDim.x) hist[x] = 0;
    __syncthreads();
#pragma unroll 1
    for (int i = threadIdx.x >> 5; i < d.n; i += blockDim.x >> 5)
#pragma unroll 1
      for (int j = i + (threadIdx.x & 31); j < d.n; j += 32) {
        const int flip = sigma_of(pb, i) ^ sigma_of(pb, j);
        if (ex && !flip) continue;
        // (j = i: the flip of site i alone)
        const double de = j == i ? ad[i] : dE64(ad[i], ad[j], P.J64[d.off_mat + (long long)i * d.n_pad + j], flip);
        const double e = __dadd_rn(Ep, de);
        if (!(e < T)) continue;
        const unsigned long long key = dkey(e);
        if (shift >= 0) {
          if (shift == 56 || key >> (shift + 8) == prefix) atomicAdd(&hist[(int)(key >> shift) & 255], 1);
        } else if (key <= prefix) {
          const int slot = atomicAdd(s_cnt, 1);
          if (slot < P.cap) *(slot < kSSV ? ssv + slot : P.surv + (long long)b * P.cap + slot) = surv_entry(i, j == i ? -1 : j);
        }
      }
    __syncthreads();
    if (shift < 0) break;
    int bin;
    find_bin(hist, rank, bin, rank);   // every warp alike
    prefix = (prefix << 8) | (unsigned)bin;
    __syncthreads();
  }
  return *s_cnt;
}

// The candidate sites of an iteration, from scratch (out of line: the first iteration of a launch, or
// when the cut guessed from the last one does not reach far enough): the sites with a_i <= cut (inf:
// every site) in a monotone bucket order of a_i. Returns their number; lo and inv are the buckets'.
// amin, amax: the range of a_i (known = false: found here).
struct LowSites {
  float *oa, *orm, *ua;
  unsigned short *os, *us;
  int *bs, *bcur;
};

static __device__ __forceinline__ void set_buckets(float amin, float amax, float cut, float& lo, float& inv) {
  const float span = __fsub_ru(fminf(cut, amax), amin);
  lo = amin;
  inv = (span > 0.f && span < INFINITY) ? __fdiv_rn((float)kSparseNB, span) : 0.f;
}

// Exclusive starts of the bucket counts in cur, into bs (kSparseNB + 1) and cur. One warp.
static __device__ __forceinline__ void bucket_starts(int* cur, int* bs) {
  const int lane = threadIdx.x & 31;
  int x[kSparseNB / 32], s = 0;
#pragma unroll
  for (int q = 0; q < kSparseNB / 32; ++q) {
    x[q] = cur[lane * (kSparseNB / 32) + q];
    s += x[q];
  }
  int inc = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += y;
  }
  int acc = inc - s;
#pragma unroll
  for (int q = 0; q < kSparseNB / 32; ++q) {
    bs[lane * (kSparseNB / 32) + q] = acc;
    cur[lane * (kSparseNB / 32) + q] = acc;
    acc += x[q];
  }
  if (lane == 31) bs[kSparseNB] = acc;
}

static __device__ __noinline__ int low_sites_again(const long long* ax, const float* rm, int n, float scale_q,
                                                   const uint64_t* pb, const LowSites& S, int* s_cn, bool known,
                                                   float& amin, float& amax, float cut, float& lo, float& inv) {
  if (!known) {
    float mn = INFINITY, mx = -INFINITY;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      const float v = __ll2float_rn(ax[k]) * scale_q;
      mn = fminf(mn, v);
      mx = fmaxf(mx, v);
    }
    block_min_max(mn, mx);
    amin = mn;
    amax = mx;
  }
  set_buckets(amin, amax, cut, lo, inv);
  __syncthreads();
  if (threadIdx.x == 0) *s_cn = 0;
  for (int x = threadIdx.x; x < kSparseNB; x += blockDim.x) S.bcur[x] = 0;
  __syncthreads();
  for (int k = threadIdx.x; k < n; k += blockDim.x) {
    const float v = __ll2float_rn(ax[k]) * scale_q;
    if (v <= cut) {
      const int e = atomicAdd(s_cn, 1);
      S.ua[e] = v;
      S.us[e] = (unsigned short)(k | (sigma_of(pb, k) << 15));
      atomicAdd(&S.bcur[sparse_bucket(v, lo, inv)], 1);
    }
  }
  __syncthreads();
  const int cn = *s_cn;
  if (threadIdx.x < 32) bucket_starts(S.bcur, S.bs);
  __syncthreads();
  for (int e = threadIdx.x; e < cn; e += blockDim.x) {
    const float v = S.ua[e];
    const unsigned short s = S.us[e];
    const int q = atomicAdd(&S.bcur[sparse_bucket(v, lo, inv)], 1);
    S.oa[q] = v;
    S.os[q] = s;
    S.orm[q] = rm[s & 0x7fff];
  }
  __syncthreads();
  return cn;
}

// FL: flip set, QIS_FLIPS_SINGLE_PAIR or QIS_FLIPS_EXCHANGE (single flips alone: qis_single.cu). One
// block of NT threads per search; 1 <= n_iters <= P.pw_n. ext: the first iteration's parent was
// picked and its fields computed by the kernels launched before this one (split modes).
// F64: the FP64 mode. The candidates are filtered as in the split modes (fixed-point fields, FP32
// copies of a_i and 4 J_ij), the survivors get the defining FP64 energies from their sites' defining
// FP64 fields.
template <int FL, bool F64, int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_search(DevPtrs P, int n_iters, int ext) {
  constexpr bool EX = FL == QIS_FLIPS_EXCHANGE;
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const int b = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K1 = P.K1, Wm = P.Wmax, cap = P.cap;
  const long long base = (long long)b * K1;
  const SearchLayout L = search_layout(P.NP, Wm, K1, cap, P.merge_cand, NW, F64);
  uint64_t* pb = reinterpret_cast<uint64_t*>(smem + L.pb);
  unsigned long long* okeyA = reinterpret_cast<unsigned long long*>(smem + L.okey0);
  unsigned long long* okeyB = reinterpret_cast<unsigned long long*>(smem + L.okey1);
  uint32_t* oflip = reinterpret_cast<uint32_t*>(smem + L.oflip);   // of a state of this launch: i | j << 16 (j = 0xffff: none)
  uint64_t* ohash = reinterpret_cast<uint64_t*>(smem + L.ohash);
  int* oslotA = reinterpret_cast<int*>(smem + L.oslot0);
  int* oslotB = reinterpret_cast<int*>(smem + L.oslot1);
  uint32_t* htab = reinterpret_cast<uint32_t*>(smem + L.htab);
  unsigned long long* ssv = reinterpret_cast<unsigned long long*>(smem + L.ssv);
  const int HT = next_pow2(2 * K1);
  uint8_t* oused = reinterpret_cast<uint8_t*>(smem + L.oused);
  uint8_t* ogen = reinterpret_cast<uint8_t*>(smem + L.ogen);
  double* ad = reinterpret_cast<double*>(smem + L.ad);   // FP64 mode: a_i of the survivors' sites
  unsigned char* scr = smem + L.scratch;
  const LowSites LS = {reinterpret_cast<float*>(smem + L.oa), reinterpret_cast<float*>(smem + L.orm),
                       reinterpret_cast<float*>(smem + L.ua), reinterpret_cast<unsigned short*>(smem + L.os),
                       reinterpret_cast<unsigned short*>(smem + L.us), reinterpret_cast<int*>(smem + L.bs),
                       reinterpret_cast<int*>(smem + L.bcur)};
  float *oa = LS.oa, *orm = LS.orm;
  unsigned short* os = LS.os;   // site | sigma << 15
  int *bs = LS.bs, *bcur = LS.bcur;
  int* pc = reinterpret_cast<int*>(smem + L.pc);
  int* vhist = pc;                                              // [256] the bound's values per bin
  unsigned* vmax = reinterpret_cast<unsigned*>(vhist + 256);    // [256] and their maxima

  __shared__ int s_sel, s_near, s_ns, s_nv, s_ocut, s_cn, s_m0, s_m1, s_set, s_nset;
  __shared__ int s_hold;   // FP64 mode: 1 + the survivors at hand before the scan, 0: none
  __shared__ float wf[2 * NW], s_u, s_thr[2];
  __shared__ int s_w[33];
  __shared__ unsigned long long s_kmm[2 * NW];
  __shared__ unsigned short s_ex[kSubSites];   // exchanges: the bound's sites of each spin class (positions)

  const int act0 = P.active[b];
  const InstDesc d = P.inst[b / P.R];
  const int n = d.n, W = d.W;
  const int t_first = P.iter_t[b] + (ext ? 0 : 1);   // the iteration of iter = 0
  const int ring_t0 = P.ring_t0[b];
  int cnt = P.lst_count[b];
  // the parent's energy: E 2^q exact, or the bits of the FP64 mode's double
  long long Epq = F64 ? 0 : P.par_q[b];
  uint64_t ph = P.par_hash[b];
  uint64_t* pw = P.pw + (long long)b * P.pw_n * Wm;   // words of the parent of iteration iter: pw + iter Wm
#pragma unroll 1
  for (int r = tid; r < K1; r += NT) {
    okeyA[r] = P.lst_key[base + r];
    oslotA[r] = P.lst_ord[base + r];
    ohash[r] = P.lst_hash[base + r];
    oused[r] = P.lst_used[base + r];
    ogen[r] = 0;   // in lst_bits (else 1 + the iteration of this launch that generated it)
  }
#pragma unroll 1
  for (int w = tid; w < W; w += NT) {
    const uint64_t x = P.par_bits[(long long)b * Wm + w];
    pb[w] = x;
    if (ext) pw[w] = x;
  }
  __syncthreads();
  // E(psi0) is still to be formed from the exact fields of its first iteration (block-uniform: the
  // list is [psi0] and psi0 is that iteration's parent)
  auto form_e0 = [&]() {
    Epq = initial_energy(P, d, pb, aq_of(P, b, t_first), reinterpret_cast<long long*>(s_kmm));
    if (tid == 0) {
      const int s0 = oslotA[0];
      const double E0 = ldexp((double)Epq, -d.q);
      okeyA[0] = qkey(Epq);
      P.lst_q[base + s0] = Epq;
      P.lst_E[base + s0] = E0;
      P.init_q[b] = Epq;
      P.init_E[b] = E0;
      P.e0_pend[b] = 0;
    }
    __syncthreads();
  };

  if (tid == 0) {
    s_u = INFINITY;
    s_hold = 0;
  }
  int act = act0, cur = 0, nprod = 0;
  int pgen = 0, pi0 = -1, pj0 = -1;   // the parent's generation in this launch and its flips
  unsigned npair = 0, nev = 0, nsurv = 0;   // of this launch (at most 128 iterations: 32 bits); npair: exchanges
  const float scale_q = (float)d.inv_scale;
  const long long* Jq = P.Jq + d.off_mat;
  const float* J4 = P.J4 + d.off_mat;
  const float* rm = P.rm4 + d.off_vec;
  unsigned long long* surv = P.surv + (long long)b * cap;
  // survivor slot s: shared memory below kSSV, the search's global buffer above (up to cap)
  auto put_surv = [&](int slot, unsigned long long e) {
    if (slot < kSSV) ssv[slot] = e;
    else if (slot < cap) surv[slot] = e;
  };
  // the cut and the buckets of the candidate sites, guessed from the last iteration (ranged)
  bool ranged = false;
  float cut = INFINITY, lo = 0.f, inv = 0.f;

  for (int iter = 0; iter < n_iters; ++iter) {
    unsigned long long* okey = cur ? okeyB : okeyA;
    unsigned long long* okeyN = cur ? okeyA : okeyB;
    int* oslot = cur ? oslotB : oslotA;
    int* oslotN = cur ? oslotA : oslotB;
    if (!act) continue;
    const int t = t_first + iter;
    // this iteration's counters (the last one's reads are behind its last barrier)
    if (tid == 0) {
      s_set = iter > 0 && s_nset && s_ns <= K1;   // (s_set, s_nset: see the bound)
      s_near = 0;
      s_ns = F64 && s_hold ? s_hold - 1 : 0;
      s_nv = 0;
      s_cn = 0;
      s_ocut = cnt;
    }
#pragma unroll 1
    for (int x = tid; x < HT; x += NT) htab[x] = kNoCand;
#pragma unroll 1
    for (int x = tid; x < kSparseNB; x += NT) bcur[x] = 0;
#pragma unroll 1
    for (int x = tid; x < 512; x += NT) vhist[x] = 0;
    float mn = INFINITY, mx = -INFINITY;   // this thread's range of a_i
    const long long* aqb = aq_of(P, b, t);
    if (F64 || iter > 0 || !ext) {
      // ------------------------------------------------------------ pick (Alg. 3)
      if (warp == 0) {
        int sel = -1;
        for (int r0 = 0; r0 < cnt && sel < 0; r0 += 32) {
          const int r = r0 + lane;
          const bool un = r < cnt && !oused[oslot[r]];
          const unsigned m = __ballot_sync(0xffffffffu, un);
          if (m) sel = r0 + __ffs(m) - 1;
        }
        if (lane == 0) s_sel = sel;
      }
      __syncthreads();
      const int sel = s_sel;
      if (sel < 0) {   // every kept state used: the search ends (block-uniform)
        act = 0;
        continue;
      }
      const int pslot = oslot[sel];
      Epq = F64 ? __double_as_longlong(dkey_inv(okey[sel])) : (long long)(okey[sel] ^ (1ull << 63));
      ph = ohash[pslot];
      // the iteration tg that generated it and its flips there
      const int gen = ogen[pslot];
      int i, j, tg;
      if (gen) {
        tg = t_first + gen - 1;
        i = (int)(oflip[pslot] & 0xffffu);
        j = (int)(short)(oflip[pslot] >> 16);
      } else {
        const uint64_t pst = P.lst_stamp[base + pslot];
        tg = (int)(pst >> 32);
        decode_candidate(n, (uint32_t)pst, i, j);
      }
      pgen = gen;
      pi0 = i;
      pj0 = j;
      // the parent's words: its own, or its generator's with the flipped bits
#pragma unroll 1
      for (int w = tid; w < W; w += NT) {
        const uint64_t x = gen ? pw[(long long)(gen - 1) * Wm + w] ^ flip_mask(w, i, j) : P.lst_bits[(base + pslot) * Wm + w];
        pb[w] = x;
        pw[(long long)iter * Wm + w] = x;
      }
      __syncthreads();   // the parent's words; every thread has read s_sel and the used flags
      if (tid == 0) oused[pslot] = 1;
      // ------------------------------------------------------------ fields
      // x = the parent, a candidate of iteration tg's parent g
      long long* ax = aq_of(P, b, t);
      if (tg >= 1 && tg > ring_t0 && tg < t && t - tg < P.ring_n) {
        const long long* ag = aq_of(P, b, tg);
        const long long* __restrict__ Ji = Jq + (long long)i * d.n_pad;   // row i = column i
        const long long* __restrict__ Jj = Jq + (long long)max(j, 0) * d.n_pad;
        // one site per thread and pass, pipelined: the next site's three loads are issued before
        // the current site's fields are formed. With s_g = -s_x at the flipped sites i, j,
        //   aq_x,k = s_x,k s_g,k aq_g,k + 4 s_x,k (s_g,i Jq_ik + s_g,j Jq_jk),
        // s_g,i = +1 where the parent's bit i is set (exact int64). The sites up to the guessed cut
        // are listed and counted into their buckets on the way.
        const bool pi = sigma_of(pb, i) != 0;
        const bool pj = j >= 0 && sigma_of(pb, j) != 0;
        long long g_n = 0, i_n = 0, j_n = 0;
        auto load = [&](int k) {
          if (k < n) {
            g_n = ag[k];
            i_n = Ji[k];
            if (j >= 0) j_n = Jj[k];
          }
        };
        load(tid);
#pragma unroll 1
        for (int k0 = 0; k0 < n; k0 += NT) {
          const int k = k0 + tid;
          const long long vg = g_n, vi = i_n, vj = j_n;
          load(k + NT);
          bool in = false;
          float v = 0.f;
          int sx = 0;
          if (k < n) {
            sx = sigma_of(pb, k);
            const long long tt = (pi ? vi : -vi) + (j >= 0 ? (pj ? vj : -vj) : 0);
            const long long aq = ((k == i || k == j) ? -vg : vg) + (sx ? -4 * tt : 4 * tt);
            v = __ll2float_rn(aq) * scale_q;
            ax[k] = aq;
            mn = fminf(mn, v);
            mx = fmaxf(mx, v);
            in = ranged && v <= cut;
          }
          const unsigned m = __ballot_sync(0xffffffffu, in);
          if (m) {
            int e = 0;
            if (lane == 0) e = atomicAdd(&s_cn, __popc(m));
            e = __shfl_sync(0xffffffffu, e, 0) + __popc(m & ((1u << lane) - 1u));
            if (in) {
              LS.ua[e] = v;
              LS.us[e] = (unsigned short)(k | (sx << 15));
              atomicAdd(&bcur[sparse_bucket(v, lo, inv)], 1);
            }
          }
        }
      } else {
        fields_full(P, d, pb, ax);   // no stored generator
        ranged = false;
      }
    } else {
      __syncthreads();   // the counters and tables are cleared
    }
    if (!F64 && iter == 0 && P.e0_pend[b]) form_e0();
    // ---------------------------------------------------------------- near states
    // the kept states one or two flips from the parent: the only candidates that can be
    // duplicates, each equal to exactly one. A state of the parent's own generation differs from it
    // by the symmetric difference of their flips. Any other's hash XOR the parent's decodes to the
    // flips it would be (near_sites), and only then are the words compared: the state is its
    // generator's words with two flips at most, so its difference from the parent has to be exactly
    // the bits that the four flips leave.
#pragma unroll 1
    for (int r = tid; r < cnt; r += NT) {
      const int g = ogen[r];
      int i, j;
      const int ci = (int)(oflip[r] & 0xffffu), cj = (int)(short)(oflip[r] >> 16);   // (of a state of this launch)
      if (g && g == pgen) {
        const bool a = ci != pi0 && ci != pj0, c = cj >= 0 && cj != pi0 && cj != pj0;
        const bool e = pi0 != ci && pi0 != cj, f = pj0 >= 0 && pj0 != ci && pj0 != cj;
        const int m = a + c + e + f;
        if (m == 0 || m > 2) continue;
        const int x = a ? ci : c ? cj : e ? pi0 : pj0;     // the first and the last of them
        const int y = f ? pj0 : e ? pi0 : c ? cj : ci;
        i = min(x, y);
        j = m == 2 ? max(x, y) : -1;
      } else {
        if (!near_sites(ohash[r] ^ ph, P.gf, P.zob, n, i, j)) continue;
        const uint64_t* src = g ? pw + (long long)(g - 1) * Wm : P.lst_bits + (base + r) * Wm;
        uint64_t diff = 0;
#pragma unroll 1
        for (int w = 0; w < W; ++w)
          diff |= src[w] ^ pb[w] ^ flip_mask(w, i, j) ^ (g ? flip_mask(w, ci, cj) : 0ull);
        if (diff) continue;
      }
      const uint32_t c = j < 0 ? (uint32_t)i : pair_index(n, i, j);
      atomicAdd(&s_near, 1);
      uint32_t pos = chash(c) & (HT - 1);
#pragma unroll 1
      while (atomicCAS(&htab[pos], kNoCand, c) != kNoCand) pos = (pos + 1) & (HT - 1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) {
      wf[warp] = mn;
      wf[NW + warp] = mx;
    }
    __syncthreads();   // the fields, their range, the listed sites and the near states are complete
    const int k = K1 + s_near;
    float amin = wf[0], amax = wf[NW];
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      amin = fminf(amin, wf[w]);
      amax = fmaxf(amax, wf[NW + w]);
    }
    // ---------------------------------------------------------------- candidate sites in order
    int cn;
    if (ranged) {   // block-uniform
      cn = s_cn;
      if (warp == 0) bucket_starts(bcur, bs);
      __syncthreads();
#pragma unroll 1
      for (int e = tid; e < cn; e += NT) {
        const float v = LS.ua[e];
        const unsigned short s = LS.us[e];
        const int q = atomicAdd(&bcur[sparse_bucket(v, lo, inv)], 1);
        oa[q] = v;
        os[q] = s;
        orm[q] = rm[s & 0x7fff];
      }
      __syncthreads();
    } else {
      cut = INFINITY;
      cn = low_sites_again(aqb, rm, n, scale_q, pb, LS, &s_cn, false, amin, amax, cut, lo, inv);
    }
    // ---------------------------------------------------------------- bound
    // an upper bound U of the k-th lowest candidate energy change: the k-th lowest among the flips of
    // the lowest listed sites (any subset of the candidates bounds it)
    int nu = 0;
    if (EX)
      for (int w = 0; w < W; ++w) nu += __popcll(pb[w]);
    const int Ccand = EX ? nu * (n - nu) : n * (n + 1) / 2;
    float Uf = s_u;
    // (s_set: in the last iteration the last kept energy was the lower threshold and left at most K+1)
    if (Ccand > k && k <= kSubMax && !s_set) {
      const int want = min(3 * k, kSubMax);
      int t0 = 0, t1 = 0;
      if (EX) {
        const int nd = n - nu;
        int m0 = max(1, (int)sqrtf((float)want));
#pragma unroll 1
        while (m0 * m0 < want) ++m0;
#pragma unroll 1
        while (m0 > 1 && (m0 - 1) * (m0 - 1) >= want) --m0;
        int mu = min(nu, m0);
        int md = min(nd, (want + mu - 1) / mu);
        mu = min(nu, (want + md - 1) / md);
        if (mu + md > kSubSites) {
          if (mu <= kSubSites / 2) md = kSubSites - mu;
          else if (md <= kSubSites / 2) mu = kSubSites - md;
          else mu = md = kSubSites / 2;
        }
        t0 = mu;   // down spins (sigma = 1)
        t1 = md;   // up spins
      } else {
        int m = max(1, (int)((sqrtf(8.f * (float)want + 1.f) - 1.f) * 0.5f));
#pragma unroll 1
        while (m * (m + 1) / 2 < want) ++m;
#pragma unroll 1
        while (m > 1 && (m - 1) * m / 2 >= want) --m;
        t0 = min(min(m, n), kSubSites);
      }
      int m0 = 0, m1 = 0;
      for (int again = 0; again < 2; ++again) {
        if (EX) {
          // the first t0 down and t1 up positions of the order
          if (warp == 0) {
            int c0 = 0, c1 = 0;
            for (int q0 = 0; q0 < cn && (c0 < t0 || c1 < t1); q0 += 32) {
              const int q = q0 + lane;
              const bool in = q < cn, dn = in && (os[q] >> 15);
              const unsigned b0 = __ballot_sync(0xffffffffu, dn), b1 = __ballot_sync(0xffffffffu, in && !dn);
              const unsigned below = (1u << lane) - 1u;
              const int p = dn ? c0 + __popc(b0 & below) : c1 + __popc(b1 & below);
              if (in && p < (dn ? t0 : t1)) s_ex[dn ? p : t0 + p] = (unsigned short)q;
              c0 += __popc(b0);
              c1 += __popc(b1);
            }
            if (lane == 0) {
              s_m0 = min(c0, t0);
              s_m1 = min(c1, t1);
            }
          }
          __syncthreads();
          m0 = s_m0;
          m1 = s_m1;
        } else {
          m0 = min(t0, cn);
        }
        if (cn == n || (m0 == t0 && (!EX || m1 == t1))) break;
        // (rare) too few listed sites: every site
        cut = INFINITY;
        cn = low_sites_again(aqb, rm, n, scale_q, pb, LS, &s_cn, true, amin, amax, cut, lo, inv);
      }
      const int M = EX ? m0 * m1 : m0 * (m0 + 1) / 2;
      if (M >= k) {   // block-uniform
        // the values are binned as they are formed, over a range that holds nearly all of them (values
        // outside clamp to the end bins, which keeps the binning monotone)
        const float top = EX ? __fadd_rn(oa[s_ex[m0 - 1]], oa[s_ex[t0 + m1 - 1]]) : 2.f * oa[m0 - 1];
        const float lo_b = __fsub_rd(__fadd_rd(amin, amin), d.j4max);
        const float scale_v = 255.99f / fmaxf(__fadd_ru(top, d.j4max) - lo_b, 1e-30f);
        auto put_value = [&](float v) {
          const int bin = min(255, max(0, (int)((v - lo_b) * scale_v)));
          atomicAdd(&vhist[bin], 1);
          atomicMax(&vmax[bin], fkey(v));
        };
        auto pair_value = [&](int x, int y) {
          const unsigned sx = os[x], sy = os[y];
          const float j4 = J4[(long long)(sx & 0x7fff) * d.n_pad + (sy & 0x7fff)];
          put_value(oa[x] + (oa[y] + (((sx ^ sy) & 0x8000u) ? -j4 : j4)));
        };
        if (!EX) {
          // the sites' own flips, then their pairs row by row: warp w takes the rows x = w, w + NW, ..
#pragma unroll 1
          for (int q = tid; q < m0; q += NT) put_value(oa[q]);
#pragma unroll 1
          for (int x = warp; x < m0; x += NW)
            for (int y = x + 1 + lane; y < m0; y += 32) pair_value(x, y);
        } else {
#pragma unroll 1
          for (int x = warp; x < m0; x += NW)
            for (int y = lane; y < m1; y += 32) pair_value(s_ex[x], s_ex[t0 + y]);
        }
        // U = the largest value in the bins up to the one holding the k-th smallest (binning is
        // monotone, so at least k values are <= U): every warp alike
        __syncthreads();
        int bsel, within;
        find_bin(vhist, k - 1, bsel, within);
        unsigned mk = 0u;
#pragma unroll 1
        for (int x = lane; x <= bsel; x += 32) mk = max(mk, vmax[x]);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) mk = max(mk, __shfl_xor_sync(0xffffffffu, mk, o));
        Uf = fminf(Uf, fkey_inv(mk));
      }
    }
    float thr;
    {
      // |dE~ - dE| <= delta: a and 4J are fl32 of exact values; the scan adds one FMA rounding
      // and one subtraction rounding (factor 8 margin). Everything in FP32 rounded up; T - Ep
      // from the exact integer keys, scaled by the power of two 2^-q. (Every thread forms the
      // same value from the same operands.)
      const unsigned long long kT = okey[K1 - 1];
      // FP64 mode: E' = fl(E_p + dE) < T needs dE < T - E_p, and E' at or below the k-th lowest needs dE
      // within an ulp of E' of its dE. An imported E_p can be any finite number, so four ulps of E_p join
      // delta (that ulp is at most two of E_p's, or below 2^-20 of |dE|); of a computed E_p they are
      // nothing beside it (|E_p| <= n (|a|max + n j4max / 4), n <= 1024), nor are the roundings of the FP64
      // fields; the grid 2^-q (2^q sum |J| >= 2^50) puts a_i + a_j off by at most 2 n 2^-q <= 2^-22 j4max,
      // half of delta's margin.
      const float tE = (cnt != K1) ? INFINITY
                       : F64 ? __double2float_ru(__dsub_ru(dkey_inv(kT), __longlong_as_double(Epq)))
                             : __fmul_ru(__ll2float_ru((long long)(kT ^ (1ull << 63)) - Epq), scale_q);
      const float tt = fminf(tE, Uf);
      const float big = __fadd_ru(__fadd_ru(__fmul_ru(3.f, fmaxf(fabsf(amin), fabsf(amax))), d.j4max),
                                  isinf(tt) ? 0.f : fabsf(tt));
      float delta = __fmul_ru(big, 0x1p-21f);
      if (F64)   // 2^(e - 1073) of E_p's exponent field e, as a float's (infinite from 2^128 on)
        delta = __fadd_ru(delta, __int_as_float(min(255, max(1, (int)(Epq >> 52 & 0x7ff) - 946)) << 23));
      thr = fminf(__fadd_ru(tE, delta), __fadd_ru(Uf, 2.f * delta));
      if (tid == 0) {
        s_nset = cnt == K1 && tE <= Uf;
        s_thr[0] = thr;
        s_thr[1] = 4.f * delta;   // (the next pass's delta is at most twice this one's)
      }
    }
    // every live row, single and partner has a_i <= need (rows: thr - a_i >= amin - rm_i, rm_i <= j4max;
    // partners below); the listed sites have to reach it
    const float need = fmaxf(thr, __fadd_ru(__fadd_ru(__fsub_ru(thr, amin), d.j4max),
                                            __fmul_ru(0x1p-20f, fabsf(amin) + d.j4max + (isinf(thr) ? 0.f : fabsf(thr)))));
    __syncthreads();   // the bound's values have been read: their place takes the rows' offsets
    if (need > cut && cn < n) {   // block-uniform, rare
      cut = need;
      cn = low_sites_again(aqb, rm, n, scale_q, pb, LS, &s_cn, true, amin, amax, cut, lo, inv);
    }
    // ---------------------------------------------------------------- scan (pairs; the single
    // flips, dE_i = a_i, no candidates under exchanges, are tested with the rows)
    {
      // the row of each pair, while the pairs fit the space of the sites as listed
      unsigned short* rowof = reinterpret_cast<unsigned short*>(smem + L.ua);
      const int rcap = P.NP * 3;
      const int cs = F64 && s_hold ? 0 : cn;
      const int per = (cs + NT - 1) / NT, q0 = min(cs, tid * per), q1 = min(cs, q0 + per);
      int sum = 0;
#pragma unroll 1
      for (int q = q0; q < q1; ++q) {
        const float ai = oa[q], r = orm[q];
        if (!EX && ai <= thr) put_surv(atomicAdd(&s_ns, 1), surv_entry(os[q] & 0x7fff, -1));
        const float c = __fsub_rn(thr, ai);
        int len = 0;
        if (c >= __fsub_rd(amin, r)) {   // a live row: its partners have a_j < nextup(c) + r
          const float up = __fadd_ru(__fmaf_ru(fabsf(c), 0x1p-23f, c), 1.2e-38f);   // >= nextup(c)
          len = max(0, bs[sparse_bucket(__fadd_ru(up, r), lo, inv) + 1] - q - 1);
        }
        pc[q] = len;
        sum += len;
      }
      int inc = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      if (lane == 31) s_w[warp] = inc;
      __syncthreads();
      int acc = inc - sum, tot = 0;
#pragma unroll
      for (int w = 0; w < NW; ++w) {
        const int x = s_w[w];
        if (w < warp) acc += x;
        tot += x;
      }
#pragma unroll 1
      for (int q = q0; q < q1; ++q) {
        const int x = pc[q];
        pc[q] = acc;
#pragma unroll 1
        for (int e = acc, e1 = min(acc + x, rcap); e < e1; ++e) rowof[e] = (unsigned short)q;
        acc += x;
      }
      __syncthreads();
      const bool direct = tot <= rcap;   // every pair's row in rowof (block-uniform)
      // one pair per thread and pass, pipelined: the coupling load of the next pass's pair is
      // issued before the current pair is tested
      int ij_n = 0;
      float cv_n = 0.f, av_n = 0.f, jv_n = 0.f;
      bool ok_n = false, neg_n = false;
      auto stage = [&](int e) {
        ok_n = false;
        if (e < tot) {
          int q = 0;
          if (direct) {
            q = rowof[e];
          } else {
            int hi = cn;
#pragma unroll 1
            while (hi - q > 1) {
              const int mid = (q + hi) >> 1;
              if (pc[mid] <= e) q = mid; else hi = mid;
            }
          }
          const int q2 = q + 1 + e - pc[q];
          const int si = os[q], sj = os[q2];
          const int i = si & 0x7fff, j = sj & 0x7fff;
          ij_n = min(i, j) | (max(i, j) << 16);
          neg_n = ((si ^ sj) & 0x8000) != 0;
          cv_n = __fsub_rn(thr, oa[q]);
          av_n = oa[q2];
          ok_n = !EX || neg_n;
          if (ok_n) jv_n = J4[(long long)i * d.n_pad + j];
        }
      };
      stage(tid);
      for (int u0 = 0; u0 < tot; u0 += NT) {
        const int ij = ij_n;
        const float cv = cv_n, av = av_n, jv = jv_n;
        const bool ok = ok_n, neg = neg_n;
        stage(u0 + NT + tid);
        bool hit = false;
        if (ok) {
          ++nev;
          hit = fmaf(neg ? -1.f : 1.f, jv, av) <= cv;
        }
        const unsigned m = __ballot_sync(0xffffffffu, hit);
        if (m) {
          const int leader = __ffs(m) - 1;
          int sb = 0;
          if (lane == leader) sb = atomicAdd(&s_ns, __popc(m));
          sb = __shfl_sync(0xffffffffu, sb, leader);
          const int slot = sb + __popc(m & ((1u << lane) - 1u));
          if (hit) put_surv(slot, surv_entry(ij & 0xffff, ij >> 16));
        }
      }
    }
    __syncthreads();   // every survivor written; the scan's scratch is free
    const int S = s_ns;
    // Block-uniform, rare: the k-th lowest dE of the cap survivors held bounds that of all candidates, and
    // the iteration runs again with it, each time over fewer (FP64 mode: where it tells none apart, with
    // the survivors by their defining energies in place of the scan's); an error only when more than the
    // buffer holds are equal
    if (S > cap) {
      const float v = kth_survivor(ssv, surv, cap, K1 + s_near, aqb, scale_q, J4, d.n_pad, pb, reinterpret_cast<int*>(pc));
      const bool lower = __fadd_ru(v, s_thr[1]) < s_thr[0];
      __syncthreads();
      int held = cap + 1;
      if (F64 && !lower)
        held = exact_survivors(P, aqb, __longlong_as_double(Epq), cnt == K1 ? dkey_inv(okey[K1 - 1]) : INFINITY, K1 + s_near, &s_ns);
      const bool again = lower || held <= cap;
      if (tid == 0) {
        if (!again) atomicOr(P.status, kStatCapacity);
        else if (!(ext && iter == 0)) oused[oslot[s_sel]] = 0;
        s_u = lower ? v : INFINITY;
        if (F64) s_hold = held <= cap ? held + 1 : 0;
      }
      if (again) --iter; else act = 0;
      __syncthreads();
      continue;
    }
    if (!(ext && iter == 0)) {   // (that one has been counted where it was picked)
      ++nprod;
      if (EX) {
        int down = 0;
#pragma unroll 1
        for (int w = 0; w < W; ++w) down += __popcll(pb[w]);
        npair += (unsigned)(down * (n - down));
      }
    }
    if (tid == 0) {
      s_u = INFINITY;
      if (F64) s_hold = 0;
    }
    // the next iteration's guess: this one's need and a quarter of its span as a margin (the bound and
    // the lowest a_i move by a few per cent of the span per iteration; a guess too low costs a second
    // pass over the sites, one too high longer lists)
    cut = need + 0.25f * (need - amin);
    set_buckets(amin, amax, cut, lo, inv);
    ranged = true;
    // ---------------------------------------------------------------- merge (Alg. 2)
    unsigned long long* sk = reinterpret_cast<unsigned long long*>(scr);
    const int PCs = search_pcs(cap, P.merge_cand);
    unsigned long long* se = sk + PCs;
    // after the keys: mem [256] candidates by bucket, rank [256], bucket sizes [kMB], every
    // warp's bucket starts [NW][kMB + 4]; keep_lowest's histogram overlaps the starts only
    int* mem = reinterpret_cast<int*>(se + PCs);
    int* bcnt = mem + 512;
    int* rhist = bcnt + 2 * kMB;                     // [256] (keep_lowest, before the buckets)
    nsurv += (unsigned)S;
    if constexpr (F64) {   // the survivors' sites (the scan's lists have been read: their place is free)
      unsigned* mark = reinterpret_cast<unsigned*>(scr);                 // [32]
      unsigned short* list = reinterpret_cast<unsigned short*>(mark + 32);   // [NP]
      if (tid < 32) mark[tid] = 0u;
      __syncthreads();
      for (int e = tid; e < S; e += NT) {
        int i, j;
        surv_sites((e < kSSV) ? ssv[e] : surv[e], i, j);
        // (a duplicate of a kept state is dropped before its energy counts: half of the survivors of a
        // list that has settled)
        const uint32_t c = (j < 0) ? (uint32_t)i : pair_index(n, i, j);
        uint32_t pos = chash(c) & (HT - 1), h = htab[pos];
        while (h != kNoCand && h != c) {
          pos = (pos + 1) & (HT - 1);
          h = htab[pos];
        }
        if (h == kNoCand) {
          atomicOr(&mark[i >> 5], 1u << (i & 31));
          if (j >= 0) atomicOr(&mark[j >> 5], 1u << (j & 31));
        }
      }
      __syncthreads();
      // every warp counts for itself; warp w lists the words w, w + NW, ..
      const unsigned mk = mark[lane];
      int inc = __popc(mk);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
      }
      const int m = __shfl_sync(0xffffffffu, inc, 31);
      for (int w = warp; w < 32; w += NW) {
        const unsigned x = __shfl_sync(0xffffffffu, mk, w);
        const int at = __shfl_sync(0xffffffffu, inc, w) - __popc(x);
        if ((x >> lane) & 1u) list[at + __popc(x & ((1u << lane) - 1u))] = (unsigned short)(w * 32 + lane);
      }
      __syncthreads();
      fields_f64(P, d, pb, aqb, list, m, ad);
      __syncthreads();
    }
#pragma unroll 1
    for (int x = tid; x < kMB; x += NT) bcnt[x] = 0;   // (after the sites' list: the places overlap)
    const bool big = S > PCs;
    if (big) {
      const long long stride = next_pow2(max(cap, 256));
      sk = P.mrg_scratch + (long long)b * 2 * stride;
      se = sk + stride;
    }
    const long long Tq = (!F64 && cnt == K1) ? (long long)(okey[K1 - 1] ^ (1ull << 63)) : LLONG_MAX;
    const double T = (F64 && cnt == K1) ? dkey_inv(okey[K1 - 1]) : INFINITY;
    unsigned long long kmn = ~0ull, kmx = 0;
    for (int u0 = 0; u0 < S; u0 += NT) {
      const int e = u0 + tid;
      bool keep = false;
      unsigned long long kk = 0, ent = 0;
      if (e < S) {
        ent = (e < kSSV) ? ssv[e] : surv[e];
        int i, j;
        surv_sites(ent, i, j);
        ent |= (j < 0) ? (uint32_t)i : pair_index(n, i, j);
        if constexpr (F64) {
          const double de = (j < 0) ? ad[i] : dE64(ad[i], ad[j], P.J64[d.off_mat + (long long)i * d.n_pad + j],
                                                   sigma_of(pb, i) ^ sigma_of(pb, j));
          const double e = __dadd_rn(__longlong_as_double(Epq), de);
          kk = dkey(e);
          keep = e < T;   // Alg. 2: strict <
        } else {
          long long de = aqb[i];
          if (j >= 0) {
            const long long jq = Jq[(long long)i * d.n_pad + j];
            de += aqb[j] + ((sigma_of(pb, i) ^ sigma_of(pb, j)) ? -4 * jq : 4 * jq);
          }
          const long long eq = Epq + de;
          kk = qkey(eq);
          keep = eq < Tq;   // Alg. 2: strict <
        }
        if (keep) {
          const uint32_t c = (uint32_t)ent;
#pragma unroll 1
          for (uint32_t pos = chash(c) & (HT - 1); htab[pos] != kNoCand; pos = (pos + 1) & (HT - 1))
            if (htab[pos] == c) {
              keep = false;   // a kept state (the binary search of Alg. 2)
              break;
            }
        }
      }
      const unsigned bal = __ballot_sync(0xffffffffu, keep);
      if (bal) {
        int wb = 0;
        if (lane == 0) wb = atomicAdd(&s_nv, __popc(bal));
        wb = __shfl_sync(0xffffffffu, wb, 0);
        if (keep) {
          const int slot = wb + __popc(bal & ((1u << lane) - 1));
          sk[slot] = kk;
          se[slot] = ent;
          kmn = min(kmn, kk);
          kmx = max(kmx, kk);
        }
      }
    }
    kmn = warp_min64(kmn);
    kmx = warp_max64(kmx);
    if (lane == 0) {
      s_kmm[warp] = kmn;
      s_kmm[NW + warp] = kmx;
    }
    __syncthreads();
    int nv = s_nv;
    // more kept candidates than the buckets take at once: only the K+1 lowest can enter the list
    if (nv > 256 && nv > K1) nv = keep_lowest(sk, se, nv, K1, rhist, s_w);
    unsigned long long kmin = s_kmm[0], kmax = s_kmm[NW];
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      kmin = min(kmin, s_kmm[w]);
      kmax = max(kmax, s_kmm[NW + w]);
    }
    // the new candidates' order (E, c) as one 64-bit value, (E - Emin) << cb | c, where the keys'
    // span leaves room for c (always but for extreme ranges); equal energies are ordered by c
    const uint32_t n_cand = (uint32_t)n + (uint32_t)((long long)n * (n - 1) / 2);
    const int cb = 32 - __clz((int)n_cand);
    const bool bucketed = nv <= 256 && ((kmax - kmin) >> (64 - cb)) == 0;   // block-uniform
    int* rnk = mem + 256;              // [256] place of each new candidate among the new ones
    int* bst = bcnt + kMB + warp * (kMB + 4);   // this warp's bucket starts [kMB + 1]
    const int sh = max(0, 64 - __clzll((long long)(((kmax - kmin) << cb) | ((1ull << cb) - 1))) - kMBits);
    if (bucketed) {
      // without sorting them: the order values packed in place, a counting sort by their top
      // bits into kMB buckets, then a count within the bucket (the values are distinct)
      constexpr int V = NT >= 256 ? 1 : 256 / NT;
      int wb[V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int p = tid + v * NT;
        wb[v] = 0;
        if (p < nv) {
          sk[p] = ((sk[p] - kmin) << cb) | (uint32_t)se[p];
          wb[v] = atomicAdd(&bcnt[(int)(sk[p] >> sh)], 1);
        }
      }
      __syncthreads();
      {   // every warp forms the bucket starts itself (no barrier)
        int x[kMB / 32], sum = 0;
#pragma unroll
        for (int q = 0; q < kMB / 32; ++q) {
          x[q] = bcnt[lane * (kMB / 32) + q];
          sum += x[q];
        }
        int inc = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += y;
        }
        int acc = inc - sum;
#pragma unroll
        for (int q = 0; q < kMB / 32; ++q) {
          bst[lane * (kMB / 32) + q] = acc;
          acc += x[q];
        }
        if (lane == 31) bst[kMB] = acc;
        __syncwarp();
      }
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const int p = tid + v * NT;
        if (p < nv) mem[bst[(int)(sk[p] >> sh)] + wb[v]] = p;
      }
      __syncthreads();
#pragma unroll 1
      for (int p = tid; p < nv; p += NT) {
        const unsigned long long vp = sk[p];
        const int bk = (int)(vp >> sh);
        int r = bst[bk];
#pragma unroll 1
        for (int q = bst[bk], q1 = bst[bk + 1]; q < q1; ++q) r += (sk[mem[q]] < vp) ? 1 : 0;
        rnk[p] = r;
      }
    } else {
      sort_pairs_any(sk, se, nv);   // rare: sorted in place, the place of p is p (nv may exceed rnk's)
    }
    // old entries: their place plus the new candidates strictly below their key
#pragma unroll 1
    for (int o = tid; o < cnt; o += NT) {
      const unsigned long long ko = okey[o];
      int lo;
      if (nv == 0 || ko <= kmin) {
        lo = 0;
      } else if (ko > kmax) {
        lo = nv;
      } else if (bucketed) {
        const unsigned long long vo = (ko - kmin) << cb;   // below every new value of energy ko
        const int bk = (int)(vo >> sh);
        lo = bst[bk];
#pragma unroll 1
        for (int q = bst[bk], q1 = bst[bk + 1]; q < q1; ++q) lo += (sk[mem[q]] < vo) ? 1 : 0;
      } else {
        lo = 0;
        int hi = nv;
#pragma unroll 1
        while (lo < hi) {
          const int mid = (lo + hi) >> 1;
          if (sk[mid] < ko) lo = mid + 1; else hi = mid;
        }
      }
      const int rank = o + lo;
      if (rank < K1) {
        oslotN[rank] = oslot[o];
        okeyN[rank] = ko;
      } else {
        atomicMin(&s_ocut, o);
      }
    }
    __syncthreads();
    const int ocut = s_ocut, n_ev = cnt - ocut;
#pragma unroll 1
    for (int p = tid; p < nv; p += NT) {
      const unsigned long long kp = bucketed ? (sk[p] >> cb) + kmin : sk[p];
      int lo = 0, hi = cnt;
#pragma unroll 1
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (okey[mid] <= kp) lo = mid + 1; else hi = mid;
      }
      const int rn = bucketed ? rnk[p] : p, rank = rn + lo;
      if (rank >= K1) continue;
      const int slot = (rn < n_ev) ? oslot[ocut + rn] : cnt + (rn - n_ev);
      int i, j;
      surv_sites(se[p], i, j);
      // the state is kept as (iteration, flips): its words are written at the end of the launch
      oflip[slot] = (uint32_t)i | ((uint32_t)j << 16);
      ohash[slot] = ph ^ P.zob[i] ^ ((j >= 0) ? P.zob[j] : 0ull);
      oused[slot] = 0;
      ogen[slot] = (uint8_t)(iter + 1);
      oslotN[rank] = slot;
      okeyN[rank] = kp;
    }
    cnt = min(K1, cnt + nv);
    cur ^= 1;
    __syncthreads();   // the new order is complete before the next pick reads it
  }
  // ------------------------------------------------------------------ write back
  const unsigned long long* okey = cur ? okeyB : okeyA;
  const int* oslot = cur ? oslotB : oslotA;
#pragma unroll 1
  for (int r = tid; r < cnt; r += NT) {
    const int slot = oslot[r];
    P.lst_key[base + r] = okey[r];
    P.lst_ord[base + r] = slot;
    P.lst_used[base + slot] = oused[slot];
    if (ogen[slot]) {
      if (F64) P.lst_E[base + slot] = dkey_inv(okey[r]);
      else P.lst_q[base + slot] = (long long)(okey[r] ^ (1ull << 63));
      const int i = (int)(oflip[slot] & 0xffffu), j = (int)(short)(oflip[slot] >> 16);
      P.lst_stamp[base + slot] = ((uint64_t)(t_first + ogen[slot] - 1) << 32) | (j < 0 ? (uint32_t)i : pair_index(n, i, j));
      P.lst_hash[base + slot] = ohash[slot];
    }
  }
#pragma unroll 1
  for (int s = warp; s < cnt; s += NW) {   // (the slots in use are 0 .. cnt - 1)
    const int g = ogen[s];
    if (!g) continue;
    const int i = (int)(oflip[s] & 0xffffu), j = (int)(short)(oflip[s] >> 16);
#pragma unroll 1
    for (int w = lane; w < W; w += 32)
      P.lst_bits[(base + s) * Wm + w] = pw[(long long)(g - 1) * Wm + w] ^ flip_mask(w, i, j);
  }
  if (act0)   // the last parent (what the per-kernel form leaves in these fields)
    for (int w = tid; w < W; w += NT) P.par_bits[(long long)b * Wm + w] = pb[w];
  if (tid == 0) {
    P.lst_count[b] = cnt;
    P.iter_t[b] = t_first + n_iters - 1;
    if (act0) {
      P.active[b] = act;
      if (F64) P.par_E[b] = __longlong_as_double(Epq);
      else P.par_q[b] = Epq;
      P.par_hash[b] = ph;
      P.nprod[b] += nprod;
      P.npair[b] += EX ? (unsigned long long)npair : (unsigned long long)nprod * (unsigned)(n * (n - 1) / 2);
      if (nsurv) atomicAdd(P.surv_tot + (b & 63), (unsigned long long)nsurv);
    }
  }
  if (act0) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) nev += __shfl_xor_sync(0xffffffffu, nev, o);
    if (lane == 0 && nev) atomicAdd(P.eval_cnt + (b & 63), (unsigned long long)nev);
  }
}

template <int FL, bool F64, int NT>
static cudaError_t launch_search_as(const DevPtrs& P, int n_iters, int ext, cudaStream_t s) {
  const SearchLayout L = search_layout(P.NP, P.Wmax, P.K1, P.cap, P.merge_cand, NT / 32, F64);
  const size_t sm = (size_t)L.total;
  const cudaError_t e = allow_smem((const void*)k_search<FL, F64, NT>, sm);
  if (e != cudaSuccess) return e;
  k_search<FL, F64, NT><<<P.B, NT, sm, s>>>(P, n_iters, ext);
  return cudaGetLastError();
}

template <bool F64, int NT>
static cudaError_t launch_search_nt(const DevPtrs& P, int n_iters, int ext, cudaStream_t s) {
  return P.flips == QIS_FLIPS_EXCHANGE ? launch_search_as<QIS_FLIPS_EXCHANGE, F64, NT>(P, n_iters, ext, s)
                                       : launch_search_as<QIS_FLIPS_SINGLE_PAIR, F64, NT>(P, n_iters, ext, s);
}

cudaError_t launch_search(const DevPtrs& P, int n_iters, int ext, cudaStream_t s) {
  if (n_iters <= 0 || P.B == 0) return cudaSuccess;
  // 256 threads shorten a search's chain of phases, 128 leave fewer of them waiting in each: 256 while
  // all blocks are resident at once with either (four of 256 per SM). 100 iterations of n = 300, K = 100
  // with 256 and 128 threads: 128 searches 1.22 and 1.65 ms, 512 1.63 and 1.87, 600 1.67 and 1.93, 640
  // 2.54 and 1.94, 1024 3.05 and 2.23; FP64 n = 100: 150 searches 1.69 and 1.99, 600 2.13 and 2.17, 640
  // 3.20 and 2.24. At n <= 128 the split modes' passes do not fill 256 threads: 600 searches of n = 60
  // 1.02 and 0.95 ms, 4 of n = 16 72 and 70 us in 8 iterations.
  const bool wide = P.B <= 4 * P.sms && (P.mode == QIS_FP64 || P.NP > kPad);
  if (P.mode == QIS_FP64)
    return wide ? launch_search_nt<true, 256>(P, n_iters, ext, s) : launch_search_nt<true, 128>(P, n_iters, ext, s);
  return wide ? launch_search_nt<false, 256>(P, n_iters, ext, s) : launch_search_nt<false, 128>(P, n_iters, ext, s);
}

}  // namespace qis
