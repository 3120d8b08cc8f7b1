// qis_single.cu -- every iteration of one search in one thread block, single flips only (the J = 1
// flip set), for any n (up to 16384 sites).
//
// The iteration of Alg. 3 as in qis_search.cu, in the split precision modes, with what single
// flips allow: the candidates are the n sites, so one histogram of a_i finds those that can enter
// the list (the sites up to the bin of the (K+1+near)-th lowest: a superset of that many lowest
// candidates, of which `near` at most are kept states already), and each is decided by its exact
// key at once. Per iteration the block
//   pick    takes the first unused kept state in key order
//   fields  forms its exact fields from its generator's (aq ring) and one coupling row, and counts
//           a_i into the histogram on the way (over the range of the previous parent: values
//           outside it fall into the end bins, which keeps the binning monotone)
//   near    finds the kept states one flip away: the Zobrist hash of site i carries i in its low
//           14 bits, so a kept state's hash XOR the parent's names the site if it is one flip away,
//           and only then are the words compared (by a warp)
//   merge   collects the candidates below the last kept energy, ranks them by buckets of their
//           packed (E, c) values, and writes the first K+1 of the old list and them
// The kept list (keys, stamps, hashes, used flags) stays in shared memory, and a new state is
// kept as (iteration, site): its words are its parent's, which are stored per iteration, with
// one bit flipped, and are written into the list once, at the end of the call. Rewriting them in
// every iteration would move up to (K+1) n / 8 bytes per iteration (150 KB at n = 10000), and
// comparing words for the near states as much again.
//
// What bounds it: the chain of dependent steps of an iteration (six barriers) where few searches
// leave one block per SM, so the block is as large as the sites can use; where the searches fill
// the SMs, the field update's 24 bytes per site (generator's fields and coupling row read, the
// parent's fields written).
#include <algorithm>

#include "qis_block.cuh"

namespace qis {

constexpr int kSgBuf = 512;            // new candidates held in shared memory

struct SingleLayout {
  int a, pb, okey0, okey1, ostamp, ohash, sk, se, oslot0, oslot1, hist, mem, bcnt, bst, dupm, oused, ogen, total;
};

__host__ __device__ inline SingleLayout single_layout(int NP, int Wmax, int K1, int warps) {
  SingleLayout L;
  int o = 0;
  auto take = [&](int bytes) {
    o = align_up(o, 16);
    const int r = o;
    o += bytes;
    return r;
  };
  L.a = take(NP * 4);
  L.pb = take(Wmax * 8);
  L.okey0 = take(K1 * 8);
  L.okey1 = take(K1 * 8);
  L.ostamp = take(K1 * 8);
  L.ohash = take(K1 * 8);
  L.sk = take(kSgBuf * 8);
  L.se = take(kSgBuf * 8);
  L.oslot0 = take(K1 * 4);
  L.oslot1 = take(K1 * 4);
  L.hist = take(256 * 4);
  L.mem = take(512 * 4);
  L.bcnt = take(kMB * 4);
  L.bst = take((warps < 8 ? warps : 8) * (kMB + 4) * 4);   // the first 256 threads rank
  L.dupm = take(NP / 8);
  L.oused = take(K1);
  L.ogen = take(K1);
  L.total = align_up(o, 16);
  return L;
}

// Fields of a parent without a stored generator, from scratch (rare): fq_k = hq_k + sum_j s_j Jq_jk.
static __device__ __noinline__ void single_fields_full(const DevPtrs& P, const InstDesc& d, const uint64_t* pb,
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

// n_iters >= 1, at most P.pw_n. ext: the first iteration's parent was picked and its fields
// computed by the kernels launched before this one.
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) k_single(DevPtrs P, int n_iters, int ext) {
  constexpr int NW = NT / 32;
  extern __shared__ __align__(16) unsigned char smem[];
  const int b = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K1 = P.K1, Wm = P.Wmax, cap = P.cap;
  const long long base = (long long)b * K1;
  const SingleLayout L = single_layout(P.NP, Wm, K1, NW);
  float* a = reinterpret_cast<float*>(smem + L.a);
  uint64_t* pb = reinterpret_cast<uint64_t*>(smem + L.pb);
  unsigned long long* okeyA = reinterpret_cast<unsigned long long*>(smem + L.okey0);
  unsigned long long* okeyB = reinterpret_cast<unsigned long long*>(smem + L.okey1);
  uint64_t* ostamp = reinterpret_cast<uint64_t*>(smem + L.ostamp);
  uint64_t* ohash = reinterpret_cast<uint64_t*>(smem + L.ohash);
  int* oslotA = reinterpret_cast<int*>(smem + L.oslot0);
  int* oslotB = reinterpret_cast<int*>(smem + L.oslot1);
  int* hist = reinterpret_cast<int*>(smem + L.hist);
  int* mem = reinterpret_cast<int*>(smem + L.mem);
  int* rnk = mem + 256;
  int* bcnt = reinterpret_cast<int*>(smem + L.bcnt);
  int* bst = reinterpret_cast<int*>(smem + L.bst) + min(warp, 7) * (kMB + 4);
  unsigned* dupm = reinterpret_cast<unsigned*>(smem + L.dupm);
  uint8_t* oused = reinterpret_cast<uint8_t*>(smem + L.oused);
  uint8_t* ogen = reinterpret_cast<uint8_t*>(smem + L.ogen);
  __shared__ int s_sel, s_near, s_nv, s_ocut, s_w[33];
  __shared__ float wf[2 * NW];
  __shared__ unsigned long long s_kmin, s_kmax, red[NW];

  const int act0 = P.active[b];
  const InstDesc d = P.inst[b / P.R];
  const int n = d.n, W = d.W;
  const int t_first = P.iter_t[b] + (ext ? 0 : 1);   // the iteration of iter = 0
  const int ring_t0 = P.ring_t0[b];
  int cnt = P.lst_count[b];
  long long Epq = P.par_q[b];
  uint64_t ph = P.par_hash[b];
  uint64_t* pw = P.pw + (long long)b * P.pw_n * Wm;   // words of the parent of iteration iter: pw + iter Wm
  for (int r = tid; r < K1; r += NT) {
    okeyA[r] = P.lst_key[base + r];
    oslotA[r] = P.lst_ord[base + r];
    ostamp[r] = P.lst_stamp[base + r];
    ohash[r] = P.lst_hash[base + r];
    oused[r] = P.lst_used[base + r];
    ogen[r] = 0;   // in lst_bits (else 1 + the iteration of this launch that generated it)
  }
  for (int w = tid; w < W; w += NT) {
    const uint64_t x = P.par_bits[(long long)b * Wm + w];
    pb[w] = x;
    if (ext) pw[w] = x;
  }
  for (int x = tid; x < 256; x += NT) hist[x] = 0;
  for (int x = tid; x < P.NP / 32; x += NT) dupm[x] = 0u;
  if (tid == 0) s_near = 0;
  float mn = INFINITY, mx = -INFINITY;   // this thread's range of a_i
  float lo = 0.f, scale = 0.f;           // the histogram's range
  bool ranged = false;
  if (act0 && ext)
    for (int i = tid; i < n; i += NT) {
      const float v = P.as32[(long long)b * P.NP + i].x;
      a[i] = v;
      mn = fminf(mn, v);
      mx = fmaxf(mx, v);
    }
  __syncthreads();
  if (act0 && ext && P.e0_pend[b]) {   // block-uniform: the list is [psi0] and psi0 is the parent
    Epq = initial_energy(P, d, pb, aq_of(P, b, t_first), reinterpret_cast<long long*>(red));
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
  }

  int act = act0, t = t_first - 1, cur = 0, nprod = 0;
  unsigned long long nsurv = 0;
  const float scale_q = (float)d.inv_scale;
  const long long* Jq = P.Jq + d.off_mat;
  auto bin_of = [&](float v) { return min(255, max(0, (int)((v - lo) * scale))); };

  for (int iter = 0; iter < n_iters; ++iter) {
    unsigned long long* okey = cur ? okeyB : okeyA;
    unsigned long long* okeyN = cur ? okeyA : okeyB;
    int* oslot = cur ? oslotB : oslotA;
    int* oslotN = cur ? oslotA : oslotB;
    t += 1;
    if (!act) continue;
    long long* ax = aq_of(P, b, t);
    if (iter > 0 || !ext) {
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
      Epq = (long long)(okey[sel] ^ (1ull << 63));
      const uint64_t pst = ostamp[pslot];
      ph = ohash[pslot];
      const int gen = ogen[pslot];
      const int tg = (int)(pst >> 32), i0 = (int)(uint32_t)pst;
      const bool stored = tg >= 1 && tg > ring_t0 && tg < t && t - tg < P.ring_n;   // the generator's fields
      for (int w = tid; w < W; w += NT) {
        const uint64_t x = gen ? pw[(long long)(gen - 1) * Wm + w] ^ ((i0 >> 6) == w ? 1ull << (i0 & 63) : 0ull)
                               : P.lst_bits[(base + pslot) * Wm + w];
        pb[w] = x;
        pw[(long long)iter * Wm + w] = x;
      }
      __syncthreads();   // the parent's words; every thread has read s_sel and the used flags
      if (tid == 0) oused[pslot] = 1;
      ++nprod;
      // ------------------------------------------------------------ fields
      // as in qis_search.cu, one flipped site i0: aq_x,k = s_x,k s_g,k aq_g,k + 4 s_x,k s_g,i0 Jq_i0k
      auto put = [&](int k, long long aq) {
        const float v = __ll2float_rn(aq) * scale_q;
        a[k] = v;
        mn = fminf(mn, v);
        mx = fmaxf(mx, v);
        if (ranged) atomicAdd(&hist[bin_of(v)], 1);
      };
      if (stored) {
        const long long* ag = aq_of(P, b, tg);   // (written by this launch)
        const long long* __restrict__ Ji = Jq + (long long)i0 * d.n_pad;
        const bool pi = sigma_of(pb, i0) != 0;
        constexpr int U = 4;   // sites per thread and pass, their loads issued together
        for (int k0 = tid; k0 < n; k0 += U * NT) {
          long long vg[U], vi[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int k = k0 + u * NT;
            vg[u] = k < n ? ag[k] : 0;
            vi[u] = k < n ? Ji[k] : 0;
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int k = k0 + u * NT;
            if (k >= n) break;
            const bool neg = (sigma_of(pb, k) != 0) == pi;   // sign of s_x,k s_g,i0
            const long long aq = (k == i0 ? -vg[u] : vg[u]) + (neg ? -4 : 4) * vi[u];
            ax[k] = aq;
            put(k, aq);
          }
        }
      } else {
        single_fields_full(P, d, pb, ax);
        for (int k = tid; k < n; k += NT) put(k, ax[k]);   // (this thread's own sites)
      }
    }
    // ---------------------------------------------------------------- kept states one flip away
    for (int r0 = warp * 32; r0 < cnt; r0 += NT) {
      const int r = r0 + lane;
      const uint64_t x = r < cnt ? ohash[r] ^ ph : 0ull;
      const int i = (int)x & kSiteMask;
      const bool hit = r < cnt && x != 0ull && i < n && P.zob[i] == x;
      for (unsigned m = __ballot_sync(0xffffffffu, hit); m; m &= m - 1) {
        const int src = __ffs(m) - 1, rr = r0 + src;
        const int site = __shfl_sync(0xffffffffu, i, src), g = ogen[rr], c = (int)(uint32_t)ostamp[rr];
        bool diff = false;
        for (int w = lane; w < W; w += 32) {
          uint64_t y = g ? pw[(long long)(g - 1) * Wm + w] : P.lst_bits[(base + rr) * Wm + w];
          if (g && (c >> 6) == w) y ^= 1ull << (c & 63);
          if ((site >> 6) == w) y ^= 1ull << (site & 63);
          diff = diff || y != pb[w];
        }
        if (!__any_sync(0xffffffffu, diff) && lane == 0) {
          atomicOr(&dupm[site >> 5], 1u << (site & 31));
          atomicAdd(&s_near, 1);
        }
      }
    }
    // ---------------------------------------------------------------- candidates
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    }
    if (lane == 0) {
      wf[warp] = mn;
      wf[NW + warp] = mx;
    }
    if (tid == 0) {
      s_nv = 0;
      s_ocut = cnt;
      s_kmin = ~0ull;
      s_kmax = 0;
    }
    for (int x = tid; x < kMB; x += NT) bcnt[x] = 0;
    __syncthreads();   // a_i, the histogram (if ranged) and the near states are complete
    float nlo = wf[0], nhi = wf[NW];
#pragma unroll
    for (int w = 1; w < NW; ++w) {
      nlo = fminf(nlo, wf[w]);
      nhi = fmaxf(nhi, wf[NW + w]);
    }
    mn = INFINITY;
    mx = -INFINITY;
    if (!ranged) {   // block-uniform: the first parent of the launch
      lo = nlo;
      scale = 255.99f / fmaxf(nhi - nlo, 1e-30f);
      for (int i = tid; i < n; i += NT) atomicAdd(&hist[bin_of(a[i])], 1);
      __syncthreads();
    }
    const int k = K1 + s_near;
    int bsel = 255, upto = n;   // the sites to decide: bins up to bsel, `upto` of them
    if (n > k) {
      int within;
      find_bin(hist, k - 1, bsel, within);
      upto = k - 1 - within + hist[bsel];
    }
    unsigned long long* sk = reinterpret_cast<unsigned long long*>(smem + L.sk);
    unsigned long long* se = reinterpret_cast<unsigned long long*>(smem + L.se);
    unsigned kth = ~0u;
    const bool fine = n > k && upto > min(kSgBuf, cap);   // block-uniform, rare (outliers, ties)
    if (fine) {
      // the bin holds too many: the k-th lowest a_i itself (radix select of the ordered keys of
      // all a_i, kept in their place), ties included
      __syncthreads();   // every thread has read the histogram
      unsigned* key = reinterpret_cast<unsigned*>(a);
      for (int i = tid; i < n; i += NT) {
        const unsigned u = __float_as_uint(a[i] + 0.f);
        key[i] = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
      }
      __syncthreads();
      kth = radix_select<unsigned>(key, n, k - 1, hist);
      int mine = 0;
      for (int i = tid; i < n; i += NT) mine += key[i] <= kth;
      int tot;
      block_exclusive_sum(mine, s_w, &tot);
      upto = tot;
    }
    if (upto > kSgBuf) {
      const long long stride = next_pow2(max(cap, 256));
      sk = P.mrg_scratch + (long long)b * 2 * stride;
      se = sk + stride;
    }
    nsurv += (unsigned long long)upto;
    // ---------------------------------------------------------------- merge (Alg. 2)
    const long long Tq = (cnt == K1) ? (long long)(okey[K1 - 1] ^ (1ull << 63)) : LLONG_MAX;
    unsigned long long kmn = ~0ull, kmx = 0;
    for (int u0 = 0; u0 < n; u0 += NT) {
      const int i = u0 + tid;
      bool keep = false;
      unsigned long long kk = 0;
      if (i < n && (fine ? reinterpret_cast<unsigned*>(a)[i] <= kth : bin_of(a[i]) <= bsel)) {
        const long long eq = Epq + ax[i];
        kk = qkey(eq);
        keep = eq < Tq && !((dupm[i >> 5] >> (i & 31)) & 1u);   // Alg. 2: strict <, not a kept state
      }
      const unsigned bal = __ballot_sync(0xffffffffu, keep);
      if (bal) {
        int wb = 0;
        if (lane == 0) wb = atomicAdd(&s_nv, __popc(bal));
        wb = __shfl_sync(0xffffffffu, wb, 0);
        const int slot = wb + __popc(bal & ((1u << lane) - 1));
        if (keep && slot < cap) {
          sk[slot] = kk;
          se[slot] = (unsigned long long)i;
          kmn = min(kmn, kk);
          kmx = max(kmx, kk);
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      kmn = min(kmn, __shfl_xor_sync(0xffffffffu, kmn, o));
      kmx = max(kmx, __shfl_xor_sync(0xffffffffu, kmx, o));
    }
    if (lane == 0 && kmn <= kmx) {
      atomicMin(&s_kmin, kmn);
      atomicMax(&s_kmax, kmx);
    }
    __syncthreads();
    int nv = s_nv;
    // (ties at the bound that cannot enter the list, however many, take no place in the buffer)
    if (nv > cap) {   // block-uniform: more candidates than the search's buffer holds
      if (tid == 0) atomicOr(P.status, kStatCapacity);
      act = 0;
      continue;
    }
    // more kept candidates than the buckets take at once: only the K+1 lowest can enter the list
    if (nv > 256 && nv > K1) nv = keep_lowest(sk, se, nv, K1, hist, s_w);
    const unsigned long long kmin = s_kmin, kmax = s_kmax;
    const int cb = 32 - __clz(n);
    const bool bucketed = nv <= 256 && ((kmax - kmin) >> (64 - cb)) == 0;   // block-uniform
    const int sh = max(0, 64 - __clzll((long long)(((kmax - kmin) << cb) | ((1ull << cb) - 1))) - kMBits);
    if (bucketed) {
      // as in qis_search.cu: the order values (E - Emin) << cb | c packed in place, a counting
      // sort by their top bits, then a count within the bucket (the values are distinct)
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
      if (warp < 8) {   // the warps that rank form the bucket starts themselves
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
      for (int p = tid; p < nv; p += NT) {
        const unsigned long long vp = sk[p];
        const int bk = (int)(vp >> sh);
        int r = bst[bk];
        for (int q = bst[bk], q1 = bst[bk + 1]; q < q1; ++q) r += (sk[mem[q]] < vp) ? 1 : 0;
        rnk[p] = r;
      }
    } else {
      sort_pairs_any(sk, se, nv);   // rare: sorted in place, the place of p is p
    }
    // old entries: their place plus the new candidates strictly below their key
    for (int o = tid; o < cnt; o += NT) {
      const unsigned long long ko = okey[o];
      int below;
      if (nv == 0 || ko <= kmin) {
        below = 0;
      } else if (ko > kmax) {
        below = nv;
      } else if (bucketed) {
        const unsigned long long vo = (ko - kmin) << cb;   // below every new value of energy ko
        const int bk = (int)(vo >> sh);
        below = bst[bk];
        for (int q = bst[bk], q1 = bst[bk + 1]; q < q1; ++q) below += (sk[mem[q]] < vo) ? 1 : 0;
      } else {
        below = 0;
        int hi = nv;
        while (below < hi) {
          const int mid = (below + hi) >> 1;
          if (sk[mid] < ko) below = mid + 1; else hi = mid;
        }
      }
      const int rank = o + below;
      if (rank < K1) {
        oslotN[rank] = oslot[o];
        okeyN[rank] = ko;
      } else {
        atomicMin(&s_ocut, o);
      }
    }
    // the next iteration's counters (this one's are read no more) and its histogram range
    for (int x = tid; x < 256; x += NT) hist[x] = 0;
    for (int x = tid; x < P.NP / 32; x += NT) dupm[x] = 0u;
    if (tid == 0) s_near = 0;
    lo = nlo;
    scale = 255.99f / fmaxf(nhi - nlo, 1e-30f);
    ranged = true;
    __syncthreads();
    const int ocut = s_ocut, n_ev = cnt - ocut;
    for (int p = tid; p < nv; p += NT) {
      const unsigned long long kp = bucketed ? (sk[p] >> cb) + kmin : sk[p];
      int lo2 = 0, hi = cnt;
      while (lo2 < hi) {
        const int mid = (lo2 + hi) >> 1;
        if (okey[mid] <= kp) lo2 = mid + 1; else hi = mid;
      }
      const int rn = bucketed ? rnk[p] : p, rank = rn + lo2;
      if (rank >= K1) continue;
      const int slot = (rn < n_ev) ? oslot[ocut + rn] : cnt + (rn - n_ev);
      const int i = (int)se[p];
      ostamp[slot] = ((uint64_t)t << 32) | (uint32_t)i;
      ohash[slot] = ph ^ P.zob[i];
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
  for (int r = tid; r < cnt; r += NT) {
    const int slot = oslot[r];
    P.lst_key[base + r] = okey[r];
    P.lst_ord[base + r] = slot;
    P.lst_used[base + slot] = oused[slot];
    if (ogen[slot]) {
      P.lst_q[base + slot] = (long long)(okey[r] ^ (1ull << 63));
      P.lst_stamp[base + slot] = ostamp[slot];
      P.lst_hash[base + slot] = ohash[slot];
    }
  }
  for (int s = warp; s < cnt; s += NW) {   // (the slots in use are 0 .. cnt - 1)
    const int g = ogen[s];
    if (!g) continue;
    const int c = (int)(uint32_t)ostamp[s];
    const uint64_t* src = pw + (long long)(g - 1) * Wm;
    for (int w = lane; w < W; w += 32)
      P.lst_bits[(base + s) * Wm + w] = src[w] ^ ((c >> 6) == w ? 1ull << (c & 63) : 0ull);
  }
  if (act0)   // the last parent (what the per-kernel form leaves in these fields)
    for (int w = tid; w < W; w += NT) P.par_bits[(long long)b * Wm + w] = pb[w];
  if (tid == 0) {
    P.lst_count[b] = cnt;
    P.iter_t[b] = t_first + n_iters - 1;
    if (act0) {
      P.active[b] = act;
      P.par_q[b] = Epq;
      P.par_hash[b] = ph;
      P.nprod[b] += nprod;
      if (nsurv) atomicAdd(P.surv_tot + (b & 63), nsurv);
    }
  }
}

template <int NT>
static cudaError_t launch_single_nt(const DevPtrs& P, int n_iters, int ext, cudaStream_t s) {
  const size_t sm = (size_t)single_layout(P.NP, P.Wmax, P.K1, NT / 32).total;
  const cudaError_t e = allow_smem((const void*)k_single<NT>, sm);
  if (e != cudaSuccess) return e;
  k_single<NT><<<P.B, NT, sm, s>>>(P, n_iters, ext);
  return cudaGetLastError();
}

// n_iters iterations, at most P.pw_n; ext: the first one's parent and fields are in place.
cudaError_t launch_single(const DevPtrs& P, int n_iters, int ext, cudaStream_t s) {
  if (n_iters <= 0 || P.B == 0) return cudaSuccess;
  // Threads per block: about two to four sites per thread, but no more than the block's share of
  // the SM's 1024 threads (64 registers each) among the blocks that are resident there. Measured
  // (120 iterations, ms at 128 / 256 / 512 / 1024 threads): 2048 searches of n = 2048 5.3 / 6.3 /
  // 8.5 / 14.6 (14 blocks per SM wait for one), 128 of n = 10000 6.8 / 4.1 / 2.7 / 2.3, 60 of
  // n = 1524 1.55 / 0.95 / 0.82 / 0.94, 286 of n = 583 0.79 / 0.70 / 0.82 / 1.5; the per-kernel
  // form took 22.8, 16.8, 5.9 and 3.3 ms.
  const int fit = std::max(1, (int)(225 * 1024 / single_layout(P.NP, P.Wmax, P.K1, 4).total));
  const int per_sm = std::min((P.B + P.sms - 1) / P.sms, fit);
  const int nt = std::min(P.NP > 2560 ? 1024 : P.NP > 1024 ? 512 : 256, 1024 / per_sm);
  if (nt >= 1024) return launch_single_nt<1024>(P, n_iters, ext, s);
  if (nt >= 512) return launch_single_nt<512>(P, n_iters, ext, s);
  if (nt >= 256) return launch_single_nt<256>(P, n_iters, ext, s);
  return launch_single_nt<128>(P, n_iters, ext, s);
}

}  // namespace qis
