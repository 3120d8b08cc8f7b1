// qis_noalloc.cu -- candidate selection of one parent state without any device allocation.
//
// Some callers cannot call cudaMalloc at the moment they need this work done: code that runs
// while a CUDA stream is being captured into a graph (an allocation there breaks the capture),
// real-time loops that must never block in the driver's allocator, and plugins that live in a
// host process whose device memory is owned by another framework's pool. For them this file
// keeps the one scratch area it needs in a file-scope __device__ array, sized at build time;
// the caller passes only its own input and output buffers.
//
// What it computes (FP64, the fields and changes of energy of the library's QIS_FP64 mode): for a
// parent state psi of an n-spin instance (J, h), every single flip i and pair flip i < j, with
// E' = E(psi) + dE, and returns the k candidates of lowest (E', c), c the candidate index
// (c = i for singles, n + rank(i, j) for pairs). This is the candidate side of one iteration
// of the QI search before duplicates against a kept list are removed.
//
// The scratch array is shared by every call on a device and keeps the last call's contents;
// every element a call reads is written earlier in that same call, so nothing needs clearing.
// Calls whose kernels overlap on the GPU (different streams, no ordering) race on the array.
//
// Two launches. The first forms the fields: the sum of a site runs over j ascending (the order of
// the FP64 mode), a chain of n dependent additions that bounds this kernel, so the rows of 16
// sites are staged in shared memory first. In the second every block bounds the k-th lowest change
// of energy by the k-th lowest of a few hundred flips of the lowest-a sites (any subset of the
// candidates bounds it from above), tests its rows' candidates against that bound and keeps
// those at or below it (the k lowest of them when there are more); the block that ends last orders
// the kept ones of all blocks. Measured at n = 300, k = 100: 5092 -> 48 us per call, of which the
// sum of E(psi) by one thread and the uncoalesced rows took 4700 and the sorts of every candidate 360;
// n = 512 and less 412 .. 5092 -> 25 .. 48 us. E(psi) from the fields is nearer the exact value than
// the pairs one by one (2e-15 against 2e-14 at n = 300).
#include <mutex>
#include <string>

#include "qis_block.cuh"

namespace qis {

constexpr int kNaMaxN = 512;       // largest n accepted
constexpr int kNaMaxK = 128;       // largest k accepted
constexpr int kNaBlocks = 64;      // candidate blocks: block b takes the rows b, b + 64, ..
constexpr int kNaSites = 16;       // sites per field block
constexpr int kNaList = kNaBlocks * kNaMaxK;   // kept candidates of all blocks at most

struct NoAllocScratch {
  double a[kNaMaxN];                         // a_i = -2 s_i f_i of the parent
  unsigned long long key[kNaBlocks][kNaMaxK];   // per-block kept candidates: order keys of E'
  uint32_t c[kNaBlocks][kNaMaxK];            // and their candidate indices
  int cnt[kNaBlocks];                        // and their number
  int done;                                  // candidate blocks that have written theirs
};

// ~100 KB; every GPU that loads the library holds it until the process exits
static __device__ __align__(256) NoAllocScratch g_na_scratch;

// f_i = (sum_{j != i} s_j J_ij, j ascending) + h_i, a_i = -2 s_i f_i, in FP64 with unfused additions.
__global__ void __launch_bounds__(256) k_na_fields(int n, const double* J, const double* h, const uint64_t* bits,
                                                   NoAllocScratch* S) {
  extern __shared__ __align__(16) unsigned char na_smem[];
  double* row = reinterpret_cast<double*>(na_smem);   // [kNaSites][n + 1], s_j J_ij
  const int i0 = blockIdx.x * kNaSites;
  if (blockIdx.x == 0 && threadIdx.x == 0) S->done = 0;
  for (int r = threadIdx.x >> 5; r < kNaSites; r += 8) {
    const int i = i0 + r;
    if (i >= n) break;
#pragma unroll 4
    for (int j = threadIdx.x & 31; j < n; j += 32) {
      const double v = J[(long long)i * n + j];
      row[r * (n + 1) + j] = sigma_of(bits, j) ? -v : v;
    }
  }
  __syncthreads();
  const int i = i0 + (int)threadIdx.x;
  if (threadIdx.x >= kNaSites || i >= n) return;
  const double* x = row + threadIdx.x * (n + 1);
  double acc = 0.0;
#pragma unroll 8
  for (int j = 0; j < n; ++j)
    if (j != i) acc = __dadd_rn(acc, x[j]);
  const double f = __dadd_rn(acc, h[i]);
  S->a[i] = sigma_of(bits, i) ? 2.0 * f : -2.0 * f;
}

__device__ void na_sort(unsigned long long* key, uint32_t* val, int n2) {
  for (int k = 2; k <= n2; k <<= 1) {
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int t = threadIdx.x; t < n2; t += blockDim.x) {
        const int u = t ^ j;
        if (u > t) {
          const unsigned long long a = key[t], c = key[u];
          const uint32_t va = val[t], vc = val[u];
          const bool gt = (a > c) || (a == c && va > vc);
          if (gt == ((t & k) == 0)) {
            key[t] = c; key[u] = a;
            val[t] = vc; val[u] = va;
          }
        }
      }
      __syncthreads();
    }
  }
}

// Sort of cnt entries in shared memory (room for the next power of two).
__device__ void na_sort_any(unsigned long long* key, uint32_t* val, int cnt) {
  const int n2 = next_pow2(cnt);
  for (int t = cnt + threadIdx.x; t < n2; t += blockDim.x) {
    key[t] = ~0ull;
    val[t] = 0xffffffffu;
  }
  __syncthreads();
  na_sort(key, val, n2);
}

__global__ void __launch_bounds__(256) k_na_select(int n, const double* J, const double* h, const uint64_t* bits, int k,
                                                   NoAllocScratch* S, double* E_out, uint32_t* c_out, double* Ep_out) {
  extern __shared__ __align__(16) unsigned char na_smem[];
  unsigned long long* key = reinterpret_cast<unsigned long long*>(na_smem);   // [kNaList]
  uint32_t* val = reinterpret_cast<uint32_t*>(key + kNaList);                 // [kNaList]
  float* sub = reinterpret_cast<float*>(na_smem);                             // [kSubMax], before the candidates
  __shared__ double a[kNaMaxN];
  __shared__ uint64_t pb[kNaMaxN / 64];
  __shared__ __align__(16) int hist[256];
  __shared__ int sites[kSubSites], off[kNaBlocks + 1];
  __shared__ int s_ns, s_bin, s_cnt, s_last;
  __shared__ double s_e[8];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid < (n + 63) / 64) pb[tid] = bits[tid];
  if (tid == 0) s_ns = s_cnt = 0;
  hist[tid] = 0;
  __syncthreads();
  // E(psi) from the fields, E = sum_i (s_i f_i + s_i h_i) / 2 with s_i f_i = -a_i / 2 (Eq. 1): sums
  // of n terms, each of a chain of n, where the pairs one by one are a chain of n^2 / 2
  double e = 0.0;
  float mn = INFINITY, mx = -INFINITY;
  for (int i = tid; i < n; i += 256) {
    const double x = S->a[i], hv = h[i];
    a[i] = x;
    e = __dadd_rn(e, __dadd_rn(sigma_of(pb, i) ? -hv : hv, -0.5 * x));
    mn = fminf(mn, (float)x);
    mx = fmaxf(mx, (float)x);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) e = __dadd_rn(e, __shfl_xor_sync(0xffffffffu, e, o));
  if (lane == 0) s_e[warp] = e;
  block_min_max(mn, mx);
  e = s_e[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) e = __dadd_rn(e, s_e[w]);
  const double Ep = 0.5 * e;
  // the bound: the m lowest-a sites (a histogram's bins), m (m + 1) / 2 >= 3 k, their flips
  const float scale = 255.99f / fmaxf(mx - mn, 1e-30f);
  auto bin_of = [&](int i) { return min(255, max(0, (int)(((float)a[i] - mn) * scale))); };
  for (int i = tid; i < n; i += 256) atomicAdd(&hist[bin_of(i)], 1);
  __syncthreads();
  int m = 1;
  while (m * (m + 1) / 2 < 3 * k) ++m;
  m = min(min(m, n), kSubSites);
  if (warp == 0) {
    int bin, within;
    find_bin(hist, m - 1, bin, within);
    if (lane == 0) s_bin = bin;
  }
  __syncthreads();
  for (int i = tid; i < n; i += 256)
    if (bin_of(i) <= s_bin) {
      const int q = atomicAdd(&s_ns, 1);
      if (q < kSubSites) sites[q] = i;
    }
  __syncthreads();
  const int mm = min(s_ns, kSubSites), M = mm * (mm + 1) / 2;
  float vlo = INFINITY, vhi = -INFINITY;
  // row x of the subset: the flip of its site x and the pairs with its later sites; a warp per row,
  // the values rounded up to FP32 (upper bounds)
  for (int x = warp; x < mm; x += 8) {
    const int at = x * mm - x * (x - 1) / 2;
    for (int y = x + lane; y < mm; y += 32) {
      const int sx = sites[x], sy = sites[y], i = min(sx, sy), j = max(sx, sy);
      const double de = x == y ? a[i] : dE64(a[i], a[j], J[(long long)i * n + j], sigma_of(pb, i) ^ sigma_of(pb, j));
      const float v = __double2float_ru(de);
      sub[at + y - x] = v;
      vlo = fminf(vlo, v);
      vhi = fmaxf(vhi, v);
    }
  }
  float U = INFINITY;
  if (M >= k) {   // block-uniform
    __syncthreads();
    U = value_select_upper(sub, M, k - 1, hist, vlo, vhi);
  }
  __syncthreads();   // the subset's values have been read: the candidates take their place
  const double cap = __dadd_rn(Ep, (double)U);   // E' = fl(E + dE) is monotone in dE
  for (int i = blockIdx.x; i < n; i += gridDim.x) {
    const double ai = a[i];
    const int si = sigma_of(pb, i);
    for (int j = i + tid; j < n; j += 256) {   // j = i: the flip of site i alone
      const double de = j == i ? ai : dE64(ai, a[j], J[(long long)i * n + j], si ^ sigma_of(pb, j));
      const double E = __dadd_rn(Ep, de);
      if (!(E > cap)) {   // (a NaN is kept, and ordered last)
        const int q = atomicAdd(&s_cnt, 1);
        key[q] = dkey(E);
        val[q] = j == i ? (uint32_t)i : pair_index(n, i, j);
      }
    }
  }
  __syncthreads();
  int cnt = s_cnt;   // at most the block's candidates: 8 rows of 512 at most
  if (cnt > k) {     // ties, or a loose bound
    na_sort_any(key, val, cnt);
    cnt = k;
  }
  for (int t = tid; t < cnt; t += 256) {
    S->key[blockIdx.x][t] = key[t];
    S->c[blockIdx.x][t] = val[t];
  }
  if (tid == 0) S->cnt[blockIdx.x] = cnt;
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(&S->done, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (tid == 0) {
    int o = 0;
    for (int b = 0; b < (int)gridDim.x; ++b) {
      off[b] = o;
      o += *(volatile int*)&S->cnt[b];
    }
    off[gridDim.x] = o;
  }
  __syncthreads();
  const int tot = off[gridDim.x];
  for (int b = warp; b < (int)gridDim.x; b += 8)
    for (int t = lane; t < off[b + 1] - off[b]; t += 32) {
      key[off[b] + t] = *(volatile unsigned long long*)&S->key[b][t];
      val[off[b] + t] = *(volatile uint32_t*)&S->c[b][t];
    }
  __syncthreads();
  if (tot <= 1024) {   // usual: the place of each by counting the ones before it (all distinct by c)
    for (int p = tid; p < tot; p += 256) {
      const unsigned long long kp = key[p];
      const uint32_t cp = val[p];
      int r = 0;
      for (int q = 0; q < tot; ++q) r += (key[q] < kp || (key[q] == kp && val[q] < cp)) ? 1 : 0;
      if (r < k) {
        E_out[r] = dkey_inv(kp);
        c_out[r] = cp;
      }
    }
  } else {
    na_sort_any(key, val, tot);
    for (int t = tid; t < min(k, tot); t += 256) {
      E_out[t] = dkey_inv(key[t]);
      c_out[t] = val[t];
    }
  }
  for (int t = tot + tid; t < k; t += 256) {   // (only where NaNs left fewer)
    E_out[t] = INFINITY;
    c_out[t] = 0xffffffffu;
  }
  if (tid == 0 && Ep_out) *Ep_out = Ep;
}

namespace {
std::mutex g_na_mu;
NoAllocScratch* g_na_ptr[64] = {nullptr};   // device address of the scratch array, per device
bool g_na_attr[64] = {false};
}  // namespace

}  // namespace qis

using namespace qis;

extern "C" int qis_select_candidates_noalloc(int n, const double* J, const double* h, const uint64_t* bits, int k,
                                             double* E_out, uint32_t* c_out, double* Ep_out, void* stream) {
  if (n < 2 || n > kNaMaxN) {
    set_global_error("qis_select_candidates_noalloc: n must be in [2, 512] (static scratch size)");
    return QIS_ERR_INVALID_ARG;
  }
  if (k < 1 || k > kNaMaxK || (long long)k > (long long)n * (n + 1) / 2) {
    set_global_error("qis_select_candidates_noalloc: k must be in [1, min(128, n(n+1)/2)] (static scratch size)");
    return QIS_ERR_INVALID_ARG;
  }
  if (!J || !h || !bits || !E_out || !c_out) {
    set_global_error("qis_select_candidates_noalloc: NULL buffer");
    return QIS_ERR_INVALID_ARG;
  }
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    set_global_error("qis_select_candidates_noalloc: no current CUDA device");
    return QIS_ERR_CUDA;
  }
  NoAllocScratch* S = nullptr;
  {
    // set-up once per device, with that device current: the host-side name of the array is a
    // stand-in, the kernels need its device address
    std::lock_guard<std::mutex> lk(g_na_mu);
    if (!g_na_ptr[dev]) {
      void* p = nullptr;
      const cudaError_t e = cudaGetSymbolAddress(&p, g_na_scratch);
      if (e != cudaSuccess || !p) {
        set_global_error((std::string("qis_select_candidates_noalloc: cudaGetSymbolAddress of the scratch array: ") +
                          cudaGetErrorString(e)).c_str());
        return QIS_ERR_CUDA;
      }
      g_na_ptr[dev] = static_cast<NoAllocScratch*>(p);
    }
    if (!g_na_attr[dev]) {
      const int sm_f = kNaSites * (kNaMaxN + 1) * 8, sm_s = kNaList * 12;
      cudaError_t e = cudaFuncSetAttribute(k_na_fields, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_f);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(k_na_select, cudaFuncAttributeMaxDynamicSharedMemorySize, sm_s);
      if (e != cudaSuccess) {
        set_global_error((std::string("qis_select_candidates_noalloc: shared-memory attribute: ") +
                          cudaGetErrorString(e)).c_str());
        return QIS_ERR_CUDA;
      }
      g_na_attr[dev] = true;
    }
    S = g_na_ptr[dev];
  }
  // Each launch's own status: cudaLaunchKernel returns the error of that launch (it does not
  // consume an error the caller's earlier work left in the runtime's last-error state).
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const auto launched = [](cudaError_t e, const char* kernel) {
    if (e == cudaSuccess) return QIS_OK;
    set_global_error((std::string("qis_select_candidates_noalloc: launch of ") + kernel + ": " +
                      cudaGetErrorString(e)).c_str());
    return QIS_ERR_CUDA;
  };
  {
    void* args[] = {&n, &J, &h, &bits, &S};
    const int rc = launched(cudaLaunchKernel((const void*)k_na_fields, dim3((n + kNaSites - 1) / kNaSites), dim3(256), args,
                                             (size_t)kNaSites * (n + 1) * 8, s), "k_na_fields");
    if (rc) return rc;
  }
  {
    void* args[] = {&n, &J, &h, &bits, &k, &S, &E_out, &c_out, &Ep_out};
    return launched(cudaLaunchKernel((const void*)k_na_select, dim3(n < kNaBlocks ? n : kNaBlocks), dim3(256), args,
                                     (size_t)kNaList * 12, s), "k_na_select");
  }
}
