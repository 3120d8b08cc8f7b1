// qis_energy.cu -- energies from scratch (Eq. 1) of many states on the tensor cores.
//
// E(s) = sum_{i<j} J_ij s_i s_j + sum_i h_i s_i = sum_{i<j<=n} A_ij s_i s_j, with the field h_i as
// the coupling A_in to an extra site n whose spin is +1. The couplings are taken as integers
// v = A 2^Q and written in balanced base-4096 digits on the way into shared memory (each digit an
// exact FP16 integer), so
//     F_d[s][i] = sum_{i<j<=n} s_j D_d[i][j]          (one FP16 MMA chain per digit)
// is exact in the FP32 accumulators (a segment sums at most 1024 columns: |F_d| <= 2^21), and
// sum_i s_i F_d[s][i] is added up in integers: the energy is exact for the integers v, whatever
// the order. Q holds the couplings exactly where their span fits 58 bits (every instance on its
// grid; its fixed-point plane Jq is read then, Q = q); otherwise Q leaves 58 bits below the largest
// coupling, an error of 2^-59 of it per coupling (an FP64 sum rounds at 2^-53 of the partial sum
// at every step).
//
// Work: a block takes 64 rows i, a segment of at most kEnSeg 64-column steps of the upper triangle
// and 128 states of one instance. States are the M = 128 rows of the accumulator, so a thread of
// the epilogue owns one state and folds s_i into its own integer sums without any shuffle; the 64
// rows are the N columns, digit d in TMEM columns 64 d.. . All 256 threads convert: a thread
// loads 8 couplings of a row (64 contiguous bytes) one step ahead, extracts their digits and
// writes one 16-byte chunk per digit; the +-1 spins of the step are expanded from the packed
// states. Two shared-memory buffers: the MMAs of one step run under the conversion of the next.
//
// What bounds it: issue of the conversion (about 60 instructions per coupling and 128 states; the
// MMAs need a fifth of that and the couplings are read once per 128 states). The form it
// replaced added every coupling to 16 states with predicated FP64 or int64 adds (FP64 has two
// lanes per SM here): 5000 states of n = 1000 from host memory 906 -> 149 us (106 of them this kernel); the merged lists of
// 32 instances of n = 2048 off their grid 18.7 -> 0.5 ms, of 2 of n = 10000 26.2 -> 0.4 ms, of 4 of
// n = 200 .. 700 1.38 -> 0.07 ms, of 120 of n = 600 on their grid 0.87 -> 0.2 ms. The block that
// completes a state's sums forms its energy (a second launch cost a small call 6 us).
#include <algorithm>

#include "qis_tc.cuh"

namespace qis {

constexpr int kEnSeg = 16;          // 64-column steps per block (1024 columns: |F_d| <= 2^21, the magic add below)
constexpr int kEnTileA = 128 * 64 * 2;   // spins of 128 states
constexpr int kEnTileD = 64 * 64 * 2;    // one digit of 64 x 64 couplings
constexpr unsigned kEnFailed = 1u << 20;  // (at most 2192 blocks share a state: their sum stays below 2^32)
constexpr float kMagic = 12582912.f;     // 1.5 2^23: x + kMagic has the integer x in its low bits, |x| <= 2^21

// Where the states of a call are, and where their integer sums go.
struct EnergyJob {
  int inst0;                 // first instance (blockIdx.z counts from it)
  int per;                   // states per instance (the stride of the sums and results)
  int k;                     // states wanted per instance (k <= per)
  int Wn;                    // words per state of `states`
  const uint64_t* states;    // [inst][per][Wn], or NULL: the merged lists (mrg_ref)
  int from_q;                // 1: the fixed-point couplings of every instance (split modes)
  unsigned long long* acc;   // [inst][per][2]: sum of the digits 2.. and of 0, 1 (zero between calls)
  int* left;                 // [inst][tile of 128 states]: blocks done, kEnFailed per failed one (zero between calls)
  double* E_out;             // [inst][per] energies (NaN: a wait gave up), or NULL: init_q and init_E of search first_search + s
  uint64_t* words_out;       // [inst][per][Wmax] the states' words (may be NULL)
};

__device__ inline int energy_count(const DevPtrs& P, const EnergyJob& E, int inst) {
  return E.states ? E.k : min(E.k, P.mrg_count[inst]);
}
__device__ inline const uint64_t* energy_state(const DevPtrs& P, const EnergyJob& E, int inst, int s) {
  if (E.states) return E.states + ((long long)(inst - E.inst0) * E.per + s) * E.Wn;
  return P.lst_bits + (long long)P.mrg_ref[inst * P.K1 + s] * P.Wmax;
}
// Blocks (64 rows, one segment) that share a state of an n-spin instance: sum over the row blocks
// of ceil(steps / kEnSeg), steps = columns' steps right of the diagonal.
__device__ inline int energy_blocks(int n) {
  auto f = [](int m) { const int q = m / kEnSeg; return kEnSeg * q * (q + 1) / 2 + (m - q * kEnSeg) * (q + 1); };
  const int steps = n / 64 + 1;
  return f(steps) - f(steps - (n + 63) / 64);
}

__global__ void __launch_bounds__(256) k_energy(DevPtrs P, EnergyJob E, int nseg_max, int digits_max, int ncols) {
  const int inst = E.inst0 + blockIdx.z;
  const InstDesc d = P.inst[inst];
  const int n = d.n, np = d.n_pad;
  const int rb = blockIdx.x / nseg_max, seg = blockIdx.x % nseg_max;
  const int i0 = rb * 64, s0 = blockIdx.y * 128;
  const int steps_all = n / 64 + 1;                       // columns 0 .. n
  const int kc0 = rb + seg * kEnSeg, kc1 = min(kc0 + kEnSeg, steps_all);
  if (i0 >= n || kc0 >= steps_all) return;                // block-uniform
  const int cnt = energy_count(P, E, inst);
  if (s0 >= cnt) return;
  const bool q_src = P.mode != QIS_FP64 && (E.from_q || !d.rounded);
  const int Q = q_src ? d.q : d.eq;
  const int D = energy_digits(d.etop, Q);

  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int stage = kEnTileA + digits_max * kEnTileD;
  __shared__ __align__(8) uint64_t done[2];
  __shared__ uint32_t tmem_base;
  __shared__ const uint64_t* st_ptr[128];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    mbar_init(&done[0], 1);
    mbar_init(&done[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 128) st_ptr[tid] = energy_state(P, E, inst, min(s0 + tid, cnt - 1));
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base)),
                 "r"(ncols));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  const uint64_t t0 = gtimer();

  // this thread's two units of a step: rows r, r + 32, the 8 columns of chunk c
  const int c = tid & 7, r = tid >> 3;
  const double* Jd = P.J64 + d.off_mat;
  const long long* Ji = P.Jq + d.off_mat;
  unsigned long long raw[2][8];
  uint64_t wd[4];   // the step's word of states r, r + 32, ..
  auto fetch = [&](int kc) {
#pragma unroll
    for (int m = 0; m < 4; ++m) wd[m] = kc < d.W ? st_ptr[r + 32 * m][kc] : 0ull;
    if (kc == n >> 6)   // the extra site: spin +1, whatever the caller's word holds there (sites past it have no couplings)
#pragma unroll
      for (int m = 0; m < 4; ++m) wd[m] &= ~(1ull << (n & 63));
    const int j0 = kc * 64 + c * 8;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const long long at = (long long)(i0 + r + 32 * u) * np + j0;
      const ulonglong2* p = reinterpret_cast<const ulonglong2*>(q_src ? reinterpret_cast<const unsigned long long*>(Ji + at)
                                                                      : reinterpret_cast<const unsigned long long*>(Jd + at));
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const ulonglong2 x = j0 < np ? p[e] : make_ulonglong2(0ull, 0ull);   // n_pad is a multiple of 128
        raw[u][2 * e] = x.x;
        raw[u][2 * e + 1] = x.y;
      }
    }
  };
  fetch(kc0);
  const uint32_t idesc = idesc_f16(64);
  bool ok = !P.wait_probe || mbar_wait(&done[0], 0, t0, P.wait_ns);   // (the probe: a wait that nothing completes)
  int it = 0;
  for (int kc = kc0; kc < kc1; ++kc, ++it) {
    const int buf = it & 1;
    unsigned char* st = smem + buf * stage;
    if (it >= 2) ok = mbar_wait(&done[buf], ((it >> 1) - 1) & 1, t0, P.wait_ns);   // the MMAs of step it - 2
    // spins of columns kc 64 .. + 63: 128 states x 8 chunks of 8 halves +-1 (0x3c00 and a sign bit)
#pragma unroll
    for (int m = 0; m < 4; ++m) {
      const int sr = r + 32 * m;
      const unsigned b = (unsigned)(wd[m] >> (8 * c)) & 255u;
      uint4 v;
      v.x = 0x3c003c00u | ((b & 1u) << 15) | ((b & 2u) << 30);
      v.y = 0x3c003c00u | ((b & 4u) << 13) | ((b & 8u) << 28);
      v.z = 0x3c003c00u | ((b & 16u) << 11) | ((b & 32u) << 26);
      v.w = 0x3c003c00u | ((b & 64u) << 9) | ((b & 128u) << 24);
      *reinterpret_cast<uint4*>(st + sr * 128 + ((c ^ (sr & 7)) << 4)) = v;
    }
    const int j0 = kc * 64 + c * 8;
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const int row = r + 32 * u, i = i0 + row;
      long long v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const int j = j0 + e;
        v[e] = 0;
        if (j > i && j < n) v[e] = q_src ? (long long)raw[u][e] : fixed_point_rn(__longlong_as_double((long long)raw[u][e]), Q);
      }
      if (n >= j0 && n < j0 + 8 && i < n) {
        const long long hv = q_src ? P.hq[d.off_vec + i]
                                   : fixed_point_rn(P.h64[d.off_vec + i], Q);
#pragma unroll
        for (int e = 0; e < 8; ++e)
          if (j0 + e == n) v[e] = hv;
      }
      unsigned char* dst = st + kEnTileA + row * 128 + ((c ^ (row & 7)) << 4);
      for (int dg = 0; dg < D; ++dg) {
        // balanced digit ((v + 2048) mod 4096) - 2048 as an exact FP16 integer; v <- the rest / 4096
        uint32_t pk[4];
#pragma unroll
        for (int e = 0; e < 8; e += 2) {
          const long long ta = v[e] + 2048, tb = v[e + 1] + 2048;
          const float fa = __uint_as_float(0x4b000000u | ((uint32_t)ta & 4095u)) - 8390656.f;   // 2^23 + 2048
          const float fb = __uint_as_float(0x4b000000u | ((uint32_t)tb & 4095u)) - 8390656.f;
          v[e] = ta >> 12;
          v[e + 1] = tb >> 12;
          asm("cvt.rn.f16x2.f32 %0, %1, %2;" : "=r"(pk[e >> 1]) : "f"(fb), "f"(fa));
        }
        *reinterpret_cast<uint4*>(dst + dg * kEnTileD) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
      }
    }
    if (kc + 1 < kc1) fetch(kc + 1);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (__syncthreads_or(!ok)) {   // block-uniform: a wait gave up
      ok = false;
      break;
    }
    if (tid == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;");
      const uint32_t a = smem_u32(st), b = a + kEnTileA;
      for (int dg = 0; dg < D; ++dg)
#pragma unroll
        for (int k4 = 0; k4 < 4; ++k4)
          mma_f16(tmem + dg * 64, sdesc(a + k4 * 32), sdesc(b + dg * kEnTileD + k4 * 32), idesc, (it | k4) != 0);
      mma_commit(&done[buf]);
    }
  }
  // every issued step complete: the last two commits (bounded like the drains of the field GEMM)
  for (int x = max(0, it - 2); x < it; ++x) {
    const bool w = mbar_wait(&done[x & 1], (x >> 1) & 1, gtimer(), ok ? (uint64_t)P.wait_ns : kDrainNs);
    ok = ok && w;
  }
  asm volatile("tcgen05.fence::after_thread_sync;");
  const int total = energy_blocks(n);
  const bool mine = tid < 128 && s0 + tid < cnt;
  long long hi = 0, lo = 0;   // this thread's state: the sums of digits 2.. and of 0, 1
  unsigned long long* a = E.acc + 2 * ((long long)blockIdx.z * E.per + s0 + tid);
  bool failed = __syncthreads_or(!ok);
  if (failed) {
    // (the host finds the NaN of given states in what it copies; the searches are none the worse)
    if (tid == 0 && !(E.E_out && E.states)) atomicOr(P.status, kStatTimeout);
  } else if (warp < 4) {
    // thread = state: T_d = sum over the 64 rows i of s_i F_d (|T_d| <= 2^27, int32)
    const uint64_t w = st_ptr[tid][rb];   // i0 < n: word rb is within the state
    for (int dg = D - 1; dg >= 0; --dg) {
      unsigned T = 0;
#pragma unroll
      for (int c0 = 0; c0 < 64; c0 += 16) {
        uint32_t v[16];
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
              "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
            : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(dg * 64 + c0)));
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        const uint32_t wb = (uint32_t)(w >> c0);
#pragma unroll
        for (int u = 0; u < 16; ++u)
          T += __float_as_uint(__uint_as_float(v[u] ^ (((wb >> u) & 1u) << 31)) + kMagic);
      }
      const long long Td = (int)(T - 64u * 0x4b400000u);
      if (dg >= 2) hi = (hi << 12) + Td; else lo = (lo << 12) + Td;
    }
    if (mine && total > 1) {
      if (hi) atomicAdd(a, (unsigned long long)hi);
      if (lo) atomicAdd(a + 1, (unsigned long long)lo);
      __threadfence();   // the sums before this block's count
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols));
  // the last block of these states turns the sums into energies and clears them for the next call
  if (total > 1) {
    __shared__ int s_last, s_failed;
    if (tid == 0) {
      int* c = E.left + (long long)blockIdx.z * gridDim.y + blockIdx.y;
      const unsigned done_before = (unsigned)atomicAdd(c, failed ? (int)(kEnFailed + 1) : 1);
      s_last = (int)(done_before & (kEnFailed - 1)) == total - 1;
      s_failed = failed || done_before >= kEnFailed;
      if (s_last) *c = 0;
    }
    __syncthreads();
    if (!s_last) return;
    failed = s_failed;
    __threadfence();
    if (mine) {
      hi = (long long)atomicExch(a, 0ull);
      lo = (long long)atomicExch(a + 1, 0ull);
    }
  }
  if (E.words_out) {
    uint64_t* out = E.words_out + ((long long)blockIdx.z * E.per + s0) * P.Wmax;
    for (int x = tid; x < min(128, cnt - s0) * P.Wmax; x += 256) {
      const int s = x / P.Wmax, k = x - s * P.Wmax;
      out[x] = k < d.W ? st_ptr[s][k] : 0ull;
    }
  }
  if (!mine) return;
  if (E.E_out) {
    // hi 2^24 + lo rounded once (hi has at most 53 bits unless the couplings need all 58)
    E.E_out[(long long)blockIdx.z * E.per + s0 + tid] =
        failed ? __longlong_as_double(0x7ff8000000000000ll) : ldexp((double)hi * 16777216.0 + (double)lo, -Q);
  } else {
    const long long b2 = (long long)d.first_search + s0 + tid, Eq = (hi << 24) + lo;   // |E 2^q| < 2^52
    P.init_q[b2] = Eq;
    P.init_E[b2] = ldexp((double)Eq, -Q);
  }
}

static cudaError_t launch_energy(const DevPtrs& P, const EnergyJob& E, int n_inst, int max_n, int digits, cudaStream_t s) {
  if (E.k <= 0 || n_inst <= 0) return cudaSuccess;
  const int rows = (max_n + 63) / 64, nseg = (max_n / 64 + 1 + kEnSeg - 1) / kEnSeg, tiles = (E.k + 127) / 128;
  int ncols = 64;
  while (ncols < 64 * digits) ncols <<= 1;
  // two blocks per SM share its 512 tensor-memory columns; five digits take them all, so that form
  // asks for more than half of the shared memory
  size_t sm = 2 * (size_t)(kEnTileA + digits * kEnTileD) + 1024;
  if (ncols > 256) sm = std::max<size_t>(sm, 120 * 1024);
  const cudaError_t ea = allow_smem((const void*)k_energy, sm);
  if (ea != cudaSuccess) return ea;
  for (int z = 0; z < n_inst; z += 65535) {   // (the grid's third dimension)
    EnergyJob F = E;
    F.inst0 = E.inst0 + z;
    if (F.states) F.states += (long long)z * E.per * E.Wn;
    F.acc += 2ll * z * E.per;
    F.left += (long long)z * tiles;
    if (F.E_out) F.E_out += (long long)z * E.per;
    if (F.words_out) F.words_out += (long long)z * E.per * P.Wmax;
    k_energy<<<dim3(rows * nseg, tiles, std::min(n_inst - z, 65535)), 256, sm, s>>>(P, F, nseg, digits, ncols);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// `count` states of instance `inst` (Wn words each, consecutive) into E_out.
cudaError_t launch_energies(const DevPtrs& P, int inst, const InstDesc& d, const uint64_t* states, int count, int Wn,
                            double* E_out, cudaStream_t s) {
  const EnergyJob E{inst, count, count, Wn, states, 0, P.en_acc, P.en_left, E_out, nullptr};
  const int q = P.mode != QIS_FP64 && !d.rounded ? d.q : d.eq;
  return launch_energy(P, E, 1, d.n, energy_digits(d.etop, q), s);
}

// The first min(k, count) states of every instance's merged list: words [inst][k][Wmax], energies [inst][k].
cudaError_t launch_energies_merged(const DevPtrs& P, int k, int max_n, int digits, uint64_t* words, double* E_out,
                                   cudaStream_t s) {
  const EnergyJob E{0, k, k, P.Wmax, nullptr, 0, P.en_acc, P.en_left, E_out, words};
  return launch_energy(P, E, P.n_inst, max_n, digits, s);
}

// E(psi0) 2^q of the initial states of instances inst0 .. inst0 + n_inst - 1 (split modes, the
// fixed-point couplings) into init_q and init_E.
cudaError_t launch_init_energy(const DevPtrs& P, int inst0, int n_inst, int max_n, int digits, cudaStream_t s) {
  const EnergyJob E{inst0, P.R, P.R, P.Wmax, P.init_bits + (long long)inst0 * P.R * P.Wmax, 1, P.en_acc, P.en_left,
                    nullptr, nullptr};
  return launch_energy(P, E, n_inst, max_n, digits, s);
}

}  // namespace qis
