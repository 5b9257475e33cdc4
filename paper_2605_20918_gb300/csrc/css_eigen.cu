// FP64 eigen-decomposition of the projected block-tridiagonal matrices, one per colour, and
// the subspace matrix function Z = U f(Lambda) U^T E_1 B_0 (paper, Eq. 5-7: exact
// diagonalisation of the Krylov-projected Hamiltonian).
//
// GB300 runs FP64 at about 1/64 of the FP32 rate and a dependent FP64 sqrt + divide costs
// ~0.6 us, so no stage here is a long sequential FP64 chain:
//   1. band -> tridiagonal by Householder bulge chasing, many sweeps in flight (8, 16 or 32
//      lanes each, a sweep waits only for the one before it to move past its window); reflectors
//      of length <= b, and a sweep's reflectors touch disjoint rows, so their action on
//      b-column blocks is applied sweep by sweep with all of a sweep's reflectors in parallel;
//   2. eigenvalues of the tridiagonal by Sturm-count bisection in FP32 (one thread per
//      eigenvalue), used only as shifts;
//   3. Rayleigh-quotient inverse iteration (two FP32 steps, two FP64): one thread per eigenvalue, then
//      one warp per cluster of close shifts (simultaneous iteration with Gram-Schmidt and a
//      Rayleigh-Ritz step inside the cluster), which gives eigenvalues and eigenvectors to
//      FP64 accuracy;
//   4. Y = U^T (Q_band^T E_1 B_0), weights w = ||Y_k||^2, and after mu is known
//      Z = Q_band U f(Lambda) Y.
#include <algorithm>

#include "css_eigen.cuh"
#include "css_pipe.cuh"

namespace {

// ------------------------------------------------------------------ band storage
// AB[col * LDB + d] = T[col + d][col], d in [0, LDB), LDB = 2 kd + 2 (room for the bulge, and an odd
// stride LDB - 1 between the entries of a row, so that a column of lanes reads distinct banks)
__global__ void k_band_build(int32_t b, int32_t m, int32_t nmax, int32_t ldb, const double* __restrict__ Ablk,
                             const double* __restrict__ Bblk, const int32_t* __restrict__ nblk,
                             double* __restrict__ AB) {
  const int32_t c = blockIdx.x;
  const int32_t n = nblk[c] * b;
  double* ab = AB + (size_t)c * nmax * ldb;
  for (int32_t t = threadIdx.x; t < nmax * ldb; t += blockDim.x) {
    int32_t col = t / ldb, d = t % ldb, row = col + d;
    double v = 0.0;
    if (col < n && row < n && d <= b) {
      int32_t jc = col / b, kc = col % b, jr = row / b, kr = row % b;
      if (jr == jc) v = Ablk[(((size_t)c * m + jc) * b + kr) * b + kc];
      else if (jr == jc + 1 && kr <= kc) v = Bblk[(((size_t)c * m + jc) * b + kr) * b + kc];
    }
    ab[t] = v;
  }
}

// Sweeps of an n x n band matrix of half-width kd, the reflectors of a sweep (one annihilating
// column i, then one per chase step whose block has at least two rows) and the first slot of sweep
// i among the colour's reflectors: sum over i' < i of 1 + (n - 3 - i') / kd, in closed form.
__device__ __forceinline__ int32_t n_sweeps(int32_t n, int32_t kd) { return kd >= 2 && n > 2 ? n - 2 : 0; }
__device__ __forceinline__ int32_t sweep_len(int32_t i, int32_t n, int32_t kd) { return 1 + (n - 3 - i) / kd; }
__device__ __forceinline__ int32_t sweep_slot(int32_t i, int32_t n, int32_t kd) {
  auto floors = [kd](int32_t x) {  // sum of r / kd over r < x
    const int32_t q = x / kd;
    return kd * (q * (q - 1) / 2) + q * (x - q * kd);
  };
  return i + floors(n - 2) - floors(n - 2 - i);
}

template <int LPS>
__device__ __forceinline__ double group_sum(double v) {
#pragma unroll
  for (int o = LPS / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Householder reflector of x (one element per lane of a group of LPS, zero past its length):
// H x = beta e_0, H = I - tau v v^T, v_0 = 1, with beta of the sign opposite to x_0 (Golub & Van
// Loan, section 5.1.3), so x_0 - beta has no cancellation and one reciprocal square root and one
// division serve tau, beta and the scaling.  Every lane of the warp calls this.
template <int LPS>
__device__ __forceinline__ double group_house(double x, int l, double& tau, double& beta) {
  const double x0 = __shfl_sync(0xffffffffu, x, 0, LPS);
  const double sig = group_sum<LPS>(l >= 1 ? x * x : 0.0);
  const double ss = fma(x0, x0, sig), r = rsqrt(ss);
  const double b = x0 >= 0.0 ? -(ss * r) : ss * r;
  const double v0 = x0 - b;
  const bool none = sig == 0.0;
  tau = none ? 0.0 : fabs(v0) * r;
  beta = none ? x0 : b;
  return l == 0 ? 1.0 : (none ? 0.0 : x * (1.0 / v0));
}

// Band -> tridiagonal with the sweeps pipelined.  Sweep i annihilates column i and chases the
// bulge.  A step works on the rows [q0, hi) of the lower triangle (its off-diagonal block B and its
// diagonal block D) and the next step on the rows from hi on.  So a step of sweep i may run once
// every later step of sweep i - 1 works on rows >= its own hi: what they touch is then disjoint, the
// same holds by induction for all earlier sweeps, and the result is the sequential order's.  Two
// steps of sweep i - 1 ahead of sweep i are enough.  Sweep i belongs to slot i mod S of the S slots
// of a colour, which publishes (sweep, first row of its next step) in one 64-bit word.
//
// Bound by FP64 issue: a warp's FP64 instruction takes 64 clocks of its scheduler (19 of the SM with
// four or more warps) whatever its active lanes, dependent or not, so what counts is the number of
// instructions of a step and how many schedulers have a step to run:
//   - LPS = 8, 16 or 32 lanes work on a sweep (kd <= LPS) and a warp holds 32 / LPS sweeps, each at
//     its own window; with one sweep per warp, 26 of 32 lanes of every FP64 instruction idled at b = 6;
//   - the two updates of the off-diagonal block are one rank-2 update, the symmetric block is
//     updated over its lower triangle only, and a reflector takes one rsqrt and one division;
//   - where the band fits (SMEM), it lives in shared memory and one CTA works on a colour;
//     otherwise it stays in L2, a step works on a shared-memory copy of its window, and a
//     cluster of CTAs (co-scheduled, so they may wait for each other) shares a colour, neighbouring
//     sweeps on different SMs.
// Measured, one CTA of 32 one-sweep warps per colour -> this: n = 920, kd = 23, 63 colours 52.9 ->
// 24.4 ms (FP64 issue alone: 16.6 ms on the 126 SMs); n = 390, kd = 13, 44 colours 13.5 -> 5.8 ms;
// n = 180, kd = 6: 27 colours 4.36 -> 1.57 ms, 504 colours 17.2 -> 2.8 ms.
// Every wait is bounded: after 2 s without progress the colour's status gets bit 2 and all its
// CTAs stop.
struct BandArgs {
  int32_t kd, nmax, ldb, rcap, cta_per_col, hold;  // hold: tests only, sweeps after the first wait for ever
  const int32_t* nblk;
  double* AB;
  double* RV;
  double* RT;
  unsigned long long* slots;  // [c][S], zeroed (tile mode)
  double *dd, *ee;
  int32_t* status;
};

// doubles of shared memory one sweep needs: vectors v, nv, tz, w and, in tile mode, an mbarrier (16
// bytes) and the band columns of its window
__host__ __device__ constexpr int band_group_doubles(int kd, int ldb, int lps, bool smem) {
  return 4 * lps + (smem ? 0 : 2 + 2 * kd * ldb);
}

template <int LPS, bool SMEM>
__global__ void __launch_bounds__(SMEM ? 1024 : 512) k_band_to_tri(const BandArgs a) {
  constexpr int SPW = 32 / LPS;
  constexpr unsigned FULL = 0xffffffffu;
  extern __shared__ __align__(16) unsigned char band_smem[];
  const int32_t kd = a.kd, ldb = a.ldb, C = a.cta_per_col;
  const int32_t c = blockIdx.x / C, rank = blockIdx.x - c * C;
  const int32_t n = a.nblk[c] * kd;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane / LPS, l = lane - g * LPS;
  const int32_t nw = blockDim.x >> 5, S = C * nw * SPW;
  double* ab = a.AB + (size_t)c * a.nmax * ldb;
  double* mem = reinterpret_cast<double*>(band_smem);
  volatile unsigned long long* slots;
  if constexpr (SMEM) {
    slots = reinterpret_cast<unsigned long long*>(mem);
    for (int32_t t = threadIdx.x; t < S; t += blockDim.x) slots[t] = 0ull;
    mem += S;
    for (int32_t t = threadIdx.x; t < n * ldb; t += blockDim.x) mem[t] = ab[t];
    ab = mem;
    mem += (size_t)a.nmax * ldb;
    __syncthreads();
  } else {
    slots = a.slots + (size_t)c * S;
  }
  mem += (size_t)(warp * SPW + g) * band_group_doubles(kd, ldb, LPS, SMEM);
  double *v = mem, *nv = mem + LPS, *tz = mem + 2 * LPS, *wv = mem + 3 * LPS;
  // tile mode: copy of the band columns of the step's window
  uint64_t* bar = reinterpret_cast<uint64_t*>(mem + 4 * LPS);
  double* win = mem + 4 * LPS + 2;
  uint32_t parity = 0;
  if constexpr (!SMEM) {
    if (l == 0) css_pipe::bar_init(bar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncwarp();
  }
  const int32_t cs = ldb - 1;  // entry (r, j) of a block: base[j * cs + r]
  const int32_t nsweep = n_sweeps(n, kd);
  // neighbouring sweeps on different CTAs of the colour
  const int32_t me = (warp * SPW + g) * C + rank;
  auto fence = [] {
    if constexpr (SMEM) __threadfence_block();
    else __threadfence();
  };
  int32_t i = me, p0 = -1, Lp = 0, k = 0;  // p0 < 0: the sweep's first step is next
  double tau = 0.0;
  uint64_t t0 = 0;
  uint32_t idle = 0;
  while (__any_sync(FULL, i < nsweep)) {
    // ------------------------------------------------ may the next step run?
    const bool live = i < nsweep, first = p0 < 0;
    const int32_t q0 = first ? i + 1 : p0 + Lp;
    const int32_t Lq = live ? min(kd, n - q0) : 0;
    bool act = live;
    if (live && i > 0) {
      const unsigned long long x = slots[(i - 1) % S];
      const int32_t id = (int32_t)(x >> 32) - 1, next_row = (int32_t)(uint32_t)x;
      act = !a.hold && (id > i - 1 || (id == i - 1 && next_row >= q0 + Lq));
    }
    if (!__any_sync(FULL, act)) {
      if (++idle == 1) t0 = css_pipe::gtime();
      if ((idle & 255u) == 0) {
        const bool stop = (*(volatile int32_t*)&a.status[c] & 2) || css_pipe::gtime() - t0 > css_pipe::kWaitNs;
        if (__any_sync(FULL, stop)) {  // the lanes leave together: those that stayed would vote without the others
          if (lane == 0) atomicOr(&a.status[c], 2);
          break;
        }
      }
      __nanosleep(20);
      continue;
    }
    idle = 0;
    fence();
    __syncwarp();
    // --------------------------------------------------- blocks of the window
    // B = A[q0 .., p0 ..] (not at the first step) and the lower triangle of D = A[q0 .., q0 ..].  In
    // tile mode the columns of the window, one contiguous run of the band, arrive by one bulk copy;
    // the step writes back only what it changed (rows past the window are other sweeps').
    const int32_t c0 = first ? i : p0;
    double* w0 = ab + (size_t)c0 * ldb;
    if constexpr (!SMEM) {
      bool late = false;
      if (act) {
        if (l == 0) {
          const uint32_t bytes = (uint32_t)((q0 + Lq - c0) * ldb) * 8u;
          asm volatile("fence.proxy.async;" ::: "memory");
          css_pipe::bar_expect(bar, bytes);
          css_pipe::bulk_g2s(win, w0, bytes, bar);
        }
        const uint64_t tc = css_pipe::gtime();
        while (!late && !css_pipe::bar_test(bar, parity)) late = css_pipe::gtime() - tc > css_pipe::kWaitNs;
        parity ^= 1;
      }
      if (__any_sync(FULL, late)) {
        if (lane == 0) atomicOr(&a.status[c], 2);
        break;
      }
      w0 = win;
    }
    double* B = w0 + (q0 - c0);                // entry (r, j) of B (column p0 + j)
    double* D = w0 + (size_t)(q0 - c0) * ldb;  // entry (r, j) of D (column q0 + j)
    double* col = w0 + 1;                      // first step: A[i + 1 .., i]
    // ------------------------------ new reflector (and the old one applied to B)
    double x = 0.0, ty = 0.0, tau2, beta;
    if (act && l < Lq) {
      if (first) {
        x = col[l];
      } else {
        double y = 0.0;
#pragma unroll 4
        for (int32_t j = 0; j < Lp; ++j) y = fma(B[j * cs + l], v[j], y);
        ty = tau * y;
        x = B[l] - ty;
      }
    }
    const double h = group_house<LPS>(x, l, tau2, beta);
    const bool grow = act && (first || Lq >= 2);  // a one-row block ends the sweep without a reflector
    const double nl = grow && l < Lq ? h : 0.0;
    nv[l] = nl;
    const double d = group_sum<LPS>(nl * ty);
    __syncwarp();
    if (act && !first) {
      // z = nv^T (B - ty v^T) for the columns j >= 1 (one per lane), then
      // B <- B - ty v^T - nv (tau2 z)^T in one pass
      double z = 0.0;
      if (grow && l >= 1 && l < Lp) {
        const double* Bc = B + l * cs;
#pragma unroll 4
        for (int32_t r = 0; r < Lq; ++r) z = fma(nv[r], Bc[r], z);
        z = tau2 * fma(-d, v[l], z);
      }
      tz[l] = z;
    }
    __syncwarp();
    if (act && l < Lq) {
      if (first) {
        (SMEM ? col : ab + (size_t)i * ldb + 1)[l] = l == 0 ? beta : 0.0;
      } else {
        double* out = SMEM ? B + l : ab + (size_t)p0 * ldb + (q0 - p0) + l;
        out[0] = grow ? (l == 0 ? beta : 0.0) : B[l] - ty;
#pragma unroll 4
        for (int32_t j = 1; j < Lp; ++j) out[(size_t)j * cs] = fma(-nl, tz[j], fma(-ty, v[j], B[j * cs + l]));
      }
    }
    // --------------------------------------------- D <- H D H on its lower triangle
    double pl = 0.0;
    if (grow && l < Lq && tau2 != 0.0) {
      double s0 = 0.0;  // one loop over the row, so that every lane runs the same Lq steps
      for (int32_t j = 0; j < Lq; ++j) s0 = fma(D[j <= l ? j * cs + l : l * cs + j], nv[j], s0);
      pl = tau2 * s0;
    }
    const double alpha = -0.5 * tau2 * group_sum<LPS>(pl * nl);
    wv[l] = fma(alpha, nl, pl);
    __syncwarp();
    if (grow) {
      const int32_t ne = Lq * (Lq + 1) / 2;
      int32_t r = 0, cc = l;
      for (int32_t e = l; e < ne; e += LPS, cc += LPS) {
        while (cc > r) {
          cc -= r + 1;
          ++r;
        }
        D[cc * cs + r] = fma(-nv[r], wv[cc], fma(-wv[r], nv[cc], D[cc * cs + r]));
      }
      const int32_t slot = sweep_slot(i, n, kd) + k;
      if (l < kd) a.RV[((size_t)c * a.rcap + slot) * kd + l] = nl;
      if (l == 0) a.RT[(size_t)c * a.rcap + slot] = tau2;
    }
    v[l] = act ? nl : v[l];
    __syncwarp();
    if constexpr (!SMEM) {  // D back to the band, a column of rows per store
      if (grow && l < Lq) {
        double* out = ab + (size_t)q0 * ldb + l;
        for (int32_t j = 0; j <= l; ++j) out[(size_t)j * cs] = D[j * cs + l];
      }
      __syncwarp();
    }
    // --------------------------------------------------------- publish, move on
    if (act) {
      if (l == 0) fence();
      tau = tau2;
      p0 = q0;
      Lp = Lq;
      ++k;
      const bool over = !grow || q0 + Lq > n - 1;  // no rows below the window
      if (l == 0)
        slots[i % S] = ((unsigned long long)(uint32_t)(i + 1) << 32) |
                       (unsigned long long)(uint32_t)(over ? 0x7fffffff : q0 + Lq);
      if (over) {
        i += S;
        p0 = -1;
        Lp = 0;
        k = 0;
      }
    }
    __syncwarp();
  }
  if constexpr (SMEM) {
    __syncthreads();
    for (int32_t t = threadIdx.x; t < n; t += blockDim.x) {
      a.dd[(size_t)c * a.nmax + t] = ab[(size_t)t * ldb];
      a.ee[(size_t)c * a.nmax + t] = t + 1 < n ? ab[(size_t)t * ldb + 1] : 0.0;
    }
  }
}

// diagonal and sub-diagonal of the reduced band (tile mode)
__global__ void k_tri_out(int32_t kd, int32_t nmax, int32_t ldb, const int32_t* __restrict__ nblk,
                          const double* __restrict__ AB, double* __restrict__ dd, double* __restrict__ ee) {
  const int32_t c = blockIdx.x, n = nblk[c] * kd;
  const double* ab = AB + (size_t)c * nmax * ldb;
  for (int32_t t = threadIdx.x; t < n; t += blockDim.x) {
    dd[(size_t)c * nmax + t] = ab[(size_t)t * ldb];
    ee[(size_t)c * nmax + t] = t + 1 < n ? ab[(size_t)t * ldb + 1] : 0.0;
  }
}

// Apply the recorded reflectors to columns of an n x b block X ([c][nmax][b]): FWD applies them in
// generation order (X <- Q^T X), otherwise in reverse (X <- Q X).  A sweep's reflectors act on
// disjoint rows, so one thread per (reflector of the sweep, column) works in parallel; the columns
// are independent, so a colour's are shared out to gridDim.y CTAs of cw columns.  The columns live in
// shared memory and the next sweep's reflectors arrive (cp.async) while this one's are applied.
// Bound by FP64 issue (2 kd FMAs per reflector and column).  One CTA per colour, reading both from
// global memory: n = 920, 63 colours 7.3 ms, n = 180 0.42 ms; now 3.6 and 0.22.
template <bool FWD>
__global__ void __launch_bounds__(1024) k_apply_refl(int32_t kd, int32_t b, int32_t cw, int32_t nmax, int32_t rcap,
                                                     const int32_t* __restrict__ nblk, const double* __restrict__ RV,
                                                     const double* __restrict__ RT, double* __restrict__ X) {
  extern __shared__ __align__(16) double refl_smem[];
  const int32_t c = blockIdx.x, j0 = blockIdx.y * cw, w = min(cw, b - j0);
  const int32_t n = nblk[c] * kd;
  const double* rv = RV + (size_t)c * rcap * kd;
  const double* rt = RT + (size_t)c * rcap;
  double* xg = X + (size_t)c * nmax * b + j0;
  const int32_t nsweep = n_sweeps(n, kd);
  const int32_t most = nmax / kd + 1, stage = most * (kd + 1);  // reflectors of a sweep, doubles of a stage
  double* x = refl_smem;  // [n][w]
  double* sv = refl_smem + (size_t)nmax * cw;
  for (int32_t t = threadIdx.x; t < n * w; t += blockDim.x) x[t] = xg[(size_t)(t / w) * b + t % w];
  auto copy8 = [](double* d, const double* g) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(css_pipe::su32(d)), "l"(g) : "memory");
  };
  auto fetch = [&](int32_t s) {  // a sweep's reflectors and their taus
    const int32_t i = FWD ? s : nsweep - 1 - s, t0 = sweep_slot(i, n, kd), len = sweep_len(i, n, kd);
    double* d = sv + (s & 1) * stage;
    for (int32_t t = threadIdx.x; t < len * kd; t += blockDim.x) copy8(d + t, rv + (size_t)t0 * kd + t);
    for (int32_t t = threadIdx.x; t < len; t += blockDim.x) copy8(d + most * kd + t, rt + t0 + t);
  };
  if (nsweep > 0) fetch(0);
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int32_t s = 0; s < nsweep; ++s) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // this sweep's reflectors are there, and the previous sweep is done
    if (s + 1 < nsweep) fetch(s + 1);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int32_t i = FWD ? s : nsweep - 1 - s, len = sweep_len(i, n, kd);
    const double* d = sv + (s & 1) * stage;
    for (int32_t t = threadIdx.x; t < len * w; t += blockDim.x) {
      const int32_t r = t / w, r0 = i + 1 + r * kd, L = min(kd, n - r0);
      const double* v = d + r * kd;
      double* xr = x + (size_t)r0 * w + (t - r * w);
      double s2 = 0.0;
#pragma unroll 4
      for (int32_t l = 0; l < L; ++l) s2 = fma(v[l], xr[l * w], s2);
      s2 *= d[most * kd + r];
#pragma unroll 4
      for (int32_t l = 0; l < L; ++l) xr[l * w] = fma(-s2, v[l], xr[l * w]);
    }
  }
  __syncthreads();
  for (int32_t t = threadIdx.x; t < n * w; t += blockDim.x) xg[(size_t)(t / w) * b + t % w] = x[t];
}

// X0 = E_1 B_0 = [B_0; 0] for a general start factor B_0 [c][b][b]
__global__ void k_x0_b0(int32_t b, int32_t nmax, const double* __restrict__ B0, double* __restrict__ X) {
  const int32_t c = blockIdx.x;
  for (int32_t t = threadIdx.x; t < nmax * b; t += blockDim.x) {
    const int32_t i = t / b, k = t % b;
    X[(size_t)c * nmax * b + t] = (i < b) ? B0[((size_t)c * b + i) * b + k] : 0.0;
  }
}

// X0 = E_1 B_0 = sqrt|c| [I_b; 0]
__global__ void k_x0(int32_t b, int32_t nmax, const int32_t* __restrict__ cnt, double* __restrict__ X) {
  const int32_t c = blockIdx.x;
  const double s = sqrt((double)cnt[c]);
  for (int32_t t = threadIdx.x; t < nmax * b; t += blockDim.x) {
    int32_t i = t / b, k = t % b;
    X[(size_t)c * nmax * b + t] = (i == k) ? s : 0.0;
  }
}

// ------------------------------------------------------------- FP32 bisection
__device__ __forceinline__ int32_t sturm32(const float* d, const float* e2, int32_t n, float x, float pivmin) {
  float qv = d[0] - x;
  int32_t cnt = qv < 0.f;
  for (int32_t i = 1; i < n; ++i) {
    if (fabsf(qv) < pivmin) qv = -pivmin;
    qv = (d[i] - x) - __fdividef(e2[i - 1], qv);
    cnt += qv < 0.f;
  }
  return cnt;
}

__global__ void k_bisect32(int32_t kd, int32_t nmax, const int32_t* __restrict__ nblk, const double* __restrict__ dd,
                           const double* __restrict__ ee, float* __restrict__ lam32, double* __restrict__ tnorm) {
  extern __shared__ float sh32[];
  const int32_t c = blockIdx.x;
  const int32_t n = nblk[c] * kd;
  float* d = sh32;
  float* e2 = sh32 + nmax;
  __shared__ double red_lo[32], red_hi[32];
  double lo = 1e300, hi = -1e300, emax = 0.0;
  for (int32_t i = threadIdx.x; i < n; i += blockDim.x) {
    double di = dd[(size_t)c * nmax + i];
    double el = i > 0 ? fabs(ee[(size_t)c * nmax + i - 1]) : 0.0;
    double er = i + 1 < n ? fabs(ee[(size_t)c * nmax + i]) : 0.0;
    lo = fmin(lo, di - el - er);
    hi = fmax(hi, di + el + er);
    d[i] = (float)di;
    double e = i + 1 < n ? ee[(size_t)c * nmax + i] : 0.0;
    e2[i] = (float)(e * e);
    emax = fmax(emax, e * e);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    emax = fmax(emax, __shfl_xor_sync(0xffffffffu, emax, o));
  }
  if ((threadIdx.x & 31) == 0) {
    red_lo[threadIdx.x >> 5] = lo;
    red_hi[threadIdx.x >> 5] = fmax(hi, -1e300);
  }
  __shared__ double semax[32];
  if ((threadIdx.x & 31) == 0) semax[threadIdx.x >> 5] = emax;
  __syncthreads();
  double glo = 1e300, ghi = -1e300, gem = 0.0;
  for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
    glo = fmin(glo, red_lo[i]);
    ghi = fmax(ghi, red_hi[i]);
    gem = fmax(gem, semax[i]);
  }
  const double span = fmax(fabs(glo), fabs(ghi));
  if (threadIdx.x == 0) tnorm[c] = fmax(span, 1e-100);
  const float flo = (float)(glo - 1e-3 * span - 1e-30), fhi = (float)(ghi + 1e-3 * span + 1e-30);
  const float pivmin = (float)fmax(1e-30, 1e-30 * gem);
  const int32_t k = blockIdx.y * blockDim.x + threadIdx.x;  // one eigenvalue per thread
  if (k < n) {
    float a = flo, z = fhi;
    for (int it = 0; it < 80; ++it) {
      float mid = 0.5f * (a + z);
      if (!(mid > a && mid < z)) break;
      if (sturm32(d, e2, n, mid, pivmin) <= k) a = mid;
      else z = mid;
    }
    lam32[(size_t)c * nmax + k] = 0.5f * (a + z);
  }
}

// ------------------------------------------------- FP64 inverse iteration
constexpr int kMaxCluster = 16;
// Convergence: the last solve (T - sigma I) y = x, ||x|| = 1, grew by ||y|| > 1 / (kResTol ||T||), so
// the returned y / ||y|| has residual ||(T - sigma I) y/||y|| || below kResTol ||T|| (128 eps);
// with the shift that close, the step damps every component outside the target eigenvector by
// at least that residual over the gap to the other eigenvalues.
constexpr double kResTol = 128.0 * 2.2e-16;

// uniform in [-1, 1)
__device__ __forceinline__ float hash_unit(uint64_t a, uint64_t b) {
  const uint64_t z = css_splitmix64(a * 0x9E3779B97F4A7C15ull + 0x5851F42D4C957F2Dull, b);
  return (float)(int32_t)(z >> 32) * 4.656612873077393e-10f;
}

constexpr int kCB = 8;  // rows per batch

// Scratch of one solve in the caller's column, nmax apart per row: the rows of U (reciprocal pivot and
// two super-diagonals) and the right-hand side / solution.
struct Col64 {
  using T = double;
  double *u0, *u1, *u2, *x;
  size_t ld;
  __device__ __forceinline__ double rhs(int32_t i) const { return x[i * ld]; }
  __device__ __forceinline__ void put(int32_t i, double a, double b, double c, double r) const {
    u0[i * ld] = a;
    u1[i * ld] = b;
    u2[i * ld] = c;
    x[i * ld] = r;
  }
  __device__ __forceinline__ void get(int32_t i, double& a, double& b, double& c, double& r) const {
    a = u0[i * ld];
    b = u1[i * ld];
    c = u2[i * ld];
    r = x[i * ld];
  }
  __device__ __forceinline__ void put_x(int32_t i, double y) const { x[i * ld] = y; }
};
// the same in FP32, in the 8-byte slots of the FP64 u0 and u1 columns
struct Col32 {
  using T = float;
  float2 *p, *q;  // {u0, u1}, {u2, x}
  size_t ld;
  __device__ __forceinline__ float rhs(int32_t i) const { return q[i * ld].y; }
  __device__ __forceinline__ void put(int32_t i, float a, float b, float c, float r) const {
    p[i * ld] = make_float2(a, b);
    q[i * ld] = make_float2(c, r);
  }
  __device__ __forceinline__ void get(int32_t i, float& a, float& b, float& c, float& r) const {
    const float2 v = p[i * ld], w = q[i * ld];
    a = v.x;
    b = v.y;
    c = w.x;
    r = w.y;
  }
  __device__ __forceinline__ void put_x(int32_t i, float y) const { q[i * ld].y = y; }
};

// |x| as an integer of the same order: an integer comparison where an FP64 one would take the FP64 pipe
__device__ __forceinline__ long long abs_bits(double x) { return __double_as_longlong(x) & 0x7fffffffffffffffll; }
__device__ __forceinline__ int abs_bits(float x) { return __float_as_int(x) & 0x7fffffff; }

// LU with partial pivoting of T - sigma I fused with the forward elimination of the column's right-hand
// side (scaled by scl), then the back substitution U y = x; y overwrites the column.  Returns ||y||^2
// and, with RQ, y^T (T - ref I) y.  Every sweep over the rows loads a batch of rows before the batch's dependent
// arithmetic, so a warp keeps several loads in flight.  Lanes with st == false store nothing.
template <bool RQ, typename Col>
__device__ typename Col::T shifted_solve(const Col& m, const typename Col::T* __restrict__ d,
                                         const typename Col::T* __restrict__ e, int32_t n, typename Col::T sigma,
                                         typename Col::T scl, typename Col::T pivmin, bool st, typename Col::T& rq,
                                         typename Col::T ref = 0) {
  using T = typename Col::T;
  T cd = d[0] - sigma, cs = n > 1 ? e[0] : T(0);
  T xc = m.rhs(0) * scl;
  for (int32_t i0 = 0; i0 + 1 < n; i0 += kCB) {
    T sub[kCB], dg[kCB], sup[kCB], xn[kCB];
#pragma unroll
    for (int q = 0; q < kCB; ++q) {
      const int32_t i = i0 + q;
      const bool ok = i + 1 < n;
      sub[q] = ok ? e[i] : T(1);
      dg[q] = ok ? d[i + 1] : T(0);
      sup[q] = (i + 2 < n) ? e[i + 1] : T(0);
      xn[q] = ok ? m.rhs(i + 1) : T(0);
    }
#pragma unroll
    for (int q = 0; q < kCB; ++q) {
      const int32_t i = i0 + q;
      if (i + 1 >= n) break;
      const T dgs = dg[q] - sigma, xs = xn[q] * scl;
      // neighbouring lanes hold neighbouring shifts and mostly agree on the pivot, so a branch costs
      // no more than the selects that would replace it
      T u0, u1, u2, rhs, ncd, ncs, nx;
      if (abs_bits(cd) >= abs_bits(sub[q])) {
        if (abs_bits(cd) < abs_bits(pivmin)) cd = cd >= T(0) ? pivmin : -pivmin;
        u0 = T(1) / cd;  // the pivot's reciprocal serves the multiplier and the back substitution
        const T l = sub[q] * u0;
        u1 = cs;
        u2 = T(0);
        rhs = xc;
        ncd = dgs - l * cs;
        ncs = sup[q];
        nx = xs - l * xc;
      } else {
        u0 = T(1) / sub[q];
        const T l = cd * u0;
        u1 = dgs;
        u2 = sup[q];
        rhs = xs;
        ncd = cs - l * dgs;
        ncs = -l * sup[q];
        nx = xc - l * xs;
      }
      if (st) m.put(i, u0, u1, u2, rhs);
      cd = ncd;
      cs = ncs;
      xc = nx;
    }
  }
  if (fabs(cd) < pivmin) cd = cd >= T(0) ? pivmin : -pivmin;
  // back substitution, rows n-1 down to 0, in batches
  T y1 = xc / cd, y2 = T(0);
  T ss = y1 * y1;
  rq = RQ ? ss * (d[n - 1] - ref) : T(0);
  if (st) m.put_x(n - 1, y1);
  for (int32_t i0 = n - 2; i0 >= 0; i0 -= kCB) {
    T r[kCB], a0[kCB], a1[kCB], a2[kCB], dv[kCB], ev[kCB];
#pragma unroll
    for (int q = 0; q < kCB; ++q) {
      const int32_t i = i0 - q, j = i >= 0 ? i : 0;
      m.get(j, a0[q], a1[q], a2[q], r[q]);
      if (RQ) {
        dv[q] = d[j];
        ev[q] = e[j];
      }
    }
#pragma unroll
    for (int q = 0; q < kCB; ++q) {
      const int32_t i = i0 - q;
      if (i < 0) break;
      const T y = (r[q] - a1[q] * y1 - a2[q] * y2) * a0[q];
      if (st) m.put_x(i, y);
      ss += y * y;
      if (RQ) rq += y * ((dv[q] - ref) * y + T(2) * (ev[q] * y1));
      y2 = y1;
      y1 = y;
    }
  }
  return ss;
}

// Phase 1 of the inverse iteration: one thread per eigenvalue, all threads of a colour in lockstep
// (same loop bounds, fixed four iterations), so the column-per-thread accesses to the scratch are
// coalesced across a warp.  The first two iterations run at the FP32 shift and in FP32: they only have
// to bring the random start vector to the eigenvector within FP32 rounding over the gap (which is at
// least 1e-4 ||T|| here), from where the two FP64 iterations with Rayleigh-quotient shifts converge
// cubically.  Eigenvalues whose shift lies within tol of a neighbour's (a cluster) and results that did
// not converge or left their window are flagged for phase 2.
// Bound by FP64 issue (64 clocks of a scheduler per instruction, ~19 a row and solve).  With all four
// iterations, the start vector and separate Rayleigh-quotient passes in FP64 n = 920, 63 colours took
// 14.8 ms and n = 180, 62 colours 1.29 ms; now 8.7 and 0.61 (four CTAs per SM: with the 168 registers
// the compiler takes otherwise, 10.3 ms).
__global__ void __launch_bounds__(128, 4) k_inviter_p1(int32_t kd, int32_t nmax, const int32_t* __restrict__ nblk,
                                                    const double* __restrict__ dd, const double* __restrict__ ee,
                                                    const float* __restrict__ lam32, const double* __restrict__ tnorm,
                                                    double rel_cluster, double* __restrict__ U,
                                                    double* __restrict__ F, double* __restrict__ lam,
                                                    int32_t* __restrict__ flag, const int32_t* __restrict__ gid) {
  extern __shared__ float p1_smem[];
  const int32_t c = blockIdx.y;
  const uint64_t cseed = gid ? (uint64_t)gid[c] : (uint64_t)c;  // the colour's own id seeds its start vectors
  const int32_t n = nblk[c] * kd;
  const int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  if (blockIdx.x * blockDim.x >= n) return;  // whole block beyond this colour's size
  const double* d = dd + (size_t)c * nmax;
  const double* e = ee + (size_t)c * nmax;
  const float* l32 = lam32 + (size_t)c * nmax;
  float *d32 = p1_smem, *e32 = p1_smem + nmax;
  for (int32_t i = threadIdx.x; i < n; i += blockDim.x) {
    d32[i] = (float)d[i];
    e32[i] = i + 1 < n ? (float)e[i] : 0.0f;
  }
  __syncthreads();
  const double tn = tnorm[c];
  const double tol = rel_cluster * tn;
  const double res_tol = kResTol * tn;
  const bool valid = k < n;
  bool in_cluster = false;
  double win_lo = 0.0, win_hi = 0.0;
  if (valid) {
    const double lk = (double)l32[k];
    const double g_lo = k > 0 ? lk - (double)l32[k - 1] : tn;
    const double g_hi = k + 1 < n ? (double)l32[k + 1] - lk : tn;
    in_cluster = g_lo <= tol || g_hi <= tol;
    win_lo = lk - 0.25 * g_lo - 2e-6 * tn;
    win_hi = lk + 0.25 * g_hi + 2e-6 * tn;
  }
  const bool work = valid && !in_cluster;
  if (!__any_sync(0xffffffffu, work)) {
    if (valid) flag[(size_t)c * nmax + k] = 1;
    return;
  }
  // idle lanes shadow the colour's last column and store nothing
  const size_t nn = (size_t)nmax * nmax, col = valid ? k : n - 1;
  double* f = F + (size_t)c * 5 * nn + col;
  const Col64 m{f, f + nn, f + 2 * nn, f + 3 * nn, (size_t)nmax};
  const Col32 m32{reinterpret_cast<float2*>(f), reinterpret_cast<float2*>(f + nn), (size_t)nmax};
  if (work)
    for (int32_t i = 0; i < n; ++i) m32.put_x(i, hash_unit(cseed * 1000003ull + (uint64_t)k, (uint64_t)i));
  float ss = (float)n * (1.0f / 3.0f), none;  // the start vector's expected square norm
  for (int it = 0; it < 2; ++it)
    ss = shifted_solve<false>(m32, d32, e32, n, l32[col], rsqrtf(ss), 1.2e-7f * (float)tn, work, none);
  // its Rayleigh quotient, and the vector in FP64
  double s2 = 0.0, rq = 0.0, prev = 0.0;
  for (int32_t i0 = 0; i0 < n; i0 += kCB) {
    float x[kCB];
#pragma unroll
    for (int q = 0; q < kCB; ++q) x[q] = i0 + q < n ? m32.rhs(i0 + q) : 0.0f;
#pragma unroll
    for (int q = 0; q < kCB; ++q) {
      const int32_t i = i0 + q;
      if (i >= n) break;
      const double y = (double)x[q];
      if (work) m.put_x(i, y);
      s2 += y * y;
      rq += y * (d[i] * y + (i > 0 ? 2.0 * (e[i - 1] * prev) : 0.0));
      prev = y;
    }
  }
  double sigma = rq / s2, scl = rsqrt(s2), growth = 0.0;
  // The eigenvalue is the last vector's quotient about its shift, whose terms cancel instead of adding up to the
  // eigenvalue: errors of the eigenvalues are half of the plain quotient's.  The shift itself stays the plain
  // quotient: the solve loses more to a pivot of rounding size than it gains from the last bits (with the finer
  // shift the errors of Z grew by 30% at n = 180).
  for (int it = 0; it < 2; ++it) {
    const double ref = it ? sigma : 0.0, y2 = shifted_solve<true>(m, d, e, n, sigma, scl, 2.2e-16 * tn, work, rq, ref);
    growth = sqrt(y2);
    scl = 1.0 / growth;
    sigma = ref + rq / y2;
  }
  if (!valid) return;
  const bool ok = work && growth * res_tol > 1.0 && sigma >= win_lo && sigma <= win_hi;
  flag[(size_t)c * nmax + k] = ok ? 0 : 1;
  if (!ok) return;
  double* u = U + (size_t)c * nn + k;
  for (int32_t i = 0; i < n; ++i) u[(size_t)i * nmax] = m.x[(size_t)i * nmax] * scl;
  lam[(size_t)c * nmax + k] = sigma;
}

// Phase 2 of the FP64 inverse iteration: one warp per cluster of close shifts (or per single
// eigenvalue that phase 1 flagged).  Lane j < kc owns member k0 + j; its iterate is column k0 + j
// of the scratch X and its LU factors columns k0 + j of U0..U2, so the lanes of a warp touch
// contiguous addresses of a row.  Every member solves with its own shift, then the members are
// orthonormalised by modified Gram-Schmidt in member order (simultaneous inverse iteration);
// Rayleigh-Ritz inside the cluster gives the final pairs.  A single eigenvalue takes its norm and
// Rayleigh quotient from the solve and skips the orthonormalisation.
// Work lists of phase 2: (colour, first member, members), one thread per shift.  CLUSTERS: every cluster of
// close shifts (runs cut every kMaxCluster members), none of which phase 1 works on; else the single
// eigenvalues that phase 1 did not finish.  The order of a list does not matter (every item writes only
// its own columns).
template <bool CLUSTERS>
__global__ void k_cl_items(int32_t kd, int32_t nmax, const int32_t* __restrict__ nblk,
                           const float* __restrict__ lam32, const double* __restrict__ tnorm, double rel_cluster,
                           const int32_t* __restrict__ flag, int32_t* __restrict__ count, int4* __restrict__ items) {
  const int32_t c = blockIdx.y;
  const int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  const int32_t n = nblk[c] * kd;
  if (k >= n) return;
  const float* l32 = lam32 + (size_t)c * nmax;
  const double tol = rel_cluster * tnorm[c];
  auto close = [&](int32_t i) { return (double)l32[i + 1] - (double)l32[i] <= tol; };  // to the next shift
  const bool cluster = (k > 0 && close(k - 1)) || (k + 1 < n && close(k));
  if (cluster != CLUSTERS) return;
  int32_t k1 = k;
  if (CLUSTERS) {
    int32_t s = k;
    while (s > 0 && close(s - 1)) --s;
    if ((k - s) % kMaxCluster != 0) return;  // not the first member of an item
    while (k1 + 1 < n && close(k1) && k1 + 1 - k < kMaxCluster) ++k1;
  } else if (flag[(size_t)c * nmax + k] == 0) {
    return;  // phase 1 finished it
  }
  items[atomicAdd(count, 1)] = make_int4(c, k, k1 - k + 1, 0);
}

// one warp, a CTA of its own, per work item of k_cl_items (CTAs past the list's length return), so that
// the items of small systems spread over the SMs: eight to a CTA, 48 items of 62 colours shared six SMs.
// With that, the shuffles of the cluster products bounded by the cluster's size and the cheaper solves:
// n = 180, 62 colours 1.84 -> 0.94 ms, n = 920, 63 colours 10.4 -> 8.2 ms
__global__ void __launch_bounds__(32) k_inviter_cl(int32_t kd, int32_t nmax, const int32_t* __restrict__ nblk,
                                                    const double* __restrict__ dd, const double* __restrict__ ee,
                                                    const float* __restrict__ lam32,
                                                    const double* __restrict__ tnorm, double rel_cluster,
                                                    double* __restrict__ U, double* __restrict__ F,
                                                    double* __restrict__ lam, int32_t* __restrict__ status,
                                                    const int32_t* __restrict__ gid, const int32_t* __restrict__ count,
                                                    const int4* __restrict__ items) {
  __shared__ double sC[kMaxCluster][kMaxCluster + 1];
  __shared__ double sV[kMaxCluster][kMaxCluster + 1];
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x;
  const int32_t item = blockIdx.x;
  if (item >= *count) return;  // uniform over the warp
  const int4 it4 = items[item];
  const int32_t c = it4.x, k0 = it4.y, kc = it4.z, k1 = k0 + kc - 1;
  const uint64_t cseed = gid ? (uint64_t)gid[c] : (uint64_t)c;
  const int32_t n = nblk[c] * kd;
  const float* l32 = lam32 + (size_t)c * nmax;
  double* u = U + (size_t)c * nmax * nmax;
  const double* d = dd + (size_t)c * nmax;
  const double* e = ee + (size_t)c * nmax;
  const size_t nn = (size_t)nmax * nmax;
  double* f0 = F + (size_t)c * 5 * nn;
  double* xm = f0 + 3 * nn;
  const double tn = tnorm[c];
  const double pivmin = 2.2e-16 * tn;
  const double res_tol = kResTol * tn;
  int32_t failed = 0;
  {
    {
      const bool act = lane < kc;
      const int32_t col = k0 + (act ? lane : 0);  // idle lanes shadow member 0 and store nothing
      const Col64 m{f0 + col, f0 + nn + col, f0 + 2 * nn + col, f0 + 3 * nn + col, (size_t)nmax};
      const double g_lo = k0 > 0 ? (double)l32[k0] - (double)l32[k0 - 1] : tn;
      const double g_hi = k1 + 1 < n ? (double)l32[k1 + 1] - (double)l32[k1] : tn;
      const double win_lo = (double)l32[k0] - 0.25 * g_lo - 2e-6 * tn;
      const double win_hi = (double)l32[k1] + 0.25 * g_hi + 2e-6 * tn;
      double lamj = 0.0;
      bool ok_all = false;
      for (int attempt = 0; attempt < 3 && !ok_all; ++attempt) {
        // start vectors (their expected norm folded into the first solve's right-hand side)
        if (act)
          for (int32_t i = 0; i < n; ++i)
            xm[(size_t)i * nmax + col] = hash_unit(cseed * 1000003ull + (uint64_t)col + 7919ull * attempt, (uint64_t)i);
        double scl = sqrt(3.0 / (double)n);
        double sigma = (double)l32[col];
        for (int it = 0; it < 8; ++it) {
          double rq1;
          const double y2 = kc > 1 ? shifted_solve<false>(m, d, e, n, sigma, scl, pivmin, act, rq1)
                                   : shifted_solve<true>(m, d, e, n, sigma, scl, pivmin, act, rq1);
          const double growth = sqrt(y2);
          if (kc == 1) {
            scl = 1.0 / growth;
            if (it >= 1) sigma = rq1 / y2;
            if (__all_sync(FULL, !act || (it >= 2 && growth * res_tol > 1.0))) break;
            continue;
          }
          // modified Gram-Schmidt in member order; pass s subtracts the projection on member s-1
          // (coefficient from pass s-1) and takes the inner products with member s
          double cprev = 0.0, nrm2 = 1.0;
          for (int32_t s = 0; s < kc; ++s) {
            double dj = 0.0;
            for (int32_t i0 = 0; i0 < n; i0 += kCB) {
              double v[kCB];
#pragma unroll
              for (int q = 0; q < kCB; ++q) v[q] = (i0 + q < n) ? xm[(size_t)(i0 + q) * nmax + col] : 0.0;
#pragma unroll
              for (int q = 0; q < kCB; ++q) {
                if (s > 0) {
                  const double xp = __shfl_sync(FULL, v[q], s - 1);
                  if (lane >= s) v[q] = fma(-cprev, xp, v[q]);
                }
                const double xs = __shfl_sync(FULL, v[q], s);
                dj = fma(xs, v[q], dj);
              }
              if (s > 0 && act && lane >= s) {
#pragma unroll
                for (int q = 0; q < kCB; ++q)
                  if (i0 + q < n) xm[(size_t)(i0 + q) * nmax + col] = v[q];
              }
            }
            const double ds = __shfl_sync(FULL, dj, s);
            if (lane == s) nrm2 = ds;
            cprev = lane > s ? dj / ds : 0.0;
          }
          // normalise and take the Rayleigh quotient x^T T x
          const double r = 1.0 / sqrt(nrm2);
          double rq = 0.0, prev = 0.0;
          for (int32_t i0 = 0; i0 < n; i0 += kCB) {
            double v[kCB], dv[kCB], ev[kCB];
#pragma unroll
            for (int q = 0; q < kCB; ++q) {
              const int32_t i = i0 + q;
              v[q] = i < n ? xm[(size_t)i * nmax + col] * r : 0.0;
              dv[q] = i < n ? d[i] : 0.0;
              ev[q] = (i > 0 && i < n) ? e[i - 1] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < kCB; ++q) {
              rq += v[q] * (dv[q] * v[q] + 2.0 * ev[q] * prev);
              prev = v[q];
              if (act && i0 + q < n) xm[(size_t)(i0 + q) * nmax + col] = v[q];
            }
          }
          scl = 1.0;
          if (it >= 1) sigma = rq;
          const bool conv = it >= 2 && growth * res_tol > 1.0;
          if (__all_sync(FULL, !act || conv)) break;
        }
        lamj = sigma;
        const double fin = kc > 1 ? 1.0 : scl;  // a single vector is normalised as it is written
        if (kc > 1) {
          // Rayleigh-Ritz inside the cluster: C = X^T T X, column j accumulated by lane j
          double cc[kMaxCluster];
#pragma unroll
          for (int a = 0; a < kMaxCluster; ++a) cc[a] = 0.0;
          double xprev = 0.0;
          double xcur = xm[col];
          for (int32_t i0 = 0; i0 < n; i0 += kCB) {
            double xnx[kCB], dv[kCB], elo[kCB], ehi[kCB];
#pragma unroll
            for (int q = 0; q < kCB; ++q) {
              const int32_t i = i0 + q;
              xnx[q] = (i + 1 < n) ? xm[(size_t)(i + 1) * nmax + col] : 0.0;
              dv[q] = i < n ? d[i] : 0.0;
              elo[q] = (i > 0 && i < n) ? e[i - 1] : 0.0;
              ehi[q] = (i + 1 < n) ? e[i] : 0.0;
            }
#pragma unroll
            for (int q = 0; q < kCB; ++q) {
              const double tx = dv[q] * xcur + elo[q] * xprev + ehi[q] * xnx[q];
#pragma unroll
              for (int a = 0; a < kMaxCluster; ++a) {
                if (a >= kc) break;  // the whole warp
                cc[a] = fma(__shfl_sync(FULL, xcur, a), tx, cc[a]);
              }
              xprev = xcur;
              xcur = xnx[q];
            }
          }
          if (act)
#pragma unroll
            for (int a = 0; a < kMaxCluster; ++a)
              if (a < kc) sC[a][lane] = cc[a];
          __syncwarp();
          if (lane == 0) {
            double (*C)[kMaxCluster + 1] = sC;
            double (*V)[kMaxCluster + 1] = sV;
            for (int32_t a = 0; a < kc; ++a)
              for (int32_t q = 0; q < kc; ++q) V[a][q] = a == q ? 1.0 : 0.0;
            for (int32_t a = 0; a < kc; ++a)
              for (int32_t q = a + 1; q < kc; ++q) {
                const double t = 0.5 * (C[a][q] + C[q][a]);
                C[a][q] = t;
                C[q][a] = t;
              }
            for (int sweep = 0; sweep < 30; ++sweep) {  // cyclic Jacobi
              double off = 0.0, on = 0.0;
              for (int32_t a = 0; a < kc; ++a)
                for (int32_t q = 0; q < kc; ++q) (a == q ? on : off) += C[a][q] * C[a][q];
              if (off <= 1e-32 * on || off == 0.0) break;
              for (int32_t a = 0; a < kc; ++a)
                for (int32_t q = a + 1; q < kc; ++q) {
                  if (C[a][q] == 0.0) continue;
                  const double theta = (C[q][q] - C[a][a]) / (2.0 * C[a][q]);
                  const double t = (theta >= 0 ? 1.0 : -1.0) / (fabs(theta) + sqrt(theta * theta + 1.0));
                  const double cs = 1.0 / sqrt(t * t + 1.0), sn = t * cs;
                  for (int32_t r2 = 0; r2 < kc; ++r2) {
                    const double ca = C[r2][a], cb = C[r2][q];
                    C[r2][a] = cs * ca - sn * cb;
                    C[r2][q] = sn * ca + cs * cb;
                  }
                  for (int32_t r2 = 0; r2 < kc; ++r2) {
                    const double ca = C[a][r2], cb = C[q][r2];
                    C[a][r2] = cs * ca - sn * cb;
                    C[q][r2] = sn * ca + cs * cb;
                  }
                  for (int32_t r2 = 0; r2 < kc; ++r2) {
                    const double va = V[r2][a], vb = V[r2][q];
                    V[r2][a] = cs * va - sn * vb;
                    V[r2][q] = sn * va + cs * vb;
                  }
                }
            }
          }
          __syncwarp();
          lamj = act ? sC[lane][lane] : 0.0;
        }
        ok_all = __all_sync(FULL, !act || (lamj >= win_lo && lamj <= win_hi));
        if (!ok_all && attempt < 2) continue;
        // write the eigenvectors: X (rotated by V inside a cluster) into U
        double vcol[kMaxCluster];
#pragma unroll
        for (int a = 0; a < kMaxCluster; ++a) vcol[a] = (kc > 1 && act && a < kc) ? sV[a][lane] : 0.0;
        for (int32_t i0 = 0; i0 < n; i0 += kCB) {
          double v[kCB];
#pragma unroll
          for (int q = 0; q < kCB; ++q) v[q] = (i0 + q < n) ? xm[(size_t)(i0 + q) * nmax + col] : 0.0;
#pragma unroll
          for (int q = 0; q < kCB; ++q) {
            double o = v[q] * fin;
            if (kc > 1) {
              o = 0.0;
#pragma unroll
              for (int a = 0; a < kMaxCluster; ++a) {
                if (a >= kc) break;  // the whole warp
                o = fma(__shfl_sync(FULL, v[q], a), vcol[a], o);
              }
            }
            if (act && i0 + q < n) u[(size_t)(i0 + q) * nmax + col] = o;
          }
        }
        if (act) lam[(size_t)c * nmax + col] = lamj;
        if (!ok_all) failed = 1;
        __syncwarp();
      }
    }
  }
  if (failed) atomicOr(&status[c], 1);  // an eigenvalue outside its window after every attempt
}

// Y[k][col] = sum_i U[i][k] X[i][col], w[k] = ||Y[k]||^2 (one thread per k).  B: the block width (0:
// any, up to 32), so that the b running sums are registers and no test of b stands between the FMAs;
// eight rows of U are loaded ahead of their FMAs.
template <int B>
__global__ void __launch_bounds__(128) k_ritz_y(int32_t kd, int32_t b_, int32_t nmax, const int32_t* __restrict__ nblk,
                                                const double* __restrict__ U, const double* __restrict__ X,
                                                double* __restrict__ Y, double* __restrict__ wgt) {
  constexpr int NB = B ? B : CSS_MAX_B;
  constexpr int CH = 64;
  __shared__ double shx[CH * NB];
  const int32_t b = B ? B : b_;
  const int32_t c = blockIdx.y;
  const int32_t n = nblk[c] * kd;
  const int32_t k = blockIdx.x * blockDim.x + threadIdx.x;
  const double* u = U + (size_t)c * nmax * nmax + min(k, nmax - 1);
  const double* x = X + (size_t)c * nmax * b;
  double acc[NB];
#pragma unroll
  for (int a = 0; a < NB; ++a) acc[a] = 0.0;
  if ((int32_t)(blockIdx.x * blockDim.x) < n)  // the whole CTA
    for (int32_t i0 = 0; i0 < n; i0 += CH) {
      const int32_t ie = min(n, i0 + CH);
      __syncthreads();
      for (int32_t t = threadIdx.x; t < (ie - i0) * b; t += blockDim.x) shx[t] = x[(size_t)i0 * b + t];
      __syncthreads();
      for (int32_t i = i0; i < ie; i += 8) {
        double uk[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) uk[q] = i + q < ie ? u[(size_t)(i + q) * nmax] : 0.0;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (i + q >= ie) break;
          const double* xr = shx + (i + q - i0) * b;
#pragma unroll
          for (int a = 0; a < NB; ++a)
            if (B || a < b) acc[a] = fma(uk[q], xr[a], acc[a]);
        }
      }
    }
  if (k < n) {
    double w = 0.0;
#pragma unroll
    for (int a = 0; a < NB; ++a)
      if (B || a < b) {
        Y[((size_t)c * nmax + k) * b + a] = acc[a];
        w = fma(acc[a], acc[a], w);
      }
    wgt[(size_t)c * nmax + k] = w;
  } else if (k < nmax) {
    wgt[(size_t)c * nmax + k] = 0.0;
  }
}

// Zt[i][col] = sum_k U[i][k] g(lam_k) Y[k][col] (one thread per row i; U in 128 x 32 tiles through
// shared memory, so that its rows are read whole).  fn bit 1: g = x^(-1/2) (inverse square root of an
// overlap, positive Ritz values; NaN otherwise) instead of the Fermi function; bit 0: g multiplied by x
// (the energy-weighted density matrix, T_c Z_c).
template <int B>
__global__ void __launch_bounds__(128) k_zt(int32_t kd, int32_t b_, int32_t nmax, const int32_t* __restrict__ nblk,
                                            const int32_t* __restrict__ sys_of_colour, const double* __restrict__ mu,
                                            const double* __restrict__ kT, const double* __restrict__ U,
                                            const double* __restrict__ lam, const double* __restrict__ Y,
                                            double* __restrict__ Z, int fn) {
  constexpr int NB = B ? B : CSS_MAX_B;
  constexpr int CH = 32, ROWS = 128;
  __shared__ double shy[CH * NB], sg[CH];
  __shared__ double su[ROWS][CH + 1];
  const int32_t b = B ? B : b_;
  const int32_t c = blockIdx.y;
  const int32_t n = nblk[c] * kd;
  const int32_t ib = blockIdx.x * ROWS, i = ib + threadIdx.x;
  const double* u = U + (size_t)c * nmax * nmax;
  const int32_t s = sys_of_colour[c];
  const double m_ = mu[s], t_ = kT[s];
  double acc[NB];
#pragma unroll
  for (int a = 0; a < NB; ++a) acc[a] = 0.0;
  if (ib < n)  // the whole CTA
    for (int32_t k0 = 0; k0 < n; k0 += CH) {
      const int32_t ke = min(n, k0 + CH);
      __syncthreads();
      if (threadIdx.x < ke - k0) {
        const double l = lam[(size_t)c * nmax + k0 + threadIdx.x];
        double fw = (fn & 2) ? (l > 0.0 ? 1.0 / sqrt(l) : __longlong_as_double(0x7ff8000000000000ll))
                             : css_fermi_dirac(l, m_, t_);
        if (fn & 1) fw *= l;
        sg[threadIdx.x] = fw;
      }
      for (int32_t t = threadIdx.x; t < ROWS * CH; t += blockDim.x) {
        const int32_t r = t / CH, k = t - r * CH;
        su[r][k] = ib + r < n && k0 + k < ke ? u[(size_t)(ib + r) * nmax + k0 + k] : 0.0;
      }
      __syncthreads();
      for (int32_t t = threadIdx.x; t < (ke - k0) * b; t += blockDim.x)
        shy[t] = sg[t / b] * Y[((size_t)c * nmax + k0) * b + t];
      __syncthreads();
      if (i < n)
#pragma unroll 4
        for (int32_t k = 0; k < ke - k0; ++k) {
          const double uk = su[threadIdx.x][k];
#pragma unroll
          for (int a = 0; a < NB; ++a)
            if (B || a < b) acc[a] = fma(uk, shy[k * b + a], acc[a]);
        }
    }
  if (i < nmax) {
#pragma unroll
    for (int a = 0; a < NB; ++a)
      if (B || a < b) Z[((size_t)c * nmax + i) * b + a] = (i < n) ? acc[a] : 0.0;
  }
}

// diagnostics: copy the FP32 shifts over the eigenvalues
__global__ void k_shifts_out(int32_t nmax, const float* __restrict__ lam32, double* __restrict__ lam) {
  for (int32_t k = threadIdx.x; k < nmax; k += blockDim.x)
    lam[(size_t)blockIdx.x * nmax + k] = (double)lam32[(size_t)blockIdx.x * nmax + k];
}

}  // namespace

namespace {

// Launch of k_apply_refl: the column split that fills the last wave of CTAs best (the largest share of
// the columns on one SM is smallest), within shared memory
template <bool FWD>
css_status launch_refl(css_ctx* ctx, const EigArgs& a, double* X, cudaStream_t st) {
  constexpr size_t kSmem = 200 * 1024;  // of a CTA
  const int32_t kd = a.b, b = a.b, nmax = a.m * a.b;
  auto bytes = [&](int32_t cw) {
    return sizeof(double) * ((size_t)nmax * cw + 2 * (size_t)(nmax / kd + 1) * (kd + 1));
  };
  int32_t best = 1;
  double least = 1e300;
  for (int32_t cw = b; cw >= 1; --cw) {
    const int64_t splits = css_ceil_div(b, cw);
    if (bytes(cw) > kSmem || splits > 12) continue;
    const double load = (double)css_ceil_div((int64_t)a.n_col * splits, ctx->n_sm) * cw;
    if (load < 0.95 * least) {
      least = load;
      best = cw;
    }
  }
  const int32_t tasks = (nmax / kd + 1) * best;
  const unsigned threads = (unsigned)std::min<int32_t>(1024, (tasks + 31) / 32 * 32);
  CSS_TRY(css_smem_limit(ctx, k_apply_refl<FWD>, kSmem));
  k_apply_refl<FWD><<<dim3((unsigned)a.n_col, (unsigned)css_ceil_div(b, best)), threads, bytes(best), st>>>(
      kd, b, best, nmax, a.rcap, a.nblk, a.RV, a.RT, X);
  CSS_LAUNCHED(ctx);
  return CSS_OK;
}

// Launch of k_band_to_tri: lanes per sweep from the band width; enough warps for the sweeps that
// can be in flight (a sweep trails the one before it by about three windows of kd rows, so two per
// sweep never starve it); the band in shared memory when it fits beside the sweeps' vectors, else
// clusters of as many CTAs per colour as the chip has SMs for (at most four).
template <int LPS>
css_status launch_band(css_ctx* ctx, const EigArgs& a, int32_t ldb, cudaStream_t st) {
  constexpr int SPW = 32 / LPS;
  constexpr size_t kSmem = 220 * 1024;
  const int32_t kd = a.b, nmax = a.m * a.b;
  const int32_t flight = nmax / (2 * kd) + 1;
  BandArgs ba{kd, nmax, ldb, a.rcap, 1, ctx->test_band_hold, a.nblk, a.AB, a.RV, a.RT, nullptr, a.d, a.e, a.status};
  auto warps = [&](int32_t ctas, bool smem) {
    return (int32_t)std::min<int64_t>(smem ? 32 : 16, css_ceil_div(flight, (int64_t)SPW * ctas) + 1);
  };
  auto bytes = [&](int32_t nw, bool smem) {
    return sizeof(double) * ((size_t)nw * SPW * (band_group_doubles(kd, ldb, LPS, smem) + (smem ? 1 : 0)) +
                             (smem ? (size_t)nmax * ldb : 0));
  };
  cudaLaunchConfig_t cfg = {};
  cfg.stream = st;
  if (bytes(warps(1, true), true) <= kSmem) {
    const int32_t nw = warps(1, true);
    cfg.gridDim = dim3((unsigned)a.n_col);
    cfg.blockDim = dim3((unsigned)(32 * nw));
    cfg.dynamicSmemBytes = bytes(nw, true);
    CSS_TRY(css_smem_limit(ctx, k_band_to_tri<LPS, true>, kSmem));
    CSS_CU(ctx, cudaLaunchKernelEx(&cfg, k_band_to_tri<LPS, true>, ba));
    CSS_LAUNCHED(ctx);
    return CSS_OK;
  }
  int32_t C = a.n_col * 4 <= ctx->n_sm ? 4 : a.n_col * 2 <= ctx->n_sm ? 2 : 1;
  int32_t nw = warps(C, false);
  while (nw > 1 && bytes(nw, false) > kSmem) --nw;  // fewer sweeps in flight, the same result
  ba.cta_per_col = C;
  const size_t S = (size_t)C * nw * SPW;
  CSS_TRY(css_ws(ctx, "e_slots", (size_t)a.n_col * S * sizeof(unsigned long long), (void**)&ba.slots));
  CSS_CU(ctx, cudaMemsetAsync(ba.slots, 0, (size_t)a.n_col * S * sizeof(unsigned long long), st));
  cfg.gridDim = dim3((unsigned)(a.n_col * C));
  cfg.blockDim = dim3((unsigned)(32 * nw));
  cfg.dynamicSmemBytes = bytes(nw, false);
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)C;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  CSS_TRY(css_smem_limit(ctx, k_band_to_tri<LPS, false>, kSmem));
  CSS_CU(ctx, cudaLaunchKernelEx(&cfg, k_band_to_tri<LPS, false>, ba));
  CSS_LAUNCHED(ctx);
  k_tri_out<<<a.n_col, 256, 0, st>>>(kd, nmax, ldb, a.nblk, a.AB, a.d, a.e);
  CSS_LAUNCHED(ctx);
  return CSS_OK;
}

}  // namespace

css_status css_eigen_ritz(css_ctx* ctx, const EigArgs& a, cudaStream_t st) {
  const int32_t nc = a.n_col, b = a.b, nmax = a.m * b, ldb = css_band_ld(b);
  k_band_build<<<nc, 256, 0, st>>>(b, a.m, nmax, ldb, a.Ablk, a.Bblk, a.nblk, a.AB);
  CSS_LAUNCHED(ctx);
  CSS_CU(ctx, cudaMemsetAsync(a.status, 0, sizeof(int32_t) * nc, st));
  if (b <= 8) CSS_TRY(launch_band<8>(ctx, a, ldb, st));
  else if (b <= 16) CSS_TRY(launch_band<16>(ctx, a, ldb, st));
  else CSS_TRY(launch_band<32>(ctx, a, ldb, st));
  if (a.B0)
    k_x0_b0<<<nc, 256, 0, st>>>(b, nmax, a.B0, a.X0);
  else
    k_x0<<<nc, 256, 0, st>>>(b, nmax, a.cnt, a.X0);
  CSS_LAUNCHED(ctx);
  int32_t* cl_count;
  int4* cl_items;
  CSS_TRY(css_ws(ctx, "e_cl_count", 256, (void**)&cl_count));
  CSS_TRY(css_ws(ctx, "e_cl_items", 2 * (size_t)nc * nmax * sizeof(int4), (void**)&cl_items));
  CSS_CU(ctx, cudaMemsetAsync(cl_count, 0, 2 * sizeof(int32_t), st));
  // Three parts that do not depend on one another run side by side: the reflectors on X0 (needed by
  // k_ritz_y only), phase 1 of the inverse iteration, and phase 2 for the clusters, which phase 1 leaves
  // alone.  Phase 2 is one warp per item, a chain of solves that leaves most of the chip idle.  Eigen stage in
  // turn -> side by side: 27 colours of 180 3.3 -> 2.5 ms, 62 of 180 3.6 -> 2.9; 63 of 920, where each part fills
  // the FP64 pipes, 48.5 -> 48.0.
  while (ctx->side.size() < 2) {
    cudaStream_t s2;
    CSS_CU(ctx, cudaStreamCreateWithFlags(&s2, cudaStreamNonBlocking));
    ctx->side.push_back(s2);
  }
  while (ctx->side_ev.size() < 4) {
    cudaEvent_t e2;
    CSS_CU(ctx, cudaEventCreateWithFlags(&e2, cudaEventDisableTiming));
    ctx->side_ev.push_back(e2);
  }
  const cudaStream_t s_refl = ctx->side[0], s_cl = ctx->side[1];
  const dim3 gk((unsigned)css_ceil_div(nmax, 128), (unsigned)nc);
  // phase 2 on a compact list: one warp per cluster (list 0) or unfinished eigenvalue (list 1) of any colour
  auto phase2 = [&](int list, cudaStream_t s) -> css_status {
    int4* items = cl_items + (size_t)list * nc * nmax;
    (list == 0 ? k_cl_items<true> : k_cl_items<false>)<<<gk, 128, 0, s>>>(b, nmax, a.nblk, a.lam32, a.tnorm, 1e-4,
                                                                          a.flag, cl_count + list, items);
    CSS_LAUNCHED(ctx);
    k_inviter_cl<<<(unsigned)(nc * nmax), 32, 0, s>>>(b, nmax, a.nblk, a.d, a.e, a.lam32, a.tnorm, 1e-4, a.U, a.F,
                                                     a.lam, a.status, a.gid, cl_count + list, items);
    CSS_LAUNCHED(ctx);
    return CSS_OK;
  };
  auto parts = [&]() -> css_status {
    CSS_CU(ctx, cudaEventRecord(ctx->side_ev[0], st));
    CSS_CU(ctx, cudaStreamWaitEvent(s_refl, ctx->side_ev[0], 0));
    CSS_TRY(launch_refl<true>(ctx, a, a.X0, s_refl));
    const size_t sh = 2 * (size_t)nmax * sizeof(float);  // 32 KB at the largest nmax, 4096
    k_bisect32<<<dim3((unsigned)nc, (unsigned)css_ceil_div(nmax, 128)), 128, sh, st>>>(b, nmax, a.nblk, a.d, a.e,
                                                                                      a.lam32, a.tnorm);
    CSS_LAUNCHED(ctx);
    CSS_CU(ctx, cudaEventRecord(ctx->side_ev[1], st));
    CSS_CU(ctx, cudaStreamWaitEvent(s_cl, ctx->side_ev[1], 0));
    CSS_TRY(phase2(0, s_cl));
    k_inviter_p1<<<gk, 128, 2 * (size_t)nmax * sizeof(float), st>>>(b, nmax, a.nblk, a.d, a.e, a.lam32, a.tnorm, 1e-4,
                                                                   a.U, a.F, a.lam, a.flag, a.gid);
    CSS_LAUNCHED(ctx);
    return phase2(1, st);
  };
  const css_status rc = parts();
  // joined on every path, so that no side stream still works on the workspace after return
  CSS_CU(ctx, cudaEventRecord(ctx->side_ev[2], s_refl));
  CSS_CU(ctx, cudaStreamWaitEvent(st, ctx->side_ev[2], 0));
  CSS_CU(ctx, cudaEventRecord(ctx->side_ev[3], s_cl));
  CSS_CU(ctx, cudaStreamWaitEvent(st, ctx->side_ev[3], 0));
  CSS_TRY(rc);
  if (ctx->debug_eig == 1) {
    k_shifts_out<<<nc, 256, 0, st>>>(nmax, a.lam32, a.lam);
    CSS_LAUNCHED(ctx);
  }
  dim3 g((unsigned)css_ceil_div(nmax, 128), (unsigned)nc);
  (b == 6 ? k_ritz_y<6> : b == 23 ? k_ritz_y<23> : k_ritz_y<0>)<<<g, 128, 0, st>>>(b, b, nmax, a.nblk, a.U, a.X0, a.Y,
                                                                                     a.wgt);
  CSS_LAUNCHED(ctx);
  return CSS_OK;
}

css_status css_eigen_z(css_ctx* ctx, const EigArgs& a, const int32_t* sys_of_colour, const double* mu,
                       const double* kT, double* Z, cudaStream_t st, int fn) {
  const int32_t nc = a.n_col, b = a.b, nmax = a.m * b;
  dim3 g((unsigned)css_ceil_div(nmax, 128), (unsigned)nc);
  (b == 6 ? k_zt<6> : b == 23 ? k_zt<23> : k_zt<0>)<<<g, 128, 0, st>>>(b, b, nmax, a.nblk, sys_of_colour, mu, kT, a.U,
                                                                         a.lam, a.Y, Z, fn);
  CSS_LAUNCHED(ctx);
  CSS_TRY(launch_refl<false>(ctx, a, Z, st));
  return CSS_OK;
}

css_status css_eigen_project(css_ctx* ctx, const EigArgs& a, double* V, double* YV, double* scratch, cudaStream_t st) {
  const int32_t nc = a.n_col, b = a.b, nmax = a.m * b;
  CSS_TRY(launch_refl<true>(ctx, a, V, st));
  dim3 g((unsigned)css_ceil_div(nmax, 128), (unsigned)nc);
  (b == 6 ? k_ritz_y<6> : b == 23 ? k_ritz_y<23> : k_ritz_y<0>)<<<g, 128, 0, st>>>(b, b, nmax, a.nblk, a.U, V, YV,
                                                                                     scratch);
  CSS_LAUNCHED(ctx);
  return CSS_OK;
}
