// FP64 H * V on the tensor cores: every entry is cut into eight 8-bit digits, the digit products are
// summed exactly, and the sums are put together in 64-bit integers (the Ozaki scheme: Ozaki, Ogita,
// Oishi & Rump, Numer. Algorithms 59 (2012) 95; its integer form: Ootomo, Ozaki & Yokota, IJHPCA 38
// (2024) 297).
//
// The GB300 runs FP64 FMAs at 1/64 of its FP32 rate (a warp instruction per 16 clocks of an SM), which
// bounded the DFMA kernel (css_lanczos.cu k_spmm): 5.38 ms a launch for 128 molecules at b = 23, 48.7 us for 64
// at b = 6.  Here they take 1.00 ms (digits of V and exponents included) and 40 us.  Whole builds are faster than with
// DFMA at every b that comes here: 2,000 molecules b = 1 19.7 -> 11.4 ms, b = 4 43.8 -> 25.6, b = 9 160 -> 90; 512
// molecules b = 13 70.8 -> 31.6, b = 16 68.3 -> 32.2, b = 24 144 -> 62; 64 molecules b = 1 6.2 -> 4.8, b = 6 6.57 -> 6.34.
// A bf16 holds an 8-bit signed digit exactly and the products of two digits sum exactly in an FP32 accumulator
// up to 2^24, so bf16 tensor-core products of digits are integer arithmetic.
//
// Digits: H is scaled by powers of two, its rows by 2^-e (2^e above the row's largest |entry|) and then its
// columns by 2^-c (so above the largest of the scaled column), and V by 2^c and each of its columns by its
// largest entry.  A scaled entry times 2^62 rounds to an integer x = sum_s d_s 256^(7 - s) with
// |d_0| <= 65 and -128 <= d_s <= 128.  Of the 64 products d_i d'_j the 43 with i + j <= 8 are taken; the others
// are below 2^-69 of the two maxima.  So an output differs from the exact sum by its own rounding and the
// rounding of the entries to 2^-63 of those maxima; the column scaling keeps that true of graded matrices
// D A D.  The sums are exact, so the result depends on neither the order of the blocks nor the other columns of
// the pass.  The ten bits below those of an FP64 sum are needed: in the recurrence the on-site terms of a row (tens
// of eV) cancel and leave couplings that an FP64 sum carries to their own 2^-53.  With seven digits (2^-56,
// 34 products; 0.79 ms) the projected blocks of 20 molecules were off by 4 (b = 13) to 12 times (b = 24) as much as
// with the DFMA kernel; now by a third to a half.
// An infinity or NaN in a row of H or a column of V makes that row or column of the result NaN.
//
// Shape: mma.sync m16n8k16 with 16 columns of V as M, the rows of an H block as N and the columns of the
// block as K.  The sums of the nine i + j and of every N tile live in registers (108 at b = 23), which a
// tcgen05 tile of M = 128 in tensor memory would need once per 24 columns of N with a K of 23 per
// block: the digit products are many small MMAs, not one large one.
// A CTA takes one block row I and eight tiles of 16 columns, a warp each.  The digits of 16 columns of H_IJ (6 KB
// at b = 23, shared by the warps) and of as many rows of V_J (4 KB per warp) arrive in MMA fragment order through a
// cp.async ring of five stages at b > 16 (all that shared memory holds), else three (six when the CTAs do not
// fill the chip and nothing else hides a copy's latency); a thread copies the very 16 bytes of V it will load.
#include <algorithm>

#include "css_lanczos.cuh"

namespace {

constexpr int kDig = 8;    // digits of an entry
constexpr int kSum = 9;    // sums S_d over i + j = d
constexpr int kWarps = 8;  // column tiles per CTA
constexpr int kTile = 16;  // columns of V per warp
// rows of H and columns of V whose largest entry is below 2^-961 keep 2^-1023 as their last digit
constexpr int kMinExp = 61;
constexpr int kMinCol = -900;    // least column scale of H
constexpr int kColBias = 4096;   // hcol holds c + kColBias, 0 for a column without entries
constexpr int kNotFinite = 4096; // exponent of a column of V with an infinity or NaN
// largest buffer of V's digits: wider blocks of columns go through it in turn, each reading H's digits
// once more (at 10,000 molecules, b = 23, eight turns)
constexpr size_t kVBytes = (size_t)1 << 30;
// largest digits of H (2 times its FP64 blocks at b = 16, 2.9 at 23, 7.1 at 6, 256 at 1): beyond, the DFMA kernel
// runs as before
constexpr size_t kHBytes = (size_t)10 << 30;

// NT tiles of 8 rows and KC tiles of 16 columns of an H block; a stage holds one K tile
template <int NT, int KC>
struct IntCfg {
  static constexpr int HB = kDig * NT * 32 * 8;  // bytes of the digits of a K tile of an H block
  static constexpr int VB = kDig * 32 * 16;      // of a V block (16 columns)
  static constexpr int smem(int stages) { return stages * (HB + kWarps * VB); }
};
inline int nt_of(int32_t b) { return (b + 7) / 8; }
inline int kc_of(int32_t b) { return (b + 15) / 16; }
inline size_t h_block_bytes(int32_t b) { return (size_t)kDig * nt_of(b) * 32 * kc_of(b) * 8; }
inline size_t v_block_bytes(int32_t b) { return (size_t)kDig * kc_of(b) * 32 * 16; }

__device__ __forceinline__ uint32_t expo(double x) { return (uint32_t)(__double2hiint(x) & 0x7ff00000) >> 20; }
// 2^(62 + c - e) for entries of biased exponent at most E: |x| < 2^e, e = E - 1022; 0 where it would be
// subnormal (no entry under it then reaches half of the last digit)
__device__ __forceinline__ double digit_scale(int E, int c) {
  return __hiloint2double(max(2107 + c - max(E, kMinExp), 0) << 20, 0);
}
__device__ __forceinline__ int col_scale(int hcol) { return hcol ? max(hcol - kColBias, kMinCol) : 0; }

// the digits of x0 and x1 (scaled integers) as pairs of bf16, most significant first
__device__ __forceinline__ void digits2(long long x0, long long x1, uint32_t (&d)[kDig]) {
#pragma unroll
  for (int s = kDig - 1; s >= 0; --s) {
    const int a = s ? (int)(signed char)x0 : (int)x0, b = s ? (int)(signed char)x1 : (int)x1;
    x0 = (x0 - a) >> 8;
    x1 = (x1 - b) >> 8;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(d[s]) : "f"((float)b), "f"((float)a));
  }
}

// largest biased exponent of every scalar row of H (a CTA per block row)
__global__ void __launch_bounds__(256) k_hrow_exp(int32_t b, const int32_t* __restrict__ row_ptr,
                                                  const double* __restrict__ H, int32_t* __restrict__ hexp) {
  const int32_t I = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t p0 = row_ptr[I], p1 = row_ptr[I + 1];
  for (int32_t a = warp; a < b; a += 8) {
    uint32_t e = 0;
    if (lane < b)
      for (int64_t p = p0; p < p1; ++p) e = max(e, expo(H[(p * b + a) * b + lane]));
    e = __reduce_max_sync(0xffffffffu, e);
    if (lane == 0) hexp[(int64_t)I * b + a] = (int32_t)e;
  }
}

// largest biased exponent of every column of the row-scaled H (hcol cleared before): a CTA per block row, a
// thread per column of a block
__global__ void __launch_bounds__(256) k_hcol_exp(int32_t b, const int32_t* __restrict__ row_ptr,
                                                  const int32_t* __restrict__ col_idx, const double* __restrict__ H,
                                                  const int32_t* __restrict__ hexp, int32_t* __restrict__ hcol) {
  const int64_t p0 = row_ptr[blockIdx.x], p1 = row_ptr[blockIdx.x + 1];
  const int32_t* e = hexp + (int64_t)blockIdx.x * b;
  for (int64_t t = p0 * b + threadIdx.x; t < p1 * b; t += 256) {
    const int64_t p = t / b;
    const int32_t k = (int32_t)(t - p * b);
    int m = -kColBias;
    for (int32_t a = 0; a < b; ++a) {
      const double h = H[(p * b + a) * b + k];
      if (h != 0.0) m = max(m, (int)expo(h) - max(e[a], kMinExp));
    }
    if (m > -kColBias) atomicMax(&hcol[(int64_t)col_idx[p] * b + k], m + kColBias);
  }
}

// digits of every H block (a CTA per block row) in the order of the B fragments:
// [block][K tile][digit][N tile][lane][2 words]
template <int NT, int KC>
__global__ void __launch_bounds__(256) k_hdigits(int32_t b, const int32_t* __restrict__ row_ptr,
                                                 const int32_t* __restrict__ col_idx, const double* __restrict__ H,
                                                 const int32_t* __restrict__ hexp, const int32_t* __restrict__ hcol,
                                                 uint32_t* __restrict__ out) {
  const int lane = threadIdx.x & 31;
  const int64_t p1 = row_ptr[blockIdx.x + 1];
  for (int64_t t = (int64_t)row_ptr[blockIdx.x] * NT + (threadIdx.x >> 5); t < p1 * NT; t += 8) {
    const int64_t p = t / NT;
    const int nt = (int)(t - p * NT), a = 8 * nt + (lane >> 2);
    const double sc = a < b ? digit_scale(hexp[(int64_t)blockIdx.x * b + a], 0) : 0.0;
    const double* h = H + (p * b + a) * b;
    const int32_t* hc = hcol + (int64_t)col_idx[p] * b;
    auto at = [&](int k) -> long long {
      if (a >= b || k >= b) return 0;
      return __double2ll_rn(h[k] * sc * __hiloint2double((1023 - col_scale(hc[k])) << 20, 0));
    };
#pragma unroll
    for (int r = 0; r < 2 * KC; ++r) {
      const int k = 8 * r + 2 * (lane & 3);
      uint32_t d[kDig];
      digits2(at(k), at(k + 1), d);
#pragma unroll
      for (int s = 0; s < kDig; ++s) out[((((p * KC + r / 2) * kDig + s) * NT + nt) * 32 + lane) * 2 + (r & 1)] = d[s];
    }
  }
}

// largest biased exponent of every column of the scaled V (vexp cleared before): 16 ng rows by 128 columns a CTA
__global__ void __launch_bounds__(128) k_vcol_exp(int64_t N, int32_t ng, int32_t w, int32_t ws, const double* __restrict__ V,
                                                  const int32_t* __restrict__ hcol, int32_t* __restrict__ vexp) {
  const int32_t col = blockIdx.y * 128 + threadIdx.x;
  if (col >= w) return;
  const int64_t r0 = (int64_t)blockIdx.x * ng * 16;
  int e = 0;
  for (int64_t r = r0; r < min(N, r0 + ng * 16); r += 16) {
    const double* v = V + (size_t)r * ws + col;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (r + i >= N) break;
      const int x = (int)expo(v[(size_t)i * ws]);
      e = max(e, x == 0x7ff ? kNotFinite : x + col_scale(hcol[r + i]));
    }
  }
  if (e) atomicMax(&vexp[col], e);
}

// digits of 16 columns of V_J (a warp each) in the order of the A fragments: [tile][J][K tile][digit][lane][4
// words]; columns from col0 on
template <int KC>
__global__ void __launch_bounds__(256) k_vdigits(int32_t nJ, int32_t b, int32_t ntile, int32_t col0, int32_t w, int32_t ws,
                                                 const double* __restrict__ V, const int32_t* __restrict__ hcol,
                                                 const int32_t* __restrict__ vexp, uint4* __restrict__ out) {
  const int64_t wi = ((int64_t)blockIdx.x * 256 + threadIdx.x) >> 5;
  if (wi >= (int64_t)nJ * ntile) return;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const int32_t J = (int32_t)(wi / ntile), tile = (int32_t)(wi - (int64_t)J * ntile);
  const int32_t c0 = col0 + tile * kTile + g, c1 = c0 + 8;
  const int E0 = c0 < w ? vexp[c0] : 0, E1 = c1 < w ? vexp[c1] : 0;
  const double* v = V + (size_t)J * b * ws;
  const int32_t* hc = hcol + (int64_t)J * b;
  auto at = [&](int k, int32_t c, int E) -> long long {
    return k < b && c < w ? __double2ll_rn(v[(size_t)k * ws + c] * digit_scale(E, col_scale(hc[k]))) : 0;
  };
#pragma unroll
  for (int kc = 0; kc < KC; ++kc) {
    uint32_t d[4][kDig];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int k = 16 * kc + 8 * (r >> 1) + 2 * t;
      const int32_t c = r & 1 ? c1 : c0;
      const int E = r & 1 ? E1 : E0;
      digits2(at(k, c, E), at(k + 1, c, E), d[r]);
    }
    uint4* o = out + (((int64_t)tile * nJ + J) * KC + kc) * kDig * 32 + lane;
#pragma unroll
    for (int s = 0; s < kDig; ++s) o[s * 32] = make_uint4(d[0][s], d[1][s], d[2][s], d[3][s]);
  }
}

__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint4& a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, "
      "%2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b0), "r"(b1));
}

// (hi 2^32 + lo) 2^S, rounded once (twice into the subnormals)
__device__ __forceinline__ double join(long long hi, long long lo, int S) {
  const double x = fma((double)hi, 4294967296.0, (double)lo);
  const int e = (int)expo(x) + S;
  if (x == 0.0) return x;
  if (e >= 1 && e <= 2046) return __hiloint2double(__double2hiint(x) + S * (1 << 20), __double2loint(x));
  const int s1 = S >> 1, s2 = S - s1;
  return x * __hiloint2double((1023 + s1) << 20, 0) * __hiloint2double((1023 + s2) << 20, 0);
}

struct IntArgs {
  int32_t b, nJ, ntile, col0, w, ws, flush, row0;
  const int32_t *row_ptr, *col_idx, *hexp, *vexp;
  const unsigned char *Hd, *Vd;
  double* W;
};

template <int NT, int KC, int kStages>
__global__ void __launch_bounds__(32 * kWarps, 1) k_hv_int(const IntArgs a) {
  using C = IntCfg<NT, KC>;
  extern __shared__ __align__(16) unsigned char sm[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t I = blockIdx.x, tile = blockIdx.y * kWarps + warp;
  const bool live = tile < a.ntile;
  const int64_t p0 = a.row_ptr[I];
  const int32_t ns = (int32_t)(a.row_ptr[I + 1] - p0) * KC;  // K tiles of the row
  const unsigned char* vt = a.Vd + (size_t)(live ? tile : 0) * a.nJ * KC * C::VB;
  auto stage_h = [&](int s) { return sm + (size_t)(s % kStages) * (C::HB + kWarps * C::VB); };
  auto stage_v = [&](int s) { return stage_h(s) + C::HB + warp * C::VB; };
  auto load = [&](int32_t s) {
    if (s < ns) {
      const unsigned char* h = a.Hd + (size_t)(p0 * KC + s) * C::HB;
      unsigned char* dh = stage_h(s);
      for (int i = threadIdx.x; i < C::HB / 16; i += 32 * kWarps) copy16(dh + 16 * i, h + 16 * i);
      if (live) {
        const unsigned char* v = vt + ((size_t)(a.col_idx[p0 + s / KC] - a.row0) * KC + s % KC) * C::VB;
        unsigned char* dv = stage_v(s);
#pragma unroll
        for (int i = 0; i < kDig; ++i) copy16(dv + 16 * (32 * i + lane), v + 16 * (32 * i + lane));
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[kSum][NT][4];
  long long hi[NT][4], lo[NT][4];  // sums 0 to 4 and 5 to 8
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      hi[n][i] = lo[n][i] = 0;
#pragma unroll
      for (int d = 0; d < kSum; ++d) acc[d][n][i] = 0.0f;
    }
  for (int s = 0; s < kStages - 1; ++s) load(s);
  int32_t left = a.flush;
#pragma unroll 1
  for (int32_t s = 0; s < ns; ++s) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();  // K tile s has arrived in every thread, s - 1 is read
    load(s + kStages - 1);
    if (live) {
      const unsigned char *dh = stage_h(s), *dv = stage_v(s);
      uint4 av[kDig];
#pragma unroll
      for (int i = 0; i < kDig; ++i) av[i] = *reinterpret_cast<const uint4*>(dv + 16 * (32 * i + lane));
#pragma unroll
      for (int j = 0; j < kDig; ++j)
#pragma unroll
        for (int n = 0; n < NT; ++n) {
          const uint2 bv = *reinterpret_cast<const uint2*>(dh + 8 * ((j * NT + n) * 32 + lane));
#pragma unroll
          for (int i = 0; i < kDig; ++i)
            if (i + j < kSum) mma_bf16(acc[i + j][n], av[i], bv.x, bv.y);
        }
      if ((s + 1) % KC == 0 && (--left == 0 || s + 1 == ns)) {  // the sums are below 2^24 so far: take them over
        left = a.flush;
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
#pragma unroll
            for (int d = 0; d < kSum; ++d) {
              (d < 5 ? hi : lo)[n][i] += (long long)(int)acc[d][n][i] * (1ll << (8 * (d < 5 ? 4 - d : 8 - d)));
              acc[d][n][i] = 0.0f;
            }
          }
      }
    }
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (!live) return;
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int32_t r = 8 * n + 2 * (lane & 3) + (i & 1), c = a.col0 + tile * kTile + (lane >> 2) + 8 * (i >> 1);
      if (r >= a.b || c >= a.w) continue;
      const int EH = a.hexp[(int64_t)I * a.b + r], EV = a.vexp[c];
      double y;
      if (EH == 0x7ff || EV == kNotFinite)
        y = __hiloint2double(0x7ff80000, 0);
      else
        y = join(hi[n][i], lo[n][i], max(EH, kMinExp) + max(EV, kMinExp) - 2 * 1022 - 76);
      a.W[((size_t)I * a.b + r) * a.ws + c] = y;
    }
}

template <int NT, int KC>
css_status launch(css_ctx* ctx, const LzArgs& a, const double* V, double* W, int32_t* vexp, uint4* vd, int32_t per,
                  cudaStream_t st) {
  using C = IntCfg<NT, KC>;
  const int32_t b = a.b, tiles = (int32_t)css_ceil_div(a.w, kTile);
  const int64_t N = (int64_t)a.n_brow * b;
  const int32_t *hexp = a.Hexp + (size_t)a.row0 * b, *hcol = hexp + a.Hexp_n;
  constexpr int deep = KC == 1 ? 6 : 5, flat = KC == 1 ? 3 : 5;
  CSS_TRY(css_smem_limit(ctx, k_hv_int<NT, KC, flat>, C::smem(flat)));
  CSS_TRY(css_smem_limit(ctx, k_hv_int<NT, KC, deep>, C::smem(deep)));
  CSS_CU(ctx, cudaMemsetAsync(vexp, 0, sizeof(int32_t) * a.w, st));
  const int32_t ng = N > 16384 ? 4 : 1;
  k_vcol_exp<<<dim3((unsigned)css_ceil_div(N, 16 * ng), (unsigned)css_ceil_div(a.w, 128)), 128, 0, st>>>(
      N, ng, a.w, a.ws, V, hcol, vexp);
  CSS_LAUNCHED(ctx);
  for (int32_t t0 = 0; t0 < tiles; t0 += per) {
    const int32_t nt = std::min(per, tiles - t0);
    k_vdigits<KC><<<(unsigned)css_ceil_div((int64_t)a.n_brow * nt, 8), 256, 0, st>>>(a.n_brow, b, nt, t0 * kTile, a.w,
                                                                                    a.ws, V, hcol, vexp, vd);
    CSS_LAUNCHED(ctx);
    IntArgs r;
    r.b = b;
    r.nJ = a.n_brow;
    r.ntile = nt;
    r.col0 = t0 * kTile;
    r.w = a.w;
    r.ws = a.ws;
    r.flush = 145 / b;  // the largest sum (d = 7): 145 (6 128^2 + 2 65 128) is below 2^24
    r.row0 = a.row0;
    r.row_ptr = a.row_ptr;
    r.col_idx = a.col_idx;
    r.hexp = hexp;
    r.vexp = vexp;
    r.Hd = static_cast<const unsigned char*>(a.Hdig);
    r.Vd = reinterpret_cast<const unsigned char*>(vd);
    r.W = W;
    const dim3 grid((unsigned)a.n_brow, (unsigned)css_ceil_div(nt, kWarps));
    if (grid.x * (int64_t)grid.y <= ctx->n_sm)
      k_hv_int<NT, KC, deep><<<grid, 32 * kWarps, C::smem(deep), st>>>(r);
    else
      k_hv_int<NT, KC, flat><<<grid, 32 * kWarps, C::smem(flat), st>>>(r);
    CSS_LAUNCHED(ctx);
  }
  return CSS_OK;
}

// column tiles of V's digits that go through the buffer at once
int32_t tiles_at_once(int32_t n_brow, int32_t b, int32_t w) {
  const size_t one = (size_t)n_brow * v_block_bytes(b);
  const int64_t fit = (int64_t)(kVBytes / std::max<size_t>(one, 1)), all = css_ceil_div(w, kTile);
  return (int32_t)std::max<int64_t>(1, std::min(fit, all));
}

}  // namespace

bool css_hv_int_supported(int32_t b, int32_t n_brow, int32_t nnzb) {
  return b <= 24 && (size_t)nnzb * h_block_bytes(b) <= kHBytes && (size_t)n_brow * v_block_bytes(b) <= kVBytes;
}

size_t css_hv_int_h_bytes(int32_t b, int32_t n_brow, int32_t nnzb) {
  return (size_t)nnzb * h_block_bytes(b) + sizeof(int32_t) * 2 * (size_t)n_brow * b;
}

size_t css_hv_int_v_bytes(int32_t n_brow, int32_t b, int32_t w) {
  const size_t exps = ((size_t)w * sizeof(int32_t) + 255) / 256 * 256;
  return exps + std::min(kVBytes, (size_t)css_ceil_div(w, kTile) * n_brow * v_block_bytes(b));
}

css_status css_hv_int_prepare(css_ctx* ctx, int32_t b, int32_t n_brow, int32_t nnzb, const int32_t* row_ptr,
                              const int32_t* col_idx, const double* H, const void** Hdig, const int32_t** Hexp,
                              cudaStream_t st) {
  uint32_t* d;
  int32_t* e;
  CSS_TRY(css_ws(ctx, "h_digits", (size_t)nnzb * h_block_bytes(b), (void**)&d));
  const size_t n = (size_t)n_brow * b;  // exponents of the rows, then of the columns
  CSS_TRY(css_ws(ctx, "h_exp", sizeof(int32_t) * 2 * n, (void**)&e));
  CSS_CU(ctx, cudaMemsetAsync(e + n, 0, sizeof(int32_t) * n, st));
  if (n_brow > 0) {
    k_hrow_exp<<<(unsigned)n_brow, 256, 0, st>>>(b, row_ptr, H, e);
    CSS_LAUNCHED(ctx);
    k_hcol_exp<<<(unsigned)n_brow, 256, 0, st>>>(b, row_ptr, col_idx, H, e, e + n);
    CSS_LAUNCHED(ctx);
    auto kern = b <= 8 ? k_hdigits<1, 1> : b <= 16 ? k_hdigits<2, 1> : k_hdigits<3, 2>;
    kern<<<(unsigned)n_brow, 256, 0, st>>>(b, row_ptr, col_idx, H, e, e + n, d);
    CSS_LAUNCHED(ctx);
  }
  *Hdig = d;
  *Hexp = e;
  return CSS_OK;
}

css_status css_hv_int(css_ctx* ctx, const LzArgs& a, const double* V, double* W, cudaStream_t st) {
  if (a.n_brow == 0 || a.w == 0) return CSS_OK;
  int32_t* vexp = static_cast<int32_t*>(a.Vdig);
  const size_t exps = ((size_t)a.w * sizeof(int32_t) + 255) / 256 * 256;
  uint4* vd = reinterpret_cast<uint4*>(static_cast<unsigned char*>(a.Vdig) + exps);
  const int32_t per = tiles_at_once(a.n_brow, a.b, a.w);
  if (a.b <= 8) return launch<1, 1>(ctx, a, V, W, vexp, vd, per, st);
  if (a.b <= 16) return launch<2, 1>(ctx, a, V, W, vexp, vd, per, st);
  return launch<3, 2>(ctx, a, V, W, vexp, vd, per, st);
}
