// Row passes of one FP64 block-Lanczos step, block widths 6 and 23 (paper: the three-term recurrence and
// block QR of the block-Lanczos paragraph after Eq. 4), without the local reorthogonalisation:
//   S1  W0 = W - Q_{j-1} B_{j-1}^T, stored;  Kq = Q_j^T W0
//   S3  W1 = W0 - Q_j Kq, stored;  Gram W1^T W1
//   T0  V = W1 R0^-1, stored;  Gram V^T V
//   T1  Q_{j+1} = V R1^-1; for a colour that needs a third CholeskyQR pass back to W instead, with its Gram
//   T2  Q_{j+1} = W R2^-1 for those colours
//
// Bound by FP64 issue: an FP64 instruction of a warp takes 64 clocks of its scheduler, so what counts is
// the number of them and that every lane of each has work; copies, shared memory and addresses hide behind
// them.  One warp takes one colour of a chunk of rows, by itself: no CTA barrier, no share of work that
// leaves schedulers uneven.  In tiles of 32 rows it multiplies a row per lane (triangular factors with
// their half of the products only) and then sums the Gram with a block of entries per lane: at b = 23
// 3 x 6 of the full one (32 lanes), 4 x 3 of the upper triangle of a symmetric one (30 lanes); at b = 6 blocks
// of 2 x 2, the rows dealt to three or five lanes per block.  A step at b = 23 is 2,701 FP64 instructions per
// 32 rows of a colour; the tiled kernels (css_lanczos.cu) issued 3,456 and more for partly filled warps, on
// six warps of four schedulers.  Row work of a step, tiled -> here: 128 molecules b = 23 1.90 -> 1.06 ms, 256
// molecules 3.67 -> 2.20, 64 molecules b = 6 88 -> 46 us (factor kernels included).
#include <algorithm>

#include "css_lanczos.cuh"

namespace {

enum { M_S1 = 0, M_S3 = 1, M_T0 = 2, M_T1 = 3, M_T2 = 4 };

template <int B>
struct R64 {
  static constexpr int P = (B + 1) | 1;         // pitch of a staged row: odd, one zero past the last column
  static constexpr int MP = (B + 1) / 2 * 2;    // pitch of the matrix: 16-byte rows
  static constexpr int T = 32 * P;              // values of a staged tile
  // a lane's block of Gram entries: full and symmetric
  static constexpr int FR = B == 23 ? 3 : 2, FC = B == 23 ? 6 : 2, SR = B == 23 ? 4 : 2, SC = B == 23 ? 3 : 2;
  static constexpr int FN = B == 23 ? 32 : 9, SN = B == 23 ? 30 : 6;  // blocks
};
__host__ __device__ constexpr int arrays(int mode) { return mode == M_S1 ? 3 : mode == M_S3 ? 2 : 1; }

template <int B, int MODE>
__global__ void __launch_bounds__(32) k_rows64(const CssRows64 a, int32_t chunk) {
  using C = R64<B>;
  constexpr int P = C::P, NA = arrays(MODE);
  constexpr bool SYM = MODE != M_S1;
  constexpr int GR = SYM ? C::SR : C::FR, GC = SYM ? C::SC : C::FC, NBK = SYM ? C::SN : C::FN, RS = 32 / NBK;
  __shared__ __align__(16) double sM[B * C::MP];
  __shared__ double sT[NA][C::T];  // W (and the result), Q_j, Q_{j-1}
  const int lane = threadIdx.x;
  const int32_t lc = blockIdx.y;
  const bool n3 = MODE >= M_T1 && a.need3[lc] != 0;
  if (MODE == M_T2 && !n3) return;
  const bool gram = MODE <= M_T0 || (MODE == M_T1 && n3);
  const bool mul = MODE != M_S1 || !a.first;
  const int64_t rbeg = (int64_t)blockIdx.x * chunk, rend = min(a.N, rbeg + chunk);
  const double* M = MODE == M_S1 ? a.M + (size_t)(a.cb0 + lc) * B * B : a.M + (size_t)lc * B * B;
  if (mul)
    for (int e = lane; e < B * B; e += 32) {  // S1: B^T, transposed here
      const int l = e / B, k = e - l * B;
      if (MODE == M_S1) sM[k * C::MP + l] = M[e];
      else sM[l * C::MP + k] = M[e];
    }
  for (int e = lane; e < NA * C::T; e += 32) (&sT[0][0])[e] = 0.0;
  // this lane's block of the Gram and its share of the rows
  const int blk = lane % NBK, part = lane / NBK;
  int bi, bj;
  if (!SYM) {
    bi = blk / ((B + C::FC - 1) / C::FC);
    bj = blk % ((B + C::FC - 1) / C::FC);
  } else if (B == 23) {  // rows of blocks start at the first that reaches the diagonal: 8, 7, 6, 4, 3, 2 of them
    bi = blk < 8 ? 0 : blk < 15 ? 1 : blk < 21 ? 2 : blk < 25 ? 3 : blk < 28 ? 4 : 5;
    bj = blk < 8 ? blk : blk < 15 ? blk - 7 : blk < 21 ? blk - 13 : blk < 25 ? blk - 17 : blk < 28 ? blk - 20 : blk - 22;
  } else {
    bi = blk < 3 ? 0 : blk < 5 ? 1 : 2;
    bj = blk < 3 ? blk : blk < 5 ? blk - 2 : 2;
  }
  const bool summing = gram && part < RS;
  double sum[GR][GC];
#pragma unroll
  for (int i = 0; i < GR; ++i)
#pragma unroll
    for (int j = 0; j < GC; ++j) sum[i][j] = 0.0;
  const double* src[3] = {a.W, a.Q, a.Qp};
  double* out = MODE >= M_T1 ? (MODE == M_T1 && n3 ? a.W : a.out) : a.W;
  __syncwarp();
#pragma unroll 1
  for (int64_t r0 = rbeg; r0 < rend; r0 += 32) {
    const int nr = (int)min((int64_t)32, rend - r0);
    const size_t g0 = (size_t)r0 * a.ws + (size_t)lc * B;
#pragma unroll
    for (int n = 0; n < NA; ++n) {
      if (n == 2 && !mul) continue;
#pragma unroll 4
      for (int e = lane; e < 32 * B; e += 32) {
        const int r = e / B, k = e - r * B;
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(&sT[n][r * P + k]);
        const double* s = src[n] + g0 + (size_t)(r < nr ? r : 0) * a.ws + k;
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(s), "r"(r < nr ? 8 : 0) : "memory");
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncwarp();
    if (mul) {  // a row per lane
      double* w = &sT[0][lane * P];
      const double* x = MODE == M_S1 ? &sT[NA - 1][lane * P] : MODE == M_S3 ? &sT[NA > 1 ? 1 : 0][lane * P] : w;
      double o[C::MP];
#pragma unroll
      for (int k = 0; k < C::MP; ++k) o[k] = MODE <= M_S3 && k < B ? w[k] : 0.0;
#pragma unroll
      for (int l = 0; l < B; ++l) {
        const double xl = MODE <= M_S3 ? -x[l] : x[l];
#pragma unroll
        for (int c = 0; c < C::MP / 2; ++c) {
          const int k = 2 * c;
          if (MODE == M_S1 && k > l) continue;      // B^T: k <= l
          if (MODE >= M_T0 && k + 1 < l) continue;  // R^-1: k >= l
          const double2 m = *reinterpret_cast<const double2*>(&sM[l * C::MP + k]);
          if (MODE < M_T0 || k >= l) o[k] = fma(xl, m.x, o[k]);
          if (k + 1 < B && (MODE != M_S1 || k + 1 <= l)) o[k + 1] = fma(xl, m.y, o[k + 1]);
        }
      }
#pragma unroll
      for (int k = 0; k < B; ++k) w[k] = o[k];
      __syncwarp();
#pragma unroll 4
      for (int e = lane; e < nr * B; e += 32) {
        const int r = e / B, k = e - r * B;
        out[g0 + (size_t)r * a.ws + k] = sT[0][r * P + k];
      }
    }
    if (summing) {  // 32 rows in a sum of their own, then into the running one
      double s[GR][GC];
#pragma unroll
      for (int i = 0; i < GR; ++i)
#pragma unroll
        for (int j = 0; j < GC; ++j) s[i][j] = 0.0;
      const double* X = &sT[SYM || NA < 2 ? 0 : 1][bi * GR];
      const double* Y = &sT[0][bj * GC];
#pragma unroll 2
      for (int r = part; r < 32; r += RS) {
        double xv[GR], yv[GC];
#pragma unroll
        for (int i = 0; i < GR; ++i) xv[i] = X[r * P + i];
#pragma unroll
        for (int j = 0; j < GC; ++j) yv[j] = Y[r * P + j];
#pragma unroll
        for (int i = 0; i < GR; ++i)
#pragma unroll
          for (int j = 0; j < GC; ++j) s[i][j] = fma(xv[i], yv[j], s[i][j]);
      }
#pragma unroll
      for (int i = 0; i < GR; ++i)
#pragma unroll
        for (int j = 0; j < GC; ++j) sum[i][j] += s[i][j];
    }
    __syncwarp();  // the tile is read
  }
  if (!gram) return;
  double* o = a.part + ((size_t)blockIdx.x * a.ncb + lc) * B * B;
#pragma unroll
  for (int i = 0; i < GR; ++i)
#pragma unroll
    for (int j = 0; j < GC; ++j) {
      double v = sum[i][j];
#pragma unroll
      for (int p = 1; p < RS; ++p) v += __shfl_sync(0xffffffffu, sum[i][j], blk + p * NBK);
      const int k = bi * GR + i, l = bj * GC + j;
      if (part != 0 || k >= B || l >= B || (SYM && l < k)) continue;
      o[k * B + l] = v;
      if (SYM && l > k) o[l * B + k] = v;
    }
}

template <int B>
css_status launch_rows64(css_ctx* ctx, int mode, const CssRows64& a, cudaStream_t st) {
  const int32_t chunk = css_rows64_chunk(a.N);
  const dim3 grid((unsigned)css_ceil_div(a.N, chunk), (unsigned)a.ncb);
  switch (mode) {
    case M_S1: k_rows64<B, M_S1><<<grid, 32, 0, st>>>(a, chunk); break;
    case M_S3: k_rows64<B, M_S3><<<grid, 32, 0, st>>>(a, chunk); break;
    case M_T0: k_rows64<B, M_T0><<<grid, 32, 0, st>>>(a, chunk); break;
    case M_T1: k_rows64<B, M_T1><<<grid, 32, 0, st>>>(a, chunk); break;
    default: k_rows64<B, M_T2><<<grid, 32, 0, st>>>(a, chunk);
  }
  CSS_LAUNCHED(ctx);
  return CSS_OK;
}

}  // namespace

// Rows of a warp's chunk: whole tiles, four waves of eight warps per SM for 64 colours (a full count: the
// chunk may not depend on the colours of the call, or a colour's sums would)
int32_t css_rows64_chunk(int64_t N) {
  const int64_t r = css_ceil_div(css_ceil_div(N * 64, 152 * 8 * 4), 32) * 32;
  return (int32_t)std::min<int64_t>(std::max<int64_t>(r, 32), 1024);
}

bool css_rows64_supported(bool fp32, int32_t b, bool reorth) { return !fp32 && !reorth && (b == 6 || b == 23); }

css_status css_rows64(css_ctx* ctx, int mode, int32_t b, const CssRows64& a, cudaStream_t st) {
  return b == 6 ? launch_rows64<6>(ctx, mode, a, st) : launch_rows64<23>(ctx, mode, a, st);
}
