// Row passes of one FP32 block-Lanczos step with local reorthogonalisation, block widths 6 and 23
// (paper: the three-term recurrence and block QR of the block-Lanczos paragraph after Eq. 4).  Each
// pass streams N x w Krylov blocks once and applies, per colour c, small b x b matrices and / or
// accumulates b x b Gram matrices:
//   S1  W0 = W - Q_{j-1} B_{j-1}^T (not stored);  Kq = Q_j^T W0,  Kp = Q_{j-1}^T W0
//   S3  W1 = W0 - Q_j Kq - Q_{j-1} Kp, over W (W0 recomputed: B_{j-1}^T + Kp in one FP32 matrix would
//       round Kp, the correction of B's own rounding, away);  Gram W1^T W1
//   T0  V = W1 R0^-1 (not stored);  Gram V^T V
//   T1  Q_{j+1} = (W1 R0^-1) R1^-1;  when some colour needs a third CholeskyQR pass also over W, with
//       its Gram
//   T2  Q_{j+1} = W R2^-1 for those colours
// S1 and T0 store nothing: W0 and V are recomputed by the next pass, with the same FMAs, which costs
// less than a pass over memory.  A step moves ten N x w blocks instead of twelve.
//
// The rows of a group of colours (a multiple of 16 bytes in every row) arrive in a ring of tiles filled
// by one or two producer warps with 16-byte cp.async copies; the same warps write finished tiles back.
// mbarriers with bounded waits connect them to the other warps.  (One bulk copy per row segment of
// ~300 bytes instead took ~62 clocks of an SM each whatever its size, 1.3 TB/s in all.)
#include <algorithm>

#include "css_lanczos.cuh"
#include "css_pipe.cuh"

namespace {

using namespace css_pipe;

enum { R_S1 = 0, R_S3 = 1, R_T0 = 2, R_T1 = 3, R_T2 = 4 };

struct RowsArgs {
  int64_t N;
  int32_t rchk, ws, ncb, cb0, G, first;
  const float* Q;        // Q_j        (S1, S3)
  const float* Qp;       // Q_{j-1}    (S1, S3; unused when first)
  const float* W;        // W or W1
  float* out;            // S3: W; T1, T2: Q_{j+1}
  float* out2;           // T1: W, when a colour of the group needs the third pass
  const double* M1;      // S3: Kq [lc]; T0, T1: R0^-1 [lc]; T2: R2^-1 [lc]
  const double* M2;      // S3: Kp [lc]; T1: R1^-1 [lc]
  const double* Bprev;   // S1, S3: B_{j-1} [cb0 + lc]
  const int32_t* need3;  // T1, T2
  double* part1;         // Gram partials [chunk][lc][b][b]
  double* part2;         // S1: Kp
  int* err;
  int32_t hold;          // tests: arrivals that a stage waits for beyond those it gets
};

__device__ __forceinline__ unsigned long long pack2(float x, float y) {
  unsigned long long r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ unsigned long long dup2(float x) { return pack2(x, x); }
__device__ __forceinline__ float lo2(unsigned long long v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float hi2(unsigned long long v) { return __uint_as_float((unsigned)(v >> 32)); }
// two IEEE FMAs, element by element
__device__ __forceinline__ void fma2(unsigned long long& c, unsigned long long a, unsigned long long b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}
// hi + lo += x (Knuth's TwoSum: the error of the sum goes to lo)
__device__ __forceinline__ void add_comp(float& hi, float& lo, float x) {
  const float t = __fadd_rn(hi, x), z = __fsub_rn(t, hi);
  lo = __fadd_rn(lo, __fadd_rn(__fsub_rn(hi, __fsub_rn(t, z)), __fsub_rn(x, z)));
  hi = t;
}
__device__ __forceinline__ void copy16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(su32(dst)), "l"(src) : "memory");
}
// this thread's arrival on b once all its copies so far have landed
__device__ __forceinline__ void arrive_copies(uint64_t* b) {
  asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(su32(b)) : "memory");
}
// words of a staged row: the group's columns, rounded so that consecutive rows are an odd number of
// 16-byte units apart (lane-per-row accesses of 16 bytes hit distinct banks)
__host__ __device__ constexpr int row_pitch(int cols) { return 4 * (((cols + 3) / 4) | 1); }

// A CTA's tiles: ns stages of NA arrays of R rows, "full" barriers (the producers' copies) and "done"
// barriers (the consumers' arrivals); NP producer warps.
template <int NA, int R, int NP>
struct Ring {
  float* base;
  uint64_t *full, *done;
  volatile int* abort;
  int* err;
  int32_t ns, pitch, ntile;
  int64_t r0, rend;
  __device__ __forceinline__ float* stage(int32_t t) const { return base + (size_t)(t % ns) * NA * R * pitch; }
  __device__ __forceinline__ int32_t rows(int32_t t) const { return (int32_t)min((int64_t)R, rend - r0 - (int64_t)t * R); }
  // for a whole warp: whether a wait gave up is one decision of its lanes, which leave the tile loop together
  __device__ __forceinline__ bool wait_full(int32_t t) const {
    return __all_sync(0xffffffffu, bar_wait(&full[t % ns], (t / ns) & 1, abort, err));
  }
  __device__ __forceinline__ void arrive(int32_t t) const { bar_arrive(&done[t % ns]); }
  __device__ __forceinline__ void init(int32_t consumers) const {  // one thread
    for (int s = 0; s < ns; ++s) {
      bar_init(&full[s], 32 * NP);
      bar_init(&done[s], consumers);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // producer warp pw: its part of every tile as the stages become free and, with OUT, of the stores of
  // the tile's array 0 to out (and out2) once the consumers are done with it.  cpr: 16-byte chunks of a
  // row's columns, which start at col0
  template <bool OUT>
  __device__ void produce(int pw, const float* const* src, int na, float* out, float* out2, int32_t ws, int32_t col0,
                          int32_t cpr) const {
    // a thread keeps its chunk of the row and walks down the rows, rp at a time, so that a copy is two
    // pointer steps (dividing a running index took ~110 clocks of the warp per copy)
    const int tid = pw * 32 + (threadIdx.x & 31), rp = 32 * NP / cpr;
    const int32_t rb = tid / cpr, c = tid - rb * cpr;
    const bool mine = rb < rp;
    const size_t go = (size_t)rb * ws + col0 + 4 * c, gs = (size_t)rp * ws;
    const int32_t so = rb * pitch + 4 * c, ss = rp * pitch;
    auto load = [&](int32_t t) {
      float* st = stage(t) + so;
      const size_t g = (size_t)(r0 + (int64_t)t * R) * ws + go;
      const int32_t nr = mine ? rows(t) : 0;
      for (int a = 0; a < na; ++a) {
        const float* s = src[a] + g;
        float* d = st + (size_t)a * R * pitch;
#pragma unroll 4
        for (int32_t r = rb; r < nr; r += rp, s += gs, d += ss) copy16(d, s);
      }
      arrive_copies(&full[t % ns]);
    };
    for (int32_t t = 0; t < ns && t < ntile; ++t) load(t);
    for (int32_t t = 0; t < ntile; ++t) {
      if (!OUT && t + ns >= ntile) break;
      const bool ok = bar_wait(&done[t % ns], (t / ns) & 1, abort, err);
      if (!__all_sync(0xffffffffu, ok)) break;
      if (OUT) {
        const float* d = stage(t) + so;
        float* o = out + ((size_t)(r0 + (int64_t)t * R) * ws + go);
        const ptrdiff_t o2 = out2 ? out2 - out : 0;
        const int32_t nr = mine ? rows(t) : 0;
#pragma unroll 4
        for (int32_t r = rb; r < nr; r += rp, o += gs, d += ss) {
          const float4 v = *reinterpret_cast<const float4*>(d);
          *reinterpret_cast<float4*>(o) = v;
          if (o2) *reinterpret_cast<float4*>(o + o2) = v;
        }
      }
      if (t + ns < ntile) load(t + ns);  // each thread refills the chunks that it stored
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
};

// ------------------------------------------------------------------------- b = 6
// One warp per colour, two rows of a tile per lane: the matrices of the colour and its Gram accumulators live in
// registers and a row's six values are three 8-byte shared loads, so 32 rows of a colour cost a warp
// ~100 packed FMAs and 9 shared loads in S1.  A lane sums 32 rows in FP32, then the 32 lanes' sums are
// added into one hi + lo pair per entry with TwoSum, widened to FP64 once per CTA.  The general tiled
// kernels (css_lanczos.cu) moved each value through 4-byte copies, staged tiles and barriers: row work
// of a step 5.33 -> 1.91 ms at 60,000 molecules (S1 339 us, S3 463, T0 125, T1 249: 4.6-5.0 TB/s of what
// each must move), 0.40 -> 0.145 at 4,001, 0.144 -> 0.067 at 512.  What it took: two rows per lane (one
// row left the waits and shared-memory latency of a tile exposed: 2.36 ms), ten colours so that a lane
// has 168 registers (twelve spilled in S1 and S3: 2.22 ms).
constexpr int B6_R = 64;      // rows per tile, two per lane
constexpr int B6_NP = 2;      // producer warps
constexpr int B6_GMAX = 10;   // colours (warps) per CTA, an even number: 16-byte columns
template <int MODE>
struct B6Cfg {
  static constexpr int NA = MODE <= R_S3 ? 3 : 1;
  static constexpr int NS = MODE <= R_S3 ? 4 : 8;
  static size_t smem(int G) {
    return (size_t)NS * NA * B6_R * row_pitch(6 * G) * 4 + (size_t)G * 18 * 33 * 4 + (2 * NS + 2) * 8;
  }
};

// index of the pair {(k, 2 i), (k, 2 i + 1)} of a symmetric 6 x 6 matrix kept for 2 i + 1 >= k
__host__ __device__ constexpr int sym_pair(int k, int i) {
  return (k >> 1 == 0 ? 3 * k : k >> 1 == 1 ? 6 + 2 * (k - 2) : 10 + (k - 4)) + i - (k >> 1);
}

template <int MODE>
__global__ void __launch_bounds__(32 * (B6_GMAX + B6_NP), 1) k_rows6(const RowsArgs a) {
  using C = B6Cfg<MODE>;
  constexpr int NA = C::NA, NS = C::NS, R = B6_R;
  constexpr bool OUT = MODE == R_S3 || MODE == R_T1 || MODE == R_T2;
  constexpr bool SYM = MODE != R_S1;
  extern __shared__ __align__(128) unsigned char rows_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t g0 = blockIdx.y * a.G, gcount = min(a.G, a.ncb - g0);
  Ring<NA, R, B6_NP> ring;
  ring.full = reinterpret_cast<uint64_t*>(rows_smem);
  ring.done = ring.full + NS;
  ring.abort = reinterpret_cast<volatile int*>(ring.done + NS);
  ring.base = reinterpret_cast<float*>(rows_smem + (2 * NS + 2) * 8);
  ring.err = a.err;
  ring.ns = NS;
  ring.pitch = row_pitch(6 * a.G);
  ring.r0 = (int64_t)blockIdx.x * a.rchk;
  ring.rend = min(a.N, ring.r0 + a.rchk);
  ring.ntile = (int32_t)((ring.rend - ring.r0 + R - 1) / R);
  bool any3 = false;
  if (MODE >= R_T1)
    for (int32_t g = 0; g < gcount; ++g) any3 = any3 || a.need3[g0 + g] != 0;
  if (MODE == R_T2 && !any3) return;  // uniform over the CTA
  if (threadIdx.x == 0) {
    ring.init(gcount + a.hold);
    *ring.abort = *(volatile int*)a.err ? 1 : 0;
  }
  __syncthreads();
  if (*ring.abort) return;
  const int32_t lc = g0 + warp;
  const bool use_p = MODE <= R_S3 && !a.first;
  constexpr int NACC = MODE == R_S1 ? 36 : 12;
  unsigned long long acc[NACC];
#pragma unroll
  for (int i = 0; i < NACC; ++i) acc[i] = 0ull;
  if (warp >= a.G) {  // producers
    const float* src[3] = {a.W, a.Q, a.Qp};
    ring.template produce<OUT>(warp - a.G, src, MODE <= R_S3 ? (use_p ? 3 : 2) : 1, a.out,
                               MODE == R_T1 && any3 ? a.out2 : nullptr, a.ws, g0 * 6, (gcount * 24 + 15) / 16);
  } else if (warp < gcount) {
    // the colour's matrices, negated where they are subtracted, as pairs over the output column
    constexpr int NM1 = MODE == R_S1 ? 1 : MODE == R_S3 ? 18 : 12, NM2 = MODE == R_S3 ? 18 : MODE == R_T1 ? 12 : 1;
    unsigned long long m1[NM1], m2[NM2], mb[MODE <= R_S3 ? 12 : 1];
    const double* M1 = MODE == R_S1 ? nullptr : a.M1 + (size_t)lc * 36;
    const double* M2 = (MODE == R_S3 || MODE == R_T1) ? a.M2 + (size_t)lc * 36 : nullptr;
    const double* Bp = MODE <= R_S3 ? a.Bprev + (size_t)(a.cb0 + lc) * 36 : nullptr;
    int n1 = 0, n2 = 0, nb = 0;
#pragma unroll
    for (int l = 0; l < 6; ++l)
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        const int k = 2 * i;
        if (MODE <= R_S3 && k <= l)  // -B^T: entries (l, k) with k <= l
          mb[nb++] = use_p ? pack2(-(float)Bp[k * 6 + l], k + 1 <= l ? -(float)Bp[(k + 1) * 6 + l] : 0.0f) : 0ull;
        if (MODE == R_S1) continue;
        if (MODE == R_S3) {
          m1[n1++] = pack2(-(float)M1[l * 6 + k], -(float)M1[l * 6 + k + 1]);
          m2[n2++] = use_p ? pack2(-(float)M2[l * 6 + k], -(float)M2[l * 6 + k + 1]) : 0ull;
        } else if (k + 1 >= l) {  // upper triangle
          m1[n1++] = pack2((float)M1[l * 6 + k], (float)M1[l * 6 + k + 1]);
          if (MODE == R_T1) m2[n2++] = pack2((float)M2[l * 6 + k], (float)M2[l * 6 + k + 1]);
        }
      }
    // y = x R^-1 over the upper triangle
    auto tri = [&](const unsigned long long (&x)[3], const unsigned long long* mm, unsigned long long (&y)[3]) {
#pragma unroll
      for (int i = 0; i < 3; ++i) y[i] = 0ull;
      int n = 0;
#pragma unroll
      for (int l = 0; l < 6; ++l) {
        const unsigned long long xl = dup2(l & 1 ? hi2(x[l >> 1]) : lo2(x[l >> 1]));
#pragma unroll
        for (int i = 0; i < 3; ++i)
          if (2 * i + 1 >= l) fma2(y[i], xl, mm[n++]);
      }
    };
    const bool n3 = MODE >= R_T1 && a.need3[lc] != 0;
    const bool gram = MODE <= R_T0 || (MODE == R_T1 && n3);
    // the lanes' sums into the entries' hi + lo pairs, rows 3 h .. 3 h + 2 of the Gram at a time: lane e
    // adds entry e of those 18 over all lanes
    float* red = ring.base + (size_t)NS * NA * R * ring.pitch + (size_t)warp * 18 * 33;
    float hi[2][2] = {}, lo[2][2] = {};
    auto flush = [&]() {
#pragma unroll
      for (int g = 0; g < (MODE == R_S1 ? 2 : 1); ++g)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          __syncwarp();
#pragma unroll
          for (int k = 3 * h; k < 3 * h + 3; ++k)
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              if (SYM && 2 * i + 1 < k) continue;
              unsigned long long& v = acc[(SYM ? sym_pair(k, i) : g * 18 + 3 * k + i) % NACC];
              red[(6 * (k - 3 * h) + 2 * i) * 33 + lane] = lo2(v);
              red[(6 * (k - 3 * h) + 2 * i + 1) * 33 + lane] = hi2(v);
              v = 0ull;
            }
          __syncwarp();
          if (lane < 18 && (!SYM || lane % 6 >= 3 * h + lane / 6)) {
#pragma unroll 8
            for (int i = 0; i < 32; ++i) add_comp(hi[g][h], lo[g][h], red[lane * 33 + i]);
          }
        }
    };
    const bool pad = OUT && warp + 1 == gcount && (gcount & 1);  // two columns past the last colour
    for (int32_t t = 0; t < ring.ntile; ++t) {
      if (!ring.wait_full(t)) break;
      const int32_t nr = ring.rows(t);
      float* row0 = ring.stage(t) + (size_t)lane * ring.pitch + 6 * warp;
      unsigned long long w2[2][3], q2[2][3], p2[2][3];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const bool valid = lane + 32 * h < nr;
        const float* row = row0 + h * 32 * ring.pitch;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          w2[h][i] = valid ? *reinterpret_cast<const unsigned long long*>(row + 2 * i) : 0ull;
          if (MODE <= R_S3) {
            q2[h][i] = valid ? *reinterpret_cast<const unsigned long long*>(row + R * ring.pitch + 2 * i) : 0ull;
            p2[h][i] = valid && use_p ? *reinterpret_cast<const unsigned long long*>(row + 2 * R * ring.pitch + 2 * i) : 0ull;
          }
        }
      }
      if (!OUT) {  // the tile is in registers: its stage is free
        __syncwarp();
        if (lane == 0) ring.arrive(t);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        unsigned long long(&w)[3] = w2[h], (&q)[3] = q2[h], (&p)[3] = p2[h], o[3];
        float* row = row0 + h * 32 * ring.pitch;
        if (MODE <= R_S3) {  // W0 = W - Q_{j-1} B^T
          int n = 0;
#pragma unroll
          for (int l = 0; l < 6; ++l) {
            const unsigned long long x = dup2(l & 1 ? hi2(p[l >> 1]) : lo2(p[l >> 1]));
#pragma unroll
            for (int i = 0; i < 3; ++i)
              if (2 * i <= l) fma2(w[i], x, mb[n++]);
          }
        }
        if (MODE == R_S1) {
#pragma unroll
          for (int k = 0; k < 6; ++k) {
            const unsigned long long xq = dup2(k & 1 ? hi2(q[k >> 1]) : lo2(q[k >> 1]));
            const unsigned long long xp = dup2(k & 1 ? hi2(p[k >> 1]) : lo2(p[k >> 1]));
#pragma unroll
            for (int i = 0; i < 3; ++i) {
              fma2(acc[(3 * k + i) % NACC], xq, w[i]);
              fma2(acc[(18 + 3 * k + i) % NACC], xp, w[i]);
            }
          }
        } else {
          if (MODE == R_S3) {
#pragma unroll
            for (int i = 0; i < 3; ++i) o[i] = w[i];
#pragma unroll
            for (int l = 0; l < 6; ++l) {
              const unsigned long long x = dup2(l & 1 ? hi2(q[l >> 1]) : lo2(q[l >> 1]));
#pragma unroll
              for (int i = 0; i < 3; ++i) fma2(o[i], x, m1[(3 * l + i) % NM1]);
            }
#pragma unroll
            for (int l = 0; l < 6; ++l) {
              const unsigned long long x = dup2(l & 1 ? hi2(p[l >> 1]) : lo2(p[l >> 1]));
#pragma unroll
              for (int i = 0; i < 3; ++i) fma2(o[i], x, m2[(3 * l + i) % NM2]);
            }
          } else {
            tri(w, m1, o);
            if (MODE == R_T1) {
              unsigned long long v[3];
#pragma unroll
              for (int i = 0; i < 3; ++i) v[i] = o[i];
              tri(v, m2, o);
            }
          }
          if (OUT) {
            if (MODE != R_T2 || n3)
#pragma unroll
              for (int i = 0; i < 3; ++i) *reinterpret_cast<unsigned long long*>(row + 2 * i) = o[i];
            if (pad) *reinterpret_cast<unsigned long long*>(row + 6) = 0ull;
            if (h == 1) {
              __syncwarp();
              if (lane == 0) ring.arrive(t);
            }
          }
          if (gram) {
#pragma unroll
            for (int k = 0; k < 6; ++k) {
              const unsigned long long x = dup2(k & 1 ? hi2(o[k >> 1]) : lo2(o[k >> 1]));
#pragma unroll
              for (int i = k >> 1; i < 3; ++i) fma2(acc[sym_pair(k, i) % NACC], x, o[i]);
            }
          }
        }
      }
      if (gram && ((t & 15) == 15 || t + 1 == ring.ntile)) flush();
    }
    if (!gram || *ring.abort || lane >= 18) return;
#pragma unroll
    for (int g = 0; g < (MODE == R_S1 ? 2 : 1); ++g) {
      double* part = (g ? a.part2 : a.part1) + ((size_t)blockIdx.x * a.ncb + lc) * 36;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int k = 3 * h + lane / 6, l = lane % 6;
        const double v = (double)hi[g][h] + (double)lo[g][h];
        if (SYM && l < k) continue;
        part[6 * k + l] = v;
        if (SYM && l > k) part[6 * l + k] = v;
      }
    }
  }
}

// ------------------------------------------------------------------------ b = 23
// Four colours (92 columns: whole 16-byte chunks) and tiles of 64 rows per CTA (S1: 32).  Warps have roles, and
// the products of a tile run beside the Grams of the one before it, with one barrier per tile:
//   products: a warp takes one colour, two rows per lane (S1: two colours, a row per lane).  A row's 23
//     values come from the ring by 16-byte loads (a colour starts at one of four offsets within a chunk:
//     four forms of the load, one of the arithmetic), the matrices by broadcast loads shared by 64 rows, an
//     output pair per packed FMA; triangular matrices skip their zero half.  Results go back to the ring for
//     the store and, 24 columns per colour, to one of two copies for the Gram.
//   Grams: a thread owns an 8 x 8 block of a colour's 24 x 24 and every 8th row (S1: the blocks of Kq
//     and of Kp together), four or six 16-byte loads for 32 or 64 packed FMAs.  After 32 rows the eight
//     lanes of a block add their sums by halves (each keeps one row of the block) into hi + lo pairs.
// Bound by the return path of shared memory (a 16-byte load is 512 bytes to a warp, broadcast or not) and the
// latency of a product's loads; HBM is at 2 to 3.3 TB/s.  The roles are separate loops, so that the Gram sums are
// not live across the products: in one loop the products spilled and a step took 0.97 ms at 1,000 molecules
// instead of 0.65.  Row work of a step at 10,000 molecules: tiled kernels 9.34 ms, both phases on the same
// warps between two barriers 6.71, now 5.35; at 1,000 1.08, 0.81, 0.65 (S1 191 us, S3 220, T0 70, T1 87).  Slower
// there: four lanes per Gram block with more producer warps 0.67, or with a row per lane on eight product
// warps 0.74; S3 in tiles of 32 rows 0.66.
constexpr int B23_G = 4, B23_GP = 100;  // colours per CTA, pitch of the Gram copies
template <int MODE>
struct B23Cfg {
  static constexpr int R = MODE == R_S1 ? 32 : 64;      // rows per tile
  static constexpr int NA = MODE <= R_S3 ? 3 : 1;
  static constexpr int NS = MODE == R_S3 ? 2 : 4;
  // twelve warps (168 registers a lane): products, Grams, producers
  static constexpr int S = 8;                           // lanes that share a Gram block
  static constexpr int PW = MODE == R_S1 ? 2 : 4, GW = (MODE == R_S1 ? 36 : 24) * S / 32, NP = 12 - PW - GW;
  static constexpr int RPL = R / 32;                    // rows per lane of a product
  static constexpr int NM = MODE == R_S3 ? 3 : MODE == R_T1 ? 2 : 1;  // matrices per colour
  static constexpr int NG = MODE == R_S1 ? 3 : MODE == R_T2 ? 0 : 1;  // Gram copies
  static constexpr size_t smem = (size_t)NS * NA * R * row_pitch(92) * 4 + (size_t)2 * NG * R * B23_GP * 4 +
                                 (size_t)NM * B23_G * 23 * 24 * 4 + (2 * NS + 2) * 8;
};

// the 23 values at chunk + O floats of a staged row, zero past them
template <int O>
__device__ __forceinline__ void load_row(const float* chunk, float (&x)[24]) {
  constexpr int NC = (O + 23 + 3) / 4;
  float4 v[NC];
#pragma unroll
  for (int i = 0; i < NC; ++i) v[i] = *reinterpret_cast<const float4*>(chunk + 4 * i);
#pragma unroll
  for (int i = 0; i < 23; ++i) {
    const float4 q = v[(i + O) / 4];
    x[i] = (i + O) % 4 == 0 ? q.x : (i + O) % 4 == 1 ? q.y : (i + O) % 4 == 2 ? q.z : q.w;
  }
  x[23] = 0.0f;
}
template <int O>
__device__ __forceinline__ void store_row(float* chunk, const unsigned long long (&o)[12]) {
  auto at = [&](int i) { return i & 1 ? hi2(o[i >> 1]) : lo2(o[i >> 1]); };
#pragma unroll
  for (int i = 0; i < 23; ++i) {
    constexpr int first = (4 - O) % 4;  // first value on a chunk boundary
    if (i >= first && (i - first) % 4 == 0 && i + 3 < 23)
      *reinterpret_cast<float4*>(chunk + O + i) = make_float4(at(i), at(i + 1), at(i + 2), at(i + 3));
    else if (i < first || i >= first + (23 - first) / 4 * 4)
      chunk[O + i] = at(i);
  }
}
__device__ __forceinline__ void load_row_of(int c, const float* row, float (&x)[24]) {  // colour c starts at 23 c
  if (c == 0) load_row<0>(row, x);
  else if (c == 1) load_row<3>(row + 20, x);
  else if (c == 2) load_row<2>(row + 44, x);
  else load_row<1>(row + 68, x);
}
__device__ __forceinline__ void store_row_of(int c, float* row, const unsigned long long (&o)[12]) {
  if (c == 0) store_row<0>(row, o);
  else if (c == 1) store_row<3>(row + 20, o);
  else if (c == 2) store_row<2>(row + 44, o);
  else store_row<1>(row + 68, o);
}
// o += x M for N rows, M [23][24] in shared memory; TRI 1: M(l, k) = 0 for k > l, TRI 2: for k < l
template <int TRI, int N>
__device__ __forceinline__ void mul_rows(unsigned long long (&o)[N][12], const float (&x)[N][24], const float* M) {
#pragma unroll
  for (int l = 0; l < 23; ++l) {
    unsigned long long xx[N];
#pragma unroll
    for (int n = 0; n < N; ++n) xx[n] = dup2(x[n][l]);
#pragma unroll
    for (int c = 0; c < 6; ++c) {
      if ((TRI == 1 && 4 * c > l) || (TRI == 2 && 4 * c + 3 < l)) continue;
      const ulonglong2 m = *reinterpret_cast<const ulonglong2*>(M + 24 * l + 4 * c);
#pragma unroll
      for (int n = 0; n < N; ++n) {
        fma2(o[n][2 * c], xx[n], m.x);
        fma2(o[n][2 * c + 1], xx[n], m.y);
      }
    }
  }
}

// The sums of an 8 x 8 block (32 pairs, row k in pairs 4 k .. 4 k + 3) over the S lanes that share it:
// each step the lanes of a pair keep one half of what is left and give away the other.  Lane s of the
// S ends with pairs 32 / S * rev(s) .. of the block, added into its hi + lo pairs; v is cleared.
template <int S>
__device__ __forceinline__ void block_flush(unsigned long long (&v)[32], float (&hi)[64 / S], float (&lo)[64 / S]) {
  const int lane = threadIdx.x & 31;
  int n = 16;
#pragma unroll
  for (int o = S / 2; o > 0; o >>= 1, n >>= 1) {
    const bool up = lane & o;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      if (i >= n) continue;
      const unsigned long long keep = up ? v[i + n] : v[i], give = up ? v[i] : v[i + n];
      const unsigned long long got = __shfl_xor_sync(0xffffffffu, give, o);
      asm("add.rn.f32x2 %0, %1, %2;" : "=l"(v[i]) : "l"(keep), "l"(got));
    }
  }
#pragma unroll
  for (int i = 0; i < 32 / S; ++i) {
    add_comp(hi[2 * i], lo[2 * i], lo2(v[i]));
    add_comp(hi[2 * i + 1], lo[2 * i + 1], hi2(v[i]));
  }
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = 0ull;
}

template <int MODE>
__global__ void __launch_bounds__(32 * 12, 1) k_rows23(const RowsArgs a) {
  using C = B23Cfg<MODE>;
  constexpr int NA = C::NA, NS = C::NS, R = C::R, RPL = C::RPL, CT = 32 * (C::PW + C::GW), MM = 23 * 24;
  constexpr int GB = C::NG * R * B23_GP;  // values of one buffer of Gram copies
  constexpr bool OUT = MODE == R_S3 || MODE == R_T1 || MODE == R_T2;
  extern __shared__ __align__(128) unsigned char rows_smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int32_t g0 = blockIdx.y * B23_G, gcount = min(B23_G, a.ncb - g0);
  Ring<NA, R, C::NP> ring;
  ring.full = reinterpret_cast<uint64_t*>(rows_smem);
  ring.done = ring.full + NS;
  ring.abort = reinterpret_cast<volatile int*>(ring.done + NS);
  ring.base = reinterpret_cast<float*>(rows_smem + (2 * NS + 2) * 8);
  ring.err = a.err;
  ring.ns = NS;
  ring.pitch = row_pitch(92);
  ring.r0 = (int64_t)blockIdx.x * a.rchk;
  ring.rend = min(a.N, ring.r0 + a.rchk);
  ring.ntile = (int32_t)((ring.rend - ring.r0 + R - 1) / R);
  float* sG = ring.base + (size_t)NS * NA * R * ring.pitch;  // Gram copies [tile & 1][array][row][24 c + k]
  float* sM = sG + (size_t)2 * GB;                           // matrices [matrix][colour][l][k]
  bool any3 = false;
  if (MODE >= R_T1)
    for (int32_t g = 0; g < gcount; ++g) any3 = any3 || a.need3[g0 + g] != 0;
  if (MODE == R_T2 && !any3) return;  // uniform over the CTA
  const bool use_p = MODE <= R_S3 && !a.first;
  const bool gram = MODE <= R_T0 || (MODE == R_T1 && any3);
  if (threadIdx.x == 0) {
    ring.init(1 + a.hold);
    *ring.abort = *(volatile int*)a.err ? 1 : 0;
  }
  // the colours' matrices (negated where they are subtracted)
  for (int32_t e = threadIdx.x; e < B23_G * MM; e += blockDim.x) {
    const int32_t g = e / MM, rem = e - g * MM, l = rem / 24, k = rem - 24 * l;
    const bool in = g < gcount && k < 23;
    const size_t o = (size_t)(g0 + (in ? g : 0)) * 529;
    if (MODE <= R_S3)  // -B^T
      sM[e] = in && use_p && k <= l ? -(float)a.Bprev[(size_t)(a.cb0 + g0 + g) * 529 + k * 23 + l] : 0.0f;
    if (MODE == R_S3) {
      sM[B23_G * MM + e] = in ? -(float)a.M1[o + l * 23 + k] : 0.0f;
      sM[2 * B23_G * MM + e] = in && use_p ? -(float)a.M2[o + l * 23 + k] : 0.0f;
    }
    if (MODE >= R_T0) sM[e] = in ? (float)a.M1[o + l * 23 + k] : 0.0f;
    if (MODE == R_T1) sM[B23_G * MM + e] = in ? (float)a.M2[o + l * 23 + k] : 0.0f;
  }
  // rows past the end of the last tile and columns past the last colour stay zero in the Gram copies
  for (int32_t e = threadIdx.x; e < 2 * GB; e += blockDim.x) sG[e] = 0.0f;
  __syncthreads();
  if (*ring.abort) return;
  if (warp >= C::PW + C::GW) {
    const float* src[3] = {a.W, a.Q, a.Qp};
    ring.template produce<OUT>(warp - C::PW - C::GW, src, MODE <= R_S3 ? (use_p ? 3 : 2) : 1, a.out,
                               MODE == R_T1 && any3 ? a.out2 : nullptr, a.ws, g0 * 23, (gcount * 23 + 3) / 4);
    return;
  }
  auto sync = [] { asm volatile("bar.sync 1, %0;" ::"n"(CT) : "memory"); };
  auto product = [&](int32_t t, int pc) {
    const bool n3 = MODE >= R_T1 && a.need3[g0 + pc] != 0;
    float* st = ring.stage(t);
    const int nr = ring.rows(t);
    float* row[RPL];
    float* grow = sG + (size_t)(t & 1) * GB + (size_t)lane * B23_GP + 24 * pc;
    float x[RPL][24];
    unsigned long long o[RPL][12];
#pragma unroll
    for (int h = 0; h < RPL; ++h) row[h] = st + (size_t)(lane + 32 * h) * ring.pitch;
    auto load = [&](int array) {  // rows past the end as zeros
#pragma unroll
      for (int h = 0; h < RPL; ++h) {
        load_row_of(pc, row[h] + (size_t)array * R * ring.pitch, x[h]);
        if (lane + 32 * h >= nr)
#pragma unroll
          for (int i = 0; i < 24; ++i) x[h][i] = 0.0f;
      }
    };
    auto to_gram = [&](int array, auto val) {
#pragma unroll
      for (int h = 0; h < RPL; ++h)
#pragma unroll
        for (int i = 0; i < 6; ++i)
          *reinterpret_cast<ulonglong2*>(grow + ((size_t)array * R + 32 * h) * B23_GP + 4 * i) =
              make_ulonglong2(val(h, 2 * i), val(h, 2 * i + 1));
    };
    auto as_x = [&](int h, int i) { return pack2(x[h][2 * i], x[h][2 * i + 1]); };
    auto as_o = [&](int h, int i) { return o[h][i]; };
    load(0);  // W
    if (MODE <= R_S3) {
#pragma unroll
      for (int h = 0; h < RPL; ++h)
#pragma unroll
        for (int i = 0; i < 12; ++i) o[h][i] = as_x(h, i);
      if (use_p) {
        load(2);  // Q_{j-1}
        mul_rows<1>(o, x, sM + pc * MM);
        if (MODE == R_S1) to_gram(2, as_x);
      }
      if (MODE == R_S1) to_gram(0, as_o);
      load(1);  // Q_j
      if (MODE == R_S1) {
        to_gram(1, as_x);
      } else {
        mul_rows<0>(o, x, sM + (B23_G + pc) * MM);
        if (use_p) {
          load(2);
          mul_rows<0>(o, x, sM + (2 * B23_G + pc) * MM);
        }
      }
    } else {
#pragma unroll
      for (int h = 0; h < RPL; ++h)
#pragma unroll
        for (int i = 0; i < 12; ++i) o[h][i] = 0ull;
      mul_rows<2>(o, x, sM + pc * MM);
      if (MODE == R_T1) {
#pragma unroll
        for (int h = 0; h < RPL; ++h)
#pragma unroll
          for (int i = 0; i < 12; ++i) {
            x[h][2 * i] = lo2(o[h][i]);
            x[h][2 * i + 1] = hi2(o[h][i]);
            o[h][i] = 0ull;
          }
        mul_rows<2>(o, x, sM + (B23_G + pc) * MM);
      }
    }
    if (OUT) {
#pragma unroll
      for (int h = 0; h < RPL; ++h) {
        if (MODE != R_T2 || n3) store_row_of(pc, row[h], o[h]);
        if (pc + 1 == gcount)
          for (int32_t i = 23 * gcount; i & 3; ++i) row[h][i] = 0.0f;  // columns past the last colour
      }
    }
    if (MODE != R_S1 && gram) to_gram(0, as_o);
  };
  // the products of tile t run beside the Grams of tile t - 1, one barrier a tile; a warp whose wait gives
  // up still runs every barrier, so that no other waits for it
  if (warp < C::PW) {
#pragma unroll 1
    for (int32_t t = 0; t <= ring.ntile; ++t) {
      if (t < ring.ntile && ring.wait_full(t))
#pragma unroll 1
        for (int pc = warp; pc < gcount; pc += C::PW) product(t, pc);
      sync();  // the Gram copies of tile t are in place, those of tile t - 1 free, the ring's stage is done with
      if (threadIdx.x == 0 && t < ring.ntile) ring.arrive(t);
    }
    return;
  }
  // Grams: this thread's block and rows
  constexpr int S = C::S;
  const int gt = (int)threadIdx.x - 32 * C::PW, gs = gt & (S - 1), blk = gt / S;
  const int gc = MODE == R_S1 ? blk / 9 : blk / 6, gb = MODE == R_S1 ? blk % 9 : blk % 6;
  const int kb = MODE == R_S1 ? gb / 3 : gb < 3 ? 0 : gb < 5 ? 1 : 2;
  const int lb = MODE == R_S1 ? gb % 3 : gb < 3 ? gb : gb < 5 ? gb - 2 : 2;
  unsigned long long vq[32], vp[MODE == R_S1 ? 32 : 1];
  float hq[64 / S] = {}, lq[64 / S] = {}, hp[MODE == R_S1 ? 8 : 1] = {}, lp[MODE == R_S1 ? 8 : 1] = {};
#pragma unroll
  for (int i = 0; i < 32; ++i) {
    vq[i] = 0ull;
    if (MODE == R_S1) vp[i % (MODE == R_S1 ? 32 : 1)] = 0ull;
  }
  auto sum_tile = [&](int32_t t) {
    const float* buf = sG + (size_t)(t & 1) * GB + (size_t)gs * B23_GP + 24 * gc;
    const float *y0 = buf + 8 * lb, *x0 = buf + 8 * kb + (MODE == R_S1 ? R * B23_GP : 0);
#pragma unroll(MODE == R_S1 ? 1 : 2)
    for (int i = 0; i < R / S; ++i, y0 += S * B23_GP, x0 += S * B23_GP) {
      const ulonglong2 ya = *reinterpret_cast<const ulonglong2*>(y0), yb = *reinterpret_cast<const ulonglong2*>(y0 + 4);
      auto rank1 = [&](const float* xr, unsigned long long* v) {
        const float4 xa = *reinterpret_cast<const float4*>(xr), xb = *reinterpret_cast<const float4*>(xr + 4);
        const float xv[8] = {xa.x, xa.y, xa.z, xa.w, xb.x, xb.y, xb.z, xb.w};
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const unsigned long long xx = dup2(xv[k]);
          fma2(v[4 * k], xx, ya.x);
          fma2(v[4 * k + 1], xx, ya.y);
          fma2(v[4 * k + 2], xx, yb.x);
          fma2(v[4 * k + 3], xx, yb.y);
        }
      };
      rank1(x0, vq);
      if constexpr (MODE == R_S1) rank1(x0 + R * B23_GP, vp);
    }
    constexpr int FL = 32 / (R / S);  // tiles of 32 rows per lane
    if (t % FL == FL - 1 || t + 1 == ring.ntile) {
      block_flush<S>(vq, hq, lq);
      if constexpr (MODE == R_S1) block_flush<S>(vp, hp, lp);
    }
  };
#pragma unroll 1
  for (int32_t t = 0; t <= ring.ntile; ++t) {
    if (t > 0 && gram) sum_tile(t - 1);
    sync();
  }
  if (!gram || *ring.abort || gc >= gcount) return;
  if (MODE == R_T1 && a.need3[g0 + gc] == 0) return;
  // the pairs block_flush left in this lane: p0, p0 + 1, ...
  int p0 = 0;
#pragma unroll
  for (int o = S / 2, n = 16; o > 0; o >>= 1, n >>= 1) p0 += gs & o ? n : 0;
#pragma unroll
  for (int gram2 = 0; gram2 < (MODE == R_S1 ? 2 : 1); ++gram2) {
    double* part = (gram2 ? a.part2 : a.part1) + ((size_t)blockIdx.x * a.ncb + g0 + gc) * 529;
#pragma unroll
    for (int i = 0; i < 64 / S; ++i) {
      const int k = 8 * kb + (p0 + i / 2) / 4, l = 8 * lb + 2 * ((p0 + i / 2) % 4) + (i & 1);
      const float h = gram2 ? hp[i % (MODE == R_S1 ? 8 : 1)] : hq[i], w = gram2 ? lp[i % (MODE == R_S1 ? 8 : 1)] : lq[i];
      if (k < 23 && l < 23) {
        const double v = (double)h + (double)w;
        part[k * 23 + l] = v;
        if (MODE != R_S1 && kb != lb) part[l * 23 + k] = v;
      }
    }
  }
}

// Rows per CTA: chunks for one to three waves of a CTA per SM over `groups` groups of colours (a full
// count: the chunk may not depend on the colours of the call, or a colour's sums would), more waves
// where a CTA still has `most` rows, so that its start and end (~5 us) stay small.
int32_t pick_chunk(int64_t N, int groups, int R, int32_t most) {
  const int64_t waves = std::min<int64_t>(3, std::max<int64_t>(1, N * groups / (152ll * most)));
  const int64_t nch = std::max<int64_t>(1, 152 * waves / groups);
  return (int32_t)std::max<int64_t>(css_ceil_div(css_ceil_div(N, nch), R) * R, R);
}

template <int MODE>
css_status launch_rows6(css_ctx* ctx, RowsArgs& r, cudaStream_t st) {
  const int32_t ngr = (int32_t)css_ceil_div(r.ncb, B6_GMAX);
  r.G = (int32_t)css_ceil_div(css_ceil_div(r.ncb, ngr), 2) * 2;  // even groups of nearly equal size
  const size_t sm = B6Cfg<MODE>::smem(r.G);
  CSS_TRY(css_smem_limit(ctx, k_rows6<MODE>, B6Cfg<MODE>::smem(B6_GMAX)));
  const dim3 grid((unsigned)css_ceil_div(r.N, r.rchk), (unsigned)css_ceil_div(r.ncb, r.G));
  k_rows6<MODE><<<grid, 32 * (r.G + B6_NP), sm, st>>>(r);
  CSS_LAUNCHED(ctx);
  return CSS_OK;
}

template <int MODE>
css_status launch_rows23(css_ctx* ctx, RowsArgs& r, cudaStream_t st) {
  using C = B23Cfg<MODE>;
  CSS_TRY(css_smem_limit(ctx, k_rows23<MODE>, C::smem));
  const dim3 grid((unsigned)css_ceil_div(r.N, r.rchk), (unsigned)css_ceil_div(r.ncb, B23_G));
  k_rows23<MODE><<<grid, 32 * 12, C::smem, st>>>(r);
  CSS_LAUNCHED(ctx);
  return CSS_OK;
}

template <int MODE>
css_status launch_rows(css_ctx* ctx, int32_t b, RowsArgs& r, cudaStream_t st) {
  return b == 6 ? launch_rows6<MODE>(ctx, r, st) : launch_rows23<MODE>(ctx, r, st);
}

}  // namespace

bool css_rows_supported(bool fp32, int32_t b) { return fp32 && (b == 6 || b == 23); }

int32_t css_rows_chunk(int64_t N, int32_t b) {
  return b == 6 ? pick_chunk(N, 7, B6_R, 2048) : pick_chunk(N, 17, 64, 2048);
}

css_status css_rows(css_ctx* ctx, int mode, const CssRows& p, cudaStream_t st) {
  RowsArgs r;
  r.N = p.N;
  r.rchk = css_rows_chunk(p.N, p.b);
  r.ws = p.ws;
  r.ncb = p.ncb;
  r.cb0 = p.cb0;
  r.G = 0;
  r.first = p.first;
  r.Q = p.Q;
  r.Qp = p.Qp;
  r.W = p.W;
  r.out = p.out;
  r.out2 = p.out2;
  r.M1 = p.M1;
  r.M2 = p.M2;
  r.Bprev = p.Bprev;
  r.need3 = p.need3;
  r.part1 = p.part1;
  r.part2 = p.part2;
  r.err = p.err;
  r.hold = ctx->test_rows_hold;
  switch (mode) {
    case R_S1: return launch_rows<R_S1>(ctx, p.b, r, st);
    case R_S3: return launch_rows<R_S3>(ctx, p.b, r, st);
    case R_T0: return launch_rows<R_T0>(ctx, p.b, r, st);
    case R_T1: return launch_rows<R_T1>(ctx, p.b, r, st);
    default: return launch_rows<R_T2>(ctx, p.b, r, st);
  }
}
