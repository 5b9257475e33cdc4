// Colour graph (cell list, exact int64 fixed-point distances), Jones-Plassmann colouring and
// CSS probe signs.  Paper: CSS construction paragraph after Eq. 2 (greedy multicolouring,
// Welsh-Powell order) and Fig. 1(b,c).
//
// Jones-Plassmann with the priority (degree desc, SplitMix64(seed, id) desc, id asc): a vertex
// is coloured once all of its higher-priority neighbours (its parents) are, with the smallest
// colour none of them uses.  That is exactly the sequential greedy colouring in priority order,
// whatever the order in which ready vertices are taken, so the result is bit-identical to it.
#include <algorithm>

#include "css_internal.cuh"
#include "css_pipe.cuh"

namespace {

constexpr int64_t kFix = 1048576;  // 2^20 per Angstrom

struct __align__(32) q4 {
  long long x, y, z, w;
};

// minimum image of the difference of two coordinates of [0, Lq): a select instead of a 64-bit
// remainder, which is tens of instructions
__device__ __forceinline__ int64_t min_image(int64_t d, int64_t Lq) {
  if (d > Lq / 2) d -= Lq;
  if (d < -(Lq / 2)) d += Lq;
  return d;
}

// u before v in the greedy order; the hashes are only taken between vertices of equal degree
__device__ __forceinline__ bool higher(uint64_t seed, int32_t du, int32_t u, int32_t dv, int32_t v) {
  if (du != dv) return du > dv;
  const uint64_t ku = css_splitmix64(seed, (uint64_t)u), kv = css_splitmix64(seed, (uint64_t)v);
  if (ku != kv) return ku > kv;
  return u < v;
}

// Fixed-point coordinates wrapped into [0, Lq)^3, and the cell of each molecule.
__global__ void k_quantise(int32_t n, const double* __restrict__ xyz, int64_t Lq, int32_t nc, q4* __restrict__ q,
                           int32_t* __restrict__ cell) {
  int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  int64_t w[3];
  for (int d = 0; d < 3; ++d) {
    w[d] = __double2ll_rn(xyz[3 * (int64_t)i + d] * (double)kFix) % Lq;
    if (w[d] < 0) w[d] += Lq;
  }
  q[i] = q4{w[0], w[1], w[2], 0};
  int32_t ci[3] = {0, 0, 0};
  if (nc >= 3)
    for (int d = 0; d < 3; ++d) {
      const int64_t t = (w[d] * nc) / Lq;
      ci[d] = (int32_t)(t >= nc ? nc - 1 : t);
    }
  cell[i] = (ci[0] * nc + ci[1]) * nc + ci[2];
}

__global__ void k_cell_count(int32_t n, const int32_t* __restrict__ cell, int32_t* __restrict__ cnt) {
  int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) atomicAdd(&cnt[cell[i]], 1);
}

__global__ void k_cell_fill(int32_t n, const int32_t* __restrict__ cell, const int32_t* __restrict__ start,
                            int32_t* __restrict__ fillpos, int32_t* __restrict__ members) {
  int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    int32_t c = cell[i];
    int32_t p = atomicAdd(&fillpos[c], 1);
    members[start[c] + p] = i;
  }
}

// Neighbours of every molecule, one warp each: the lanes test the candidates of the 27 cells
// around it (or of all molecules when the box holds fewer than 3 cells per edge) 32 at a time.
// Pass 0 counts them into deg; pass 1 writes those of higher priority (the parents, in any order)
// from adj_ptr[i] on and their number to np[i].  A thread per molecule left the chip idle below
// ~10^5 molecules (2.1 ms a pass at 4,001 molecules).
template <int PASS>
__global__ void k_neighbours(int32_t n, const q4* __restrict__ q, const int32_t* __restrict__ cell, int32_t nc,
                             const int32_t* __restrict__ cstart, const int32_t* __restrict__ members, int64_t Lq,
                             int64_t R2, uint64_t seed, int32_t* __restrict__ deg,
                             const int32_t* __restrict__ adj_ptr, int32_t* __restrict__ np, int32_t* __restrict__ adj) {
  const int32_t i = (int32_t)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (i >= n) return;  // whole warp
  const q4 qi = q[i];
  const int32_t di = PASS ? deg[i] : 0;
  int32_t count = 0;  // PASS 0: this lane's neighbours; PASS 1: parents written by the warp
  const int32_t out = PASS ? adj_ptr[i] : 0;
  // every lane of the warp calls this; j < 0: no candidate
  auto test = [&](int32_t j) {
    bool take = false;
    if (j >= 0 && j != i) {
      const q4 qj = q[j];
      const int64_t dx = min_image(qi.x - qj.x, Lq), dy = min_image(qi.y - qj.y, Lq), dz = min_image(qi.z - qj.z, Lq);
      take = dx * dx + dy * dy + dz * dz < R2;
    }
    if (!PASS) {
      count += take;
      return;
    }
    take = take && higher(seed, deg[j], j, di, i);
    const unsigned m = __ballot_sync(0xffffffffu, take);
    if (take) adj[out + count + __popc(m & ((1u << lane) - 1u))] = j;
    count += __popc(m);
  };
  if (nc < 3) {
    for (int32_t j = 0; j < n; j += 32) test(j + lane < n ? j + lane : -1);
  } else {
    const int32_t c = cell[i];
    const int32_t cx = c / (nc * nc), cy = (c / nc) % nc, cz = c % nc;
    for (int dx = -1; dx <= 1; ++dx)
      for (int dy = -1; dy <= 1; ++dy)
        for (int dz = -1; dz <= 1; ++dz) {
          const int32_t x = (cx + dx + nc) % nc, y = (cy + dy + nc) % nc, z = (cz + dz + nc) % nc;
          const int32_t cc = (x * nc + y) * nc + z;
          const int32_t e = cstart[cc + 1];
          for (int32_t k = cstart[cc]; k < e; k += 32) test(k + lane < e ? members[k + lane] : -1);
        }
  }
  if (!PASS) {
    for (int o = 16; o > 0; o >>= 1) count += __shfl_xor_sync(0xffffffffu, count, o);
    if (lane == 0) deg[i] = count;
  } else if (lane == 0) {
    np[i] = count;
  }
}

// ---------------------------------------------------------------- exclusive scan
__global__ void k_scan_block(const int32_t* __restrict__ in, int32_t* __restrict__ out, int64_t n,
                             int32_t* __restrict__ block_sums) {
  __shared__ int32_t s[1024];
  int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
  int32_t v = i < n ? in[i] : 0;
  s[threadIdx.x] = v;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    int32_t t = threadIdx.x >= off ? s[threadIdx.x - off] : 0;
    __syncthreads();
    s[threadIdx.x] += t;
    __syncthreads();
  }
  if (i < n) out[i] = s[threadIdx.x] - v;
  if (threadIdx.x == 1023 && block_sums) block_sums[blockIdx.x] = s[1023];
}

__global__ void k_scan_add(int32_t* __restrict__ out, int64_t n, const int32_t* __restrict__ offs) {
  int64_t i = (int64_t)blockIdx.x * 1024 + threadIdx.x;
  if (i < n) out[i] += offs[blockIdx.x];
}

}  // namespace

// exclusive scan of n int32 values into out[0..n) and out[n] = total (out has n+1 slots)
css_status css_scan_i32(css_ctx* ctx, const int32_t* in, int32_t* out, int64_t n, cudaStream_t st, int depth = 0) {
  if (n <= 0) {
    CSS_CU(ctx, cudaMemsetAsync(out, 0, sizeof(int32_t), st));
    return CSS_OK;
  }
  int64_t nb = css_ceil_div(n, 1024);
  if (nb == 1) {  // one block: its total is the grand total
    k_scan_block<<<1, 1024, 0, st>>>(in, out, n, out + n);
    CSS_LAUNCHED(ctx);
    return CSS_OK;
  }
  char name[32];
  snprintf(name, sizeof(name), "scan_sums_%d", depth);
  int32_t* sums = nullptr;
  CSS_TRY(css_ws(ctx, name, sizeof(int32_t) * (nb + 1), (void**)&sums));
  k_scan_block<<<(unsigned)nb, 1024, 0, st>>>(in, out, n, sums);
  CSS_LAUNCHED(ctx);
  char name2[32];
  snprintf(name2, sizeof(name2), "scan_offs_%d", depth);
  int32_t* offs = nullptr;
  CSS_TRY(css_ws(ctx, name2, sizeof(int32_t) * (nb + 1), (void**)&offs));
  CSS_TRY(css_scan_i32(ctx, sums, offs, nb, st, depth + 1));
  k_scan_add<<<(unsigned)nb, 1024, 0, st>>>(out, n, offs);
  CSS_LAUNCHED(ctx);
  // total = offs[nb]
  CSS_CU(ctx, cudaMemcpyAsync(out + n, offs + nb, sizeof(int32_t), cudaMemcpyDeviceToDevice, st));
  return CSS_OK;
}

namespace {

// ---------------------------------------------------------------- Jones-Plassmann
// Degrees of an explicit graph, and the parents of every vertex (one warp each) from adj_ptr[v]
// on with their number in np[v].
__global__ void k_degrees(int32_t n, const int32_t* __restrict__ adj_ptr, int32_t* __restrict__ deg) {
  const int32_t v = blockIdx.x * blockDim.x + threadIdx.x;
  if (v < n) deg[v] = adj_ptr[v + 1] - adj_ptr[v];
}
__global__ void k_parents(int32_t n, const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj,
                          uint64_t seed, const int32_t* __restrict__ deg, int32_t* __restrict__ np,
                          int32_t* __restrict__ padj) {
  const int32_t v = (int32_t)(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5);
  const int lane = threadIdx.x & 31;
  if (v >= n) return;
  const int32_t s = adj_ptr[v], e = adj_ptr[v + 1], dv = deg[v];
  int32_t count = 0;
  for (int32_t k = s; k < e; k += 32) {
    const int32_t u = k + lane < e ? adj[k + lane] : -1;
    const bool take = u >= 0 && higher(seed, deg[u], u, dv, v);
    const unsigned m = __ballot_sync(0xffffffffu, take);
    if (take) padj[s + count + __popc(m & ((1u << lane) - 1u))] = u;
    count += __popc(m);
  }
  if (lane == 0) np[v] = count;
}

// The whole colouring in one cooperative launch (all CTAs resident, so a vertex may wait for any
// other).  Warp w owns vertices [w per, w per + per); each lane watches one parent of its vertex
// that is not coloured yet (wait[v]: its index among v's parents).  When that parent has its
// colour, the warp looks at the vertex's remaining parents 32 at a time, moves the watch to the
// next uncoloured one, or, when there is none, takes the smallest colour none of the parents uses
// (256 colours at a time, the lanes' bit masks OR-reduced) and publishes it.  A colour is one
// word that never changes once set, so no ordering between words is needed.
// Bound by latency: one published colour seen by its dependants is ~1.5 us, and the longest chain
// of parents is a few hundred vertices.  With one launch per step of that chain, each scanning
// every vertex, a colouring of 20,000 molecules took 10.0 ms (445 launches); now 1.42 ms in all.
// Every wait is bounded: a warp that sees 4 s pass without any vertex of the graph being coloured
// (*done counts them) sets *err and leaves.  hold: a vertex that is never taken (tests), -1 for none.
constexpr uint64_t kColourNs = 4000000000ull;
__global__ void __launch_bounds__(256) k_jp_flow(int32_t n, int32_t per, const int32_t* __restrict__ adj_ptr,
                                                 const int32_t* __restrict__ np, const int32_t* __restrict__ padj,
                                                 int32_t* __restrict__ wait, volatile int32_t* colour,
                                                 int32_t* __restrict__ max_colour, int32_t* done,
                                                 int32_t* __restrict__ err, int32_t hold) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t v0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per;
  if (v0 >= n) return;
  const int32_t mine = (int32_t)(n - v0 < per ? n - v0 : per);
  int32_t left = mine, top = -1, seen = -1;
  uint64_t t0 = css_pipe::gtime();
  for (uint32_t sweep = 0; left > 0; ++sweep) {
    bool moved = false;
    for (int32_t g = 0; g < mine; g += 32) {
      const int32_t vl = (int32_t)v0 + g + lane;
      const bool own = g + lane < mine;
      int32_t wl = own ? wait[vl] : -1;  // -1: coloured
      const int32_t sl = own ? adj_ptr[vl] : 0, nl = own ? np[vl] : 0;
      const bool go = wl >= 0 && vl != hold && (wl >= nl || colour[padj[sl + wl]] >= 0);
      unsigned todo = __ballot_sync(FULL, go);
      moved = moved || todo != 0;
      while (todo) {
        const int src = __ffs(todo) - 1;
        todo &= todo - 1;
        const int32_t v = __shfl_sync(FULL, vl, src), s = __shfl_sync(FULL, sl, src), k = __shfl_sync(FULL, nl, src);
        int32_t w = __shfl_sync(FULL, wl, src);
        for (; w < k; w += 32) {
          const bool open = w + lane < k && colour[padj[s + w + lane]] < 0;
          const unsigned m = __ballot_sync(FULL, open);
          if (m) {
            w += __ffs(m) - 1;
            break;
          }
        }
        if (w >= k) {  // every parent has its colour
          int32_t c = -1;
          for (int32_t base = 0; c < 0; base += 256) {
            uint64_t used[4] = {0, 0, 0, 0};
            for (int32_t q = lane; q < k; q += 32) {
              const int32_t cu = colour[padj[s + q]] - base;
#pragma unroll
              for (int z = 0; z < 4; ++z)
                if (cu >= 64 * z && cu < 64 * (z + 1)) used[z] |= 1ull << (cu & 63);
            }
#pragma unroll
            for (int z = 0; z < 4; ++z) {
              for (int o = 16; o > 0; o >>= 1) used[z] |= __shfl_xor_sync(FULL, used[z], o);
              if (c < 0 && ~used[z]) c = base + 64 * z + __ffsll((long long)~used[z]) - 1;
            }
          }
          if (lane == 0) {
            colour[v] = c;
            atomicAdd(done, 1);
          }
          top = max(top, c);
          w = -1;
          --left;
        }
        if (lane == src) wait[v] = w;
        __syncwarp();
      }
    }
    if (!moved && (sweep & 255) == 255) {
      const int32_t now = __shfl_sync(FULL, *(volatile int32_t*)done, 0);
      const bool late = now == seen && css_pipe::gtime() - t0 > kColourNs;
      if (now != seen) {
        seen = now;
        t0 = css_pipe::gtime();
      }
      if (__any_sync(FULL, late)) {  // the lanes leave together: those that stayed would vote without the others
        if (lane == 0) atomicOr(err, 1);
        return;
      }
    }
  }
  if (lane == 0) atomicMax(max_colour, top);
}

// An explicit graph must have adj_ptr[0] = 0, non-decreasing adj_ptr and every neighbour in
// [0, n): vertex i checks its own row and sets *bad otherwise (its entries are then not read)
__global__ void k_graph_check(int32_t n, const int32_t* __restrict__ adj_ptr, const int32_t* __restrict__ adj,
                              int32_t* __restrict__ bad) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int32_t s = adj_ptr[i], e = adj_ptr[i + 1];
  if ((i == 0 && s != 0) || e < s) {
    atomicOr(bad, 1);
    return;
  }
  for (int32_t k = s; k < e; ++k) {
    const int32_t u = adj[k];
    if (u < 0 || u >= n) {
      atomicOr(bad, 1);
      return;
    }
  }
}

__global__ void k_probe_signs(int64_t count, uint64_t seed, int ones, int8_t* __restrict__ sign) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= count) return;
  sign[i] = ones ? (int8_t)1 : ((css_splitmix64(seed, (uint64_t)i) & 1ull) ? (int8_t)-1 : (int8_t)1);
}

// Molecule centres in fixed point, binned into a periodic grid of cells at least r_col wide
// (any coarser grid is also correct), the members of a cell in no particular order (neighbour
// counts, parent sets and conflict counts do not depend on it).  nc = 1 (one cell) when the box holds fewer than 3 cells per edge.
struct CellList {
  q4* q;
  int32_t *cell, *cstart, *members;
  int32_t nc;
  int64_t Lq, R2;
};

css_status build_cells(css_ctx* ctx, int32_t n, const double* xyz, double box, double r_col, CellList* cl,
                       cudaStream_t st) {
  const int T = 256;
  const unsigned nbk = (unsigned)css_ceil_div(n, T);
  const int64_t Lq = llrint(box * (double)kFix);
  const int64_t Rq = llrint(r_col * (double)kFix);
  int64_t nc64 = Rq > 0 ? Lq / Rq : 1024;
  int64_t nc_cap = (int64_t)cbrt((double)n) + 1;
  if (nc64 > nc_cap) nc64 = nc_cap;
  if (nc64 > 1024) nc64 = 1024;
  const int32_t nc = nc64 < 3 ? 1 : (int32_t)nc64;
  const int32_t ncells = nc >= 3 ? nc * nc * nc : 1;
  int32_t *ccnt, *cfill;
  CSS_TRY(css_ws(ctx, "col_q", sizeof(q4) * n, (void**)&cl->q));
  CSS_TRY(css_ws(ctx, "col_cell", sizeof(int32_t) * n, (void**)&cl->cell));
  CSS_TRY(css_ws(ctx, "col_ccnt", sizeof(int32_t) * (ncells + 1), (void**)&ccnt));
  CSS_TRY(css_ws(ctx, "col_cstart", sizeof(int32_t) * (ncells + 1), (void**)&cl->cstart));
  CSS_TRY(css_ws(ctx, "col_cfill", sizeof(int32_t) * (ncells + 1), (void**)&cfill));
  CSS_TRY(css_ws(ctx, "col_members", sizeof(int32_t) * n, (void**)&cl->members));
  k_quantise<<<nbk, T, 0, st>>>(n, xyz, Lq, nc, cl->q, cl->cell);
  CSS_LAUNCHED(ctx);
  CSS_CU(ctx, cudaMemsetAsync(ccnt, 0, sizeof(int32_t) * (ncells + 1), st));
  CSS_CU(ctx, cudaMemsetAsync(cfill, 0, sizeof(int32_t) * (ncells + 1), st));
  k_cell_count<<<nbk, T, 0, st>>>(n, cl->cell, ccnt);
  CSS_LAUNCHED(ctx);
  CSS_TRY(css_scan_i32(ctx, ccnt, cl->cstart, ncells, st));
  k_cell_fill<<<nbk, T, 0, st>>>(n, cl->cell, cl->cstart, cfill, cl->members);
  CSS_LAUNCHED(ctx);
  cl->nc = nc;
  cl->Lq = Lq;
  cl->R2 = Rq * Rq;
  return CSS_OK;
}

// Same-coloured pairs {i, j}, i < j, closer than r_col: thread i walks the 27 cells around
// molecule i (or all molecules when there is one cell).  Colours outside [0, n_colours) set
// *bad.  Per-warp sums are added into *count.
__global__ void k_conflicts(int32_t n, const q4* __restrict__ q, const int32_t* __restrict__ cell, int32_t nc,
                            const int32_t* __restrict__ cstart, const int32_t* __restrict__ members, int64_t Lq,
                            int64_t R2, const int32_t* __restrict__ colour, int32_t n_colours,
                            unsigned long long* __restrict__ count, int32_t* __restrict__ bad) {
  const int32_t i = blockIdx.x * blockDim.x + threadIdx.x;
  unsigned long long k = 0;
  if (i < n) {
    const int32_t ci = colour[i];
    if (ci < 0 || ci >= n_colours) atomicOr(bad, 1);
    const q4 qi = q[i];
    auto test = [&](int32_t j) {
      if (j <= i || colour[j] != ci) return;
      const q4 qj = q[j];
      const int64_t dx = min_image(qi.x - qj.x, Lq), dy = min_image(qi.y - qj.y, Lq),
                    dz = min_image(qi.z - qj.z, Lq);
      if (dx * dx + dy * dy + dz * dz < R2) ++k;
    };
    if (nc < 3) {
      for (int32_t j = i + 1; j < n; ++j) test(j);
    } else {
      const int32_t c = cell[i];
      const int32_t cx = c / (nc * nc), cy = (c / nc) % nc, cz = c % nc;
      for (int dx = -1; dx <= 1; ++dx)
        for (int dy = -1; dy <= 1; ++dy)
          for (int dz = -1; dz <= 1; ++dz) {
            const int32_t x = (cx + dx + nc) % nc, y = (cy + dy + nc) % nc, z = (cz + dz + nc) % nc;
            const int32_t cc = (x * nc + y) * nc + z;
            for (int32_t p = cstart[cc]; p < cstart[cc + 1]; ++p) test(members[p]);
          }
    }
  }
  for (int o = 16; o > 0; o >>= 1) k += __shfl_xor_sync(0xffffffffu, k, o);
  if ((threadIdx.x & 31) == 0 && k) atomicAdd(count, k);
}

// conflicts of a colouring on a geometry (blocking); *bad = 1 when a colour is out of range
css_status count_conflicts(css_ctx* ctx, const css_geom* geom, double r_col, const int32_t* colour,
                           int32_t n_colours, int64_t* count, int32_t* bad, cudaStream_t st) {
  const int32_t n = geom->n_mol;
  CellList cl;
  CSS_TRY(build_cells(ctx, n, geom->xyz, geom->box, r_col, &cl, st));
  unsigned long long* dcount;
  int32_t* dbad;
  CSS_TRY(css_ws(ctx, "chk_count", 2 * sizeof(unsigned long long), (void**)&dcount));
  dbad = (int32_t*)(dcount + 1);
  CSS_CU(ctx, cudaMemsetAsync(dcount, 0, 2 * sizeof(unsigned long long), st));
  k_conflicts<<<(unsigned)css_ceil_div(n, 256), 256, 0, st>>>(n, cl.q, cl.cell, cl.nc, cl.cstart, cl.members, cl.Lq,
                                                               cl.R2, colour, n_colours, dcount, dbad);
  CSS_LAUNCHED(ctx);
  unsigned long long* h;
  CSS_TRY(css_pinned(ctx, 64, (void**)&h));
  CSS_CU(ctx, cudaMemcpyAsync(h, dcount, 2 * sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
  CSS_CU(ctx, cudaStreamSynchronize(st));
  *count = (int64_t)h[0];
  *bad = *(const int32_t*)(h + 1) != 0 ? 1 : 0;
  return CSS_OK;
}

css_status check_geom(css_ctx* ctx, const css_geom* geom, double r_col, const char* what) {
  if (geom->n_mol < 1 || !(geom->box > 0.0) || geom->box > 1000.0 || !(r_col >= 0.0) || r_col > 1000.0)
    return css_set_arg_error(ctx, what);
  return CSS_OK;
}

}  // namespace

// Colour either a geometry (xyz != nullptr) or an explicit CSR graph.
css_status css_color_impl(css_ctx* ctx, int32_t n, const double* xyz, double box, double r_col, uint64_t seed,
                          const int32_t* adj_ptr_in, const int32_t* adj_in, int32_t* colour, int32_t* n_colours,
                          cudaStream_t st) {
  const int T = 256;
  const unsigned nbk = (unsigned)css_ceil_div(n, T), nwk = (unsigned)css_ceil_div((int64_t)n * 32, T);
  int32_t *hbuf, *deg, *np, *wait, *counters, *ptr = nullptr, *padj;
  CSS_TRY(css_pinned(ctx, 64, (void**)&hbuf));
  CSS_TRY(css_ws(ctx, "col_deg", sizeof(int32_t) * (n + 1), (void**)&deg));
  CSS_TRY(css_ws(ctx, "col_np", sizeof(int32_t) * n, (void**)&np));
  CSS_TRY(css_ws(ctx, "col_wait", sizeof(int32_t) * n, (void**)&wait));
  CSS_TRY(css_ws(ctx, "jp_counters", sizeof(int32_t) * 64, (void**)&counters));
  CSS_CU(ctx, cudaMemsetAsync(counters, 0, sizeof(int32_t) * 4, st));  // error, malformed graph, -, coloured
  const int32_t* adj_ptr = adj_ptr_in;
  if (xyz) {
    CellList cl;
    CSS_TRY(build_cells(ctx, n, xyz, box, r_col, &cl, st));
    CSS_TRY(css_ws(ctx, "col_adjptr", sizeof(int32_t) * (n + 1), (void**)&ptr));
    k_neighbours<0><<<nwk, T, 0, st>>>(n, cl.q, cl.cell, cl.nc, cl.cstart, cl.members, cl.Lq, cl.R2, seed, deg,
                                       nullptr, nullptr, nullptr);
    CSS_LAUNCHED(ctx);
    CSS_TRY(css_scan_i32(ctx, deg, ptr, n, st));
    adj_ptr = ptr;
    CSS_CU(ctx, cudaMemcpyAsync(hbuf, ptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CSS_CU(ctx, cudaStreamSynchronize(st));
    CSS_TRY(css_ws(ctx, "col_adj", sizeof(int32_t) * (size_t)std::max(hbuf[0], 1), (void**)&padj));
    k_neighbours<1><<<nwk, T, 0, st>>>(n, cl.q, cl.cell, cl.nc, cl.cstart, cl.members, cl.Lq, cl.R2, seed, deg,
                                       adj_ptr, np, padj);
    CSS_LAUNCHED(ctx);
  } else {  // a caller's graph: refuse a malformed pattern before anything reads through it
    k_graph_check<<<nbk, T, 0, st>>>(n, adj_ptr, adj_in, counters + 1);
    CSS_LAUNCHED(ctx);
    CSS_CU(ctx, cudaMemcpyAsync(hbuf, counters + 1, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CSS_CU(ctx, cudaMemcpyAsync(hbuf + 1, adj_ptr + n, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CSS_CU(ctx, cudaStreamSynchronize(st));
    if (hbuf[0] != 0)
      return css_set_arg_error(ctx, "css_color_graph: adj_ptr not non-decreasing from 0 or a neighbour outside [0, n)");
    CSS_TRY(css_ws(ctx, "col_adj", sizeof(int32_t) * (size_t)std::max(hbuf[1], 1), (void**)&padj));
    k_degrees<<<nbk, T, 0, st>>>(n, adj_ptr, deg);
    CSS_LAUNCHED(ctx);
    k_parents<<<nwk, T, 0, st>>>(n, adj_ptr, adj_in, seed, deg, np, padj);
    CSS_LAUNCHED(ctx);
  }
  CSS_CU(ctx, cudaMemsetAsync(wait, 0, sizeof(int32_t) * n, st));
  CSS_CU(ctx, cudaMemsetAsync(colour, 0xff, sizeof(int32_t) * n, st));
  CSS_CU(ctx, cudaMemsetAsync(counters + 2, 0xff, sizeof(int32_t), st));  // largest colour
  // as many warps as the chip holds at once, a vertex each as far as they go
  int occ = 0;
  CSS_CU(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_jp_flow, T, 0));
  const int64_t warps = std::min((int64_t)std::max(occ, 1) * ctx->n_sm, css_ceil_div(n, T / 32)) * (T / 32);
  int32_t per = (int32_t)css_ceil_div(n, warps), n_ = n;
  volatile int32_t* col_ = colour;
  int32_t *maxc = counters + 2, *done = counters + 3, *err = counters;
  int32_t hold_ = ctx->test_colour_hold ? 0 : -1;
  void* args[] = {&n_, &per, &adj_ptr, &np, &padj, &wait, &col_, &maxc, &done, &err, &hold_};
  CSS_CU(ctx, cudaLaunchCooperativeKernel((void*)k_jp_flow, dim3((unsigned)(warps / (T / 32))), dim3(T), args, 0, st));
  ++ctx->kernel_launches;
  CSS_CU(ctx, cudaMemcpyAsync(hbuf, counters, 3 * sizeof(int32_t), cudaMemcpyDeviceToHost, st));
  CSS_CU(ctx, cudaStreamSynchronize(st));
  if (hbuf[0]) {
    ctx->last_error = "css_color: the colouring did not finish within its time limit";
    return CSS_ERR_TIMEOUT;
  }
  *n_colours = hbuf[2] + 1;
  return CSS_OK;
}

extern "C" {

css_status css_color(css_ctx* ctx, const css_geom* geom, double r_col, uint64_t seed, int32_t* colour,
                     int32_t* n_colours, void* stream) {
  if (!ctx || !geom || !geom->xyz || !colour || !n_colours) return css_set_arg_error(ctx, "css_color: null pointer");
  if (geom->n_mol < 1 || !(geom->box > 0.0) || geom->box > 1000.0 || !(r_col >= 0.0) || r_col > 1000.0)
    return css_set_arg_error(ctx, "css_color: n_mol < 1, box not in (0, 1000] or r_col not in [0, 1000]");
  CSS_CU(ctx, cudaSetDevice(ctx->device));
  return css_color_impl(ctx, geom->n_mol, geom->xyz, geom->box, r_col, seed, nullptr, nullptr, colour, n_colours,
                        (cudaStream_t)stream);
}

css_status css_color_graph(css_ctx* ctx, int32_t n, const int32_t* adj_ptr, const int32_t* adj, uint64_t seed,
                           int32_t* colour, int32_t* n_colours, void* stream) {
  if (!ctx || !adj_ptr || !colour || !n_colours || n < 1) return css_set_arg_error(ctx, "css_color_graph: bad argument");
  CSS_CU(ctx, cudaSetDevice(ctx->device));
  return css_color_impl(ctx, n, nullptr, 0.0, 0.0, seed, adj_ptr, adj, colour, n_colours, (cudaStream_t)stream);
}

css_status css_color_check(css_ctx* ctx, const css_geom* geom, double r_col, const int32_t* colour,
                           int32_t n_colours, int64_t* n_conflicts, void* stream) {
  if (!ctx || !geom || !geom->xyz || !colour || !n_conflicts) return css_set_arg_error(ctx, "css_color_check: null pointer");
  CSS_TRY(check_geom(ctx, geom, r_col, "css_color_check: n_mol < 1, box not in (0, 1000] or r_col not in [0, 1000]"));
  if (n_colours < 1) return css_set_arg_error(ctx, "css_color_check: n_colours < 1");
  CSS_CU(ctx, cudaSetDevice(ctx->device));
  int64_t k = 0;
  int32_t bad = 0;
  CSS_TRY(count_conflicts(ctx, geom, r_col, colour, n_colours, &k, &bad, (cudaStream_t)stream));
  if (bad) return css_set_arg_error(ctx, "css_color_check: colour outside [0, n_colours)");
  *n_conflicts = k;
  return CSS_OK;
}

css_status css_color_update(css_ctx* ctx, const css_geom* geom, double r_col, double skin, uint64_t seed,
                            int32_t* colour, int32_t* n_colours, int32_t* recoloured, void* stream) {
  if (!ctx || !geom || !geom->xyz || !colour || !n_colours) return css_set_arg_error(ctx, "css_color_update: null pointer");
  if (!(skin >= 0.0)) return css_set_arg_error(ctx, "css_color_update: skin < 0");
  CSS_TRY(check_geom(ctx, geom, r_col + skin,
                     "css_color_update: n_mol < 1, box not in (0, 1000] or r_col + skin not in [0, 1000]"));
  CSS_CU(ctx, cudaSetDevice(ctx->device));
  cudaStream_t st = (cudaStream_t)stream;
  if (*n_colours >= 1) {
    int64_t k = 0;
    int32_t bad = 0;
    CSS_TRY(count_conflicts(ctx, geom, r_col, colour, *n_colours, &k, &bad, st));
    if (k == 0 && !bad) {
      if (recoloured) *recoloured = 0;
      return CSS_OK;
    }
  }
  int32_t nc = 0;
  CSS_TRY(css_color_impl(ctx, geom->n_mol, geom->xyz, geom->box, r_col + skin, seed, nullptr, nullptr, colour, &nc,
                         st));
  *n_colours = nc;
  if (recoloured) *recoloured = 1;
  return CSS_OK;
}

css_status css_probes(css_ctx* ctx, const int32_t* colour, int32_t n_mol, int32_t b, uint64_t sign_seed,
                      uint32_t flags, int8_t* sign, void* stream) {
  (void)colour;
  if (!ctx || !sign || n_mol < 1 || b < 1 || b > CSS_MAX_B) return css_set_arg_error(ctx, "css_probes: bad argument");
  CSS_CU(ctx, cudaSetDevice(ctx->device));
  int64_t count = (int64_t)n_mol * b;
  k_probe_signs<<<(unsigned)css_ceil_div(count, 256), 256, 0, (cudaStream_t)stream>>>(
      count, sign_seed, (flags & CSS_SIGNS_ONES) ? 1 : 0, sign);
  CSS_LAUNCHED(ctx);
  return CSS_OK;
}

}  // extern "C"
