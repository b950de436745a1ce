// CUDA kernels of the HHG multigrid for sm_103a.
//
// Every level-wide operation is one launch of 256-thread CTAs (32 x 8), as many
// as the GPU holds at once, walking a list of work units: chunks of free
// interface (face / edge / vertex) nodes, one node per thread, and row-pair
// tiles of the volume interiors of the active macros (the chunks first, or in
// large stencil launches spread evenly among the tiles).
//
// Volume work: in slice k of a macro's lattice the interior rows are
// j = 1..J (J = N - 2 - k) and row j holds N - 1 - j - k nodes.  Rows are
// paired as (1 + p, J - p), whose lengths add up to N - 1 - k, and a tile
// holds enough pairs for about 512 nodes of one colour in 8 consecutive
// slices; per slice the CTA flattens the nodes (or 4-node slots) of all its
// pairs into one index range, so lanes stay busy although the rows shrink
// across the triangle, and the rows it loads for one slice are still in L1
// when it processes the next.  On GB300 the FP64 pipe
// retires 2 DFMA per clock per SM and is charged per warp instruction, so
// idle lanes cost as much as busy ones.  Consecutive lanes read consecutive
// slots of one colour segment, so stencil neighbours are contiguous accesses.
//
// Flat kernels (k_gs_flat, k_res_flat, k_restrict_flat, k_prolong_flat; the
// default): no tiles, one work item per thread from a per-level table (a
// 16-byte vector of same-colour slots, or a slot of four nodes), one CTA per
// 256 items, so a launch has no CTA barrier and no CTA walking a long tile; the
// per-item arithmetic is the tile kernels', hence the same results bit for bit.
// One V(3,3) cycle, tile -> flat kernels: 7-point box of 3x2x1 sub-cubes
// refined 6 times 1.41 -> 1.06 ms, 2x2x2 refined 7 times 3.96 -> 3.00 ms;
// 15-point (sheared) refined 7 and 8 times 6.85 -> 5.35 and 35.7 -> 32.9 ms.
// The tile kernels stay for norms of more than FLAT_NORM_MAX CTAs (faster
// there), for a launch limit, for the streaming and batch forms, and for levels
// beyond the tables' range.
//
// Interface work: a node's stencil is the sum of the sub-stencils of the
// macros around it (§3.2, Fig. 4); the kernel updates the master in the
// interface container and writes the value into the ghost shell of every
// adjacent block (the local half of the ghost update of §3.1).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <type_traits>
#include <map>
#include <mutex>
#include <utility>

#include "hhg_kernels.h"

#include "cg_scalar.cuh"

namespace hhg {

std::atomic<long long> g_kernel_launches{0};

namespace {

constexpr int CTA = TILE_ROWS * TILE_SLOTS;   // 256 threads, 32 x 8

// Programmatic dependent launch: the kernels of a cycle are launched so that a
// kernel's CTAs may start while its predecessor in the stream drains
// (launch_next lets the successor start as early as that).  after_previous
// returns when the predecessor has completed and its writes are visible; before
// it a kernel touches only tables written at set-up (work items, active macros,
// lists, copy pointers, stencil weights), whose writing the host waited for.
// Every kernel launched so calls it, and completion stays in stream order; the
// forms with DEP = false are launched without, after their predecessor's end.
//
// The vectors (iterates, loads, residuals, partial sums) may change while such
// a kernel is resident and waits.  So its vector parameters are not
// __restrict__ (the compiler could move their loads above the wait, or send
// them through the read-only path, which is defined for data that stays the
// same as long as the kernel lives), and they are read with plain loads: the
// read-only path is left to launches that do not overlap (NC = !DEP below).
// The functions called after the wait may declare theirs __restrict__ again,
// which says nothing about the time before the call.
__device__ __forceinline__ void launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// 7-point structure: only the three chain axes (and negatives) are non-zero.
__host__ __device__ constexpr bool used_dir(int d, bool s7) {
  return !s7 || d == 1 || d == 2 || d == 3 || d == 8 || d == 9 || d == 10;
}

// Offset of node (i, j, k) inside a macro block (32-bit: a block holds fewer
// than 2^31 nodes for N <= 1024); rs is the level's slice-start table.
__device__ __forceinline__ int lidx32(const int* __restrict__ rs, int N, int i, int j, int k) {
  const int M = N + 1 - k;
  return ((i + 2 * j + 3 * k) & 3) * __ldg(rs + N + 2) + __ldg(rs + k) + slot_prefix(M) - slot_prefix(M - j) +
         (i >> 2);
}

// Base slot of row j of slice k of a level (colour array 0).
__device__ __forceinline__ int row_base(const int* __restrict__ rs, int N, int j, int k) {
  const int M = N + 1 - k;
  return __ldg(rs + k) + slot_prefix(M) - slot_prefix(M - j);
}

// Offsets of the 7-point neighbourhood of node (i, j, k), colour c, in one
// go: the five rows involved are derived from a single slot_prefix(M - j).
// nb[d] for d in {1, 2, 3, 8, 9, 10}; me = the node itself.
struct Slice {
  int N, k, M, CS, SLm, SL0, SLp, SMm, SM0, SMp;
};
__device__ __forceinline__ Slice slice_consts(const int* __restrict__ rs, int N, int k) {
  Slice s;
  s.N = N;
  s.k = k;
  s.M = N + 1 - k;
  s.CS = __ldg(rs + N + 2);
  s.SLm = k > 0 ? __ldg(rs + k - 1) : 0;
  s.SL0 = __ldg(rs + k);
  s.SLp = __ldg(rs + k + 1);
  s.SMm = slot_prefix(s.M - 1);
  s.SM0 = slot_prefix(s.M);
  s.SMp = slot_prefix(s.M + 1);
  return s;
}
struct Nb7 {
  int me, nb1, nb8, nb2, nb9, nb3, nb10;
};
__device__ __forceinline__ Nb7 nb7(const Slice& s, int i, int j) {
  const int X = slot_prefix(s.M - j);
  const int L = s.M - j;
  const int r0 = s.SL0 + s.SM0 - X;           // row (j, k)
  const int rjp = r0 + row_slots(L);          // row (j + 1, k)
  const int rjm = r0 - row_slots(L + 1);      // row (j - 1, k)
  const int rkp = s.SLp + s.SMm - X;          // row (j - 1, k + 1)
  const int rkm = s.SLm + s.SMp - X;          // row (j + 1, k - 1)
  const int c = (i + 2 * j + 3 * s.k) & 3;
  const int cp = ((c + 1) & 3) * s.CS, cm = ((c + 3) & 3) * s.CS;
  Nb7 n;
  n.me = c * s.CS + r0 + (i >> 2);
  n.nb1 = cp + r0 + ((i + 1) >> 2);           // ( 1,  0, 0)
  n.nb8 = cm + r0 + ((i - 1) >> 2);           // (-1,  0, 0)
  n.nb2 = cp + rjp + ((i - 1) >> 2);          // (-1,  1, 0)
  n.nb9 = cm + rjm + ((i + 1) >> 2);          // ( 1, -1, 0)
  n.nb3 = cp + rkp + (i >> 2);                // ( 0, -1, 1)
  n.nb10 = cm + rkm + (i >> 2);               // ( 0,  1, -1)
  return n;
}

__device__ __forceinline__ int tid256() { return threadIdx.y * TILE_SLOTS + threadIdx.x; }

// Sum over the CTA (any shape up to 1024 threads); result valid in thread 0.
__device__ __forceinline__ double block_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x + threadIdx.y * blockDim.x;
  const int nthreads = blockDim.x * blockDim.y;
  __syncthreads();
  if ((lane & 31) == 0) sh[lane >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (lane < 32) {
    s = (lane < (nthreads + 31) / 32) ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  return s;
}

// Colour-c nodes of interior row j of slice k: slots m = mlo .. mlo + n - 1
// (i = 4m + ic, 1 <= i <= N - 1 - j - k).
__device__ __forceinline__ void colour_row(int N, int j, int k, int c, int& ic, int& mlo, int& n) {
  ic = (c - 2 * j - 3 * k) & 3;
  const int L = N - 1 - j - k;
  mlo = ic == 0;
  n = L >= ic ? ((L - ic) >> 2) - mlo + 1 : 0;
}

// Work items of interior row j: its colour-c nodes (colour kernels; with
// vw > 1 its groups of vw consecutive slots holding them, slots vw g .. vw g
// + vw - 1) or its slots of four consecutive nodes (all-colour kernels).
__device__ __forceinline__ int row_items(int N, int j, int k, int c, bool colour, int vw = 1) {
  if (colour) {
    int ic, mlo, n;
    colour_row(N, j, k, c, ic, mlo, n);
    if (vw == 1) return n;
    return n > 0 ? (mlo + n - 1) / vw + 1 : 0;
  }
  return ((N - 1 - j - k) >> 2) + 1;
}

// An interior tile holds row pairs p = t.j0 .. t.j0 + t.m0 - 1 of slices t.k ..
// t.k + t.pad - 1, pair p being rows 1 + p and J - p of a slice (J = N - 2 -
// k).  The CTA flattens the items of all its pairs and slices into one range
// so that every lane has work: s_pre[s][q] = items of pairs t.j0 .. t.j0 + q -
// 1 in slice t.k + s (one warp per slice computes it with a warp scan), and
// s_tot[s] the items of slices t.k .. t.k + s - 1.  One CTA barrier for the
// whole tile, so that the threads stream through the items of all its slices
// without waiting for each other.  Returns the tile's item count.  All
// threads must call it.
constexpr int MAX_SLABS = 16;
__device__ __forceinline__ int flat_setup_slabs(const Tile& t, int N, int c, bool colour, int vw,
                                                int (*s_pre)[33], int* s_tot) {
  const int J0 = N - 2;
  for (int sl = threadIdx.y; sl < t.pad; sl += TILE_ROWS) {
    const int k = t.k + sl, J = J0 - k;
    const int q = threadIdx.x;
    int len = 0;
    if (q < t.m0) {
      const int j1 = 1 + t.j0 + q, j2 = J - t.j0 - q;
      if (j1 <= j2) {
        len = row_items(N, j1, k, c, colour, vw);
        if (j2 > j1) len += row_items(N, j2, k, c, colour, vw);
      }
    }
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, len, o);
      if (q >= o) len += y;
    }
    s_pre[sl][q + 1] = len;
    if (q == 0) s_pre[sl][0] = 0;
  }
  __syncthreads();
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    int acc = 0;
    for (int sl = 0; sl < t.pad; ++sl) {
      s_tot[sl] = acc;
      acc += s_pre[sl][t.m0];
    }
    s_tot[t.pad] = acc;
  }
  __syncthreads();
  return s_tot[t.pad];
}

// Item tt of a flattened tile -> its row j and index v within the row.
__device__ __forceinline__ void flat_item(const Tile& t, int N, int c, bool colour, const int* s_pre, int tt, int& j,
                                          int& v, int vw = 1) {
  int lo = 0, hi = t.m0;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (s_pre[mid] <= tt) lo = mid;
    else hi = mid;
  }
  const int j1 = 1 + t.j0 + lo;
  const int w = tt - s_pre[lo];
  const int n1 = row_items(N, j1, t.k, c, colour, vw);
  if (w < n1) {
    j = j1;
    v = w;
  } else {
    j = N - 2 - t.k - t.j0 - lo;
    v = w - n1;
  }
}

// Loop over the interior nodes of a tile, four consecutive nodes
// i = 4m .. 4m + 3 (one per colour array) per item, the items of all the
// tile's slices in one range (one CTA barrier per tile); the body sees i, j, k
// and the slice constants sc of the iterated level.  The kernel declares
// s_pre2[MAX_SLABS][33] and s_pre_tot[MAX_SLABS + 1] in shared memory.
#define HHG_TILE_NODES(NN, RS, t, s_pre, ...)                                        \
  {                                                                                  \
    const int total_ = flat_setup_slabs((t), (NN), 0, false, 1, s_pre##2, s_pre##_tot); \
    int sl_ = 0;                                                                     \
    for (int tt = tid256(); tt < total_; tt += CTA) {                                \
      while (tt >= s_pre##_tot[sl_ + 1]) ++sl_;                                      \
      const int k = (t).k + sl_;                                                     \
      const Tile ts_{k, (t).j0, (t).m0, 1};                                          \
      int j, m;                                                                      \
      flat_item(ts_, (NN), 0, false, s_pre##2[sl_], tt - s_pre##_tot[sl_], j, m);    \
      const Slice sc = slice_consts((RS), (NN), k);                                  \
      (void)sc;                                                                      \
      const int L = (NN) - 1 - j - k;                                                \
      _Pragma("unroll") for (int qq = 0; qq < 4; ++qq) {                             \
        const int i = 4 * m + qq;                                                    \
        if (i < 1 || i > L) continue;                                                \
        __VA_ARGS__                                                                  \
      }                                                                              \
    }                                                                                \
    __syncthreads();                                                                 \
  }

// Work units of a fused launch: units [0, n_if_units) are chunks of 256
// interface list entries, the rest (tile, active macro) pairs (large stencil
// launches map walk positions to units through spread_unit instead).  CTAs
// walk the units with a grid stride, so a launch has a few CTAs per SM
// whatever the level size.
#define HHG_UNITS(n_if_units, n_tiles, n_act)                                                     \
  for (int unit = blockIdx.x, n_units_ = (n_if_units) + (n_tiles) * (n_act); unit < n_units_;     \
       unit += gridDim.x)

// Interface chunk at position u of the walk (-1: a volume unit).
__device__ __forceinline__ int if_chunk(int u, int n_if_units) { return u < n_if_units ? u : -1; }
// Index of the volume unit at position u (not an interface chunk).
__device__ __forceinline__ int vol_index(int u, int n_if_units) { return u - n_if_units; }

// Walk over the same units, dynamic for large launches: CTA b starts with
// unit b; with at least DYN_UNITS_PER_CTA units per CTA, later units come from
// the problem's counter sched[0] (unit = gridDim.x + counter), so the units
// (tiles by decreasing work, the interface chunks spread among them, see
// spread_unit) are handed out greedily and the launch ends with the smallest
// tiles; smaller launches keep the grid
// stride (measured faster there, e.g. the local recovery cycles of a few
// macros).  Thread 0 takes the next unit one unit ahead, so the atomic's
// latency hides behind the work.  The CTA that finishes last (counted in
// sched[1]) puts both counters back to zero for the problem's next launch and
// counts the completed dynamic launch in sched[2] (read back by tests to show
// that the dynamic branch ran); a problem's kernels run one after another on
// one stream, so launches never share a counter.
constexpr int DYN_UNITS_PER_CTA = 4;
__device__ __forceinline__ bool walk_dynamic(int n_units) { return n_units >= DYN_UNITS_PER_CTA * (int)gridDim.x; }
__device__ __forceinline__ int walk_after(int cur, int n_units, int* sched) {
  if (cur >= n_units) return n_units;
  return walk_dynamic(n_units) ? (int)gridDim.x + atomicAdd(sched, 1) : cur + (int)gridDim.x;
}
__device__ __forceinline__ int walk_first(int n_units, int* sched, int* s_unit, int& nxt) {
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    nxt = walk_after((int)blockIdx.x, n_units, sched);
    *s_unit = blockIdx.x;
  }
  __syncthreads();
  return *s_unit;
}
__device__ __forceinline__ int walk_next(int n_units, int* sched, int* s_unit, int& nxt) {
  __syncthreads();                              // every thread has read the last unit
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    const int cur = nxt;
    nxt = walk_after(cur, n_units, sched);
    *s_unit = cur;
  }
  __syncthreads();
  return *s_unit;
}
__device__ __forceinline__ void finish_units(int* sched, int n_units) {
  if (!walk_dynamic(n_units)) return;
  if (threadIdx.x == 0 && threadIdx.y == 0) {
    __threadfence();
    if (atomicAdd(sched + 1, 1) == (int)gridDim.x - 1) {
      atomicExch(sched, 0);
      atomicExch(sched + 1, 0);
      atomicAdd(sched + 2, 1);
    }
  }
}
#define HHG_UNITS_DYN(n_if_units, n_tiles, n_act, sched, s_unit)                                      \
  for (int n_units_ = (n_if_units) + (n_tiles) * (n_act), nxt_ = 0,                                    \
           unit = walk_first(n_units_, (sched), (s_unit), nxt_);                                       \
       unit < n_units_; unit = walk_next(n_units_, (sched), (s_unit), nxt_))

// Position u of a stencil launch's walk -> its interface chunk (returned, or
// -1 for a volume unit, whose index is written to vol).  Launches that take
// the dynamic walk interleave the n_if interface chunks with the n_vol volume
// units (spread_position in hhg_internal.h: one chunk after every
// R = n_vol / n_if volume units).  An interface chunk gathers scattered
// neighbours and does little arithmetic, a volume tile streams contiguous
// rows through the FP64 (or load) pipe, so CTAs of the two kinds side by side
// on an SM keep the pipe busier than a launch whose first units are all
// interface chunks (finest FP64 Gauss-Seidel launch at refinement 8: 0.416
// against 0.442 ms).  Smaller launches keep the chunks first (measured faster
// on the coarse levels).  Every unit still runs once.
__device__ __forceinline__ int spread_unit(int u, int n_if, int n_vol, int& vol) {
  if (!walk_dynamic(n_if + n_vol)) {
    vol = u - n_if;
    return u < n_if ? u : -1;
  }
  return spread_position(u, n_if, n_vol, vol);
}

// Volume unit -> (tile, macro).  The macro index runs fastest and the tile
// lists are sorted by decreasing work, so the last units of a grid-stride walk
// are the smallest tiles of all macros (a short tail).
__device__ __forceinline__ void vol_unit(int b, int n_act, const Tile* __restrict__ tiles,
                                         const int* __restrict__ act, Tile& t, int& macro) {
  t = tiles[b / n_act];
  macro = act[b % n_act];
}

// The restriction walks each coarse tile as RESTRICT_SPLIT units of
// consecutive slices: a coarse level has an eighth of the fine level's nodes
// and its tiles give a few heavy units per CTA, whose tail left SMs idle.
constexpr int RESTRICT_SPLIT = 4;

// Volume unit b of a walk over split tiles: part (b / n_act) % split of tile
// (b / n_act) / split, for active macro b % n_act.
__device__ __forceinline__ void vol_subunit(int b, int n_act, int split, const Tile* __restrict__ tiles,
                                            const int* __restrict__ act, Tile& t, int& macro) {
  const int tp = b / n_act;
  macro = act[b % n_act];
  t = tiles[tp / split];
  const int part = tp % split;
  const int s0 = t.pad * part / split, s1 = t.pad * (part + 1) / split;
  t.k += s0;
  t.pad = s1 - s0;
}

// Off-diagonal part of an interface node's stencil applied to u, and the sum
// of the diagonal weights, over all copies of the node.
template <class T, bool S7>
__device__ __forceinline__ void if_stencil(int N, const int* __restrict__ rs, int64_t block, const T* __restrict__ u,
                                           const T* __restrict__ W, const Copy* __restrict__ cps, int c0, int c1,
                                           T& off, T& diag) {
  for (int c = c0; c < c1; ++c) {
    const Copy cp = cps[c];
    const T* w = W + ((size_t)cp.macro * 16 + node_class(cp.i, cp.j, cp.k, N)) * NDIR;
    const T* ub = u + (size_t)cp.macro * block;
    diag += w[0];
#pragma unroll
    for (int d = 1; d < NDIR; ++d) {
      if (!used_dir(d, S7)) continue;
      const T wd = w[d];
      // 15-point: skip the many zero weights; 7-point: no load waits on a weight
      if (!S7 && wd == T(0)) continue;
      int di, dj, dk;
      dir_ijk(d, di, dj, dk);
      const int ni = cp.i + di, nj = cp.j + dj, nk = cp.k + dk;
      if (!in_lattice(ni, nj, nk, N)) continue;
      off += wd * ub[lidx32(rs, N, ni, nj, nk)];
    }
  }
}

// Writes val into the copies c0 .. c1 - 1 of an interface node: at their
// precomputed block offsets cpo when given, else at the offsets computed from
// (macro, i, j, k).
template <class T>
__device__ __forceinline__ void write_copies(int N, const int* __restrict__ rs, int64_t block, T* __restrict__ u,
                                             const Copy* __restrict__ cps, const uint32_t* __restrict__ cpo, int c0,
                                             int c1, T val) {
  if (cpo) {
    for (int c = c0; c < c1; ++c) u[cpo[c]] = val;
    return;
  }
  for (int c = c0; c < c1; ++c) {
    const Copy cp = cps[c];
    u[(size_t)cp.macro * block + lidx32(rs, N, cp.i, cp.j, cp.k)] = val;
  }
}

// Interface stencil table of a problem level (build_if_tables): for list
// entry q the K distinct neighbours of the node's summed stencil, entry e at
// e * n + q (block offset nb, weight w), its diagonal and inverse diagonal.
template <class T>
struct IfTab {
  const uint32_t* nb;
  const T* w;
  const T* diag;
  const T* dinv;
  int n;
  // general connectivity (build_general_if_tables): entry e of list entry q at
  // ptr[q] + 32 e, len[q] entries (a multiple of four)
  const uint32_t* ptr;
  const int* len;
};
constexpr int if_tab_k(bool s7) { return s7 ? 6 : 14; }

// Off-diagonal part of the stencil of list entry q applied to u.
template <class T, int K>
__device__ __forceinline__ T if_offdiag(const IfTab<T>& t, const T* __restrict__ u, int q) {
  T s = T(0);
  if (K == 14 && t.ptr) {
    const int n = t.len[q];
    const uint32_t* nb = t.nb + t.ptr[q];
    const T* w = t.w + t.ptr[q];
    for (int e = 0; e < n; e += 4) {
#pragma unroll
      for (int x = 0; x < 4; ++x) s += w[32 * (e + x)] * u[nb[32 * (e + x)]];
    }
    return s;
  }
#pragma unroll
  for (int e = 0; e < K; ++e) s += t.w[(size_t)e * t.n + q] * u[t.nb[(size_t)e * t.n + q]];
  return s;
}

// ---------------------------------------------------------------------------
// Gauss-Seidel, one colour (§2.1 smoother)
// ---------------------------------------------------------------------------
// 16-byte vectors of a row: 4 FP32 or 2 FP64 consecutive slots.
template <class T>
struct Vec;
// load<true>() goes through the read-only path: a Gauss-Seidel colour
// kernel reads only arrays it does not write (the other colours and f).
// load<false>() is a plain coherent load, for code that reads data written
// earlier in the same launch (the persistent batch executor) or while the
// launch waited for its predecessor (DEP kernels).
template <>
struct Vec<float> {
  static constexpr int n = 4;
  template <bool NC = true>
  __device__ static void load(const float* p, float* v) {
    const float4 q = NC ? __ldg(reinterpret_cast<const float4*>(p)) : *reinterpret_cast<const float4*>(p);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
  }
  __device__ static void store(float* p, const float* v) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <>
struct Vec<double> {
  static constexpr int n = 2;
  template <bool NC = true>
  __device__ static void load(const double* p, double* v) {
    const double2 q = NC ? __ldg(reinterpret_cast<const double2*>(p)) : *reinterpret_cast<const double2*>(p);
    v[0] = q.x;
    v[1] = q.y;
  }
  __device__ static void store(double* p, const double* v) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  }
};

// Slots m0 + s .. m0 + s + VW - 1 (s = +1 when up, -1 when dn, else 0) of a
// row, from the aligned vector at p = &row[m0] and one extra element.
template <class T, bool NC = true>
__device__ __forceinline__ void load_shifted(const T* __restrict__ p, bool up, bool dn, T* v) {
  constexpr int VW = Vec<T>::n;
  Vec<T>::template load<NC>(p, v);
  if (up) {
    const T e = NC ? __ldg(p + VW) : p[VW];
#pragma unroll
    for (int t = 0; t < VW - 1; ++t) v[t] = v[t + 1];
    v[VW - 1] = e;
  } else if (dn) {
    const T e = NC ? __ldg(p - 1) : p[-1];
#pragma unroll
    for (int t = VW - 1; t > 0; --t) v[t] = v[t - 1];
    v[0] = e;
  }
}

// 7-point update of the colour-c nodes in slots m0 .. m0 + VW - 1 of interior
// row j of slice k (one aligned vector per stencil direction, plus one element
// where the neighbour's slot is shifted by one); only the interior nodes among
// them are written.  SCALED: the weights w and the load fb are already divided
// by the centre weight (u = f~ - sum w~ u, six FMAs per node), else the sum is
// multiplied by inv, the inverse centre weight.
template <class T, bool SCALED, bool NC = true>
__device__ __forceinline__ void gs_group7(const Slice& sc, int N, int j, int g, int c, T* __restrict__ ub,
                                          const T* __restrict__ fb, const T* __restrict__ w, T inv) {
  constexpr int VW = Vec<T>::n;
  int ic, mlo, n;
  colour_row(N, j, sc.k, c, ic, mlo, n);
  const int m0 = g * VW;
  const int X = slot_prefix(sc.M - j);
  const int L = sc.M - j;
  const int r0 = sc.SL0 + sc.SM0 - X;           // row (j, k)
  const int rjp = r0 + row_slots(L);             // row (j + 1, k)
  const int rjm = r0 - row_slots(L + 1);         // row (j - 1, k)
  const int rkp = sc.SLp + sc.SMm - X;           // row (j - 1, k + 1)
  const int rkm = sc.SLm + sc.SMp - X;           // row (j + 1, k - 1)
  const int cc = c * sc.CS, cp = ((c + 1) & 3) * sc.CS, cm = ((c + 3) & 3) * sc.CS;
  const bool e1 = ic == 3, e0 = ic == 0;         // slot of i + 1 is m + e1, of i - 1 is m - e0
  T acc[VW], a[VW];
  Vec<T>::template load<NC>(fb + cc + r0 + m0, acc);
  load_shifted<T, NC>(ub + cp + r0 + m0, e1, false, a);    // ( 1,  0,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[1] * a[t];
  load_shifted<T, NC>(ub + cp + rjp + m0, false, e0, a);   // (-1,  1,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[2] * a[t];
  Vec<T>::template load<NC>(ub + cp + rkp + m0, a);              // ( 0, -1,  1)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[3] * a[t];
  load_shifted<T, NC>(ub + cm + r0 + m0, false, e0, a);    // (-1,  0,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[8] * a[t];
  load_shifted<T, NC>(ub + cm + rjm + m0, e1, false, a);   // ( 1, -1,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[9] * a[t];
  Vec<T>::template load<NC>(ub + cm + rkm + m0, a);              // ( 0,  1, -1)
#pragma unroll
  for (int t = 0; t < VW; ++t) {
    if (SCALED) acc[t] -= w[10] * a[t];         // weights and f already divided by the centre weight
    else acc[t] = (acc[t] - w[10] * a[t]) * inv;
  }
  T* out = ub + cc + r0 + m0;
  const int lo = max(mlo - m0, 0), hi = min(mlo + n - m0, VW);
  if (lo == 0 && hi == VW) {
    Vec<T>::store(out, acc);
  } else {
#pragma unroll
    for (int t = 0; t < VW; ++t)
      if (t >= lo && t < hi) out[t] = acc[t];
  }
}

// 7-point residual r = f - A u of the colour-c nodes in slots m0 .. m0 + VW - 1
// of interior row j of slice k (same vectors as gs_group7 plus the centre);
// writes the interior nodes among them to rb and/or adds their squares to ss.
// ZERO: the residual of these nodes is known to vanish (their colour was the
// last one smoothed); zeros are written and nothing is read.
// Stores the lanes lo .. hi - 1 of a VW-vector (all lanes at once when the
// vector is complete).
template <class T>
__device__ __forceinline__ void store_lanes(T* __restrict__ out, const T* acc, int lo, int hi) {
  constexpr int VW = Vec<T>::n;
  if (lo == 0 && hi == VW) {
    Vec<T>::store(out, acc);
  } else {
#pragma unroll
    for (int t = 0; t < VW; ++t)
      if (t >= lo && t < hi) out[t] = acc[t];
  }
}

template <class T, bool WRITE, bool NORM, bool ZERO = false, bool NC = true>
__device__ __forceinline__ void res_group7(const Slice& sc, int N, int j, int g, int c, const T* __restrict__ ub,
                                           const T* __restrict__ fb, T* __restrict__ rb, const T* __restrict__ w,
                                           double& ss) {
  constexpr int VW = Vec<T>::n;
  int ic, mlo, n;
  colour_row(N, j, sc.k, c, ic, mlo, n);
  const int m0 = g * VW;
  const int X = slot_prefix(sc.M - j);
  const int L = sc.M - j;
  const int r0 = sc.SL0 + sc.SM0 - X;
  const int rjp = r0 + row_slots(L);
  const int rjm = r0 - row_slots(L + 1);
  const int rkp = sc.SLp + sc.SMm - X;
  const int rkm = sc.SLm + sc.SMp - X;
  const int cc = c * sc.CS, cp = ((c + 1) & 3) * sc.CS, cm = ((c + 3) & 3) * sc.CS;
  const bool e1 = ic == 3, e0 = ic == 0;
  T acc[VW], a[VW];
  if (ZERO) {
#pragma unroll
    for (int t = 0; t < VW; ++t) acc[t] = T(0);
    if (WRITE) store_lanes(rb + cc + r0 + m0, acc, max(mlo - m0, 0), min(mlo + n - m0, VW));
    return;
  }
  Vec<T>::template load<NC>(fb + cc + r0 + m0, acc);
  Vec<T>::template load<NC>(ub + cc + r0 + m0, a);               // centre
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[0] * a[t];
  load_shifted<T, NC>(ub + cp + r0 + m0, e1, false, a);    // ( 1,  0,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[1] * a[t];
  load_shifted<T, NC>(ub + cp + rjp + m0, false, e0, a);   // (-1,  1,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[2] * a[t];
  Vec<T>::template load<NC>(ub + cp + rkp + m0, a);              // ( 0, -1,  1)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[3] * a[t];
  load_shifted<T, NC>(ub + cm + r0 + m0, false, e0, a);    // (-1,  0,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[8] * a[t];
  load_shifted<T, NC>(ub + cm + rjm + m0, e1, false, a);   // ( 1, -1,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[9] * a[t];
  Vec<T>::template load<NC>(ub + cm + rkm + m0, a);              // ( 0,  1, -1)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[10] * a[t];
  const int lo = max(mlo - m0, 0), hi = min(mlo + n - m0, VW);
  if (NORM) {
#pragma unroll
    for (int t = 0; t < VW; ++t)
      if (t >= lo && t < hi) ss += (double)acc[t] * (double)acc[t];
  }
  if (WRITE) store_lanes(rb + cc + r0 + m0, acc, lo, hi);
}

// Base slots (colour array 0) of the seven rows (j + dj, k + dk) a 15-point
// stencil at row j of slice k touches, from one slot_prefix evaluation.
struct Rows15 {
  int r00, rp0, rm0, rmp, r0p, rpm, r0m;   // p: +1, m: -1, in the order (dj, dk)
};
__device__ __forceinline__ Rows15 rows15(const Slice& sc, int j) {
  const int L = sc.M - j, X = slot_prefix(L);
  Rows15 r;
  r.r00 = sc.SL0 + sc.SM0 - X;
  r.rp0 = r.r00 + row_slots(L);
  r.rm0 = r.r00 - row_slots(L + 1);
  r.rmp = sc.SLp + sc.SMm - X;
  r.r0p = r.rmp + row_slots(L);
  r.rpm = sc.SLm + sc.SMp - X;
  r.r0m = r.rpm - row_slots(L + 1);
  return r;
}

// acc -= w_d u_d over the 14 neighbours, in the order of the directions (the
// order of the tile kernels), for the colour-c nodes in slots m0 .. m0 + VW - 1
// of row j: one aligned vector per direction, and one element more where the
// neighbour's slot is shifted by one.
template <class T, bool NC>
__device__ __forceinline__ void sub_group15(const Slice& sc, int j, int c, int ic, int m0, const T* __restrict__ ub,
                                            const T* __restrict__ w, T* acc) {
  constexpr int VW = Vec<T>::n;
  const Rows15 r = rows15(sc, j);
  const bool e1 = ic == 3, e0 = ic == 0;   // slot of i + 1 is m + e1, of i - 1 is m - e0
  const T* c1 = ub + ((c + 1) & 3) * sc.CS + m0;
  const T* c2 = ub + ((c + 2) & 3) * sc.CS + m0;
  const T* c3 = ub + ((c + 3) & 3) * sc.CS + m0;
  const T* ptr[NDIR - 1] = {c1 + r.r00, c1 + r.rp0, c1 + r.rmp, c2 + r.rp0, c2 + r.r0p, c2 + r.rmp, c3 + r.r0p,
                            c3 + r.r00, c3 + r.rm0, c3 + r.rpm, c2 + r.rm0, c2 + r.r0m, c2 + r.rpm, c1 + r.r0m};
#pragma unroll
  for (int d = 1; d < NDIR; ++d) {
    int di, dj, dk;
    dir_ijk(d, di, dj, dk);
    T a[VW];
    load_shifted<T, NC>(ptr[d - 1], di > 0 && e1, di < 0 && e0, a);
    const T wd = w[d];
#pragma unroll
    for (int t = 0; t < VW; ++t) acc[t] -= wd * a[t];
  }
}

// 15-point update and residual of an item, as gs_group7 / res_group7.
template <class T, bool NC = true>
__device__ __forceinline__ void gs_group15(const Slice& sc, int N, int j, int g, int c, T* __restrict__ ub,
                                           const T* __restrict__ fb, const T* __restrict__ w, T inv) {
  constexpr int VW = Vec<T>::n;
  int ic, mlo, n;
  colour_row(N, j, sc.k, c, ic, mlo, n);
  const int m0 = g * VW, me = c * sc.CS + sc.SL0 + sc.SM0 - slot_prefix(sc.M - j) + m0;
  T acc[VW];
  Vec<T>::template load<NC>(fb + me, acc);
  sub_group15<T, NC>(sc, j, c, ic, m0, ub, w, acc);
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] *= inv;
  store_lanes(ub + me, acc, max(mlo - m0, 0), min(mlo + n - m0, VW));
}
template <class T, bool WRITE, bool NORM, bool ZERO = false, bool NC = true>
__device__ __forceinline__ void res_group15(const Slice& sc, int N, int j, int g, int c, const T* __restrict__ ub,
                                            const T* __restrict__ fb, T* __restrict__ rb, const T* __restrict__ w,
                                            double& ss) {
  constexpr int VW = Vec<T>::n;
  int ic, mlo, n;
  colour_row(N, j, sc.k, c, ic, mlo, n);
  const int m0 = g * VW, me = c * sc.CS + sc.SL0 + sc.SM0 - slot_prefix(sc.M - j) + m0;
  T acc[VW], a[VW];
  if (ZERO) {
#pragma unroll
    for (int t = 0; t < VW; ++t) acc[t] = T(0);
  } else {
    Vec<T>::template load<NC>(fb + me, acc);
    Vec<T>::template load<NC>(ub + me, a);
#pragma unroll
    for (int t = 0; t < VW; ++t) acc[t] -= w[0] * a[t];
    sub_group15<T, NC>(sc, j, c, ic, m0, ub, w, acc);
  }
  const int lo = max(mlo - m0, 0), hi = min(mlo + n - m0, VW);
  if (NORM) {
#pragma unroll
    for (int t = 0; t < VW; ++t)
      if (t >= lo && t < hi) ss += (double)acc[t] * (double)acc[t];
  }
  if (WRITE) store_lanes(rb + me, acc, lo, hi);
}

// The 7-point colour-c items of one tile: groups of VW consecutive same-colour
// slots per thread, the items of all the tile's slices streamed in one pass.
template <class T, bool SCALED, bool NC = true>
__device__ __forceinline__ void gs_tile7(const Tile& t, int N, const int* __restrict__ rs, int colour,
                                         T* __restrict__ ub, const T* __restrict__ fb, const T* __restrict__ w, T inv,
                                         int (*s_pre2)[33], int* s_pre_tot) {
  constexpr int VW = Vec<T>::n;
  const T wr[11] = {T(0), w[1], w[2], w[3], T(0), T(0), T(0), T(0), w[8], w[9], w[10]};
  const int total = flat_setup_slabs(t, N, colour, true, VW, s_pre2, s_pre_tot);
  int sl = 0;
  for (int tt = tid256(); tt < total; tt += CTA) {
    while (tt >= s_pre_tot[sl + 1]) ++sl;    // items only grow: the slice only advances
    const int k = t.k + sl;
    const Tile ts{k, t.j0, t.m0, 1};
    int j, g;
    flat_item(ts, N, colour, true, s_pre2[sl], tt - s_pre_tot[sl], j, g, VW);
    gs_group7<T, SCALED, NC>(slice_consts(rs, N, k), N, j, g, colour, ub, fb, wr, inv);
  }
}

// fs / Wsc (7-point only, may be null): the volume nodes read f and the
// interior weights already divided by their macro's centre weight.
template <class T, bool S7, bool DEP>
__global__ void __launch_bounds__(CTA, 5) k_gs(int N, const int* __restrict__ rs, int64_t block, T* u, T* uI,
                                            const T* f, const T* fI,
                                            const T* __restrict__ W, const T* __restrict__ Winv,
                                            const T* fs, const T* __restrict__ Wsc,
                                            const Tile* __restrict__ tiles, int n_tiles, const int* __restrict__ act,
                                            int n_act, int colour, const int* __restrict__ cptr,
                                            const Copy* __restrict__ cps, const uint32_t* __restrict__ cpo,
                                            const int* __restrict__ list, int n_list, IfTab<T> tab,
                                            int n_if_units, int* sched) {
  if (DEP) launch_next();
  if (DEP) after_previous();
  __shared__ int s_pre2[MAX_SLABS][33];
  __shared__ int s_pre_tot[MAX_SLABS + 1];
  __shared__ int s_unit;
  HHG_UNITS_DYN(n_if_units, n_tiles, n_act, sched, &s_unit) {
    int vol_ = 0;
    if (const int ic_ = spread_unit(unit, n_if_units, n_tiles * n_act, vol_); ic_ >= 0) {
      const int q = ic_ * CTA + tid256();
      if (q < n_list) {
        const int node = list[q];
        const int c0 = cptr[node], c1 = cptr[node + 1];
        T val;
        if (tab.nb) {
          val = (fI[node] - if_offdiag<T, if_tab_k(S7)>(tab, u, q)) * tab.dinv[q];
        } else {
          T off = T(0), diag = T(0);
          if_stencil<T, S7>(N, rs, block, u, W, cps, c0, c1, off, diag);
          val = (fI[node] - off) / diag;
        }
        uI[node] = val;
        write_copies(N, rs, block, u, cps, cpo, c0, c1, val);
      }
      continue;
    }
    Tile t;
    int macro;
    vol_unit(vol_, n_act, tiles, act, t, macro);
    T* ub = u + (size_t)macro * block;
    const T* fb = f + (size_t)macro * block;
    const T* w = W + (size_t)macro * 16 * NDIR;
    const T inv = Winv[macro];
    if (S7) {
      if (Wsc)
        gs_tile7<T, true, !DEP>(t, N, rs, colour, ub, fs + (size_t)macro * block, Wsc + (size_t)macro * 16 * NDIR,
                                T(1), s_pre2, s_pre_tot);
      else
        gs_tile7<T, false, !DEP>(t, N, rs, colour, ub, fb, w, inv, s_pre2, s_pre_tot);
    } else {
      // 15-point: one colour-c node per item
      const int total = flat_setup_slabs(t, N, colour, true, 1, s_pre2, s_pre_tot);
      int sl = 0;
      for (int tt = tid256(); tt < total; tt += CTA) {
        while (tt >= s_pre_tot[sl + 1]) ++sl;
        const int k = t.k + sl;
        const Tile ts{k, t.j0, t.m0, 1};
        int j, v, ic, mlo, n;
        flat_item(ts, N, colour, true, s_pre2[sl], tt - s_pre_tot[sl], j, v);
        colour_row(N, j, k, colour, ic, mlo, n);
        const int i = 4 * (mlo + v) + ic;
        const int me = lidx32(rs, N, i, j, k);
        T acc = fb[me];
#pragma unroll
        for (int d = 1; d < NDIR; ++d) {
          int di, dj, dk;
          dir_ijk(d, di, dj, dk);
          acc -= w[d] * ub[lidx32(rs, N, i + di, j + dj, k + dk)];
        }
        ub[me] = acc * inv;
      }
    }
    __syncthreads();
  }
  finish_units(sched, n_if_units + n_tiles * n_act);
}

// Flat Gauss-Seidel, one colour: one work item (one
// 16-byte vector of same-colour slots of one row) per thread, no tiles, no
// CTA barrier.  items[it] = (j << 20) | (k << 10) | g lists the colour's
// items of one macro interior, slice by slice and row by row, so consecutive
// threads take consecutive vectors of a row; a thread's global index runs
// over the active macros (item it of macro act[a]).  CTAs of interface nodes
// (one node per thread, as in k_gs) are spread among the volume CTAs
// (spread_position over CTAs).  fv / Wv: the volume's load and weights (f and
// W, or with SCALED both divided by the centre weight).  On a coarse level the tile kernel's launch
// waits for a few CTAs each walking a whole tile; here every thread has one
// item and the launch lasts about one item's latency.  Same arithmetic per
// item as gs_tile7, so the iterate equals the tile kernel's bit for bit.
// Resident CTAs per SM: the FP64 7-point form is held to 8 (32 registers;
// measured 1.2% faster at refinement 8); the FP32 form is left to the compiler
// (0: no bound; 3% slower held to 8, 6% slower held to 6).  Launches that
// overlap their predecessor keep the interface entries in registers: the FP64
// 15-point form is held to 3 CTAs (100 registers and 2 CTAs otherwise: solve
// with moved corners 11.97 instead of 11.71 ms); the FP32 7-point form is not
// held to 6 (spills: a mixed cycle of 2x2x2 sub-cubes refined 6 times 693
// instead of 629 us).
template <class T>
constexpr int flat_min_ctas(bool s7, bool dep) {
  const bool f64 = sizeof(T) == 8;
  return !f64 ? 0 : dep ? (s7 ? 0 : 3) : (s7 ? 8 : 0);
}

// Interface node of a launch that overlaps its predecessor: the stencil entries
// (all six of the 7-point form, up to 16 else) and the first two copies'
// offsets are loaded before the wait, so that after it only the neighbours and
// the right-hand side come from memory (a launch of a general mesh's interface
// class 4.0 -> 3.0 us from one to the next; general solve 18.8 -> 14.5 ms,
// solve with moved corners 14.3 -> 11.7 ms, box 860 -> 807 us a cycle).  Same
// sum in the same order as if_offdiag.
template <class T, bool S7>
__device__ __forceinline__ void gs_if_prefetched(const IfTab<T>& tab, int q, int node, int c0, int c1,
                                                 const uint32_t* __restrict__ cpo, T* u,
                                                 T* uI, const T* fI) {
  constexpr int PRE = S7 ? 6 : 16;
  const bool var = !S7 && tab.ptr;
  const int n = var ? tab.len[q] : if_tab_k(S7);
  const size_t at = var ? tab.ptr[q] : q, step = var ? 32 : tab.n;
  uint32_t nb[PRE];
  T w[PRE];
#pragma unroll
  for (int e = 0; e < PRE; ++e) {
    if (!S7 && e >= n) break;
    nb[e] = tab.nb[at + e * step];
    w[e] = tab.w[at + e * step];
  }
  const T di = tab.dinv[q];
  const uint32_t o0 = cpo[c0], o1 = c0 + 1 < c1 ? cpo[c0 + 1] : o0;
  after_previous();
  T s = T(0), x[PRE];
#pragma unroll
  for (int e = 0; e < PRE; ++e) {
    if (!S7 && e >= n) break;
    x[e] = u[nb[e]];
  }
  const T fv = fI[node];
#pragma unroll
  for (int e = 0; e < PRE; ++e) {
    if (!S7 && e >= n) break;
    s += w[e] * x[e];
  }
  if (!S7)
    for (int e = PRE; e < n; ++e) s += tab.w[at + e * step] * u[tab.nb[at + e * step]];
  const T val = (fv - s) * di;
  uI[node] = val;
  u[o0] = val;
  if (c0 + 1 < c1) u[o1] = val;
  for (int c = c0 + 2; c < c1; ++c) u[cpo[c]] = val;
}

template <class T, bool S7, bool SCALED, bool DEP>
__global__ void __launch_bounds__(CTA, flat_min_ctas<T>(S7, DEP)) k_gs_flat(int N, const int* __restrict__ rs, int64_t block, T* u,
                                                 T* uI, const T* fI,
                                                 const T* __restrict__ W, const T* __restrict__ Winv,
                                                 const T* fv, const T* __restrict__ Wv,
                                                 const uint32_t* __restrict__ items, int n_items,
                                                 const int* __restrict__ act, int n_act, int colour,
                                                 const int* __restrict__ cptr, const Copy* __restrict__ cps,
                                                 const uint32_t* __restrict__ cpo, const int* __restrict__ list,
                                                 int n_list, IfTab<T> tab, int n_if_ctas, int n_vol_ctas) {
  if (DEP) launch_next();
  int vb = 0;
  const int ib = spread_position((int)blockIdx.x, n_if_ctas, n_vol_ctas, vb);
  if (ib >= 0) {
    const int q = ib * CTA + tid256();
    if (q < n_list) {
      const int node = list[q];
      const int c0 = cptr[node], c1 = cptr[node + 1];
      if constexpr (DEP) {
        if (tab.nb && cpo) {
          gs_if_prefetched<T, S7>(tab, q, node, c0, c1, cpo, u, uI, fI);
          return;
        }
        after_previous();
      }
      T val;
      if (tab.nb) {
        val = (fI[node] - if_offdiag<T, if_tab_k(S7)>(tab, u, q)) * tab.dinv[q];
      } else {
        T off = T(0), diag = T(0);
        if_stencil<T, S7>(N, rs, block, u, W, cps, c0, c1, off, diag);
        val = (fI[node] - off) / diag;
      }
      uI[node] = val;
      write_copies(N, rs, block, u, cps, cpo, c0, c1, val);
    }
    return;
  }
  const int v = vb * CTA + tid256();
  if (v >= n_items * n_act) return;
  const int a = v / n_items, it = v - a * n_items;
  const int macro = act[a];
  const uint32_t d = items[it];
  const int j = (int)(d >> 20), k = (int)((d >> 10) & 1023u), g = (int)(d & 1023u);
  const T* w = Wv + (size_t)macro * 16 * NDIR;
  if constexpr (S7) {
    const T wr[11] = {T(0), w[1], w[2], w[3], T(0), T(0), T(0), T(0), w[8], w[9], w[10]};
    if constexpr (DEP) {
      const Slice sc = slice_consts(rs, N, k);
      const T inv = SCALED ? T(1) : Winv[macro];
      after_previous();
      gs_group7<T, SCALED, !DEP>(sc, N, j, g, colour, u + (size_t)macro * block, fv + (size_t)macro * block, wr, inv);
    } else {
      gs_group7<T, SCALED, !DEP>(slice_consts(rs, N, k), N, j, g, colour, u + (size_t)macro * block,
                           fv + (size_t)macro * block, wr, SCALED ? T(1) : Winv[macro]);
    }
  } else {
    const Slice sc = slice_consts(rs, N, k);
    if (DEP) after_previous();
    gs_group15<T, !DEP>(sc, N, j, g, colour, u + (size_t)macro * block, fv + (size_t)macro * block, w, Winv[macro]);
  }
}

// ---------------------------------------------------------------------------
// Streaming Gauss-Seidel, one colour, 7-point structure (levels with at least
// STREAM_MIN_N intervals).  In the colour-split layout the rows of a slice
// follow each other, so a band of rows of one slice and colour is one
// contiguous range of memory.  A unit (StreamTile) sweeps the band j0..j1 of
// one macro through the slices ka..kb.  The colour-c update of slice k reads
// colour c+1 in slices k and k+1, colour c-1 in slices k-1 and k, and f of
// colour c in slice k.  A producer warp copies these ranges into shared
// memory with bulk asynchronous copies (rings of three slices per neighbour
// colour, two for f) that complete on a "full" mbarrier per step; eight
// consumer warps wait on it, update their share of the slice's colour-c
// nodes straight into global memory and arrive on the step's "empty"
// mbarrier, which frees the slots the producer refills two steps later.  No
// CTA-wide barrier separates the steps of a unit, so warps and copies
// overlap; each neighbour value crosses HBM about once per launch (plus one
// row on either side of the band and one slice at either end of the unit).
// Interface chunks are updated by the consumer threads as in k_gs.  Every
// wait on an mbarrier is bounded: when one runs out the CTA sets *err, lets
// its copies in flight land (bounded) and stops taking units.
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}
__device__ __forceinline__ void fence_async_shared() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_addr(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Wait for the phase of bar with the given parity; false after `limit`
// unsuccessful tries (the first 32 back to back, then about 64 ns apart).
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, int limit) {
  for (int it = 0; it < limit; ++it) {
    if (mbar_test(bar, parity)) return true;
    if (it >= 32) __nanosleep(64);
  }
  return false;
}
constexpr int DRAIN_LIMIT = 1 << 24;

// First slot and slot count, inside one colour array, of rows ja..jb of
// slice k (clipped to the slice's closed lattice, rows 0..N-k).
__device__ __forceinline__ void band_range(const int* __restrict__ rs, int N, int k, int ja, int jb, int& off,
                                           int& len) {
  const int M = N + 1 - k;
  jb = min(jb, N - k);
  off = __ldg(rs + k) + slot_prefix(M) - slot_prefix(M - ja);
  len = jb >= ja ? slot_prefix(M - ja) - slot_prefix(M - jb - 1) : 0;
}

// 16-byte vector of a staged row in shared memory (16-byte aligned), shifted
// by one slot as in load_shifted.
template <class T>
struct SVec;
template <>
struct SVec<float> {
  __device__ static void load(const float* p, float* v) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    v[0] = q.x;
    v[1] = q.y;
    v[2] = q.z;
    v[3] = q.w;
  }
};
template <>
struct SVec<double> {
  __device__ static void load(const double* p, double* v) {
    const double2 q = *reinterpret_cast<const double2*>(p);
    v[0] = q.x;
    v[1] = q.y;
  }
};
template <class T>
__device__ __forceinline__ void lds_shifted(const T* p, bool up, bool dn, T* v) {
  constexpr int VW = Vec<T>::n;
  SVec<T>::load(p, v);
  if (up) {
    const T e = p[VW];
#pragma unroll
    for (int t = 0; t < VW - 1; ++t) v[t] = v[t + 1];
    v[VW - 1] = e;
  } else if (dn) {
    const T e = p[-1];
#pragma unroll
    for (int t = VW - 1; t > 0; --t) v[t] = v[t - 1];
    v[0] = e;
  }
}

// The update of gs_group7 with its operands read from the staged rows: a0 /
// a0p = colour c+1 rows j and j+1 of slice k, a1m = colour c+1 row j-1 of
// slice k+1, b0 / b0m = colour c-1 rows j and j-1 of slice k, bmp = colour
// c-1 row j+1 of slice k-1, fr = row j of f (all pointing at slot m0); out
// is row j of colour c in global memory at slot m0.  Same operations in the
// same order as gs_group7.
template <class T, bool SCALED>
__device__ __forceinline__ void gs_group7_staged(const T* a0, const T* a0p, const T* a1m, const T* b0, const T* b0m,
                                                 const T* bmp, const T* fr, T* __restrict__ out, bool e0, bool e1,
                                                 int lo, int hi, const T* w, T inv) {
  constexpr int VW = Vec<T>::n;
  T acc[VW], a[VW];
  SVec<T>::load(fr, acc);
  lds_shifted(a0, e1, false, a);    // ( 1,  0,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[1] * a[t];
  lds_shifted(a0p, false, e0, a);   // (-1,  1,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[2] * a[t];
  SVec<T>::load(a1m, a);            // ( 0, -1,  1)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[3] * a[t];
  lds_shifted(b0, false, e0, a);    // (-1,  0,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[8] * a[t];
  lds_shifted(b0m, e1, false, a);   // ( 1, -1,  0)
#pragma unroll
  for (int t = 0; t < VW; ++t) acc[t] -= w[9] * a[t];
  SVec<T>::load(bmp, a);            // ( 0,  1, -1)
#pragma unroll
  for (int t = 0; t < VW; ++t) {
    if (SCALED) acc[t] -= w[10] * a[t];
    else acc[t] = (acc[t] - w[10] * a[t]) * inv;
  }
  if (lo == 0 && hi == VW) {
    Vec<T>::store(out, acc);
  } else {
#pragma unroll
    for (int t = 0; t < VW; ++t)
      if (t >= lo && t < hi) out[t] = acc[t];
  }
}

// Shared memory of the streaming kernel: 8 staging slots of `slot` elements
// (3 for colour c+1, 3 for colour c-1, 2 for f) between pads of STREAM_PAD
// elements, so that the one-slot shifts of lanes outside the interior stay
// inside the allocation.  The CTA is 8 consumer warps and 1 producer warp.
constexpr int STREAM_PAD = 32;
constexpr int STREAM_NSLOT = 8;
constexpr int STREAM_CONSUMERS = 8;
constexpr int STREAM_CTA = 32 * (STREAM_CONSUMERS + 1);

template <class T, bool SCALED>
__global__ void __launch_bounds__(STREAM_CTA) k_gs_stream(
    int N, const int* __restrict__ rs, int64_t block, T* u, T* uI,
    const T* fI, const T* __restrict__ W, const T* __restrict__ Winv, const T* fv,
    const T* __restrict__ Wv, const StreamTile* __restrict__ tiles, int n_tiles, const int* __restrict__ act,
    int n_act, int colour, const int* __restrict__ cptr, const Copy* __restrict__ cps,
    const uint32_t* __restrict__ cpo, const int* __restrict__ list, int n_list, IfTab<T> tab, int n_if_units,
    int* sched, int slot, int wait_limit, int* err) {
  launch_next();
  after_previous();
  extern __shared__ __align__(128) unsigned char s_dyn[];
  T* const buf = reinterpret_cast<T*>(s_dyn) + STREAM_PAD;
  __shared__ __align__(8) uint64_t full[3], empty[3];
  __shared__ int s_pre[STREAM_SLICES][STREAM_BAND32 + 1];
  __shared__ int s_unit;
  __shared__ int s_fail;
  const int tid = tid256();
  const int warp = threadIdx.y, lane = threadIdx.x;
  const bool producer = warp == STREAM_CONSUMERS;
  if (tid == 0) s_fail = 0;
  constexpr int VW = Vec<T>::n;
  const int CS = __ldg(rs + N + 2);
  const int c = colour, cA = (c + 1) & 3, cB = (c + 3) & 3;
  bool failed = false;
  HHG_UNITS_DYN(n_if_units, n_tiles, n_act, sched, &s_unit) {
    if (const int ic_ = if_chunk(unit, n_if_units); ic_ >= 0) {
      const int q = ic_ * CTA + tid;
      if (!producer && q < n_list) {
        const int node = list[q];
        const int c0 = cptr[node], c1 = cptr[node + 1];
        T val;
        if (tab.nb) {
          val = (fI[node] - if_offdiag<T, 6>(tab, u, q)) * tab.dinv[q];
        } else {
          T off = T(0), diag = T(0);
          if_stencil<T, true>(N, rs, block, u, W, cps, c0, c1, off, diag);
          val = (fI[node] - off) / diag;
        }
        uI[node] = val;
        write_copies(N, rs, block, u, cps, cpo, c0, c1, val);
      }
      continue;
    }
    const int vb = vol_index(unit, n_if_units);
    const StreamTile st = tiles[vb / n_act];
    const int macro = act[vb % n_act];
    const int nst = st.kb - st.ka + 1;
    // fresh barriers per unit (every phase of the previous unit completed:
    // its steps were all consumed and released), and the items per row of
    // every step of the unit
    if (tid == 0)
      for (int b = 0; b < 3; ++b) {
        mbar_init(&full[b], 1);
        mbar_init(&empty[b], STREAM_CONSUMERS);
      }
    for (int sidx = warp; sidx < nst; sidx += STREAM_CONSUMERS + 1) {
      const int k = st.ka + sidx;
      const int nr = min(st.j1, N - 2 - k) - st.j0 + 1;
      int len = lane < nr ? row_items(N, st.j0 + lane, k, c, true, VW) : 0;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, len, o);
        if (lane >= o) len += y;
      }
      if (lane < nr) s_pre[sidx][lane + 1] = len;
      if (lane == 0) s_pre[sidx][0] = 0;
    }
    __syncthreads();
    T* ub = u + (size_t)macro * block;
    const int ja = st.j0 - 1, jbA = st.j1 + 1;
    if (producer) {
      if (lane == 0) {
        const T* gA = ub + (size_t)cA * CS;
        const T* gB = ub + (size_t)cB * CS;
        const T* gF = fv + (size_t)macro * block + (size_t)c * CS;
        int issued = 0;
        for (int sidx = 0; sidx < nst; ++sidx) {
          // step sidx refills the slots of step sidx - 2 (released on its empty barrier)
          if (sidx >= 2 && !mbar_wait(&empty[(sidx - 2) % 3], ((sidx - 2) / 3) & 1, wait_limit)) {
            atomicExch(err, 1);
            atomicExch(&s_fail, 1);
          }
          if (*(volatile int*)&s_fail) break;
          const int k = st.ka + sidx;
          int oA1, lA1, oB0, lB0, oF, lF, oA0 = 0, lA0 = 0, oBm = 0, lBm = 0;
          band_range(rs, N, k + 1, ja, jbA, oA1, lA1);
          band_range(rs, N, k, ja, jbA, oB0, lB0);
          band_range(rs, N, k, st.j0, min(st.j1, N - 2 - k), oF, lF);
          if (sidx == 0) {
            band_range(rs, N, k, ja, jbA, oA0, lA0);
            band_range(rs, N, k - 1, ja, jbA, oBm, lBm);
          }
          if (max(max(max(lA1, lB0), max(lF, lA0)), lBm) > slot) {   // never for the host's slot size
            atomicExch(err, 2);
            lA1 = min(lA1, slot);
            lB0 = min(lB0, slot);
            lF = min(lF, slot);
            lA0 = min(lA0, slot);
            lBm = min(lBm, slot);
          }
          fence_async_shared();
          uint64_t* b = &full[sidx % 3];
          mbar_expect(b, (uint32_t)(lA1 + lB0 + lF + lA0 + lBm) * (uint32_t)sizeof(T));
          if (lA1) bulk_load(buf + ((k + 1) % 3) * slot, gA + oA1, lA1 * (uint32_t)sizeof(T), b);
          if (lB0) bulk_load(buf + (3 + k % 3) * slot, gB + oB0, lB0 * (uint32_t)sizeof(T), b);
          if (lF) bulk_load(buf + (6 + k % 2) * slot, gF + oF, lF * (uint32_t)sizeof(T), b);
          if (lA0) bulk_load(buf + (k % 3) * slot, gA + oA0, lA0 * (uint32_t)sizeof(T), b);
          if (lBm) bulk_load(buf + (3 + (k + 2) % 3) * slot, gB + oBm, lBm * (uint32_t)sizeof(T), b);
          issued = sidx + 1;
        }
        if (*(volatile int*)&s_fail) {
          // the copies of the last step issued on each barrier may still be in flight
          for (int b = 0; b < 3; ++b) {
            int last = -1;
            for (int q = 0; q < issued; ++q)
              if (q % 3 == b) last = q;
            if (last >= 0) mbar_wait(&full[b], (last / 3) & 1, DRAIN_LIMIT);
          }
        }
      }
    } else {
      T* gU = ub + (size_t)c * CS;
      const T* wm = Wv + (size_t)macro * 16 * NDIR;
      const T w[11] = {T(0), wm[1], wm[2], wm[3], T(0), T(0), T(0), T(0), wm[8], wm[9], wm[10]};
      const T inv = SCALED ? T(1) : Winv[macro];
      for (int sidx = 0; sidx < nst; ++sidx) {
        if (!mbar_wait(&full[sidx % 3], (sidx / 3) & 1, wait_limit)) {
          if (lane == 0) {
            atomicExch(err, 1);
            atomicExch(&s_fail, 1);
          }
          break;   // no arrival on empty: the producer stops at its next wait
        }
        const int k = st.ka + sidx;
        const int nr = min(st.j1, N - 2 - k) - st.j0 + 1;
        const int* pre = s_pre[sidx];
        const int total = pre[nr];
        const int M = N + 1 - k, M1 = N - k, Mm = N + 2 - k;
        const T* sA0 = buf + (k % 3) * slot;
        const T* sA1 = buf + ((k + 1) % 3) * slot;
        const T* sB0 = buf + (3 + k % 3) * slot;
        const T* sBm = buf + (3 + (k + 2) % 3) * slot;
        const T* sF = buf + (6 + k % 2) * slot;
        const int PA = slot_prefix(M - ja), PA1 = slot_prefix(M1 - ja), PAm = slot_prefix(Mm - ja);
        const int PF = slot_prefix(M - st.j0);
        const int gbase = __ldg(rs + k) + slot_prefix(M);
        for (int tt = tid; tt < total; tt += CTA) {
          int lo_r = 0, hi_r = nr;
          while (hi_r - lo_r > 1) {
            const int mid = (lo_r + hi_r) >> 1;
            if (pre[mid] <= tt) lo_r = mid;
            else hi_r = mid;
          }
          const int j = st.j0 + lo_r;
          const int g = tt - pre[lo_r];
          int ic, mlo, n;
          colour_row(N, j, k, c, ic, mlo, n);
          const int m0 = g * VW;
          const int X = slot_prefix(M - j);
          const T* a0 = sA0 + (PA - X) + m0;
          const T* a0p = sA0 + (PA - slot_prefix(M - j - 1)) + m0;
          const T* a1m = sA1 + (PA1 - slot_prefix(M1 - j + 1)) + m0;
          const T* b0 = sB0 + (PA - X) + m0;
          const T* b0m = sB0 + (PA - slot_prefix(M - j + 1)) + m0;
          const T* bmp = sBm + (PAm - slot_prefix(Mm - j - 1)) + m0;
          const T* fr = sF + (PF - X) + m0;
          const int lo = max(mlo - m0, 0), hi = min(mlo + n - m0, VW);
          gs_group7_staged<T, SCALED>(a0, a0p, a1m, b0, b0m, bmp, fr, gU + (gbase - X) + m0, ic == 0, ic == 3,
                                      lo, hi, w, inv);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[sidx % 3]);
      }
    }
    __syncthreads();
    if (*(volatile int*)&s_fail) {
      failed = true;
      break;
    }
  }
  (void)failed;
  finish_units(sched, n_if_units + n_tiles * n_act);
}

// ---------------------------------------------------------------------------
// Residual r = f - A u on the free nodes (all colours); optional write of r
// (zero at the problem's frozen ghost copies) and per-CTA partial sums of r^2
// ---------------------------------------------------------------------------
// The 15-point items of one tile: four nodes of one slot each.
template <class T, bool WRITE, bool NORM>
__device__ __forceinline__ void res_tile15(const Tile& t, int N, const int* __restrict__ rs,
                                           const T* __restrict__ ub, const T* __restrict__ fb, T* __restrict__ rb,
                                           const T* __restrict__ w, int skip, double& ss, int (*s_pre2)[33],
                                           int* s_pre_tot) {
  HHG_TILE_NODES(N, rs, t, s_pre, {
    const int me = lidx32(rs, N, i, j, k);
    T acc = T(0);
    if (((i + 2 * j + 3 * k) & 3) != skip) {
      acc = fb[me] - w[0] * ub[me];
_Pragma("unroll")
      for (int d = 1; d < NDIR; ++d) {
        int di, dj, dk;
        dir_ijk(d, di, dj, dk);
        acc -= w[d] * ub[lidx32(rs, N, i + di, j + dj, k + dk)];
      }
    }
    if (WRITE) rb[me] = acc;
    if (NORM) ss += (double)acc * (double)acc;
  })
}

template <class T, bool S7, bool WRITE, bool NORM, bool DEP>
__global__ void __launch_bounds__(CTA, 4) k_res(int N, const int* __restrict__ rs, int64_t block, const T* u,
                                             const T* uI, const T* f,
                                             const T* fI, T* r, const T* __restrict__ W,
                                             const Tile* __restrict__ tiles, int n_tiles, const int* __restrict__ act,
                                             int n_act, const int* __restrict__ cptr, const Copy* __restrict__ cps,
                                             const uint32_t* __restrict__ cpo, const int* __restrict__ list,
                                             int n_list, IfTab<T> tab,
                                             const int64_t* __restrict__ zero_off, int n_zero, int n_if_units,
                                             double* partial, int* sched, int skip,
                                             int skip_lo, int skip_hi) {
  if (DEP) launch_next();
  if (DEP) after_previous();
  __shared__ int s_pre2[MAX_SLABS][33];
  __shared__ int s_pre_tot[MAX_SLABS + 1];
  __shared__ double sh[32];
  double ss = 0.0;
  __shared__ int s_unit;
  HHG_UNITS_DYN(n_if_units, n_tiles, n_act, sched, &s_unit) {
    int vol_ = 0;
    if (const int ic_ = spread_unit(unit, n_if_units, n_tiles * n_act, vol_); ic_ >= 0) {
      const int q = ic_ * CTA + tid256();
      if (q < n_list) {
        const int node = list[q];
        const int c0 = cptr[node], c1 = cptr[node + 1];
        T res;
        if (q >= skip_lo && q < skip_hi) {
          res = T(0);                              // the colour smoothed last
        } else if (tab.nb) {
          res = fI[node] - tab.diag[q] * uI[node] - if_offdiag<T, if_tab_k(S7)>(tab, u, q);
        } else {
          T off = T(0), diag = T(0);
          if_stencil<T, S7>(N, rs, block, u, W, cps, c0, c1, off, diag);
          res = fI[node] - diag * uI[node] - off;
        }
        if (WRITE) write_copies(N, rs, block, r, cps, cpo, c0, c1, res);
        if (NORM) ss += (double)res * (double)res;
      } else if (WRITE && q < n_list + n_zero) {
        r[zero_off[q - n_list]] = T(0);
      }
      continue;
    }
    Tile t;
    int macro;
    vol_unit(vol_, n_act, tiles, act, t, macro);
    const T* ub = u + (size_t)macro * block;
    const T* fb = f + (size_t)macro * block;
    T* rb = r + (size_t)macro * block;
    const T* w = W + (size_t)macro * 16 * NDIR;
    if (S7) {
      // one colour after another, groups of VW same-colour slots per thread
      constexpr int VW = Vec<T>::n;
      const T wr[11] = {w[0], w[1], w[2], w[3], T(0), T(0), T(0), T(0), w[8], w[9], w[10]};
      for (int c = 0; c < 4; ++c) {
        if (!WRITE && c == skip) continue;         // norm only: the skipped colour adds nothing
        const int total = flat_setup_slabs(t, N, c, true, VW, s_pre2, s_pre_tot);
        int sl = 0;
        for (int tt = tid256(); tt < total; tt += CTA) {
          while (tt >= s_pre_tot[sl + 1]) ++sl;
          const int k = t.k + sl;
          const Tile ts{k, t.j0, t.m0, 1};
          int j, g;
          flat_item(ts, N, c, true, s_pre2[sl], tt - s_pre_tot[sl], j, g, VW);
          if (c == skip)
            res_group7<T, WRITE, NORM, true>(slice_consts(rs, N, k), N, j, g, c, ub, fb, rb, wr, ss);
          else
            res_group7<T, WRITE, NORM, false, !DEP>(slice_consts(rs, N, k), N, j, g, c, ub, fb, rb, wr, ss);
        }
        __syncthreads();
      }
      continue;
    }
    res_tile15<T, WRITE, NORM>(t, N, rs, ub, fb, rb, w, skip, ss, s_pre2, s_pre_tot);
  }
  finish_units(sched, n_if_units + n_tiles * n_act);
  if (NORM) {
    const double s = block_sum(ss, sh);
    if (threadIdx.x == 0 && threadIdx.y == 0) partial[blockIdx.x] = s;
  }
}

// Flat residual: the items of all four colours of the flat
// Gauss-Seidel tables (colour c's at off[c] .. off[c + 1]) for every active
// macro, and the interface entries, in chunks of 256 walked with a grid
// stride (launched with one chunk per CTA), interface chunks spread among the
// volume chunks; no tiles and no CTA barrier before the final norm
// reduction.  Same arithmetic per item as k_res (res_group7), so r is the
// same bit for bit; the norm's partial sums follow the grid.  n_items:
// items per macro taken (off[4], or off[3] for a norm-only launch that skips
// colour 3).
template <class T, bool S7, bool WRITE, bool NORM, bool DEP>
__global__ void __launch_bounds__(CTA) k_res_flat(int N, const int* __restrict__ rs, int64_t block,
                                                  const T* u, const T* uI,
                                                  const T* f, const T* fI, T* r,
                                                  const T* __restrict__ W, const uint32_t* __restrict__ items,
                                                  int4 off, int n_items, const int* __restrict__ act, int n_act,
                                                  const int* __restrict__ cptr, const Copy* __restrict__ cps,
                                                  const uint32_t* __restrict__ cpo, const int* __restrict__ list,
                                                  int n_list, IfTab<T> tab, const int64_t* __restrict__ zero_off,
                                                  int n_zero, int n_if_chunks, int n_vol_chunks,
                                                  double* partial, int skip, int skip_lo, int skip_hi) {
  __shared__ double sh[32];
  double ss = 0.0;
  const int n_vol = n_items * n_act;
  if (DEP) launch_next();
  if (DEP) after_previous();
  for (int chunk = blockIdx.x; chunk < n_if_chunks + n_vol_chunks; chunk += gridDim.x) {
    int vc = 0;
    const int ic = spread_position(chunk, n_if_chunks, n_vol_chunks, vc);
    if (ic >= 0) {
      const int q = ic * CTA + tid256();
      if (q < n_list) {
        const int node = list[q];
        const int c0 = cptr[node], c1 = cptr[node + 1];
        T res;
        if (q >= skip_lo && q < skip_hi) {
          res = T(0);                              // the colour smoothed last
        } else if (tab.nb) {
          res = fI[node] - tab.diag[q] * uI[node] - if_offdiag<T, if_tab_k(S7)>(tab, u, q);
        } else {
          T off_ = T(0), diag = T(0);
          if_stencil<T, S7>(N, rs, block, u, W, cps, c0, c1, off_, diag);
          res = fI[node] - diag * uI[node] - off_;
        }
        if (WRITE) write_copies(N, rs, block, r, cps, cpo, c0, c1, res);
        if (NORM) ss += (double)res * (double)res;
      } else if (WRITE && q < n_list + n_zero) {
        r[zero_off[q - n_list]] = T(0);
      }
      continue;
    }
    const int v = vc * CTA + tid256();
    if (v >= n_vol) continue;
    const int a = v / n_items, it = v - a * n_items;
    const int c = it < off.y ? 0 : it < off.z ? 1 : it < off.w ? 2 : 3;
    if (!WRITE && c == skip) continue;             // norm only: the skipped colour adds nothing
    const int macro = act[a];
    const uint32_t d = items[it];
    const int j = (int)(d >> 20), k = (int)((d >> 10) & 1023u), g = (int)(d & 1023u);
    const T* w = W + (size_t)macro * 16 * NDIR;
    const size_t mb = (size_t)macro * block;
    // 7 points: slice_consts inside each branch on the skipped colour: before it
    // the constants stay live through both, 48 registers instead of 40 and five
    // CTAs per SM instead of six
    if constexpr (S7) {
      const T wr[11] = {w[0], w[1], w[2], w[3], T(0), T(0), T(0), T(0), w[8], w[9], w[10]};
      if (c == skip) res_group7<T, WRITE, NORM, true>(slice_consts(rs, N, k), N, j, g, c, u + mb, f + mb, r + mb, wr, ss);
      else res_group7<T, WRITE, NORM, false, !DEP>(slice_consts(rs, N, k), N, j, g, c, u + mb, f + mb, r + mb, wr, ss);
    } else {
      const Slice sc = slice_consts(rs, N, k);
      if (c == skip) res_group15<T, WRITE, NORM, true>(sc, N, j, g, c, u + mb, f + mb, r + mb, w, ss);
      else res_group15<T, WRITE, NORM, false, !DEP>(sc, N, j, g, c, u + mb, f + mb, r + mb, w, ss);
    }
  }
  if (NORM) {
    const double s = block_sum(ss, sh);
    if (threadIdx.x == 0 && threadIdx.y == 0) partial[blockIdx.x] = s;
  }
}

// ---------------------------------------------------------------------------
// Restriction R = P^T onto the coarse level (§2.1); zero the coarse correction
// ---------------------------------------------------------------------------
// Calls body(j, k, m) for every item of a tile: slot m of interior row j of
// slice k, i.e. the nodes i = 4m .. 4m + 3 (one per colour array), the items
// of all the tile's slices in one range (one CTA barrier per tile, as for the
// stencil kernels); ends with a CTA barrier.  The kernel declares
// s_pre2[MAX_SLABS][33] and s_pre_tot[MAX_SLABS + 1] in shared memory.
template <class F>
__device__ __forceinline__ void for_tile_slots(const Tile& t, int N, int (*s_pre2)[33], int* s_pre_tot, F&& body) {
  const int total = flat_setup_slabs(t, N, 0, false, 1, s_pre2, s_pre_tot);
  int sl = 0;
  for (int tt = tid256(); tt < total; tt += CTA) {
    while (tt >= s_pre_tot[sl + 1]) ++sl;
    const int k = t.k + sl;
    const Tile ts{k, t.j0, t.m0, 1};
    int j, m;
    flat_item(ts, N, 0, false, s_pre2[sl], tt - s_pre_tot[sl], j, m);
    body(j, k, m);
  }
  __syncthreads();
}

// Full-weighting restriction f_c = r(2I) + 1/2 sum_d r(2I + d) (d over the 14
// stencil directions, summed in their order) of the coarse nodes I = 4M ..
// 4M + 3 of interior row J of coarse slice K (one per colour array); the
// coarse correction there is zeroed.  The seven fine rows (2J + dj, 2K + dk)
// are located once per item; fine node i' = 8M + 2q + di lies in colour
// array (2q + di + 2 jf + 3 kf) & 3 at slot 2M + ((2q + di) >> 2), so every
// load is a row base plus constants.  All colours of the item in one pass
// keep the fine rows in cache for the four coarse nodes.  Plain loads when
// NC is false (data written in this launch).
template <class T, bool NC>
__device__ __forceinline__ void restrict_slot(int Nc, const int* __restrict__ rsc, int Nf,
                                              const int* __restrict__ rsf, int J, int K, int M,
                                              const T* __restrict__ rb, T* __restrict__ fcb, T* __restrict__ ucb) {
  const int Lc = Nc - 1 - J - K;
  const int CSf = __ldg(rsf + Nf + 2);
  int base[NDIR], col[NDIR];
#pragma unroll
  for (int d = 0; d < NDIR; ++d) {
    int di, dj, dk;
    dir_ijk(d, di, dj, dk);
    const int jf = 2 * J + dj, kf = 2 * K + dk;
    base[d] = row_base(rsf, Nf, jf, kf) + 2 * M;
    col[d] = 2 * jf + 3 * kf;
  }
  const int CSc = __ldg(rsc + Nc + 2);
  const int rbc = row_base(rsc, Nc, J, K) + M;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int I = 4 * M + q;
    if (I < 1 || I > Lc) continue;
    T cen = T(0), acc = T(0);
#pragma unroll
    for (int d = 0; d < NDIR; ++d) {
      int di, dj, dk;
      dir_ijk(d, di, dj, dk);
      const int o = ((2 * q + di + col[d]) & 3) * CSf + base[d] + ((2 * q + di) >> 2);
      const T x = NC ? __ldg(rb + o) : rb[o];
      if (d == 0) cen = x;
      else acc += x;
    }
    const int me = ((q + 2 * J + 3 * K) & 3) * CSc + rbc;
    fcb[me] = fma(T(0.5), acc, cen);   // the halving is exact: same value as a separate multiply
    ucb[me] = T(0);
  }
}

// Volume restriction of a coarse tile.
template <class T, bool NC>
__device__ __forceinline__ void restrict_tile(const Tile& t, int Nc, const int* __restrict__ rsc, int Nf,
                                              const int* __restrict__ rsf, const T* __restrict__ rb,
                                              T* __restrict__ fcb, T* __restrict__ ucb, int (*s_pre2)[33],
                                              int* s_pre_tot) {
  for_tile_slots(t, Nc, s_pre2, s_pre_tot, [&](int J, int K, int M) {
    restrict_slot<T, NC>(Nc, rsc, Nf, rsf, J, K, M, rb, fcb, ucb);
  });
}

template <class T, bool DEP>
__global__ void __launch_bounds__(CTA, 4) k_restrict(int Nc, const int* __restrict__ rsc, int64_t bc, T* fc, T* fIc,
                                                  T* uc, T* uIc, int Nf, const int* __restrict__ rsf, int64_t bf,
                                                  const T* rf, const Tile* __restrict__ tiles, int n_tiles,
                                                  const int* __restrict__ act, int n_act,
                                                  const int* __restrict__ cptr, const Copy* __restrict__ cps,
                                                  const uint32_t* __restrict__ cpo,
                                                  const int* __restrict__ list, int n_list,
                                                  const int64_t* __restrict__ gather,
                                                  const int64_t* __restrict__ zero_off, int n_zero, int n_if_units, int* sched) {
  if (DEP) launch_next();
  if (DEP) after_previous();
  __shared__ int s_pre2[MAX_SLABS][33];
  __shared__ int s_pre_tot[MAX_SLABS + 1];
  __shared__ int s_unit;
  HHG_UNITS_DYN(n_if_units, n_tiles * RESTRICT_SPLIT, n_act, sched, &s_unit) {
    if (const int ic_ = if_chunk(unit, n_if_units); ic_ >= 0) {
      const int q = ic_ * CTA + tid256();
      if (q < n_list) {
        const int node = list[q];
        const int64_t* g = gather + (size_t)q * NDIR;
        T acc = T(0);
        for (int e = 1; e < NDIR; ++e) {
          const int64_t o = g[e];
          if (o >= 0) acc += rf[o];
        }
        fIc[node] = rf[g[0]] + T(0.5) * acc;
        uIc[node] = T(0);
        write_copies(Nc, rsc, bc, uc, cps, cpo, cptr[node], cptr[node + 1], T(0));
      } else if (q < n_list + n_zero) {
        uc[zero_off[q - n_list]] = T(0);
      }
      continue;
    }
    Tile t;
    int macro;
    vol_subunit(vol_index(unit, n_if_units), n_act, RESTRICT_SPLIT, tiles, act, t, macro);
    restrict_tile<T, !DEP>(t, Nc, rsc, Nf, rsf, rf + (size_t)macro * bf, fc + (size_t)macro * bc,
                           uc + (size_t)macro * bc, s_pre2, s_pre_tot);
  }
  finish_units(sched, n_if_units + n_tiles * RESTRICT_SPLIT * n_act);
}

// ---------------------------------------------------------------------------
// Prolongation u_f += P u_c (linear interpolation, §2.1)
// ---------------------------------------------------------------------------
template <class T>
__device__ __forceinline__ T interp(const T* __restrict__ cb, int Nc, const int* __restrict__ rsc, int i, int j, int k) {
  const int pi = i & 1, pj = j & 1, pk = k & 1;
  if (!(pi | pj | pk)) return cb[lidx32(rsc, Nc, i >> 1, j >> 1, k >> 1)];
  // the coarse edge through a fine midpoint: parity -> local direction
  int di, dj, dk;
  const int code = pi | (pj << 1) | (pk << 2);
  switch (code) {
    case 1: di = 1; dj = 0; dk = 0; break;
    case 2: di = 0; dj = 1; dk = 0; break;
    case 4: di = 0; dj = 0; dk = 1; break;
    case 3: di = -1; dj = 1; dk = 0; break;
    case 5: di = -1; dj = 0; dk = 1; break;
    case 6: di = 0; dj = -1; dk = 1; break;
    default: di = 1; dj = -1; dk = 1; break;
  }
  const T a = cb[lidx32(rsc, Nc, (i - di) >> 1, (j - dj) >> 1, (k - dk) >> 1)];
  const T b = cb[lidx32(rsc, Nc, (i + di) >> 1, (j + dj) >> 1, (k + dk) >> 1)];
  return T(0.5) * (a + b);
}

// Coarse edge through a fine node of parities (pi, pj, pk), not all zero: the
// fine node is the midpoint of coarse nodes (i -+ di, j -+ dj, k -+ dk) / 2.
__device__ __forceinline__ void edge_dir(int code, int& di, int& dj, int& dk) {
  switch (code) {
    case 1: di = 1; dj = 0; dk = 0; break;
    case 2: di = 0; dj = 1; dk = 0; break;
    case 4: di = 0; dj = 0; dk = 1; break;
    case 3: di = -1; dj = 1; dk = 0; break;
    case 5: di = -1; dj = 0; dk = 1; break;
    case 6: di = 0; dj = -1; dk = 1; break;
    default: di = 1; dj = -1; dk = 1; break;
  }
}

// Prolongation u_f += P u_c of the fine nodes i = 4m .. 4m + 3 of interior
// row j of fine slice k (one per colour array; fine block fb, coarse block
// cb).  The parities of a node are (q & 1, j & 1, k & 1), so an item has two
// interpolation cases (even and odd i): the coarse node (i/2, j/2, k/2) when
// all parities are even, else the mean of the coarse edge's two ends.  Their
// coarse rows are located once per item; coarse node I = 2m + const lies in
// colour array (I + 2J + 3K) & 3 at slot I >> 2.  Plain loads for the fine
// values (written by this launch), the read-only path for the coarse ones
// when NC.  Nodes of colour skip are left out (-1: none).
template <class T, bool NC>
__device__ __forceinline__ void prolong_slot(int Nf, const int* __restrict__ rsf, int Nc, const int* __restrict__ rsc,
                                             int j, int k, int m, T* __restrict__ fb, const T* __restrict__ cb,
                                             int skip) {
  const int L = Nf - 1 - j - k;
  const int CSf = __ldg(rsf + Nf + 2), CSc = __ldg(rsc + Nc + 2);
  const int rbf = row_base(rsf, Nf, j, k) + m;
  const int cf = 2 * j + 3 * k;
  // per parity of i: direction, the two coarse rows and their colour terms
  int di[2], rba[2], rbb[2], ca[2], cbb[2], code[2];
#pragma unroll
  for (int par = 0; par < 2; ++par) {
    code[par] = par | ((j & 1) << 1) | ((k & 1) << 2);
    int dj = 0, dk = 0;
    di[par] = 0;
    if (code[par]) edge_dir(code[par], di[par], dj, dk);
    const int JA = (j - dj) >> 1, KA = (k - dk) >> 1, JB = (j + dj) >> 1, KB = (k + dk) >> 1;
    rba[par] = row_base(rsc, Nc, JA, KA);
    rbb[par] = row_base(rsc, Nc, JB, KB);
    ca[par] = 2 * JA + 3 * KA;
    cbb[par] = 2 * JB + 3 * KB;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = 4 * m + q;
    if (i < 1 || i > L || ((q + cf) & 3) == skip) continue;
    const int par = q & 1;
    T* out = fb + ((q + cf) & 3) * CSf + rbf;
    const T u = *out;
    if (code[par] == 0) {
      const int I = 2 * m + (q >> 1);
      const int o = ((I + ca[par]) & 3) * CSc + rba[par] + (I >> 2);
      *out = u + (NC ? __ldg(cb + o) : cb[o]);
    } else {
      const int IA = 2 * m + ((q - di[par]) >> 1), IB = 2 * m + ((q + di[par]) >> 1);
      const int oa = ((IA + ca[par]) & 3) * CSc + rba[par] + (IA >> 2);
      const int ob = ((IB + cbb[par]) & 3) * CSc + rbb[par] + (IB >> 2);
      const T a = NC ? __ldg(cb + oa) : cb[oa];
      const T b = NC ? __ldg(cb + ob) : cb[ob];
      *out = fma(T(0.5), a + b, u);   // the halving is exact: same value as a separate multiply
    }
  }
}

// The same prolongation for the colour-c nodes in slots m0 .. m0 + VW - 1 of
// interior row j of fine slice k, one 16-byte vector of fine values: all
// nodes i = 4m + ic of a colour row share their parities, hence one case.
template <class T, bool NC>
__device__ __forceinline__ void prolong_group(int Nf, const int* __restrict__ rsf, int Nc, const int* __restrict__ rsc,
                                              int j, int k, int g, int c, T* __restrict__ fb,
                                              const T* __restrict__ cb) {
  constexpr int VW = Vec<T>::n;
  int ic, mlo, n;
  colour_row(Nf, j, k, c, ic, mlo, n);
  const int m0 = g * VW;
  const int lo = max(mlo - m0, 0), hi = min(mlo + n - m0, VW);
  T* out = fb + c * __ldg(rsf + Nf + 2) + row_base(rsf, Nf, j, k) + m0;
  T v[VW];
  Vec<T>::template load<false>(out, v);
  const int CSc = __ldg(rsc + Nc + 2);
  const int code = (ic & 1) | ((j & 1) << 1) | ((k & 1) << 2);
  int di = 0, dj = 0, dk = 0;
  if (code) edge_dir(code, di, dj, dk);
  const int JA = (j - dj) >> 1, KA = (k - dk) >> 1, ia = (ic - di) >> 1;
  const int JB = (j + dj) >> 1, KB = (k + dk) >> 1, ib = (ic + di) >> 1;
  const int rba = row_base(rsc, Nc, JA, KA), rbb = row_base(rsc, Nc, JB, KB);
  const int ca = ia + 2 * JA + 3 * KA, cbb = ib + 2 * JB + 3 * KB;
#pragma unroll
  for (int q = 0; q < VW; ++q) {
    if (q < lo || q >= hi) continue;
    const int two_m = 2 * (m0 + q);
    const int oa = ((ca + two_m) & 3) * CSc + rba + ((two_m + ia) >> 2);
    const T a = NC ? __ldg(cb + oa) : cb[oa];
    if (code == 0) {
      v[q] += a;
    } else {
      const int ob = ((cbb + two_m) & 3) * CSc + rbb + ((two_m + ib) >> 2);
      const T b = NC ? __ldg(cb + ob) : cb[ob];
      v[q] = fma(T(0.5), a + b, v[q]);   // the halving is exact: same value as a separate multiply
    }
  }
  store_lanes(out, v, lo, hi);
}

// Volume prolongation of a fine tile: FP64 one item per slot (four nodes,
// all colours), FP32 colour by colour in 16-byte vectors (measured faster for
// each precision); colour skip left out (-1: none).
template <class T, bool NC>
__device__ __forceinline__ void prolong_tile(const Tile& t, int Nf, const int* __restrict__ rsf, int Nc,
                                             const int* __restrict__ rsc, T* __restrict__ fb, const T* __restrict__ cb,
                                             int skip, int (*s_pre2)[33], int* s_pre_tot) {
  if constexpr (std::is_same<T, float>::value) {
    constexpr int VW = Vec<T>::n;
    for (int c = 0; c < 4; ++c) {
      if (c == skip) continue;
      const int total = flat_setup_slabs(t, Nf, c, true, VW, s_pre2, s_pre_tot);
      int sl = 0;
      for (int tt = tid256(); tt < total; tt += CTA) {
        while (tt >= s_pre_tot[sl + 1]) ++sl;
        const int k = t.k + sl;
        const Tile ts{k, t.j0, t.m0, 1};
        int j, g;
        flat_item(ts, Nf, c, true, s_pre2[sl], tt - s_pre_tot[sl], j, g, VW);
        prolong_group<T, NC>(Nf, rsf, Nc, rsc, j, k, g, c, fb, cb);
      }
      __syncthreads();
    }
  } else {
    for_tile_slots(t, Nf, s_pre2, s_pre_tot, [&](int j, int k, int m) {
      prolong_slot<T, NC>(Nf, rsf, Nc, rsc, j, k, m, fb, cb, skip);
    });
  }
}

template <class T, bool DEP>
__global__ void __launch_bounds__(CTA) k_prolong(int Nf, const int* __restrict__ rsf, int64_t bf, T* uf, T* uIf,
                                                 int Nc, const int* __restrict__ rsc, int64_t bc, const T* uc,
                                                 const Tile* __restrict__ tiles, int n_tiles,
                                                 const int* __restrict__ act, int n_act, const int* __restrict__ cptr,
                                                 const Copy* __restrict__ cps, const uint32_t* __restrict__ cpo,
                                                 const int* __restrict__ list,
                                                 int n_list, int n_if_units, int* sched, int skip,
                                                 int if_lo, int if_hi) {
  if (DEP) launch_next();
  if (DEP) after_previous();
  __shared__ int s_pre2[MAX_SLABS][33];
  __shared__ int s_pre_tot[MAX_SLABS + 1];
  __shared__ int s_unit;
  HHG_UNITS_DYN(n_if_units, n_tiles, n_act, sched, &s_unit) {
    if (const int ic_ = if_chunk(unit, n_if_units); ic_ >= 0) {
      const int q = ic_ * CTA + tid256();
      if (q < n_list && (q < if_lo || q >= if_hi)) {
        const int node = list[q];
        const int c0 = cptr[node], c1 = cptr[node + 1];
        const Copy cp = cps[c0];
        const T val = uIf[node] + interp(uc + (size_t)cp.macro * bc, Nc, rsc, cp.i, cp.j, cp.k);
        uIf[node] = val;
        write_copies(Nf, rsf, bf, uf, cps, cpo, c0, c1, val);
      }
      continue;
    }
    Tile t;
    int macro;
    vol_unit(vol_index(unit, n_if_units), n_act, tiles, act, t, macro);
    prolong_tile<T, !DEP>(t, Nf, rsf, Nc, rsc, uf + (size_t)macro * bf, uc + (size_t)macro * bc, skip, s_pre2,
                          s_pre_tot);
  }
  finish_units(sched, n_if_units + n_tiles * n_act);
}

// Flat transfers (levels on the flat kernels): one thread per item, no tiles
// and no CTA barrier, CTAs of interface nodes spread among the volume CTAs.
// The restriction takes the coarse level's slot items (four coarse nodes of
// one row per thread, restrict_slot); the prolongation takes the fine level's
// Gauss-Seidel items of the colours it updates (one 16-byte vector of
// same-colour fine nodes per thread, prolong_group).  Same arithmetic per
// node as k_restrict / k_prolong, so the same values bit for bit.
template <class T, bool DEP>
__global__ void __launch_bounds__(CTA) k_restrict_flat(int Nc, const int* __restrict__ rsc, int64_t bc,
                                                       T* fc, T* fIc, T* uc,
                                                       T* uIc, int Nf, const int* __restrict__ rsf,
                                                       int64_t bf, const T* rf,
                                                       const uint32_t* __restrict__ slots, int n_slots,
                                                       const int* __restrict__ act, int n_act,
                                                       const int* __restrict__ cptr, const Copy* __restrict__ cps,
                                                       const uint32_t* __restrict__ cpo, const int* __restrict__ list,
                                                       int n_list, const int64_t* __restrict__ gather,
                                                       const int64_t* __restrict__ zero_off, int n_zero,
                                                       int n_if_ctas, int n_vol_ctas) {
  if (DEP) launch_next();
  int vb = 0;
  const int ib = spread_position((int)blockIdx.x, n_if_ctas, n_vol_ctas, vb);
  if (ib >= 0) {
    if (DEP) after_previous();
    const int q = ib * CTA + tid256();
    if (q < n_list) {
      const int node = list[q];
      const int64_t* g = gather + (size_t)q * NDIR;
      T acc = T(0);
      for (int e = 1; e < NDIR; ++e) {
        const int64_t o = g[e];
        if (o >= 0) acc += rf[o];
      }
      fIc[node] = rf[g[0]] + T(0.5) * acc;
      uIc[node] = T(0);
      write_copies(Nc, rsc, bc, uc, cps, cpo, cptr[node], cptr[node + 1], T(0));
    } else if (q < n_list + n_zero) {
      uc[zero_off[q - n_list]] = T(0);
    }
    return;
  }
  const int v = vb * CTA + tid256();
  if (v >= n_slots * n_act) return;
  const int a = v / n_slots, it = v - a * n_slots;
  const int macro = act[a];
  const uint32_t d = slots[it];
  if (DEP) after_previous();
  restrict_slot<T, !DEP>(Nc, rsc, Nf, rsf, (int)(d >> 20), (int)((d >> 10) & 1023u), (int)(d & 1023u),
                         rf + (size_t)macro * bf, fc + (size_t)macro * bc, uc + (size_t)macro * bc);
}

// items / n_items: the fine level's Gauss-Seidel items of colours first_c ..
// 3 (colour-major, from off[first_c] on); off holds the starts of the later
// colours relative to that (n_items where there is none), to find an item's
// colour.
template <class T, bool DEP>
__global__ void __launch_bounds__(CTA) k_prolong_flat(int Nf, const int* __restrict__ rsf, int64_t bf,
                                                      T* uf, T* uIf, int Nc,
                                                      const int* __restrict__ rsc, int64_t bc,
                                                      const T* uc, const uint32_t* __restrict__ items,
                                                      int n_items, int first_c, int3 off,
                                                      const int* __restrict__ act, int n_act,
                                                      const int* __restrict__ cptr, const Copy* __restrict__ cps,
                                                      const uint32_t* __restrict__ cpo,
                                                      const int* __restrict__ list, int n_list, int if_lo, int if_hi,
                                                      int n_if_ctas, int n_vol_ctas) {
  if (DEP) launch_next();
  int vb = 0;
  const int ib = spread_position((int)blockIdx.x, n_if_ctas, n_vol_ctas, vb);
  if (ib >= 0) {
    if (DEP) after_previous();
    const int q = ib * CTA + tid256();
    if (q < n_list && (q < if_lo || q >= if_hi)) {
      const int node = list[q];
      const int c0 = cptr[node], c1 = cptr[node + 1];
      const Copy cp = cps[c0];
      const T val = uIf[node] + interp(uc + (size_t)cp.macro * bc, Nc, rsc, cp.i, cp.j, cp.k);
      uIf[node] = val;
      write_copies(Nf, rsf, bf, uf, cps, cpo, c0, c1, val);
    }
    return;
  }
  const int v = vb * CTA + tid256();
  if (v >= n_items * n_act) return;
  const int a = v / n_items, it = v - a * n_items;
  const int c = first_c + (it >= off.x) + (it >= off.y) + (it >= off.z);
  const int macro = act[a];
  const uint32_t d = items[it];
  if (DEP) after_previous();
  prolong_group<T, !DEP>(Nf, rsf, Nc, rsc, (int)(d >> 20), (int)((d >> 10) & 1023u), (int)(d & 1023u), c,
                         uf + (size_t)macro * bf, uc + (size_t)macro * bc);
}

// ---------------------------------------------------------------------------
// Mixed precision: FP64 residual handed to the FP32 cycle as its right-hand
// side (with partial sums of r^2), and the FP64 update u += e
// ---------------------------------------------------------------------------
template <bool S7>
__device__ __forceinline__ void res_f32_tile(const Tile& t, int N, const int* __restrict__ rs,
                                             const double* __restrict__ ub, const double* __restrict__ fb,
                                             float* __restrict__ ob, const double* __restrict__ w, double& ss,
                                             int (*s_pre2)[33], int* s_pre_tot) {
  HHG_TILE_NODES(N, rs, t, s_pre, {
    int me;
    double acc;
    if (S7) {
      const Nb7 q = nb7(sc, i, j);
      me = q.me;
      acc = fb[me] - w[0] * ub[me];
      acc -= w[1] * ub[q.nb1];
      acc -= w[2] * ub[q.nb2];
      acc -= w[3] * ub[q.nb3];
      acc -= w[8] * ub[q.nb8];
      acc -= w[9] * ub[q.nb9];
      acc -= w[10] * ub[q.nb10];
    } else {
      me = lidx32(rs, N, i, j, k);
      acc = fb[me] - w[0] * ub[me];
_Pragma("unroll")
      for (int d = 1; d < NDIR; ++d) {
        int di, dj, dk;
        dir_ijk(d, di, dj, dk);
        acc -= w[d] * ub[lidx32(rs, N, i + di, j + dj, k + dk)];
      }
    }
    ob[me] = (float)acc;
    ss += acc * acc;
  })
}

template <bool S7>
__global__ void __launch_bounds__(CTA) k_res_f32(int N, const int* __restrict__ rs, int64_t block, const double* u,
                                                 const double* uI, const double* f,
                                                 const double* fI, float* f32,
                                                 float* fI32, const double* __restrict__ W,
                                                 const Tile* __restrict__ tiles, int n_tiles,
                                                 const int* __restrict__ act, int n_act,
                                                 const int* __restrict__ cptr, const Copy* __restrict__ cps,
                                                 const int* __restrict__ list, int n_list, IfTab<double> tab,
                                                 int n_if_units, double* partial,
                                                 int* sched) {
  launch_next();
  after_previous();
  __shared__ int s_pre2[MAX_SLABS][33];
  __shared__ int s_pre_tot[MAX_SLABS + 1];
  __shared__ double sh[32];
  double ss = 0.0;
  __shared__ int s_unit;
  HHG_UNITS_DYN(n_if_units, n_tiles, n_act, sched, &s_unit) {
    int vol_ = 0;
    if (const int ic_ = spread_unit(unit, n_if_units, n_tiles * n_act, vol_); ic_ >= 0) {
      const int q = ic_ * CTA + tid256();
      if (q < n_list) {
        const int node = list[q];
        double res;
        if (tab.nb) {
          res = fI[node] - tab.diag[q] * uI[node] - if_offdiag<double, if_tab_k(S7)>(tab, u, q);
        } else {
          double off = 0.0, diag = 0.0;
          if_stencil<double, S7>(N, rs, block, u, W, cps, cptr[node], cptr[node + 1], off, diag);
          res = fI[node] - diag * uI[node] - off;
        }
        fI32[node] = (float)res;
        ss += res * res;
      }
      continue;
    }
    Tile t;
    int macro;
    vol_unit(vol_, n_act, tiles, act, t, macro);
    const double* ub = u + (size_t)macro * block;
    const double* fb = f + (size_t)macro * block;
    float* ob = f32 + (size_t)macro * block;
    const double* w = W + (size_t)macro * 16 * NDIR;
    res_f32_tile<S7>(t, N, rs, ub, fb, ob, w, ss, s_pre2, s_pre_tot);
  }
  finish_units(sched, n_if_units + n_tiles * n_act);
  const double s = block_sum(ss, sh);
  if (threadIdx.x == 0 && threadIdx.y == 0) partial[blockIdx.x] = s;
}

// u64 += e32 over whole active blocks, two slots per thread and step: the
// FP32 correction is zero at every slot the cycle does not own (Dirichlet and
// frozen copies, padding; the blocks are cleared before the cycle), and each
// ghost copy of a free interface node holds the master's correction, so the
// copies stay equal to their masters.  Blocks are multiples of 256 slots.
__device__ __forceinline__ void add_corr(double2* __restrict__ ub, const float2* __restrict__ eb, int64_t n) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
    double2 x = ub[q];
    const float2 d = eb[q];
    x.x += (double)d.x;
    x.y += (double)d.y;
    ub[q] = x;
  }
}
__global__ void __launch_bounds__(256) k_add_corr_blocks(double* u, const float* e, int64_t block,
                                                        const int* __restrict__ act) {
  launch_next();
  after_previous();
  const size_t base = (size_t)act[blockIdx.y] * block;
  add_corr(reinterpret_cast<double2*>(u + base), reinterpret_cast<const float2*>(e + base), block / 2);
}

// uI[list[q]] += eI[list[q]] for the free interface masters.
__global__ void k_add_corr_masters(double* uI, const float* eI, const int* __restrict__ list,
                                   int n) {
  launch_next();
  after_previous();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) {
    const int node = list[q];
    uI[node] += (double)eI[node];
  }
}

// ---------------------------------------------------------------------------
// Coarse-level CG, one CTA (FP64; §2.1 coarse solver)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double cta_sum(double v, double* sh) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    // only the first blockDim.x / 32 entries were written
    double s = threadIdx.x < (blockDim.x + 31) / 32 ? sh[threadIdx.x] : 0.0;
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) sh[32] = s;
  }
  __syncthreads();
  return sh[32];
}

constexpr int CG_THREADS = 256;
constexpr int CG_WARPS = CG_THREADS / 32;

// Sum over the warp, the same bits in every lane: both partners of a step add
// the same two rounded values (__dadd_rn keeps the compiler from fusing a
// lane's own product into its first add).
__device__ __forceinline__ double warp_sum_xor(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// The CG's sums have one order whatever the launch: rows in blocks of 32 (or
// 128, see cg_block_shift), a block summed by the shuffle tree above (missing
// rows count 0), block b added
// to bucket b mod 32 in ascending order, the 32 buckets summed by the same
// tree.  So the one-CTA form below (also run by the persistent batch executor
// and the allocation-free cycle) and the cluster form give the same iterates
// bit for bit.
//
// One CTA of CG_THREADS threads: warp w takes the blocks w, w + 8, ..., four
// at a time.  Their four trees run as one: after the step over 16 lanes each
// half of the warp holds two of them, after the step over 8 each quarter one,
// so four blocks cost six additions instead of twenty (one CTA is bound by the
// FP64 pipe, 2 lanes a clock and about 17 operations a row and iteration: a
// cycle of 4x4x4 sub-cubes refined 3 times, 3375 coarse rows, takes 3.45 ms in
// the executor, 4.45 with a tree per block).  Quarter e of the warp ends with block
// e's sum, the same bits as warp_sum_xor, and holds bucket w + 8 e.
__device__ __forceinline__ double warp_sum4(const double (&v)[4]) {
  const bool h16 = (threadIdx.x & 16) != 0, h8 = (threadIdx.x & 8) != 0;
  const double a = __dadd_rn(h16 ? v[2] : v[0], __shfl_xor_sync(0xffffffffu, h16 ? v[0] : v[2], 16));
  const double b = __dadd_rn(h16 ? v[3] : v[1], __shfl_xor_sync(0xffffffffu, h16 ? v[1] : v[3], 16));
  double s = __dadd_rn(h8 ? b : a, __shfl_xor_sync(0xffffffffu, h8 ? a : b, 8));
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) s = __dadd_rn(s, __shfl_xor_sync(0xffffffffu, s, o));
  return s;
}

// Rows per lane of a block (as a shift): from 16385 rows on a block has 128
// rows, lane l's rows l, l + 32, l + 64, l + 96 being added first, which
// leaves a quarter of the tree's operations.
__host__ __device__ __forceinline__ int cg_block_shift(int n) { return n > 16384 ? 2 : 0; }

// Calls body(q) -> double for the rows q of the warp's blocks and returns the
// sum over all rows (to every thread).  buf: 32 doubles; consecutive sums
// alternate between two buffers.
template <class F>
__device__ __forceinline__ double cg_rows_sum(int n, double* buf, F&& body) {
  const int t = threadIdx.y * blockDim.x + threadIdx.x;   // 1-D or (32, 8) CTAs
  const int lane = t & 31, w = t >> 5;
  const int sh = cg_block_shift(n);
  const int nb = ((n - 1) >> (5 + sh)) + 1;
  double acc = 0.0;
  for (int b0 = w; b0 < nb; b0 += 32) {
    double v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int b = b0 + CG_WARPS * e;
      v[e] = 0.0;
      for (int g = 0; b < nb && g < 1 << sh; ++g) {
        const int q = ((b << sh) + g) * 32 + lane;
        if (q < n) v[e] = g ? __dadd_rn(v[e], body(q)) : body(q);
      }
    }
    acc += warp_sum4(v);
  }
  if ((lane & 7) == 0) buf[w + CG_WARPS * (lane >> 3)] = acc;
  __syncthreads();
  return warp_sum_xor(buf[lane]);
}

// CG on the compact free nodes of the coarsest level from x = 0 until
// ||r|| <= rtol ||b|| or maxit iterations, with z = r, or, given the
// reciprocal diagonal, z = r / diag (Jacobi preconditioning; below r.r stands
// for r.z, the stopping test keeps r.r).  The direction's image s = A p is
// carried along, s <- A r + beta s, so that the product A r does not wait for
// beta.  One iteration: p.s, alpha = r.r / p.s, x += alpha p, r -= alpha s,
// r.r, beta = r.r / old r.r (the reciprocal formed beside the critical path), p <- r + beta p, s <- A r + beta s.  A row's product is summed in two
// chains, even and odd entries.
//
// One CTA of CG_THREADS threads; x, r, p and s live in global memory (4 n
// doubles); a row belongs to one thread throughout.  dinv: the
// reciprocal diagonal, or null.  red: 64 doubles of shared memory.
template <class T>
__device__ __forceinline__ void cg_one_cta(int n, const int* rowptr, const int* col, const double* val,
                                           const int64_t* fsrc, const T* f, const T* fI, const int* uptr,
                                           const int64_t* udst, const int* umaster, T* u, T* uI, double* x, double* r,
                                           double* p, double* s, const double* dinv, double rtol, int maxit,
                                           int* iters, double* red) {
  const int t = threadIdx.y * blockDim.x + threadIdx.x;
  auto z = [&](int q) { return dinv ? dinv[q] * r[q] : r[q]; };
  auto row_times = [&](int q) {   // entries four at a time, their loads together
    double a0 = 0.0, a1 = 0.0;
    const int e0 = rowptr[q], e1 = rowptr[q + 1];
    for (int e = e0; e < e1; e += 4) {
      double zv[4], wv[4];
#pragma unroll
      for (int x = 0; x < 4; ++x) {
        const int at = e + x < e1 ? e + x : e;
        wv[x] = val[at];
        zv[x] = z(col[at]);
      }
      a0 = fma(wv[0], zv[0], a0);
      if (e + 1 < e1) a1 = fma(wv[1], zv[1], a1);
      if (e + 2 < e1) a0 = fma(wv[2], zv[2], a0);
      if (e + 3 < e1) a1 = fma(wv[3], zv[3], a1);
    }
    return a0 + a1;
  };
  auto squares = [&]() { return cg_rows_sum(n, red + 32, [&](int q) { return r[q] * r[q]; }); };
  double rz = cg_rows_sum(n, red, [&](int q) {
    const int64_t src = fsrc[q];
    const double b = src >= 0 ? (double)f[src] : (double)fI[-1 - src];
    x[q] = p[q] = s[q] = 0.0;
    r[q] = b;
    return b * z(q);
  });
  double rr = dinv ? squares() : rz;
  double back = 1.0;
  if (!cg_in_range(rr)) {   // cg_shift
    uint32_t m = 0;
    for (int q = t; q < n; q += CG_THREADS) m = max(m, cg_exponent(r[q]));
    m = __reduce_max_sync(0xffffffffu, m);
    __syncthreads();   // the totals have been read
    if ((t & 31) == 0) red[t >> 5] = (double)m;
    __syncthreads();
    for (int w = 0; w < CG_WARPS; ++w) m = max(m, (uint32_t)red[w]);
    const double up = cg_shift(m);
    back = 1.0 / up;
    for (int q = t; q < n; q += CG_THREADS) r[q] *= up;
    __syncthreads();
    rz = cg_rows_sum(n, red, [&](int q) { return r[q] * z(q); });
    rr = dinv ? squares() : rz;
  }
  const double bnorm = sqrt(rr);
  const CgTest test = cg_test(rtol * bnorm);
  int it = 0;
  double beta = 0.0;
  while (bnorm > 0.0 && it < maxit && cg_above(rr, test)) {
    __syncthreads();   // every r entry is written, every total read
    const double pAp = cg_rows_sum(n, red + 32, [&](int q) {
      const double p0 = p[q], s0 = s[q], zq = z(q);   // zero in the first iteration, as beta
      const double w = row_times(q);
      const double pq = fma(beta, p0, zq);
      const double sq = fma(beta, s0, w);
      p[q] = pq;
      s[q] = sq;
      return pq * sq;
    });
    const double alpha = rz * cg_recip(pAp);
    const double inv = cg_recip(rz);
    const double rz_new = cg_rows_sum(n, red, [&](int q) {
      x[q] = fma(alpha, p[q], x[q]);
      r[q] = fma(-alpha, s[q], r[q]);
      return r[q] * z(q);
    });
    rr = rz_new;
    if (dinv) {
      __syncthreads();   // the last total has been read
      rr = squares();
    }
    beta = rz_new * inv;
    rz = rz_new;
    ++it;
  }
  for (int q = t; q < n; q += CG_THREADS) {
    const T v = (T)(x[q] * back);
    for (int e = uptr[q]; e < uptr[q + 1]; ++e) u[udst[e]] = v;
    if (umaster[q] >= 0) uI[umaster[q]] = v;
  }
  if (t == 0 && iters) *iters = it;
}

template <class T>
__global__ void __launch_bounds__(CG_THREADS) k_cg(int n, const int* __restrict__ rowptr, const int* __restrict__ col,
                                                   const double* __restrict__ val, const int64_t* __restrict__ fsrc,
                                                   const T* f, const T* fI,
                                                   const int* __restrict__ uptr, const int64_t* __restrict__ udst,
                                                   const int* __restrict__ umaster, T* u,
                                                   T* uI, double* work,
                                                   const double* __restrict__ dinv, double rtol, int maxit,
                                                   int* iters) {
  launch_next();
  after_previous();
  __shared__ double red[64];
  cg_one_cta<T>(n, rowptr, col, val, fsrc, f, fI, uptr, udst, umaster, u, uI, work, work + n, work + 2 * (size_t)n,
                work + 3 * (size_t)n, dinv, rtol, maxit, iters, red);
}

// --- the same CG on a thread-block cluster --------------------------------
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_map(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ double cluster_load(uint32_t addr) {
  double v;
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(addr));   // ordered by the barriers' asm
  return v;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(addr), "d"(v) : "memory");
}
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\nbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Row block b belongs to CTA b mod C (C CTAs, a power of two), there to block
// b / C: warp (b / C) mod W of its W row warps; one more warp forms the totals
// and the scalars.  Shared memory of a CTA: its rows' r, the block sums of
// both reductions (every CTA holds all of them: a warp that has summed a block
// writes the sum to the C CTAs, one lane each), and its matrix rows, K entries
// each, entry-major: weight and cluster address of the r entry.  Per iteration
// two cluster barriers: after p.s, and after r and r.r.  Every CTA takes the
// same decisions from the same bits, so all leave the loop together; the
// decision to stop is formed by the scalar warp during the next p.s and read
// after its barrier.
//
// What bounds it is latency: two shuffle trees (86 clocks a step), two totals,
// a reciprocal and two cluster barriers (370 clocks) in one chain of about 2.5
// us per iteration.  Beyond about 60 rows per SM the FP64 pipe (2 lanes a
// clock): a row costs about 20 operations with its share of the trees.
// Measured per solve to 1e-12, one 256-thread CTA with the CSR matrix in
// global memory before -> now: 343 rows 187 -> 92 us, 1331 rows 960 -> 183 us,
// 3375 rows with lognormal coefficients 9025 -> 1065 us, 250047 rows 820 -> 32 ms.
struct CgArgs {
  int n, K, maxit, blocks_per_cta;
  const int *rowptr, *col;
  const double* val;
  const int64_t* fsrc;
  const int* uptr;
  const int64_t* udst;
  const int* umaster;
  const double* dinv;   // null, or the reciprocal diagonal (NB > 0)
  double rtol;
  int* iters;
  double* work;   // 4 n doubles (NB = 0)
};

// Sum of the nb block sums in the order stated above, to every lane.  With at
// most 16 blocks the tree's upper steps would only add zeros: the lanes hold
// copies of the smallest power of two of buckets and skip them.
__device__ __forceinline__ double cg_total(const double* sums, int nb) {
  const int m = nb > 16 ? 32 : nb > 8 ? 16 : nb > 4 ? 8 : nb > 2 ? 4 : nb > 1 ? 2 : 1;
  double v = 0.0;
  for (int b = threadIdx.x & (m - 1); b < nb; b += 32) v += sums[b];
  if (nb > 16) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 16));
  if (nb > 8) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 8));
  if (nb > 4) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 4));
  if (nb > 2) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 2));
  if (nb > 1) v = __dadd_rn(v, __shfl_xor_sync(0xffffffffu, v, 1));
  return v;
}

// NB > 0: row blocks per warp at most, the vectors in registers; KC > 0 (NB = 1
// only): rows of at most KC entries, held in registers too, else K entries per
// row in shared memory.  NB = 0 (large coarse problems): any number of blocks,
// x, p, s and A r in the work array and the matrix read from its CSR arrays.
template <class T, int NB, int KC, bool JAC>
__global__ void __launch_bounds__(NB > 0 ? CG_THREADS + 32 : 1024) k_cg_cluster(CgArgs A, const T* f,
                                                                const T* fI, T* u,
                                                                T* uI) {
  launch_next();
  extern __shared__ double s_cg[];
  __shared__ double s_alpha, s_beta;
  __shared__ int s_go;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, W = (blockDim.x >> 5) - 1;
  uint32_t C;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(C));
  const uint32_t rank = cluster_rank();
  const bool solo = C == 1;
  auto barrier = [&]() {
    if (solo) __syncthreads();
    else cluster_barrier();
  };
  const int sh = NB > 0 ? 0 : cg_block_shift(A.n);
  const int nb = ((A.n - 1) >> (5 + sh)) + 1, rows = A.blocks_per_cta << (5 + sh), K = A.K;
  double* sr = s_cg;
  double* sum0 = sr + rows;
  double* sum1 = sum0 + nb;
  constexpr bool jac = NB > 0 && JAC;
  double* sum2 = sum1 + nb;   // r.r beside r.z
  double* mv = sum2 + (jac ? nb : 0);
  uint32_t* ma = reinterpret_cast<uint32_t*>(mv + (size_t)K * rows);
  const bool scalar = warp == W;
  const uint32_t r_addr = smem_addr(sr);
  const uint32_t peer0 = cluster_map(smem_addr(sum0), lane % C), peer1 = cluster_map(smem_addr(sum1), lane % C),
                 peer2 = cluster_map(smem_addr(sum2), lane % C);
  constexpr int NR = NB > 0 ? NB : 1;
  const int ni = NB > 0 ? NB : (A.blocks_per_cta + W - 1) / W;
  double xr[NR], rr_[NR], pr[NR], srow[NR], wr[NR], dr[NR];
  double rv[KC > 0 ? KC : 1];
  uint32_t ra[KC > 0 ? KC : 1];
  // the warp's i-th block: local block warp + i W, global block that * C +
  // rank; its g-th row of this lane
  auto mine = [&](int i) { return !scalar && warp + i * W < A.blocks_per_cta; };
  auto slot = [&](int i, int g) { return (((warp + i * W) << sh) + g) * 32 + lane; };
  auto row_of = [&](int i, int g) {
    const int q = ((((warp + i * W) * (int)C + (int)rank) << sh) + g) * 32 + lane;
    return mine(i) && q < A.n ? q : -1;
  };
  auto addr_of = [&](int c) {   // cluster address of row c's r entry
    const uint32_t b = (uint32_t)c >> (5 + sh), in = (uint32_t)c & ((32u << sh) - 1);
    return cluster_map(r_addr + (((b / C) << (5 + sh)) + in) * 8, b % C);
  };
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    xr[i] = rr_[i] = pr[i] = srow[i] = wr[i] = 0.0;
    dr[i] = 1.0;
    if (!mine(i)) continue;
    const int q = row_of(i, 0), o = slot(i, 0);
    if (jac && q >= 0) dr[i] = A.dinv[q];
    const int e0 = q >= 0 ? A.rowptr[q] : 0, e1 = q >= 0 ? A.rowptr[q + 1] : 0;
    auto entry = [&](int e, double& v, uint32_t& addr) {
      const bool in = e0 + e < e1;
      const int c = in ? __ldg(A.col + e0 + e) : 0;
      v = in ? __ldg(A.val + e0 + e) : 0.0;
      addr = in ? addr_of(c) : cluster_map(r_addr + (uint32_t)o * 8, rank);   // padding: weight 0 on the row's own entry
    };
    if (KC > 0) {
#pragma unroll
      for (int e = 0; e < KC; ++e) entry(e, rv[e], ra[e]);
    } else {
#pragma unroll 4
      for (int e = 0; e < K; ++e) entry(e, mv[(size_t)e * rows + o], ma[(size_t)e * rows + o]);
    }
  }
  auto times = [&](int i, int q) {   // (A r) of the row
    double a0 = 0.0, a1 = 0.0;
    if (NB == 0) {
      const int e1 = q >= 0 ? __ldg(A.rowptr + q + 1) : 0;
      for (int e = q >= 0 ? __ldg(A.rowptr + q) : 0; e < e1; e += 2) {
        a0 = fma(__ldg(A.val + e), cluster_load(addr_of(__ldg(A.col + e))), a0);
        if (e + 1 < e1) a1 = fma(__ldg(A.val + e + 1), cluster_load(addr_of(__ldg(A.col + e + 1))), a1);
      }
    } else if (KC > 0) {
      double v[KC > 0 ? KC : 1];
#pragma unroll
      for (int e = 0; e < KC; ++e) v[e] = cluster_load(ra[e]);
#pragma unroll
      for (int e = 0; e < KC; e += 2) {
        a0 = fma(rv[e], v[e], a0);
        if (e + 1 < KC) a1 = fma(rv[e + 1], v[e + 1], a1);
      }
    } else {
      const int o = slot(i, 0);
#pragma unroll 4
      for (int e = 0; e < K; e += 2) {
        a0 = fma(mv[(size_t)e * rows + o], cluster_load(ma[(size_t)e * rows + o]), a0);
        if (e + 1 < K) a1 = fma(mv[(size_t)(e + 1) * rows + o], cluster_load(ma[(size_t)(e + 1) * rows + o]), a1);
      }
    }
    return a0 + a1;
  };
  // Calls body(i, g, q) for the rows of the warp's blocks.
  auto each = [&](auto&& body) {
    if (scalar) return;
    if constexpr (NB > 0) {
#pragma unroll
      for (int i = 0; i < NB; ++i)
        if (mine(i)) body(i, 0, row_of(i, 0));
    } else {
      for (int i = 0; i < ni; ++i)
        for (int g = 0; mine(i) && g < 1 << sh; ++g) body(i, g, row_of(i, g));
    }
  };
  // The same with the blocks' sums of body's values written to every CTA.
  auto each_sum = [&](uint32_t peer, auto&& body) {
    if (scalar) return;
#pragma unroll
    for (int i = 0; i < ni; ++i) {
      if (!mine(i)) continue;
      double v = body(i, 0, row_of(i, 0));
      if constexpr (NB == 0)
        for (int g = 1; g < 1 << sh; ++g) v = __dadd_rn(v, body(i, g, row_of(i, g)));
      const int b = (warp + i * W) * (int)C + (int)rank;
      const double sb = warp_sum_xor(v);
      if (b < nb && lane < (int)C) cluster_store(peer + (uint32_t)b * 8, sb);
    }
  };
  auto z = [&](int i, double r) { return jac ? dr[i] * r : r; };
  // r.r of the warp's rows, to every CTA
  auto squares = [&]() {
    if (jac) each_sum(peer2, [&](int i, int, int) { return rr_[i] * rr_[i]; });
  };
  double* gx = A.work;
  double* gp = gx + (NB > 0 ? 0 : (size_t)A.n);
  double* gs = gp + (NB > 0 ? 0 : (size_t)A.n);
  double* gw = gs + (NB > 0 ? 0 : (size_t)A.n);
  after_previous();
  barrier();   // every CTA of the cluster runs before its memory is written
  double up = 1.0;   // cg_shift; all CTAs decide alike
  for (bool first = true;; first = false) {
    each_sum(peer0, [&](int i, int g, int q) {
      double v = 0.0;
      if (q >= 0) {
        const int64_t src = A.fsrc[q];
        v = up * (src >= 0 ? (double)f[src] : (double)fI[-1 - src]);
        if (NB == 0) gx[q] = 0.0;
      }
      if (NB > 0) rr_[i] = v;
      const double zv = z(i, v);
      sr[slot(i, g)] = zv;
      return v * zv;
    });
    squares();
    barrier();   // b.b summed; every r entry written
    if (!first || cg_in_range(cg_total(jac ? sum2 : sum0, nb))) break;
#pragma unroll
    for (int i = 0; i < ni; ++i) {
      if (!mine(i)) continue;
      uint32_t m = NB > 0 ? cg_exponent(rr_[NB > 0 ? i : 0]) : 0;
      if constexpr (NB == 0)
        for (int g = 0; g < 1 << sh; ++g) m = max(m, cg_exponent(sr[slot(i, g)]));
      m = __reduce_max_sync(0xffffffffu, m);
      const int b = (warp + i * W) * (int)C + (int)rank;
      if (b < nb && lane < (int)C) cluster_store(peer1 + (uint32_t)b * 8, (double)m);
    }
    barrier();   // the blocks' exponents are written, the sums have been read
    uint32_t m = 0;
    for (int b = lane; b < nb; b += 32) m = max(m, (uint32_t)sum1[b]);
    up = cg_shift(__reduce_max_sync(0xffffffffu, m));
  }
  double rz = 0.0, rr = 0.0, inv = 0.0;   // scalar warp
  CgTest test{0.0, 0, 0};
  bool any = false;
  int it = 0;
  for (;;) {
    // r and r.r are complete: A r by the row warps, the scalars beside it
    if (scalar) {
      rz = cg_total(sum0, nb);
      if (lane == 0) s_beta = rz * inv;
    }
    each([&](int i, int, int q) {
      const double w = times(i, q);
      if (NB > 0) wr[i] = w;
      else if (q >= 0) gw[q] = w;
    });
    __syncthreads();
    if (scalar) {
      rr = jac ? cg_total(sum2, nb) : rz;
      if (it == 0) {
        const double bnorm = sqrt(rr);
        any = bnorm > 0.0;
        test = cg_test(A.rtol * bnorm);
      }
      const bool go = any && it < A.maxit && cg_above(rr, test);
      if (lane == 0) s_go = go;
      inv = cg_recip(rz);
    }
    const double beta = s_beta;
    each_sum(peer1, [&](int i, int g, int q) {
      double pq = 0.0, sq = 0.0;
      if (NB > 0) {
        const double zv = z(i, rr_[i]);
        pr[i] = pq = it ? fma(beta, pr[i], zv) : zv;
        srow[i] = sq = it ? fma(beta, srow[i], wr[i]) : wr[i];
      } else if (q >= 0) {
        const double r = sr[slot(i, g)], w = gw[q];
        gp[q] = pq = it ? fma(beta, gp[q], r) : r;
        gs[q] = sq = it ? fma(beta, gs[q], w) : w;
      }
      return pq * sq;
    });
    barrier();   // p.s summed; every read of r done; s_go written
    if (!s_go) break;
    if (scalar) {
      const double al = rz * cg_recip(cg_total(sum1, nb));
      if (lane == 0) s_alpha = al;
    }
    __syncthreads();
    const double alpha = s_alpha;
    each_sum(peer0, [&](int i, int g, int q) {
      double r = 0.0;
      if (NB > 0) {
        xr[i] = fma(alpha, pr[i], xr[i]);
        rr_[i] = r = fma(-alpha, srow[i], rr_[i]);
      } else if (q >= 0) {
        gx[q] = fma(alpha, gp[q], gx[q]);
        r = fma(-alpha, gs[q], sr[slot(i, g)]);
      }
      const double zv = z(i, r);
      sr[slot(i, g)] = zv;
      return r * zv;
    });
    squares();
    ++it;
    barrier();   // r.r summed; every r entry written
  }
  const double back = 1.0 / up;
  each([&](int i, int, int q) {
    if (q < 0) return;
    const T v = (T)((NB > 0 ? xr[i] : gx[q]) * back);
    for (int e = A.uptr[q]; e < A.uptr[q + 1]; ++e) u[A.udst[e]] = v;
    if (A.umaster[q] >= 0) uI[A.umaster[q]] = v;
  });
  if (rank == 0 && threadIdx.x == 0 && A.iters) *A.iters = it;
}

// Coefficient gradient (per macro, closed lattice): sum of lam_p times the
// macro's own sub-stencil at p applied to u, i.e. lam^T (A_T u) up to the
// factor k_T.
__global__ void __launch_bounds__(CTA) k_grad(int N, const int* __restrict__ rs, int64_t block,
                                              const double* u, const double* lam,
                                              const double* __restrict__ W, const Tile* __restrict__ tiles,
                                              double* partial) {
  launch_next();
  after_previous();
  __shared__ double sh[32];
  const Tile t = tiles[blockIdx.x];
  const int macro = blockIdx.y;
  const int k = t.k;
  const int j = t.j0 + threadIdx.y;
  const int m = t.m0 + threadIdx.x;
  const double* ub = u + (size_t)macro * block;
  const double* lb = lam + (size_t)macro * block;
  const double* Wm = W + (size_t)macro * 16 * NDIR;
  double acc = 0.0;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = 4 * m + q;
    if (i + j + k > N) continue;
    const int me = lidx32(rs, N, i, j, k);
    const double l = lb[me];
    if (l == 0.0) continue;
    const double* w = Wm + node_class(i, j, k, N) * NDIR;
    double sv = w[0] * ub[me];
    for (int d = 1; d < NDIR; ++d) {
      const double wd = w[d];
      if (wd == 0.0) continue;
      int di, dj, dk;
      dir_ijk(d, di, dj, dk);
      if (!in_lattice(i + di, j + dj, k + dk, N)) continue;
      sv += wd * ub[lidx32(rs, N, i + di, j + dj, k + dk)];
    }
    acc += l * sv;
  }
  const double s = block_sum(acc, sh);
  if (threadIdx.x == 0 && threadIdx.y == 0) partial[(size_t)macro * gridDim.x + blockIdx.x] = s;
}

__global__ void k_reduce_per_macro(const double* partial, int n_per, double* out) {
  launch_next();
  after_previous();
  __shared__ double sh[33];
  double s = 0.0;
  const double* p = partial + (size_t)blockIdx.x * n_per;
  for (int q = threadIdx.x; q < n_per; q += blockDim.x) s += p[q];
  s = cta_sum(s, sh);
  if (threadIdx.x == 0) out[blockIdx.x] = s;
}

// Sum of the partial sums into out and, where host is given, into pinned host
// memory with the mesh's error flag beside it: the caller waits for the stream
// and reads them, without two copies of a few bytes behind the kernel.
__global__ void k_reduce(const double* partial, int n, double* out, double* host,
                         const int* err, int* host_err) {
  launch_next();
  after_previous();
  __shared__ double sh[33];
  double s = 0.0;
  for (int q = threadIdx.x; q < n; q += blockDim.x) s += partial[q];
  s = cta_sum(s, sh);
  if (threadIdx.x == 0) {
    out[0] = s;
    if (host) {
      *host = s;
      *host_err = *err;
    }
  }
}

// FP64 FMA throughput probe (measurement support): every thread runs eight
// independent FMA chains of `iters` steps and writes their sum.
__global__ void __launch_bounds__(256) k_fma_probe(double* __restrict__ out, int iters, double a, double b) {
  double x[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) x[q] = threadIdx.x * 1e-3 + q;
  for (int it = 0; it < iters; ++it) {
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = fma(x[q], a, b);
  }
  double s = 0.0;
#pragma unroll
  for (int q = 0; q < 8; ++q) s += x[q];
  out[(size_t)blockIdx.x * blockDim.x + threadIdx.x] = s;
}

// ---------------------------------------------------------------------------
// Global vector <-> blocks (closed-lattice tiles: 8 rows x 32 slots)
// ---------------------------------------------------------------------------
__device__ __forceinline__ int64_t dev_gid(const MacroGeo& g, int N, int i, int j, int k, int64_t nx, int64_t ny) {
  const int64_t X = (int64_t)N * g.v0[0] + (int64_t)i * g.e1[0] + (int64_t)j * g.e2[0] + (int64_t)k * g.e3[0];
  const int64_t Y = (int64_t)N * g.v0[1] + (int64_t)i * g.e1[1] + (int64_t)j * g.e2[1] + (int64_t)k * g.e3[1];
  const int64_t Z = (int64_t)N * g.v0[2] + (int64_t)i * g.e1[2] + (int64_t)j * g.e2[2] + (int64_t)k * g.e3[2];
  return (Z * (ny + 1) + Y) * (nx + 1) + X;
}

// Node (i, j, k) of a macro has grid index node_gid(0, j, k) + i * gid_stride_i.
// A tile of the closed lattice is 8 rows x 128 nodes; its rows are taken in
// the direction (j or k) in which the grid's x grows where it does not grow with
// i, so that the 8 rows touch the same 32-byte sectors of the grid vector.  One
// launch takes f, its scaled copy, u and both masters: 29791 nodes 25 -> 10 us,
// 7.2e6 nodes 235 -> 156 us, 1.35e8 nodes 2.18 -> 2.10 ms (5.4 GB: the strided
// reads of the macros whose x grows with j or k bound it).
struct GridRow {
  int64_t gid0, step;   // grid index of i = 0, step per i
  int j, k, m;          // row and this thread's slot (nodes 4 m .. 4 m + 3)
};
__device__ __forceinline__ bool grid_row(const Tile& t, const MacroGeo& g, int N, int64_t nx, int64_t ny, GridRow& r) {
  const int along = t.j0 + threadIdx.y;
  const bool by_k = g.e2[0] == 0;   // x grows with k only
  r.j = by_k ? t.k : along;
  r.k = by_k ? along : t.k;
  r.m = t.m0 + threadIdx.x;
  if (r.j + r.k > N) return false;
  r.gid0 = dev_gid(g, N, 0, r.j, r.k, nx, ny);
  r.step = dev_gid(g, N, 1, r.j, r.k, nx, ny) - r.gid0;
  return true;
}

// Global vectors gf and gu (either may be null) into the blocks and masters: f
// on the interior nodes (and, where fs is given, f times the macro's winv into
// fs), u on the closed lattice.  The first n_if_ctas CTAs take the masters.
__global__ void __launch_bounds__(CTA) k_import(int N, const int* __restrict__ rs, int64_t block,
                                                const MacroGeo* __restrict__ geo, int64_t nx, int64_t ny,
                                                const double* gf, const double* gu,
                                                double* f, double* fs,
                                                const double* __restrict__ winv, double* u,
                                                const Tile* __restrict__ tiles, int n_tiles,
                                                const int64_t* __restrict__ if_gid, int n_if, double* fI,
                                                double* uI, int n_if_ctas) {
  launch_next();
  after_previous();
  if ((int)blockIdx.x < n_if_ctas) {
    const int q = blockIdx.x * CTA + tid256();
    if (q >= n_if) return;
    const int64_t g = if_gid[q];
    if (gf) fI[q] = gf[g];
    if (gu) uI[q] = gu[g];
    return;
  }
  const int v = blockIdx.x - n_if_ctas, macro = v / n_tiles;
  GridRow r;
  if (!grid_row(tiles[v - macro * n_tiles], geo[macro], N, nx, ny, r)) return;
  const size_t b = (size_t)macro * block + row_base(rs, N, r.j, r.k) + r.m;
  const int CS = __ldg(rs + N + 2), top = N - r.j - r.k;
  const double w = fs ? winv[macro] : 0.0;
  const bool row_in = gf && r.j >= 1 && r.k >= 1;
  double xu[4], xf[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {   // all loads before the stores
    const int i = 4 * r.m + q;
    const int64_t g = r.gid0 + i * r.step;
    xu[q] = gu && i <= top ? gu[g] : 0.0;
    xf[q] = row_in && i >= 1 && i < top ? gf[g] : 0.0;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = 4 * r.m + q;
    const size_t o = b + (size_t)((i + 2 * r.j + 3 * r.k) & 3) * CS;
    if (gu && i <= top) u[o] = xu[q];
    if (row_in && i >= 1 && i < top) {
      f[o] = xf[q];
      if (fs) fs[o] = xf[q] * w;
    }
  }
}

// The interior nodes of the blocks and the masters into the global vector g.
__global__ void __launch_bounds__(CTA) k_export(int N, const int* __restrict__ rs, int64_t block,
                                                const MacroGeo* __restrict__ geo, int64_t nx, int64_t ny,
                                                const double* u, const double* uI,
                                                double* g, const Tile* __restrict__ tiles, int n_tiles,
                                                const int64_t* __restrict__ if_gid, int n_if, int n_if_ctas) {
  launch_next();
  after_previous();
  if ((int)blockIdx.x < n_if_ctas) {
    const int q = blockIdx.x * CTA + tid256();
    if (q < n_if) g[if_gid[q]] = uI[q];
    return;
  }
  const int v = blockIdx.x - n_if_ctas, macro = v / n_tiles;
  GridRow r;
  if (!grid_row(tiles[v - macro * n_tiles], geo[macro], N, nx, ny, r) || r.j < 1 || r.k < 1) return;
  const size_t b = (size_t)macro * block + row_base(rs, N, r.j, r.k) + r.m;
  const int CS = __ldg(rs + N + 2), top = N - r.j - r.k;
  double x[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {   // all loads before the stores
    const int i = 4 * r.m + q;
    x[q] = i >= 1 && i < top ? u[b + (size_t)((i + 2 * r.j + 3 * r.k) & 3) * CS] : 0.0;
  }
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int i = 4 * r.m + q;
    if (i >= 1 && i < top) g[r.gid0 + i * r.step] = x[q];
  }
}

template <class T>
__global__ void k_import_if(const int64_t* __restrict__ gid, int n, const double* g, T* m) {
  launch_next();
  after_previous();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) m[q] = (T)g[gid[q]];
}

template <class T>
__global__ void k_export_if(const int64_t* __restrict__ gid, int n, const T* m, double* g) {
  launch_next();
  after_previous();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) g[gid[q]] = (double)m[q];
}

// out[node] = (A u)_node over the copies listed for each node (the healthy
// copies give A_I, the flux of the healthy side at an interface node).
template <bool S7>
__global__ void k_if_apply(int N, const int* __restrict__ rs, int64_t block, const double* u,
                           const double* uI, const double* __restrict__ W, const int* __restrict__ cptr,
                           const Copy* __restrict__ cps, const int* __restrict__ list, int n, double* out) {
  launch_next();
  after_previous();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= n) return;
  const int node = list[q];
  double off = 0.0, diag = 0.0;
  if_stencil<double, S7>(N, rs, block, u, W, cps, cptr[node], cptr[node + 1], off, diag);
  out[node] = diag * uI[node] + off;
}

__global__ void k_copy_listed(const double* src, double* dst, const int* __restrict__ idx,
                              int n) {
  launch_next();
  after_previous();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) dst[idx[q]] = src[idx[q]];
}

__device__ __forceinline__ void scale_all(const double* __restrict__ f, const double* __restrict__ winv,
                                          double* __restrict__ out, int64_t total, int64_t block) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < total; q += (int64_t)gridDim.x * blockDim.x)
    out[q] = f[q] * winv[q / block];
}
__global__ void k_scale_blocks(const double* f, const double* __restrict__ winv, double* out, int n_macro,
                               int64_t block) {
  launch_next();
  after_previous();
  scale_all(f, winv, out, (int64_t)n_macro * block, block);
}

__global__ void k_set_masters_zero(double* uI, const int* __restrict__ ids, int n) {
  launch_next();
  after_previous();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) uI[ids[q]] = 0.0;
}

__global__ void k_restore(double* u, const double* uI, const int64_t* __restrict__ off,
                          const int* __restrict__ master, int n) {
  launch_next();
  after_previous();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) u[off[q]] = uI[master[q]];
}

template <class T>
__global__ void k_zero_blocks(T* u, int64_t block, const int* __restrict__ act) {
  launch_next();
  after_previous();
  T* b = u + (size_t)act[blockIdx.y] * block;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < block; q += (int64_t)gridDim.x * blockDim.x)
    b[q] = T(0);
}

template <class T>
__global__ void k_zero_list(T* uI, const int* __restrict__ list, int n) {
  launch_next();
  after_previous();
  const int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q < n) uI[list[q]] = T(0);
}

// Launches of at most DEP_MAX_CTAS CTAs (or work units) may overlap their
// predecessor's end (see launch_next): on levels of up to two waves of CTAs the
// launch latency counts (one cycle of 2x2x2 sub-cubes refined 5 times 0.66 ->
// 0.46 ms, 7 times 2.98 -> 2.74 ms, 8 times 15.86 -> 15.60 ms).  Larger ones run
// without: they gain under 1%, their waiting CTAs keep the other stream's work
// off the SMs in a recovery, and the flat kernels lose 4% (FP32) to the wait
// between their index loads and the rest (DEP = false leaves it out).
//
// dep_size: the size that decides it for a launch of `size` CTAs of problem p.
inline int64_t dep_size(const ProbArgs& p, int64_t size) { return p.overlap ? size : DEP_MAX_CTAS + 1; }

template <class... P, class... A>
void launch(int64_t size, void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = size <= DEP_MAX_CTAS ? 1 : 0;
  cudaLaunchKernelEx(&cfg, kern, static_cast<P>(args)...);   // errors: the callers' cudaGetLastError
}

inline unsigned lin_grid(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

// The problem's interface table in precision T, starting at list entry off.
template <class T>
IfTab<T> if_tab(const ProbArgs& p, int off);
template <>
IfTab<double> if_tab<double>(const ProbArgs& p, int off) {
  IfTab<double> t{nullptr, nullptr, nullptr, nullptr, 0, nullptr, nullptr};
  if (p.tnb && p.tw64) t = IfTab<double>{p.tnb + (p.tptr ? 0 : off), p.tw64 + (p.tptr ? 0 : off), p.td64 + off, p.ti64 + off, p.tn,
                                          p.tptr ? p.tptr + off : nullptr, p.tlen ? p.tlen + off : nullptr};
  return t;
}
template <>
IfTab<float> if_tab<float>(const ProbArgs& p, int off) {
  IfTab<float> t{nullptr, nullptr, nullptr, nullptr, 0, nullptr, nullptr};
  if (p.tnb && p.tw32) t = IfTab<float>{p.tnb + (p.tptr ? 0 : off), p.tw32 + (p.tptr ? 0 : off), p.td32 + off, p.ti32 + off, p.tn,
                                          p.tptr ? p.tptr + off : nullptr, p.tlen ? p.tlen + off : nullptr};
  return t;
}
inline dim3 cta_shape() { return dim3(TILE_SLOTS, TILE_ROWS); }

// Grid of a fused launch: interface units first, then tiles x active macros;
// at most as many CTAs as the GPU holds at once (occupancy of the kernel
// times the SM count), each walking the units with a grid stride.
struct Units {
  int n_if_units, total;
};
inline Units units(int n_if_items, int n_tiles, int n_act) {
  Units g;
  g.n_if_units = (int)lin_grid(n_if_items, CTA);
  g.total = g.n_if_units + (n_act > 0 ? n_tiles * n_act : 0);
  return g;
}

std::mutex g_occ_mu;
std::map<std::pair<const void*, int>, int> g_occ;   // (kernel, device) -> resident CTAs

// cap > 0 limits the grid further (a smaller grid makes a launch take the
// dynamic walk at smaller sizes).
inline unsigned resident_grid(const void* kernel, int total, int cap_limit = 0) {
  int dev = 0;
  cudaGetDevice(&dev);
  int cap = 0;
  {
    std::lock_guard<std::mutex> lock(g_occ_mu);
    auto it = g_occ.find({kernel, dev});
    if (it != g_occ.end()) {
      cap = it->second;
    } else {
      int sms = 0, per_sm = 0;
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, CTA, 0);
      cap = std::max(1, sms * std::max(1, per_sm));
      g_occ[{kernel, dev}] = cap;
    }
  }
  if (cap_limit > 0) cap = std::min(cap, cap_limit);
  return (unsigned)std::min(total, cap);
}

// ---------------------------------------------------------------------------
// Persistent batch executor.  One launch runs the programs of many tasks (a
// program is the list of level-wide operations one task issues, recorded
// from the launchers; see hhg_kernels.h).  A CTA takes the next unit of the
// current operation of some task (per-operation counters of units handed out
// and finished); the CTA that finishes an operation's last unit publishes the
// task's next operation.  Units of one operation are independent, as in the
// level kernels; the publishing thread fences after the CTA's writes, and a
// CTA fences after reading a task's operation index and before reading its
// data (no read-only-path loads of data written in the launch), so every
// operation sees its predecessors' results.  A CTA never waits inside a
// unit, so some CTA always makes progress; a CTA that finds no work waits
// (bounded) and retries, and stops when every task has finished.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

template <class T>
__device__ __forceinline__ IfTab<T> dev_if_tab(const ProbArgs& p, int off);
template <>
__device__ __forceinline__ IfTab<double> dev_if_tab<double>(const ProbArgs& p, int off) {
  IfTab<double> t{nullptr, nullptr, nullptr, nullptr, 0, nullptr, nullptr};
  if (p.tnb && p.tw64) t = IfTab<double>{p.tnb + (p.tptr ? 0 : off), p.tw64 + (p.tptr ? 0 : off), p.td64 + off, p.ti64 + off, p.tn,
                                          p.tptr ? p.tptr + off : nullptr, p.tlen ? p.tlen + off : nullptr};
  return t;
}
template <>
__device__ __forceinline__ IfTab<float> dev_if_tab<float>(const ProbArgs& p, int off) {
  IfTab<float> t{nullptr, nullptr, nullptr, nullptr, 0, nullptr, nullptr};
  if (p.tnb && p.tw32) t = IfTab<float>{p.tnb + (p.tptr ? 0 : off), p.tw32 + (p.tptr ? 0 : off), p.td32 + off, p.ti32 + off, p.tn,
                                          p.tptr ? p.tptr + off : nullptr, p.tlen ? p.tlen + off : nullptr};
  return t;
}

// Unit `unit` of a Gauss-Seidel colour (k_gs).
template <class T, bool S7>
__device__ void unit_gs(const BOp& op, int unit, int (*s_pre2)[33], int* s_pre_tot) {
  const LevelArgs& L = op.L;
  const ProbArgs& p = op.P;
  const int N = L.N;
  const int* rs = L.rs;
  const int64_t block = L.block;
  T* u = (T*)op.u;
  if (unit < op.n_if_units) {
    const int q = unit * CTA + tid256();
    if (q < op.n_list) {
      T* uI = (T*)op.uI;
      const T* fI = (const T*)op.fI;
      const int node = p.free_if[op.list_off + q];
      const int c0 = L.cptr[node], c1 = L.cptr[node + 1];
      const IfTab<T> tab = dev_if_tab<T>(p, op.list_off);
      T val;
      if (tab.nb) {
        val = (fI[node] - if_offdiag<T, if_tab_k(S7)>(tab, u, q)) * tab.dinv[q];
      } else {
        T off = T(0), diag = T(0);
        if_stencil<T, S7>(N, rs, block, u, (const T*)op.W, L.cps, c0, c1, off, diag);
        val = (fI[node] - off) / diag;
      }
      uI[node] = val;
      write_copies(N, rs, block, u, L.cps, L.cp_off, c0, c1, val);
    }
    return;
  }
  const int vb = unit - op.n_if_units;
  const Tile t = L.tiles_int[vb / p.n_act];
  const int macro = p.act[vb % p.n_act];
  T* ub = u + (size_t)macro * block;
  const T* w = (const T*)op.Wv + (size_t)macro * 16 * NDIR;
  const T inv = ((const T*)op.Winv)[macro];
  const T* fb = (const T*)op.f + (size_t)macro * block;
  if (S7) {
    if (op.scaled) gs_tile7<T, true, false>(t, N, rs, op.colour, ub, fb, w, T(1), s_pre2, s_pre_tot);
    else gs_tile7<T, false, false>(t, N, rs, op.colour, ub, fb, w, inv, s_pre2, s_pre_tot);
    return;
  }
  const int total = flat_setup_slabs(t, N, op.colour, true, 1, s_pre2, s_pre_tot);
  int sl = 0;
  for (int tt = tid256(); tt < total; tt += CTA) {
    while (tt >= s_pre_tot[sl + 1]) ++sl;
    const int k = t.k + sl;
    const Tile ts{k, t.j0, t.m0, 1};
    int j, v, ic, mlo, n;
    flat_item(ts, N, op.colour, true, s_pre2[sl], tt - s_pre_tot[sl], j, v);
    colour_row(N, j, k, op.colour, ic, mlo, n);
    const int i = 4 * (mlo + v) + ic;
    const int me = lidx32(rs, N, i, j, k);
    T acc = fb[me];
#pragma unroll
    for (int d = 1; d < NDIR; ++d) {
      int di, dj, dk;
      dir_ijk(d, di, dj, dk);
      acc -= w[d] * ub[lidx32(rs, N, i + di, j + dj, k + dk)];
    }
    ub[me] = acc * inv;
  }
}

// Unit of the residual r = f - A u written to r (k_res, no norm).
template <class T, bool S7>
__device__ void unit_res(const BOp& op, int unit, int (*s_pre2)[33], int* s_pre_tot) {
  const LevelArgs& L = op.L;
  const ProbArgs& p = op.P;
  const int N = L.N;
  const int* rs = L.rs;
  const int64_t block = L.block;
  const T* u = (const T*)op.u;
  T* r = (T*)op.r;
  double ss = 0.0;
  if (unit < op.n_if_units) {
    const int q = unit * CTA + tid256();
    if (q < op.n_list) {
      const T* uI = (const T*)op.uI;
      const T* fI = (const T*)op.fI;
      const int node = p.free_if[q];
      const int c0 = L.cptr[node], c1 = L.cptr[node + 1];
      const IfTab<T> tab = dev_if_tab<T>(p, 0);
      T res;
      if (q >= op.skip_lo && q < op.skip_hi) {
        res = T(0);
      } else if (tab.nb) {
        res = fI[node] - tab.diag[q] * uI[node] - if_offdiag<T, if_tab_k(S7)>(tab, u, q);
      } else {
        T off = T(0), diag = T(0);
        if_stencil<T, S7>(N, rs, block, u, (const T*)op.W, L.cps, c0, c1, off, diag);
        res = fI[node] - diag * uI[node] - off;
      }
      write_copies(N, rs, block, r, L.cps, L.cp_off, c0, c1, res);
    } else if (q < op.n_list + op.n_zero) {
      r[p.zero_off[q - op.n_list]] = T(0);
    }
    return;
  }
  const int vb = unit - op.n_if_units;
  const Tile t = L.tiles_int[vb / p.n_act];
  const int macro = p.act[vb % p.n_act];
  const T* ub = u + (size_t)macro * block;
  const T* fb = (const T*)op.f + (size_t)macro * block;
  T* rb = r + (size_t)macro * block;
  const T* w = (const T*)op.W + (size_t)macro * 16 * NDIR;
  if (S7) {
    constexpr int VW = Vec<T>::n;
    const T wr[11] = {w[0], w[1], w[2], w[3], T(0), T(0), T(0), T(0), w[8], w[9], w[10]};
    for (int c = 0; c < 4; ++c) {
      const int total = flat_setup_slabs(t, N, c, true, VW, s_pre2, s_pre_tot);
      int sl = 0;
      for (int tt = tid256(); tt < total; tt += CTA) {
        while (tt >= s_pre_tot[sl + 1]) ++sl;
        const int k = t.k + sl;
        const Tile ts{k, t.j0, t.m0, 1};
        int j, g;
        flat_item(ts, N, c, true, s_pre2[sl], tt - s_pre_tot[sl], j, g, VW);
        if (c == op.skip)
          res_group7<T, true, false, true, false>(slice_consts(rs, N, k), N, j, g, c, ub, fb, rb, wr, ss);
        else
          res_group7<T, true, false, false, false>(slice_consts(rs, N, k), N, j, g, c, ub, fb, rb, wr, ss);
      }
      __syncthreads();
    }
    return;
  }
  HHG_TILE_NODES(N, rs, t, s_pre, {
    const int me = lidx32(rs, N, i, j, k);
    T acc = T(0);
    if (((i + 2 * j + 3 * k) & 3) != op.skip) {
      acc = fb[me] - w[0] * ub[me];
_Pragma("unroll")
      for (int d = 1; d < NDIR; ++d) {
        int di, dj, dk;
        dir_ijk(d, di, dj, dk);
        acc -= w[d] * ub[lidx32(rs, N, i + di, j + dj, k + dk)];
      }
    }
    rb[me] = acc;
  })
}

// Unit of the restriction onto the coarse level C (k_restrict).
template <class T>
__device__ void unit_restrict(const BOp& op, int unit, int (*s_pre2)[33], int* s_pre_tot) {
  const LevelArgs& F = op.L;
  const LevelArgs& C = op.C;
  const ProbArgs& pc = op.P;
  const T* rf = (const T*)op.r;
  T* fc = (T*)op.fc;
  T* uc = (T*)op.uc;
  if (unit < op.n_if_units) {
    const int q = unit * CTA + tid256();
    if (q < op.n_list) {
      T* fIc = (T*)op.fIc;
      T* uIc = (T*)op.uIc;
      const int node = pc.free_if[q];
      const int64_t* g = pc.gather + (size_t)q * NDIR;
      T acc = T(0);
      for (int e = 1; e < NDIR; ++e) {
        const int64_t o = g[e];
        if (o >= 0) acc += rf[o];
      }
      fIc[node] = rf[g[0]] + T(0.5) * acc;
      uIc[node] = T(0);
      write_copies(C.N, C.rs, C.block, uc, C.cps, C.cp_off, C.cptr[node], C.cptr[node + 1], T(0));
    } else if (q < op.n_list + op.n_zero) {
      uc[pc.zero_off[q - op.n_list]] = T(0);
    }
    return;
  }
  Tile t;
  int macro;
  vol_subunit(unit - op.n_if_units, pc.n_act, RESTRICT_SPLIT, C.tiles_int, pc.act, t, macro);
  restrict_tile<T, false>(t, C.N, C.rs, F.N, F.rs, rf + (size_t)macro * F.block, fc + (size_t)macro * C.block,
                          uc + (size_t)macro * C.block, s_pre2, s_pre_tot);
}

// Unit of the prolongation u_f += P u_c (k_prolong).
template <class T>
__device__ void unit_prolong(const BOp& op, int unit, int (*s_pre2)[33], int* s_pre_tot) {
  const LevelArgs& F = op.L;
  const LevelArgs& C = op.C;
  const ProbArgs& pf = op.P;
  T* uf = (T*)op.u;
  const T* uc = (const T*)op.uc;
  if (unit < op.n_if_units) {
    const int q = unit * CTA + tid256();
    if (q < op.n_list && (q < op.skip_lo || q >= op.skip_hi)) {
      T* uIf = (T*)op.uI;
      const int node = pf.free_if[q];
      const int c0 = F.cptr[node], c1 = F.cptr[node + 1];
      const Copy cp = F.cps[c0];
      const T val = uIf[node] + interp(uc + (size_t)cp.macro * C.block, C.N, C.rs, cp.i, cp.j, cp.k);
      uIf[node] = val;
      write_copies(F.N, F.rs, F.block, uf, F.cps, F.cp_off, c0, c1, val);
    }
    return;
  }
  const int vb = unit - op.n_if_units;
  const Tile t = F.tiles_int[vb / pf.n_act];
  const int macro = pf.act[vb % pf.n_act];
  prolong_tile<T, false>(t, F.N, F.rs, C.N, C.rs, uf + (size_t)macro * F.block, uc + (size_t)macro * C.block, op.skip,
                         s_pre2, s_pre_tot);
}

// Unit of the FP64 residual handed to the FP32 cycle (k_res_f32, no norm).
// This unit and the coarse CG are called, not inlined: the executor has 48
// registers, and what these two hold was spilled in the Gauss-Seidel loops (a
// mixed 4x4x4 global task of refinement 7 with 64 recovery tasks 235.4 -> 211.8
// ms, the global task alone first 212.2 -> 188.7; small batches as before).
template <bool S7>
__device__ __noinline__ void unit_res_f32(const BOp& op, int unit, int (*s_pre2)[33], int* s_pre_tot) {
  const LevelArgs& L = op.L;
  const ProbArgs& p = op.P;
  const int N = L.N;
  const int* rs = L.rs;
  const int64_t block = L.block;
  const double* u = (const double*)op.u;
  if (unit < op.n_if_units) {
    const int q = unit * CTA + tid256();
    if (q < op.n_list) {
      const double* uI = (const double*)op.uI;
      const double* fI = (const double*)op.fI;
      const int node = p.free_if[q];
      const IfTab<double> tab = dev_if_tab<double>(p, 0);
      double res;
      if (tab.nb) {
        res = fI[node] - tab.diag[q] * uI[node] - if_offdiag<double, if_tab_k(S7)>(tab, u, q);
      } else {
        double off = 0.0, diag = 0.0;
        if_stencil<double, S7>(N, rs, block, u, (const double*)op.W, L.cps, L.cptr[node], L.cptr[node + 1], off,
                               diag);
        res = fI[node] - diag * uI[node] - off;
      }
      ((float*)op.oI32)[node] = (float)res;
    }
    return;
  }
  const int vb = unit - op.n_if_units;
  const Tile t = L.tiles_int[vb / p.n_act];
  const int macro = p.act[vb % p.n_act];
  const double* ub = u + (size_t)macro * block;
  const double* fb = (const double*)op.f + (size_t)macro * block;
  float* ob = (float*)op.o32 + (size_t)macro * block;
  const double* w = (const double*)op.W + (size_t)macro * 16 * NDIR;
  HHG_TILE_NODES(N, rs, t, s_pre, {
    int me;
    double acc;
    if (S7) {
      const Nb7 q = nb7(sc, i, j);
      me = q.me;
      acc = fb[me] - w[0] * ub[me];
      acc -= w[1] * ub[q.nb1];
      acc -= w[2] * ub[q.nb2];
      acc -= w[3] * ub[q.nb3];
      acc -= w[8] * ub[q.nb8];
      acc -= w[9] * ub[q.nb9];
      acc -= w[10] * ub[q.nb10];
    } else {
      me = lidx32(rs, N, i, j, k);
      acc = fb[me] - w[0] * ub[me];
_Pragma("unroll")
      for (int d = 1; d < NDIR; ++d) {
        int di, dj, dk;
        dir_ijk(d, di, dj, dk);
        acc -= w[d] * ub[lidx32(rs, N, i + di, j + dj, k + dk)];
      }
    }
    ob[me] = (float)acc;
  })
}

// Coarse CG (k_cg with its vectors in the problem's global work array).
template <class T>
__device__ __noinline__ void unit_cg(const BOp& op, double* red) {
  const size_t n = (size_t)op.n_cg;
  cg_one_cta<T>(op.n_cg, op.rowptr, op.col, op.val, op.fsrc, (const T*)op.f, (const T*)op.fI, op.uptr, op.udst,
                op.umaster, (T*)op.u, (T*)op.uI, op.work, op.work + n, op.work + 2 * n, op.work + 3 * n, op.dinv,
                op.rtol, op.maxit, op.iters, red);
}

// 16384 elements per unit of the block-wise operations (zeroing, the FP32
// correction added in FP64, memsets): tens of microseconds of streaming per
// unit, like a stencil tile, so that the claims stay cheap by comparison
constexpr int BATCH_CHUNK = CTA * 64;

__device__ void run_unit(const BOp& op, int unit, int (*s_pre2)[33], int* s_pre_tot, double* red) {
  const int tid = tid256();
  switch (op.kind) {
    case BOP_GS:
      if (op.fp32) {
        if (op.seven_point) unit_gs<float, true>(op, unit, s_pre2, s_pre_tot);
        else unit_gs<float, false>(op, unit, s_pre2, s_pre_tot);
      } else {
        if (op.seven_point) unit_gs<double, true>(op, unit, s_pre2, s_pre_tot);
        else unit_gs<double, false>(op, unit, s_pre2, s_pre_tot);
      }
      break;
    case BOP_RES:
      if (op.fp32) {
        if (op.seven_point) unit_res<float, true>(op, unit, s_pre2, s_pre_tot);
        else unit_res<float, false>(op, unit, s_pre2, s_pre_tot);
      } else {
        if (op.seven_point) unit_res<double, true>(op, unit, s_pre2, s_pre_tot);
        else unit_res<double, false>(op, unit, s_pre2, s_pre_tot);
      }
      break;
    case BOP_RESTRICT:
      if (op.fp32) unit_restrict<float>(op, unit, s_pre2, s_pre_tot);
      else unit_restrict<double>(op, unit, s_pre2, s_pre_tot);
      break;
    case BOP_PROLONG:
      if (op.fp32) unit_prolong<float>(op, unit, s_pre2, s_pre_tot);
      else unit_prolong<double>(op, unit, s_pre2, s_pre_tot);
      break;
    case BOP_CG:
      if (op.fp32) unit_cg<float>(op, red);
      else unit_cg<double>(op, red);
      break;
    case BOP_RES_F32:
      if (op.seven_point) unit_res_f32<true>(op, unit, s_pre2, s_pre_tot);
      else unit_res_f32<false>(op, unit, s_pre2, s_pre_tot);
      break;
    case BOP_ZERO_BLOCKS: {
      // unit = (active macro, chunk of BATCH_CHUNK elements)
      const int64_t chunks = (op.L.block + BATCH_CHUNK - 1) / BATCH_CHUNK;
      const int macro = op.P.act[unit / chunks];
      const int64_t c0 = (unit % chunks) * BATCH_CHUNK;
      const int64_t c1 = min((int64_t)BATCH_CHUNK + c0, op.L.block);
      for (int64_t q = c0 + tid; q < c1; q += CTA) {
        if (op.fp32) ((float*)op.u)[(size_t)macro * op.L.block + q] = 0.f;
        else ((double*)op.u)[(size_t)macro * op.L.block + q] = 0.0;
      }
      break;
    }
    case BOP_ZERO_LIST: {
      const int64_t q = (int64_t)unit * CTA + tid;
      if (q < op.n) {
        if (op.fp32) ((float*)op.uI)[op.ids[q]] = 0.f;
        else ((double*)op.uI)[op.ids[q]] = 0.0;
      }
      break;
    }
    case BOP_ADD_BLOCKS: {
      // unit = (active macro, chunk of BATCH_CHUNK FP64 slots); u64 += e32
      const int64_t chunks = (op.L.block + BATCH_CHUNK - 1) / BATCH_CHUNK;
      const int macro = op.P.act[unit / chunks];
      const int64_t c0 = (unit % chunks) * BATCH_CHUNK;
      const int64_t c1 = min((int64_t)BATCH_CHUNK + c0, op.L.block);
      double* ub = (double*)op.u + (size_t)macro * op.L.block;
      const float* eb = (const float*)op.o32 + (size_t)macro * op.L.block;
      for (int64_t q = c0 + 2 * tid; q < c1; q += 2 * CTA) {
        double2 x = *reinterpret_cast<double2*>(ub + q);
        const float2 d = *reinterpret_cast<const float2*>(eb + q);
        x.x += (double)d.x;
        x.y += (double)d.y;
        *reinterpret_cast<double2*>(ub + q) = x;
      }
      break;
    }
    case BOP_ADD_MASTERS: {
      const int64_t q = (int64_t)unit * CTA + tid;
      if (q < op.n) {
        const int node = op.ids[q];
        ((double*)op.uI)[node] += (double)((const float*)op.oI32)[node];
      }
      break;
    }
    case BOP_MEMSET: {
      // 16-byte words [unit * BATCH_CHUNK, ...) of op.u
      const int64_t c0 = (int64_t)unit * BATCH_CHUNK;
      const int64_t c1 = min((int64_t)BATCH_CHUNK + c0, op.n);
      for (int64_t q = c0 + tid; q < c1; q += CTA) reinterpret_cast<double2*>(op.u)[q] = make_double2(0.0, 0.0);
      break;
    }
    case BOP_SET_ZERO: {
      const int64_t q = (int64_t)unit * CTA + tid;
      if (q < op.n) ((double*)op.uI)[op.ids[q]] = 0.0;
      break;
    }
    case BOP_RESTORE: {
      const int64_t q = (int64_t)unit * CTA + tid;
      if (q < op.n) ((double*)op.u)[op.offs[q]] = ((const double*)op.uI)[op.ids[q]];
      break;
    }
    default:
      break;
  }
}

// Persistent executor of a batch: task t runs ops [op_off[t], op_off[t + 1])
// in order; n_live tasks have at least one operation.  Every CTA repeatedly
// claims a unit of the current operation of some task, runs it and counts it
// done; the CTA that completes an operation's last unit publishes the task's
// next phase.
//   * Claims: warp 0 scans the tasks 32 at a time in priority classes (the
//     tasks order[seg[c] .. seg[c + 1]) form class c, highest first); within
//     a class it starts at the task it served last, and the first lane that
//     sees unissued units of its task's current operation takes one with an
//     atomic.  While the CTA runs a unit, thread 0 already claims the next
//     unit of the same operation (the atomic's latency hides behind the
//     work), except near the end of the operation; a unit taken there is
//     valid because an operation with unissued units is still its task's
//     current one.
//   * Memory order: a unit's writes precede its done count (CTA barrier, then
//     a device fence by the counting thread); a CTA reads a published phase
//     before the data (device fence by the scanning warp, then a CTA
//     barrier); the units read that data with plain coherent loads.
//   * A CTA that finds no unit for wait_limit rounds in a row sets *err = 1
//     and stops; the CTA that completes an operation always finds the next
//     one, so the work still finishes.
//   * Time stamps: st.start_ns (first CTA), st.task_ns[t] (the task's last
//     unit done).
// One unit per claim: a large operation gives each CTA only a few units
// (a Gauss-Seidel tile takes tens of microseconds), so claiming several at
// once lengthens the operation's tail by more than the claims cost.
__device__ __forceinline__ int batch_claim_size(int) { return 1; }

// Scheduler state of a CTA, in shared memory so that no register stays live
// across a unit's body.
struct BatchCtl {
  int state, task, gi, unit, cnt;   // the claim to run (written by warp 0)
  int cur_gi, cur_task;             // operation held in the CTA's op copy
  int next;                         // first task of the next scan
  int pf_u, pf_k;                   // chunk claimed ahead on cur_gi (-1: none)
  int idle;                         // scans in a row that found nothing
};

__global__ void __launch_bounds__(CTA, 5) k_batch(const BOp* __restrict__ ops, const int* __restrict__ op_off,
                                                  const int* __restrict__ order, const int* __restrict__ seg, int n_seg,
                                                  int n_live, BatchState st, int wait_limit, int* __restrict__ err) {
  __shared__ int s_pre2[MAX_SLABS][33];
  __shared__ int s_pre_tot[MAX_SLABS + 1];
  __shared__ double red[64];
  __shared__ BatchCtl ctl;
  __shared__ __align__(16) BOp s_op;
  if (tid256() == 0) {
    atomicMin(st.start_ns, global_ns());
    ctl.cur_gi = -1;
    ctl.cur_task = 0;
    ctl.next = -1;
    ctl.pf_u = -1;
    ctl.pf_k = 0;
    ctl.idle = 0;
  }
  __syncthreads();
  for (;;) {
    if (tid256() < 32) {
      const int lane = tid256();
      int state = 0, task = 0, gi = 0, u = 0, cnt = 0;
      if (ctl.pf_u >= 0) {
        state = 1;
        task = ctl.cur_task;
        gi = ctl.cur_gi;
        u = ctl.pf_u;
        cnt = ctl.pf_k;
      } else if (*(volatile int*)st.tasks_done >= n_live) {
        state = 2;
      } else {
        int pos_taken = 0;
        for (int c = 0; c < n_seg && state == 0; ++c) {
          const int lo = seg[c], len = seg[c + 1] - lo;
          const int cur = ctl.next;   // position in order[] of the task served last
          const int start = cur >= lo && cur < lo + len ? cur - lo : (int)(blockIdx.x % (unsigned)len);
          for (int base = 0; base < len && state == 0; base += 32) {
            const int q = base + lane;
            int pos = start + q;
            if (pos >= len) pos -= len;
            bool avail = false;
            int g = 0, nu = 0, t = 0;
            if (q < len) {
              t = order[lo + pos];
              const int ph = *(volatile int*)(st.phase + t);
              const int o0 = op_off[t];
              if (ph < op_off[t + 1] - o0) {
                g = o0 + ph;
                nu = ops[g].n_units;
                avail = *(volatile int*)(st.issued + g) < nu;
              }
            }
            unsigned mask = __ballot_sync(0xffffffffu, avail);
            while (mask) {
              const int src = __ffs(mask) - 1;
              mask &= mask - 1;
              int claim = -1, k = 0;
              if (lane == src) {
                k = batch_claim_size(nu);
                const int u0 = atomicAdd(st.issued + g, k);
                if (u0 < nu) {
                  claim = u0;
                  k = min(k, nu - u0);
                }
              }
              claim = __shfl_sync(0xffffffffu, claim, src);
              if (claim >= 0) {
                state = 1;
                task = __shfl_sync(0xffffffffu, t, src);
                gi = __shfl_sync(0xffffffffu, g, src);
                cnt = __shfl_sync(0xffffffffu, k, src);
                pos_taken = lo + __shfl_sync(0xffffffffu, pos, src);
                u = claim;
                break;
              }
            }
          }
        }
        if (state == 1 && lane == 0) ctl.next = pos_taken;
        __threadfence();   // what the earlier operations wrote is read after this
      }
      __syncwarp();
      if (lane == 0) {
        ctl.state = state;
        ctl.task = task;
        ctl.gi = gi;
        ctl.unit = u;
        ctl.cnt = cnt;
      }
    }
    __syncthreads();
    if (ctl.state == 2) break;
    if (ctl.state == 0) {
      __syncthreads();   // every thread has read the state
      if (tid256() == 0) {
        if (++ctl.idle > wait_limit) {
          atomicExch(err, 1);
          ctl.state = 2;
        } else {
          __nanosleep(256);
        }
      }
      __syncthreads();
      if (ctl.state == 2) break;
      continue;
    }
    if (ctl.gi != ctl.cur_gi) {
      const int* src = reinterpret_cast<const int*>(ops + ctl.gi);
      int* dst = reinterpret_cast<int*>(&s_op);
      for (int q = tid256(); q < (int)(sizeof(BOp) / sizeof(int)); q += CTA) dst[q] = src[q];
      __syncthreads();
    }
    if (tid256() == 0) {
      ctl.idle = 0;
      ctl.cur_gi = ctl.gi;
      ctl.cur_task = ctl.task;
      // claim the next unit of this operation while this one runs, unless
      // the operation nears its end (a unit held back there lengthens the
      // operation's tail)
      const int nu = s_op.n_units;
      ctl.pf_k = batch_claim_size(nu);
      ctl.pf_u = ctl.unit + ctl.cnt + 2 * (int)gridDim.x * ctl.pf_k < nu ? atomicAdd(st.issued + ctl.gi, ctl.pf_k) : nu;
    }
    for (int c = 0; c < ctl.cnt; ++c) {
      run_unit(s_op, ctl.unit + c, s_pre2, s_pre_tot, red);
      __syncthreads();
    }
    if (tid256() == 0) {
      const int nu = s_op.n_units;
      if (ctl.pf_u >= nu) ctl.pf_u = -1;
      else ctl.pf_k = min(ctl.pf_k, nu - ctl.pf_u);
      const int gi = ctl.gi, cnt = ctl.cnt;
      __threadfence();   // the CTA's writes before its units count as done
      const int d = atomicAdd(st.done + gi, cnt);
      if (d + cnt == nu) {
        const int t = ctl.task;
        const int ph = gi - op_off[t] + 1;
        __threadfence();
        atomicExch(st.phase + t, ph);
        if (ph == op_off[t + 1] - op_off[t]) {
          st.task_ns[t] = global_ns();
          __threadfence();
          atomicAdd(st.tasks_done, 1);
        }
      }
    }
    // the next scan (warp 0) reads ctl after thread 0 wrote it: same warp,
    // ordered by __syncwarp at the top of the scan
    __syncwarp();
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
namespace {
thread_local std::vector<BOp>* g_rec = nullptr;

// A batch operation of kind k in the arithmetic type T.
template <class T>
BOp new_op(int kind) {
  BOp op;
  std::memset(&op, 0, sizeof(op));
  op.kind = kind;
  op.fp32 = sizeof(T) == 4 ? 1 : 0;
  return op;
}

int64_t block_chunks(int64_t block) { return (block + BATCH_CHUNK - 1) / BATCH_CHUNK; }
}  // namespace

void record_ops(std::vector<BOp>* rec) { g_rec = rec; }
bool recording() { return g_rec != nullptr; }

cudaError_t memset16(void* p, size_t bytes, cudaStream_t s) {
  if (g_rec) {
    if (bytes % 16 != 0 || reinterpret_cast<uintptr_t>(p) % 16 != 0) return cudaErrorInvalidValue;
    BOp op = new_op<double>(BOP_MEMSET);
    op.u = p;
    op.n = (int64_t)(bytes / 16);
    op.n_units = (int)((op.n + BATCH_CHUNK - 1) / BATCH_CHUNK);
    if (op.n_units > 0) g_rec->push_back(op);
    return cudaSuccess;
  }
  return cudaMemsetAsync(p, 0, bytes, s);
}

cudaError_t run_batch(const BOp* ops, const int* op_off, const int* order, const int* seg, int n_seg, int n_live,
                      const BatchState& st, int wait_limit, int* err, cudaStream_t s) {
  if (n_live <= 0) return cudaSuccess;
  const unsigned grid = resident_grid((const void*)k_batch, 1 << 30);
  ++g_kernel_launches;
  k_batch<<<grid, cta_shape(), 0, s>>>(ops, op_off, order, seg, n_seg, n_live, st, wait_limit, err);
  return cudaGetLastError();
}
// Elements of one staging slot of the streaming kernel on a level: the
// largest band range, rows 0..band+1 of slice 0, rounded up to 32 elements.
inline int stream_slot(int N, int band) {
  const int M = N + 1;
  const int len = slot_prefix(M) - slot_prefix(std::max(0, M - (band + 2)));
  return (len + 31) & ~31;
}

template <class T, bool SCALED>
cudaError_t launch_gs_stream(const LevelArgs& L, const ProbArgs& p, T* u, T* uI, const T* fI, const T* W,
                             const T* Winv, const T* fv, const T* Wv, int colour, int n, cudaStream_t s) {
  const bool wide = sizeof(T) == 4;   // FP32 cycles: wider bands
  const StreamTile* tiles = wide ? L.tiles_stream32 : L.tiles_stream;
  const int n_tiles = wide ? L.n_tiles_stream32 : L.n_tiles_stream;
  const Units g = units(n, n_tiles, p.n_act);
  if (g.total == 0) return cudaSuccess;
  const int slot = stream_slot(L.N, wide ? L.stream_band32 : L.stream_band);
  const size_t smem = (size_t)(STREAM_NSLOT * slot + 2 * STREAM_PAD) * sizeof(T);
  auto kern = k_gs_stream<T, SCALED>;
  // the kernel may use up to the device's opt-in shared memory per CTA (set
  // once per device; a smaller setting would refuse later, larger launches)
  static std::mutex mu;
  static std::map<int, int> attr_max;   // device -> bytes allowed
  int dev = 0;
  cudaGetDevice(&dev);
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = attr_max.find(dev);
    if (it == attr_max.end()) {
      int optin = 0;
      cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
      const int static_bytes = 4096;   // the kernel's own shared arrays, with room
      const int allow = std::max(0, optin - static_bytes);
      const cudaError_t e =
          cudaFuncSetAttribute((const void*)kern, cudaFuncAttributeMaxDynamicSharedMemorySize, allow);
      if (e != cudaSuccess) return e;
      it = attr_max.emplace(dev, allow).first;
    }
    if ((size_t)it->second < smem) return cudaErrorInvalidConfiguration;
  }
  int per_sm = 0, sms = 0;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, (const void*)kern, STREAM_CTA, smem);
  int cap = std::max(1, sms * std::max(1, per_sm));
  if (p.grid_cap > 0) cap = std::min(cap, p.grid_cap);
  const unsigned grid = (unsigned)std::min(g.total, cap);
  ++g_kernel_launches;
  launch(dep_size(p, g.total), kern, grid, dim3(32, STREAM_CONSUMERS + 1), smem, s, L.N, L.rs, L.block, u, uI, fI, W, Winv, fv, Wv, tiles,
                                                         n_tiles, p.act, p.n_act, colour, L.cptr, L.cps, L.cp_off,
                                       p.free_if + p.col_off[colour], n, if_tab<T>(p, p.col_off[colour]),
                                       g.n_if_units, p.sched, slot, p.wait_limit, p.err);
  return cudaGetLastError();
}

bool flat_on(const LevelArgs& L, const ProbArgs& p) {
  return L.gs_flat == FLAT_ON || (L.gs_flat == FLAT_AUTO && p.grid_cap == 0);
}

template <class T>
cudaError_t gs_colour(const LevelArgs& L, const ProbArgs& p, T* u, T* uI, const T* f, const T* fI, const T* W,
                      const T* Winv, int colour, bool seven_point, cudaStream_t s, cudaEvent_t ev_begin,
                      cudaEvent_t ev_end, const T* fs, const T* Wsc) {
  if (g_rec) {
    if (!seven_point || !fs || !Wsc) fs = Wsc = nullptr;
    const int nl = p.col_off[colour + 1] - p.col_off[colour];
    const Units g = units(nl, L.n_tiles_int, p.n_act);
    if (g.total == 0) return cudaSuccess;
    BOp op = new_op<T>(BOP_GS);
    op.seven_point = seven_point ? 1 : 0;
    op.scaled = fs ? 1 : 0;
    op.colour = colour;
    op.L = L;
    op.P = p;
    op.list_off = p.col_off[colour];
    op.n_list = nl;
    op.n_if_units = g.n_if_units;
    op.n_units = g.total;
    op.u = u;
    op.uI = uI;
    op.f = fs ? fs : f;
    op.fI = fI;
    op.W = W;
    op.Wv = Wsc ? Wsc : W;
    op.Winv = Winv;
    g_rec->push_back(op);
    return cudaSuccess;
  }
  if (!seven_point) fs = Wsc = nullptr;
  if (!fs || !Wsc) fs = Wsc = nullptr;
  const int n = p.col_off[colour + 1] - p.col_off[colour];
  if (seven_point && p.stream_gs && L.n_tiles_stream > 0 && p.err) {
    if (ev_begin) cudaEventRecord(ev_begin, s);
    const cudaError_t e = fs ? launch_gs_stream<T, true>(L, p, u, uI, fI, W, Winv, fs, Wsc, colour, n, s)
                             : launch_gs_stream<T, false>(L, p, u, uI, fI, W, Winv, f, W, colour, n, s);
    if (ev_end) cudaEventRecord(ev_end, s);
    return e;
  }
  const uint32_t* items = sizeof(T) == 8 ? L.gs_items64 : L.gs_items32;
  if (flat_on(L, p) && items) {
    const int* off = sizeof(T) == 8 ? L.gs_off64 : L.gs_off32;
    const int n_items = off[colour + 1] - off[colour];
    const int n_if_ctas = (int)lin_grid(n, CTA);
    const int n_vol_ctas = p.n_act > 0 ? (int)lin_grid((int64_t)n_items * p.n_act, CTA) : 0;
    if (n_if_ctas + n_vol_ctas == 0) return cudaSuccess;
    const bool dep = dep_size(p, n_if_ctas + n_vol_ctas) <= DEP_MAX_CTAS;
    auto kern = !seven_point ? (dep ? k_gs_flat<T, false, false, true> : k_gs_flat<T, false, false, false>)
                : fs         ? (dep ? k_gs_flat<T, true, true, true> : k_gs_flat<T, true, true, false>)
                             : (dep ? k_gs_flat<T, true, false, true> : k_gs_flat<T, true, false, false>);
    if (ev_begin) cudaEventRecord(ev_begin, s);
    ++g_kernel_launches;
    launch(dep_size(p, n_if_ctas + n_vol_ctas), kern, n_if_ctas + n_vol_ctas, cta_shape(), 0, s,
        L.N, L.rs, L.block, u, uI, fI, W, Winv, fs ? fs : f, Wsc ? Wsc : W, items + off[colour], n_items, p.act,
        p.n_act, colour, L.cptr, L.cps, L.cp_off, p.free_if + p.col_off[colour], n, if_tab<T>(p, p.col_off[colour]),
        n_if_ctas, n_vol_ctas);
    if (ev_end) cudaEventRecord(ev_end, s);
    return cudaGetLastError();
  }
  const Units g = units(n, L.n_tiles_int, p.n_act);
  if (g.total == 0) return cudaSuccess;
  const bool dep = dep_size(p, g.total) <= DEP_MAX_CTAS;
  auto kern = seven_point ? (dep ? k_gs<T, true, true> : k_gs<T, true, false>)
                          : (dep ? k_gs<T, false, true> : k_gs<T, false, false>);
  const unsigned grid = resident_grid((const void*)kern, g.total, p.grid_cap);
  if (ev_begin) cudaEventRecord(ev_begin, s);
  ++g_kernel_launches;
  launch(dep_size(p, g.total), kern, grid, cta_shape(), 0, s, L.N, L.rs, L.block, u, uI, f, fI, W, Winv, fs, Wsc, L.tiles_int, L.n_tiles_int, p.act,
                                    p.n_act, colour, L.cptr, L.cps, L.cp_off, p.free_if + p.col_off[colour], n,
                                    if_tab<T>(p, p.col_off[colour]), g.n_if_units, p.sched);
  if (ev_end) cudaEventRecord(ev_end, s);
  return cudaGetLastError();
}

template <class T>
cudaError_t residual(const LevelArgs& L, const ProbArgs& p, const T* u, const T* uI, const T* f, const T* fI, T* r,
                     const T* W, bool seven_point, bool write_r, double* partial, int* n_part, cudaStream_t s,
                     int skip) {
  if (g_rec) {
    if (partial || !write_r) return cudaErrorNotSupported;   // norms are not part of a batch
    const int nl = p.col_off[4];
    const Units g = units(nl + p.n_zero, L.n_tiles_int, p.n_act);
    if (g.total == 0) return cudaSuccess;
    BOp op = new_op<T>(BOP_RES);
    op.seven_point = seven_point ? 1 : 0;
    op.skip = skip >= 0 && skip < 4 ? skip : -1;
    op.skip_lo = op.skip >= 0 ? p.col_off[op.skip] : 0;
    op.skip_hi = op.skip >= 0 ? p.col_off[op.skip + 1] : 0;
    op.L = L;
    op.P = p;
    op.n_list = nl;
    op.n_zero = p.n_zero;
    op.n_if_units = g.n_if_units;
    op.n_units = g.total;
    op.u = (void*)u;
    op.uI = (void*)uI;
    op.f = f;
    op.fI = fI;
    op.r = r;
    op.W = W;
    g_rec->push_back(op);
    return cudaSuccess;
  }
  const bool norm = partial != nullptr;
  const int n = p.col_off[4];
  const int n_zero = write_r ? p.n_zero : 0;
  const Units g = units(n + n_zero, L.n_tiles_int, p.n_act);
  if (n_part) *n_part = 0;
  if (g.total == 0) return cudaSuccess;
  const uint32_t* items = sizeof(T) == 8 ? L.gs_items64 : L.gs_items32;
  if (flat_on(L, p) && items && write_r && !norm) {
    // the residual before a restriction, on levels whose Gauss-Seidel runs
    // flat: one chunk per CTA
    const int* off = sizeof(T) == 8 ? L.gs_off64 : L.gs_off32;
    const int sk = skip >= 0 && skip < 4 ? skip : -1;
    const int n_items = off[4];
    const int n_if_chunks = (int)lin_grid(n + n_zero, CTA);
    const int n_vol_chunks = p.n_act > 0 ? (int)lin_grid((int64_t)n_items * p.n_act, CTA) : 0;
    ++g_kernel_launches;
    const bool dep = dep_size(p, n_if_chunks + n_vol_chunks) <= DEP_MAX_CTAS;
    auto kern = seven_point ? (dep ? k_res_flat<T, true, true, false, true> : k_res_flat<T, true, true, false, false>)
                            : (dep ? k_res_flat<T, false, true, false, true> : k_res_flat<T, false, true, false, false>);
    launch(dep_size(p, n_if_chunks + n_vol_chunks), kern, n_if_chunks + n_vol_chunks, cta_shape(), 0, s,
        L.N, L.rs, L.block, u, uI, f, fI, r, W, items, make_int4(off[0], off[1], off[2], off[3]), n_items, p.act,
        p.n_act, L.cptr, L.cps, L.cp_off, p.free_if, n, if_tab<T>(p, 0), p.zero_off, n_zero, n_if_chunks,
        n_vol_chunks, nullptr, sk, sk >= 0 ? p.col_off[sk] : 0, sk >= 0 ? p.col_off[sk + 1] : 0);
    return cudaGetLastError();
  }
  if (flat_on(L, p) && items && norm && !write_r) {
    // the stopping test's norm on small and medium levels: one chunk per CTA,
    // whose partial sums a reduction of up to FLAT_NORM_MAX terms adds up
    const int* off = sizeof(T) == 8 ? L.gs_off64 : L.gs_off32;
    const int sk = skip >= 0 && skip < 4 ? skip : -1;
    const int n_items = sk == 3 ? off[3] : off[4];
    const int n_if_chunks = (int)lin_grid(n, CTA);
    const int n_vol_chunks = p.n_act > 0 ? (int)lin_grid((int64_t)n_items * p.n_act, CTA) : 0;
    const int chunks = n_if_chunks + n_vol_chunks;
    if (chunks <= FLAT_NORM_MAX) {
      if (n_part) *n_part = chunks;
      const bool dep = dep_size(p, chunks) <= DEP_MAX_CTAS;
      auto kern = seven_point ? (dep ? k_res_flat<T, true, false, true, true> : k_res_flat<T, true, false, true, false>)
                              : (dep ? k_res_flat<T, false, false, true, true> : k_res_flat<T, false, false, true, false>);
      ++g_kernel_launches;
      launch(dep_size(p, chunks), kern, chunks, cta_shape(), 0, s, L.N, L.rs, L.block, u, uI, f, fI, r, W, items,
             make_int4(off[0], off[1], off[2], off[3]), n_items, p.act, p.n_act, L.cptr, L.cps, L.cp_off, p.free_if, n,
             if_tab<T>(p, 0), p.zero_off, 0, n_if_chunks, n_vol_chunks, partial, sk, sk >= 0 ? p.col_off[sk] : 0,
             sk >= 0 ? p.col_off[sk + 1] : 0);
      return cudaGetLastError();
    }
  }
  void (*kern)(int, const int*, int64_t, const T*, const T*, const T*, const T*, T*, const T*, const Tile*, int, const int*,
               int, const int*, const Copy*, const uint32_t*, const int*, int, IfTab<T>, const int64_t*, int, int,
               double*, int*, int, int, int);
  const int skip_lo = skip >= 0 && skip < 4 ? p.col_off[skip] : 0;
  const int skip_hi = skip >= 0 && skip < 4 ? p.col_off[skip + 1] : 0;
  const bool dep = dep_size(p, g.total) <= DEP_MAX_CTAS;
  if (write_r && norm) return cudaErrorNotSupported;   // no caller wants both
  if (seven_point)
    kern = write_r ? (dep ? k_res<T, true, true, false, true> : k_res<T, true, true, false, false>)
                   : (dep ? k_res<T, true, false, true, true> : k_res<T, true, false, true, false>);
  else
    kern = write_r ? (dep ? k_res<T, false, true, false, true> : k_res<T, false, true, false, false>)
                   : (dep ? k_res<T, false, false, true, true> : k_res<T, false, false, true, false>);
  const unsigned grid = resident_grid((const void*)kern, g.total, p.grid_cap);
  if (n_part && norm) *n_part = (int)grid;
  ++g_kernel_launches;
  launch(dep_size(p, g.total), kern, grid, cta_shape(), 0, s, L.N, L.rs, L.block, u, uI, f, fI, r, W, L.tiles_int, L.n_tiles_int, p.act,
                                    p.n_act, L.cptr, L.cps, L.cp_off, p.free_if, n, if_tab<T>(p, 0), p.zero_off, n_zero,
                                    g.n_if_units, partial, p.sched, skip >= 0 && skip < 4 ? skip : -1, skip_lo, skip_hi);
  return cudaGetLastError();
}

template <class T>
cudaError_t restrict_to(const LevelArgs& C, const LevelArgs& F, const ProbArgs& pc, const T* rf, T* fc, T* fIc, T* uc,
                        T* uIc, cudaStream_t s) {
  if (g_rec) {
    const int nl = pc.col_off[4];
    const Units g = units(nl + pc.n_zero, C.n_tiles_int * RESTRICT_SPLIT, pc.n_act);
    if (g.total == 0) return cudaSuccess;
    BOp op = new_op<T>(BOP_RESTRICT);
    op.L = F;
    op.C = C;
    op.P = pc;
    op.n_list = nl;
    op.n_zero = pc.n_zero;
    op.n_if_units = g.n_if_units;
    op.n_units = g.total;
    op.r = (void*)rf;
    op.fc = fc;
    op.fIc = fIc;
    op.uc = uc;
    op.uIc = uIc;
    g_rec->push_back(op);
    return cudaSuccess;
  }
  const int n = pc.col_off[4];
  const Units g = units(n + pc.n_zero, C.n_tiles_int * RESTRICT_SPLIT, pc.n_act);
  if (g.total == 0) return cudaSuccess;
  if (flat_on(C, pc) && C.slot_items) {
    const int n_if_ctas = (int)lin_grid(n + pc.n_zero, CTA);
    const int n_vol_ctas = pc.n_act > 0 ? (int)lin_grid((int64_t)C.n_slots * pc.n_act, CTA) : 0;
    ++g_kernel_launches;
    const int64_t size = dep_size(pc, n_if_ctas + n_vol_ctas);
    auto kern = size <= DEP_MAX_CTAS ? k_restrict_flat<T, true> : k_restrict_flat<T, false>;
    launch(size, kern, n_if_ctas + n_vol_ctas, cta_shape(), 0, s,
        C.N, C.rs, C.block, fc, fIc, uc, uIc, F.N, F.rs, F.block, rf, C.slot_items, C.n_slots, pc.act, pc.n_act,
        C.cptr, C.cps, C.cp_off, pc.free_if, n, pc.gather, pc.zero_off, pc.n_zero, n_if_ctas, n_vol_ctas);
    return cudaGetLastError();
  }
  const int64_t size = dep_size(pc, g.total);
  auto kern = size <= DEP_MAX_CTAS ? k_restrict<T, true> : k_restrict<T, false>;
  const unsigned grid = resident_grid((const void*)kern, g.total, pc.grid_cap);
  ++g_kernel_launches;
  launch(size, kern, grid, cta_shape(), 0, s, C.N, C.rs, C.block, fc, fIc, uc, uIc, F.N, F.rs, F.block, rf, C.tiles_int,
                                             C.n_tiles_int, pc.act, pc.n_act, C.cptr, C.cps, C.cp_off, pc.free_if, n,
                                             pc.gather, pc.zero_off, pc.n_zero, g.n_if_units, pc.sched);
  return cudaGetLastError();
}

template <class T>
cudaError_t prolong_add(const LevelArgs& F, const LevelArgs& C, const ProbArgs& pf, T* uf, T* uIf, const T* uc,
                        cudaStream_t s, int skip, int if_lo, int if_hi) {
  skip = skip >= 0 && skip < 4 ? skip : -1;
  if (if_hi <= if_lo) if_lo = if_hi = 0;
  if (g_rec) {
    const int nl = pf.col_off[4];
    const Units g = units(nl, F.n_tiles_int, pf.n_act);
    if (g.total == 0) return cudaSuccess;
    BOp op = new_op<T>(BOP_PROLONG);
    op.skip = skip;
    op.skip_lo = if_lo;
    op.skip_hi = if_hi;
    op.L = F;
    op.C = C;
    op.P = pf;
    op.n_list = nl;
    op.n_if_units = g.n_if_units;
    op.n_units = g.total;
    op.u = uf;
    op.uI = uIf;
    op.uc = (void*)uc;
    g_rec->push_back(op);
    return cudaSuccess;
  }
  const int n = pf.col_off[4];
  const Units g = units(n, F.n_tiles_int, pf.n_act);
  if (g.total == 0) return cudaSuccess;
  const uint32_t* items = sizeof(T) == 8 ? F.gs_items64 : F.gs_items32;
  if (flat_on(F, pf) && items && (skip == -1 || skip == 0)) {
    // the fine level's items of the colours updated: all, or 1..3 when the
    // first post-smoothing sweep overwrites colour 0
    const int* off = sizeof(T) == 8 ? F.gs_off64 : F.gs_off32;
    const int first_c = skip == 0 ? 1 : 0;
    const int n_items = off[4] - off[first_c];
    int rel[3];   // starts of the colours after first_c, relative to off[first_c]
    for (int t = 0; t < 3; ++t) {
      const int cc = first_c + 1 + t;
      rel[t] = cc <= 3 ? off[cc] - off[first_c] : n_items;
    }
    const int n_if_ctas = (int)lin_grid(n, CTA);
    const int n_vol_ctas = pf.n_act > 0 ? (int)lin_grid((int64_t)n_items * pf.n_act, CTA) : 0;
    ++g_kernel_launches;
    const int64_t size = dep_size(pf, n_if_ctas + n_vol_ctas);
    auto kern = size <= DEP_MAX_CTAS ? k_prolong_flat<T, true> : k_prolong_flat<T, false>;
    launch(size, kern, n_if_ctas + n_vol_ctas, cta_shape(), 0, s,
        F.N, F.rs, F.block, uf, uIf, C.N, C.rs, C.block, uc, items + off[first_c], n_items, first_c,
        make_int3(rel[0], rel[1], rel[2]), pf.act,
        pf.n_act, F.cptr, F.cps, F.cp_off, pf.free_if, n, if_lo, if_hi, n_if_ctas, n_vol_ctas);
    return cudaGetLastError();
  }
  const int64_t size = dep_size(pf, g.total);
  auto kern = size <= DEP_MAX_CTAS ? k_prolong<T, true> : k_prolong<T, false>;
  const unsigned grid = resident_grid((const void*)kern, g.total, pf.grid_cap);
  ++g_kernel_launches;
  launch(size, kern, grid, cta_shape(), 0, s, F.N, F.rs, F.block, uf, uIf, C.N, C.rs, C.block, uc, F.tiles_int,
                                            F.n_tiles_int, pf.act, pf.n_act, F.cptr, F.cps, F.cp_off, pf.free_if, n,
                                            g.n_if_units, pf.sched, skip, if_lo, if_hi);
  return cudaGetLastError();
}

// Launch shape of the cluster CG for n rows of at most K entries; clusters
// == 0: it does not fit (or the device holds no such cluster).
constexpr int CG_MAX_NB = 4;
struct CgShape {
  int clusters, ctas, warps, blocks_per_cta, blocks_per_warp;
  size_t smem;
};
// The register form of a shape (see k_cg_cluster).
template <class T, bool JAC>
auto cg_kernel(const CgShape& sh, int K) {
  return sh.blocks_per_warp > 1 ? k_cg_cluster<T, CG_MAX_NB, 0, JAC>
         : K <= 7               ? k_cg_cluster<T, 1, 7, JAC>
         : K <= 15              ? k_cg_cluster<T, 1, 15, JAC>
                                : k_cg_cluster<T, 1, 0, JAC>;
}
// Dynamic shared bytes a CTA may have and CTAs per cluster (16 where the device
// schedules such clusters) on the current device.
std::pair<int, int> cg_limits() {
  static std::mutex mu;
  static std::map<int, std::pair<int, int>> known;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  auto it = known.find(dev);
  if (it != known.end()) return it->second;
  int optin = 0;
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  int a = std::max(0, optin - 2048), c = 16;
  std::vector<const void*> kern = {(const void*)k_cg_cluster<float, 0, 0, false>,
                                   (const void*)k_cg_cluster<double, 0, 0, false>};
  for (int nbw : {1, CG_MAX_NB})
    for (int K : {7, 15, 16}) {
      const CgShape sh{1, 1, 1, 1, nbw, 0};
      kern.push_back((const void*)cg_kernel<float, false>(sh, K));
      kern.push_back((const void*)cg_kernel<float, true>(sh, K));
      kern.push_back((const void*)cg_kernel<double, false>(sh, K));
      kern.push_back((const void*)cg_kernel<double, true>(sh, K));
    }
  for (const void* k : kern)
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, a) != cudaSuccess ||
        cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
      a = 0;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof(cfg));
  cfg.gridDim = dim3(16);
  cfg.blockDim = dim3(1024);
  cfg.dynamicSmemBytes = (size_t)a;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 16;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, (const void*)k_cg_cluster<double, 0, 0, false>, &cfg) != cudaSuccess ||
      clusters < 1)
    c = 8;
  cudaGetLastError();
  return known.emplace(dev, std::make_pair(a, c)).first->second;
}
CgShape cg_shape(int n, int K, bool jac) {
  const std::pair<int, int> lim = cg_limits();
  CgShape g{0, 1, 1, 1, 1, 0};
  const int nb = (n + 31) / 32;
  // measured (us per solve to 1e-12): 5 blocks 79 on one CTA, 88 on 8; 11
  // blocks 162 / 92 / 97 on 1 / 8 / 16; 17 blocks 139 / 147 on 8 / 16; 42
  // blocks 187 / 183; 106 blocks 446 / 334
  const int C = std::min(nb <= 5 ? 1 : nb <= 32 ? 8 : 16, lim.second);
  int bpc = (nb + C - 1) / C;
  int W = std::min(bpc, CG_WARPS);
  int nbw = (bpc + W - 1) / W;
  const size_t sums = (jac ? 3 : 2) * (size_t)nb * 8;
  size_t smem = (size_t)bpc * 32 * 8 + sums + (nbw == 1 && K <= 15 ? 0 : (size_t)K * bpc * 32 * 12);
  if (n > 16384 || nbw > CG_MAX_NB || smem > (size_t)lim.first) {
    const int sh = cg_block_shift(n), nbl = ((n - 1) >> (5 + sh)) + 1;
    bpc = (nbl + C - 1) / C;
    W = std::min(bpc, 31);
    nbw = 0;
    smem = ((size_t)bpc << (5 + sh)) * 8 + 2 * (size_t)nbl * 8;
    if (smem > (size_t)lim.first) return g;
  }
  return CgShape{1, C, W, bpc, nbw, smem};
}

// The preconditioner is used where the diagonal varies (the host then stores
// its reciprocal), the rows fit the register forms, and the iteration runs to
// the default tolerance: a caller that caps the iterations or loosens the
// tolerance gets that many steps of plain CG.
const double* cg_precond(const DevProblem& p, double rtol, int maxit) {
  if (!p.cg_dinv || rtol > 1e-12 || maxit < 1000 || p.n_cg > 16384) return nullptr;
  return cg_shape(p.n_cg, p.cg_width, true).blocks_per_warp > 0 ? p.cg_dinv : nullptr;
}

template <class T>
cudaError_t coarse_cg(const DevProblem& p, const T* f, const T* fI, T* u, T* uI, double rtol, int maxit,
                      cudaStream_t s, double* work) {
  rtol = std::max(rtol, CG_RTOL_MIN);
  if (g_rec) {
    if (p.n_cg == 0) return cudaSuccess;
    BOp op = new_op<T>(BOP_CG);
    op.n_units = 1;
    op.n_cg = p.n_cg;
    op.rowptr = p.rowptr;
    op.col = p.col;
    op.val = p.val;
    op.fsrc = p.fsrc;
    op.uptr = p.uptr;
    op.udst = p.udst;
    op.umaster = p.umaster;
    op.work = work ? work : p.cg_work;
    op.dinv = cg_precond(p, rtol, maxit);
    op.iters = p.cg_iters;
    op.rtol = rtol;
    op.maxit = maxit;
    op.f = f;
    op.fI = fI;
    op.u = u;
    op.uI = uI;
    g_rec->push_back(op);
    return cudaSuccess;
  }
  if (p.n_cg == 0) return cudaSuccess;
  const double* dinv = cg_precond(p, rtol, maxit);
  const CgShape sh = cg_shape(p.n_cg, p.cg_width, dinv != nullptr);
  if (sh.clusters > 0) {
    CgArgs A;
    A.n = p.n_cg;
    A.K = p.cg_width;
    A.maxit = maxit;
    A.blocks_per_cta = sh.blocks_per_cta;
    A.rowptr = p.rowptr;
    A.col = p.col;
    A.val = p.val;
    A.fsrc = p.fsrc;
    A.uptr = p.uptr;
    A.udst = p.udst;
    A.umaster = p.umaster;
    A.dinv = dinv;
    A.rtol = rtol;
    A.iters = p.cg_iters;
    A.work = work ? work : p.cg_work;
    cudaLaunchConfig_t cfg;
    std::memset(&cfg, 0, sizeof(cfg));
    cfg.gridDim = dim3(sh.ctas);
    cfg.blockDim = dim3(32 * (sh.warps + 1));   // and the scalar warp
    cfg.dynamicSmemBytes = sh.smem;
    cfg.stream = s;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = sh.ctas;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = p.overlap ? 2 : 1;
    ++g_kernel_launches;
    const auto kern = sh.blocks_per_warp == 0 ? k_cg_cluster<T, 0, 0, false>
                      : dinv                  ? cg_kernel<T, true>(sh, A.K)
                                              : cg_kernel<T, false>(sh, A.K);
    return cudaLaunchKernelEx(&cfg, kern, A, f, fI, u, uI);
  }
  ++g_kernel_launches;
  launch(p.overlap ? 1 : DEP_MAX_CTAS + 1, k_cg<T>, 1, CG_THREADS, 0, s, p.n_cg, p.rowptr, p.col, p.val, p.fsrc, f, fI, p.uptr, p.udst, p.umaster, u, uI,
                                   work ? work : p.cg_work, dinv, rtol, maxit, p.cg_iters);
  return cudaGetLastError();
}

cudaError_t fma_probe(double* out, int blocks, int iters, cudaStream_t s) {
  ++g_kernel_launches;
  k_fma_probe<<<blocks, 256, 0, s>>>(out, iters, 0.999999, 1e-7);
  return cudaGetLastError();
}

cudaError_t reduce_partials(const double* partial, int n, double* out, cudaStream_t s, double* host, const int* err,
                            int* host_err) {
  if (g_rec) return cudaSuccess;   // a batch needs no norms
  ++g_kernel_launches;
  launch(1, k_reduce, 1, 1024, 0, s, partial, n, out, host, err, host_err);
  return cudaGetLastError();
}

cudaError_t import_problem(const LevelArgs& L, const MacroGeo* geo, int n_macro, int64_t nx, int64_t ny,
                           const double* gf, const double* gu, double* f, double* fs, const double* winv, double* u,
                           const int64_t* if_gid, int n_if, double* fI, double* uI, cudaStream_t s) {
  const int n_if_ctas = (int)lin_grid(n_if, CTA);
  const int64_t grid = n_if_ctas + (int64_t)L.n_tiles_all * n_macro;
  if (grid == 0) return cudaSuccess;
  if (grid > INT32_MAX) return cudaErrorInvalidConfiguration;
  ++g_kernel_launches;
  launch(grid, k_import, (unsigned)grid, cta_shape(), 0, s, L.N, L.rs, L.block, geo, nx, ny, gf, gu, f, fs, winv, u,
         L.tiles_all, L.n_tiles_all, if_gid, n_if, fI, uI, n_if_ctas);
  return cudaGetLastError();
}

cudaError_t export_solution(const LevelArgs& L, const MacroGeo* geo, int n_macro, int64_t nx, int64_t ny,
                            const double* u, const double* uI, const int64_t* if_gid, int n_if, double* g,
                            cudaStream_t s) {
  const int n_if_ctas = (int)lin_grid(n_if, CTA);
  const int64_t grid = n_if_ctas + (int64_t)L.n_tiles_all * n_macro;
  if (grid == 0) return cudaSuccess;
  if (grid > INT32_MAX) return cudaErrorInvalidConfiguration;
  ++g_kernel_launches;
  launch(grid, k_export, (unsigned)grid, cta_shape(), 0, s, L.N, L.rs, L.block, geo, nx, ny, u, uI, g, L.tiles_all,
         L.n_tiles_all, if_gid, n_if, n_if_ctas);
  return cudaGetLastError();
}

template <class T>
cudaError_t import_masters(const int64_t* gid, int n, const double* g, T* m, cudaStream_t s) {
  if (n > 0) {
    ++g_kernel_launches;
    launch(lin_grid(n, 256), k_import_if<T>, lin_grid(n, 256), 256, 0, s, gid, n, g, m);
  }
  return cudaGetLastError();
}

template <class T>
cudaError_t export_masters(const int64_t* gid, int n, const T* m, double* g, cudaStream_t s) {
  if (n > 0) {
    ++g_kernel_launches;
    launch(lin_grid(n, 256), k_export_if<T>, lin_grid(n, 256), 256, 0, s, gid, n, m, g);
  }
  return cudaGetLastError();
}

cudaError_t grad_partials(const LevelArgs& L, int n_macro, const double* u, const double* lam, const double* W,
                          double* partial, cudaStream_t s) {
  if (L.n_tiles_all > 0 && n_macro > 0) {
    ++g_kernel_launches;
    launch((int64_t)L.n_tiles_all * n_macro, k_grad, dim3((unsigned)L.n_tiles_all, (unsigned)n_macro), cta_shape(), 0, s, L.N, L.rs, L.block, u, lam, W,
                                                                                   L.tiles_all, partial);
  }
  return cudaGetLastError();
}

cudaError_t reduce_per_macro(const double* partial, int n_per, int n_macro, double* out, cudaStream_t s) {
  if (n_macro > 0) {
    ++g_kernel_launches;
    launch(n_macro, k_reduce_per_macro, n_macro, 256, 0, s, partial, n_per, out);
  }
  return cudaGetLastError();
}

cudaError_t apply_if_nodes(const LevelArgs& L, const double* u, const double* uI, const double* W, bool seven_point,
                           const int* list, int n, double* out, cudaStream_t s) {
  if (n > 0) {
    ++g_kernel_launches;
    if (seven_point)
      launch(lin_grid(n, 128), k_if_apply<true>, lin_grid(n, 128), 128, 0, s, L.N, L.rs, L.block, u, uI, W, L.cptr, L.cps, list, n, out);
    else
      launch(lin_grid(n, 128), k_if_apply<false>, lin_grid(n, 128), 128, 0, s, L.N, L.rs, L.block, u, uI, W, L.cptr, L.cps, list, n, out);
  }
  return cudaGetLastError();
}

cudaError_t copy_listed(const double* src, double* dst, const int* idx, int n, cudaStream_t s) {
  if (n > 0) {
    ++g_kernel_launches;
    launch(lin_grid(n, 256), k_copy_listed, lin_grid(n, 256), 256, 0, s, src, dst, idx, n);
  }
  return cudaGetLastError();
}

cudaError_t set_masters_zero(double* uI, const int* ids, int n, cudaStream_t s) {
  if (g_rec) {
    if (n <= 0) return cudaSuccess;
    BOp op = new_op<double>(BOP_SET_ZERO);
    op.uI = uI;
    op.ids = ids;
    op.n = n;
    op.n_units = (int)lin_grid(n, CTA);
    g_rec->push_back(op);
    return cudaSuccess;
  }
  if (n > 0) {
    ++g_kernel_launches;
    launch(lin_grid(n, 256), k_set_masters_zero, lin_grid(n, 256), 256, 0, s, uI, ids, n);
  }
  return cudaGetLastError();
}

cudaError_t scale_blocks(const double* f, const double* winv, double* out, int n_macro, int64_t block,
                         cudaStream_t s) {
  const int64_t total = (int64_t)n_macro * block;
  if (total > 0) {
    ++g_kernel_launches;
    launch(lin_grid(total, 256), k_scale_blocks, (unsigned)std::min<int64_t>(lin_grid(total, 256), 152 * 16), 256, 0, s, f, winv, out, n_macro,
                                                                                               block);
  }
  return cudaGetLastError();
}

cudaError_t restore_copies(double* u, const double* uI, const int64_t* off, const int* master, int n, cudaStream_t s) {
  if (g_rec) {
    if (n <= 0) return cudaSuccess;
    BOp op = new_op<double>(BOP_RESTORE);
    op.u = u;
    op.uI = (void*)uI;
    op.offs = off;
    op.ids = master;
    op.n = n;
    op.n_units = (int)lin_grid(n, CTA);
    g_rec->push_back(op);
    return cudaSuccess;
  }
  if (n > 0) {
    ++g_kernel_launches;
    launch(lin_grid(n, 256), k_restore, lin_grid(n, 256), 256, 0, s, u, uI, off, master, n);
  }
  return cudaGetLastError();
}

cudaError_t residual_to_f32(const LevelArgs& L, const ProbArgs& p, const double* u, const double* uI, const double* f,
                            const double* fI, float* f32, float* fI32, const double* W, bool seven_point,
                            double* partial, int* n_part, cudaStream_t s) {
  if (g_rec) {
    const int nl = p.col_off[4];
    const Units g = units(nl, L.n_tiles_int, p.n_act);
    if (n_part) *n_part = 0;
    if (g.total == 0) return cudaSuccess;
    BOp op = new_op<double>(BOP_RES_F32);
    op.seven_point = seven_point ? 1 : 0;
    op.L = L;
    op.P = p;
    op.n_list = nl;
    op.n_if_units = g.n_if_units;
    op.n_units = g.total;
    op.u = (void*)u;
    op.uI = (void*)uI;
    op.f = f;
    op.fI = fI;
    op.o32 = f32;
    op.oI32 = fI32;
    op.W = W;
    g_rec->push_back(op);
    return cudaSuccess;
  }
  const int n = p.col_off[4];
  const Units g = units(n, L.n_tiles_int, p.n_act);
  if (n_part) *n_part = 0;
  if (g.total == 0) return cudaSuccess;
  auto kern = seven_point ? k_res_f32<true> : k_res_f32<false>;
  const unsigned grid = resident_grid((const void*)kern, g.total, p.grid_cap);
  if (n_part) *n_part = (int)grid;
  ++g_kernel_launches;
  launch(dep_size(p, g.total), kern, grid, cta_shape(), 0, s, L.N, L.rs, L.block, u, uI, f, fI, f32, fI32, W, L.tiles_int, L.n_tiles_int, p.act,
                                    p.n_act, L.cptr, L.cps, p.free_if, n, if_tab<double>(p, 0), g.n_if_units, partial,
                                    p.sched);
  return cudaGetLastError();
}

cudaError_t add_correction(const LevelArgs& L, const ProbArgs& p, double* u, double* uI, const float* e,
                           const float* eI, cudaStream_t s) {
  if (g_rec) {
    if (p.n_act > 0) {
      BOp op = new_op<double>(BOP_ADD_BLOCKS);
      op.L = L;
      op.P = p;
      op.u = u;
      op.o32 = (void*)e;
      op.n_units = (int)(p.n_act * block_chunks(L.block));
      g_rec->push_back(op);
    }
    if (p.col_off[4] > 0) {
      BOp op = new_op<double>(BOP_ADD_MASTERS);
      op.uI = uI;
      op.oI32 = (void*)eI;
      op.ids = p.free_if;
      op.n = p.col_off[4];
      op.n_units = (int)lin_grid(op.n, CTA);
      g_rec->push_back(op);
    }
    return cudaSuccess;
  }
  if (p.n_act > 0) {
    const int64_t per = 256 * 8;
    const unsigned gx = (unsigned)std::min<int64_t>((L.block / 2 + per - 1) / per, 4096);
    ++g_kernel_launches;
    launch(dep_size(p, (int64_t)gx * p.n_act), k_add_corr_blocks, dim3(gx, (unsigned)p.n_act), 256, 0, s, u, e, L.block, p.act);
  }
  const int n = p.col_off[4];
  if (n > 0) {
    ++g_kernel_launches;
    launch(dep_size(p, lin_grid(n, 256)), k_add_corr_masters, lin_grid(n, 256), 256, 0, s, uI, eI, p.free_if, n);
  }
  return cudaGetLastError();
}

template <class T>
cudaError_t zero_problem_blocks(const LevelArgs& L, const ProbArgs& p, T* u, T* uI, cudaStream_t s) {
  if (g_rec) {
    if (p.n_act > 0) {
      BOp op = new_op<T>(BOP_ZERO_BLOCKS);
      op.L = L;
      op.P = p;
      op.u = u;
      op.n_units = (int)(p.n_act * block_chunks(L.block));
      g_rec->push_back(op);
    }
    if (p.col_off[4] > 0) {
      BOp op = new_op<T>(BOP_ZERO_LIST);
      op.uI = uI;
      op.ids = p.free_if;
      op.n = p.col_off[4];
      op.n_units = (int)lin_grid(op.n, CTA);
      g_rec->push_back(op);
    }
    return cudaSuccess;
  }
  if (p.n_act > 0) {
    const int64_t per = 256 * 8;
    unsigned gx = (unsigned)std::min<int64_t>((L.block + per - 1) / per, 4096);
    ++g_kernel_launches;
    launch(dep_size(p, (int64_t)gx * p.n_act), k_zero_blocks<T>, dim3(gx, p.n_act), 256, 0, s, u, L.block, p.act);
  }
  const int n = p.col_off[4];
  if (n > 0) {
    ++g_kernel_launches;
    launch(dep_size(p, lin_grid(n, 256)), k_zero_list<T>, lin_grid(n, 256), 256, 0, s, uI, p.free_if, n);
  }
  return cudaGetLastError();
}

#define HHG_INSTANTIATE(T)                                                                                        \
  template cudaError_t gs_colour<T>(const LevelArgs&, const ProbArgs&, T*, T*, const T*, const T*, const T*,   \
                                    const T*, int, bool, cudaStream_t, cudaEvent_t, cudaEvent_t, const T*,      \
                                    const T*);                                                                  \
  template cudaError_t residual<T>(const LevelArgs&, const ProbArgs&, const T*, const T*, const T*, const T*, T*, \
                                   const T*, bool, bool, double*, int*, cudaStream_t, int);                    \
  template cudaError_t restrict_to<T>(const LevelArgs&, const LevelArgs&, const ProbArgs&, const T*, T*, T*, T*, \
                                      T*, cudaStream_t);                                                       \
  template cudaError_t prolong_add<T>(const LevelArgs&, const LevelArgs&, const ProbArgs&, T*, T*, const T*,     \
                                      cudaStream_t, int, int, int);                                            \
  template cudaError_t coarse_cg<T>(const DevProblem&, const T*, const T*, T*, T*, double, int, cudaStream_t,     \
                                    double*);                                                                  \
  template cudaError_t import_masters<T>(const int64_t*, int, const double*, T*, cudaStream_t);                  \
  template cudaError_t export_masters<T>(const int64_t*, int, const T*, double*, cudaStream_t);                  \
  template cudaError_t zero_problem_blocks<T>(const LevelArgs&, const ProbArgs&, T*, T*, cudaStream_t);

HHG_INSTANTIATE(double)
HHG_INSTANTIATE(float)

}  // namespace hhg
