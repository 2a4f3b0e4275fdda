// 3D friends-of-friends over a periodic snapshot (Section "Parallelization": every process runs
// 3D FoF on its particles before subhalo finding).
//
// Pipeline (one stream, no host round trip except the optional group count):
//   k_cell_keys   cell key per particle on a grid of sub-cells of side sc <= 0.99 ll / sqrt(3)
//                 (so two particles in one sub-cell are always linked) -> mixed-radix key
//                 (z ns + y) ns + x; value = particle index
//   radix sort    (key, index), ceil(log2 ns^3) key bits (32 for ns = 1600, not 3*11)
//   k_cell_heads, k_cells   the occupied sub-cells in key order: first particle, row (z ns + y), x,
//                 and every particle's cell; sorted positions as float4
//   k_row_cells   dense table of the first cell of every row
//   k_link_cells  union-find over the occupied cells (every sub-cell is a clique, so one linked
//                 pair joins two cells): first the adjacent cells, then, after a compression, the
//                 rest of the half stencil of R sub-cells, where most cells in reach already share
//                 a root. A thread per cell tests a few pairs of two large cells and lists them for
//   k_link_pairs  (a block per listed pair of cells, if their roots still differ)
//   k_cell_min    each cell's smallest id; k_group_min lowers every root's to its group's
//   k_fof_labels  label of every particle in input order
//
// A thread per particle searching the stencil repeated each search for all particles of a dense cell,
// with two root searches per visited cell. Measured on 2^24 particles in L = 256 Mpc/h: link kernels
// 6.4 -> 2.0 ms, the whole call 8.8 -> 4.2 ms; 2^27 particles in L = 512: 51 -> 15 ms. In the 2^24 case (ncu) the
// far pass has its issue slots busy 75% of the cycles (row searches); the near pass 52%, its warps waiting 14
// cycles an instruction for gathers. Searching the rows of one z side by side, to overlap their loads, was
// slower: 20 ms.
#include <cmath>

#include "rs_common.cuh"

namespace {

constexpr int kThreads = 256;

struct Grid3 {
  int ns;        // sub-cells per axis
  int R;         // stencil radius in sub-cells
  bool full;     // 2R+1 > ns: visit every cell once instead of the half stencil
  float inv_sc;  // ns / L
};

int make_grid(rs_ctx* ctx, float L, float ll, Grid3* g) {
  if (!(L > 0.f) || !(ll > 0.f) || !std::isfinite(L) || !std::isfinite(ll))
    return rs::set_error(ctx, RS_ERR_INVALID_ARG, "box_L and link_len must be positive");
  const double sc_target = 0.99 * double(ll) / std::sqrt(3.0);
  double nsd = std::ceil(double(L) / sc_target);
  if (nsd < 1) nsd = 1;
  if (nsd > 4096)
    return rs::set_error(ctx, RS_ERR_INVALID_ARG,
                         "box_L / link_len = %g needs more than 4096 sub-cells per axis",
                         double(L) / double(ll));
  g->ns = int(nsd);
  const double sc = double(L) / g->ns;
  int R = 1;
  while (R * sc <= double(ll) * (1.0 + 1e-3)) ++R;
  g->R = R;
  g->full = (2 * R + 1) > g->ns;
  g->inv_sc = float(double(g->ns) / double(L));
  return RS_OK;
}

__global__ void __launch_bounds__(kThreads)
k_cell_keys(int64_t n, const float* __restrict__ pos, float inv_sc, int ns,
            uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  uint32_t c[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    const float x = pos[3 * i + d];
    int k = int(__fmul_rn(x, inv_sc));
    k = k < 0 ? 0 : (k >= ns ? ns - 1 : k);
    c[d] = uint32_t(k);
  }
  keys[i] = (uint64_t(c[2]) * uint64_t(ns) + c[1]) * uint64_t(ns) + c[0];  // mixed radix
  vals[i] = uint32_t(i);
}

// Occupied cells: a head is a sorted position whose key differs from the one before. Tiles of
// kHeadTile positions: k_cell_heads counts a tile's heads, k_cells (after a scan of the counts)
// numbers them.
constexpr int kHeadPer = 8;
constexpr int kHeadTile = kThreads * kHeadPer;

__device__ __forceinline__ bool is_head(const uint64_t* __restrict__ keys, int64_t i, uint64_t key) {
  return i == 0 || keys[i - 1] != key;
}

__global__ void __launch_bounds__(kThreads)
k_cell_heads(int64_t n, const uint64_t* __restrict__ keys, int64_t* __restrict__ count) {
  __shared__ int wsum[kThreads / 32];
  int c = 0;
#pragma unroll
  for (int k = 0; k < kHeadPer; ++k) {
    const int64_t i = int64_t(blockIdx.x) * kHeadTile + k * kThreads + threadIdx.x;
    c += __popc(__ballot_sync(0xffffffffu, i < n && is_head(keys, i, keys[i])));
  }
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < kThreads / 32; ++w) t += wsum[w];
    count[blockIdx.x] = t;
  }
}

struct Cells {
  const int64_t* count;       // occupied cells (device)
  uint32_t* start;            // [cells + 1] first sorted particle
  uint32_t* row;              // z ns + y
  uint16_t* x;
  uint32_t* parent;           // union-find
  const uint32_t* row_cell;   // [ns^2 + 1] first cell of each row
  const float4* pos;          // sorted positions
};

// Cell tables, the cell of every sorted particle, and the sorted positions.
__global__ void __launch_bounds__(kThreads)
k_cells(int64_t n, const uint64_t* __restrict__ keys, const uint32_t* __restrict__ idx,
        const float* __restrict__ pos, int ns, const int64_t* __restrict__ tile_off, Cells C,
        float4* __restrict__ posS, uint32_t* __restrict__ cell_of) {
  __shared__ int wsum[kHeadPer][kThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t key[kHeadPer];
  unsigned heads[kHeadPer];
#pragma unroll
  for (int k = 0; k < kHeadPer; ++k) {
    const int64_t i = int64_t(blockIdx.x) * kHeadTile + k * kThreads + threadIdx.x;
    key[k] = i < n ? keys[i] : 0ull;
    heads[k] = __ballot_sync(0xffffffffu, i < n && is_head(keys, i, key[k]));
    if (lane == 0) wsum[k][warp] = __popc(heads[k]);
  }
  __syncthreads();
  if (threadIdx.x < 32) {  // exclusive scan of the 64 warp counts, in position order
    int* w = &wsum[0][0];
    static_assert(kHeadPer * (kThreads / 32) == 64, "two counts a lane");
    const int a = w[2 * lane], b = w[2 * lane + 1];
    int incl = a + b;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += t;
    }
    w[2 * lane] = incl - a - b;
    w[2 * lane + 1] = incl - b;
  }
  __syncthreads();
  const uint32_t base = uint32_t(tile_off[blockIdx.x]);
#pragma unroll
  for (int k = 0; k < kHeadPer; ++k) {
    const int64_t i = int64_t(blockIdx.x) * kHeadTile + k * kThreads + threadIdx.x;
    if (i >= n) continue;
    // heads up to and including this position, minus one
    const uint32_t c = base + uint32_t(wsum[k][warp] + __popc(heads[k] & (0xffffffffu >> (31 - lane)))) - 1u;
    cell_of[i] = c;
    const int64_t s = idx[i];
    posS[i] = make_float4(pos[3 * s], pos[3 * s + 1], pos[3 * s + 2], 0.f);
    if ((heads[k] >> lane) & 1u) {
      uint32_t row, x;
      if (key[k] < (uint64_t(1) << 32)) {  // 32-bit division whenever ns^3 fits (ns <= 1625)
        row = uint32_t(key[k]) / uint32_t(ns);
        x = uint32_t(key[k]) - row * uint32_t(ns);
      } else {
        row = uint32_t(key[k] / uint64_t(ns));
        x = uint32_t(key[k] - uint64_t(row) * uint64_t(ns));
      }
      C.start[c] = uint32_t(i);
      C.row[c] = row;
      C.x[c] = uint16_t(x);
      C.parent[c] = c;
    }
    if (i == n - 1) C.start[c + 1] = uint32_t(n);
  }
}

// row_cell[r] = first cell of a row >= r, r in [0, rows]: one thread per row, binary search over the
// cells (neighbouring rows share search paths).
__global__ void __launch_bounds__(kThreads)
k_row_cells(Cells C, int64_t rows, uint32_t* __restrict__ row_cell) {
  const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r > rows) return;
  uint32_t lo = 0, hi = uint32_t(*C.count);
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if (C.row[mid] < uint32_t(r)) lo = mid + 1; else hi = mid;
  }
  row_cell[r] = lo;
}

// A listed pair of cells: the particles [chunk, chunk + 1) kPairChunk of cell a against cell b.
struct PairItem {
  uint32_t a, b, chunk;
};
constexpr uint32_t kPairChunk = 1024;

// Pairs whose larger cell holds at most kSmallPair particles share the first `cap` items; when those are
// full a thread tests the pair by itself. The other pairs have items of their own after them, enough for
// all there can be (pair_items), so that no thread is left with the pairs of two large cells: a call with
// 1e8 pairs of particles beside a full list took 22 s on one thread, 7 ms in this form.
constexpr uint32_t kSmallPair = 512;

// Most items of pairs with a cell above kSmallPair. A pair takes ceil(s / kPairChunk) items, s its larger
// cell's particles; a cell has at most `reach` others in its stencil, and all pairs of a few cells are few.
int64_t pair_items(int64_t n, int ns, int R) {
  const int64_t cells = rsd::min64(n, int64_t(ns) * ns * ns), d = rsd::min64(2 * int64_t(R) + 1, ns);
  const int64_t reach = d * d * d - 1;
  const double per_cell = double(reach) * double(n) * (1.0 / kPairChunk + 1.0 / kSmallPair);
  const double all_pairs = double(cells) * (double(n) / kPairChunk + 0.5 * double(cells));
  return int64_t(std::min(per_cell, all_pairs)) + 1;
}

struct LinkArgs {
  Cells C;
  int ns, R;
  bool full;
  float L, hL, ll2;
  PairItem* items;
  unsigned long long* n_items;  // [0] of small pairs, [1] of the others
  unsigned long long cap;
};

__device__ __forceinline__ bool linked(const LinkArgs& A, float4 p, float4 q) {
  return rsd::sq3(rsd::wrap_diff(p.x, q.x, A.L, A.hL), rsd::wrap_diff(p.y, q.y, A.L, A.hL),
                  rsd::wrap_diff(p.z, q.z, A.L, A.hL)) <= A.ll2;
}

// Cells a and b with different roots: unite them if one pair of their particles is linked. All pairs
// when there are at most kInline of them; otherwise a 4 x 4 sample first (two dense adjacent cells are
// linked by almost any pair), and the pair of cells is listed when the sample has no link.
constexpr uint32_t kInline = 64;

__device__ __forceinline__ void test_cells(const LinkArgs& A, uint32_t a, uint32_t b) {
  const uint32_t a0 = A.C.start[a], na = A.C.start[a + 1] - a0, b0 = A.C.start[b], nb = A.C.start[b + 1] - b0;
  const bool small = uint64_t(na) * nb <= kInline;
  const uint32_t sa = small ? 1u : max(na / 4u, 1u), sb = small ? 1u : max(nb / 4u, 1u);
  for (uint32_t i = 0; i < na; i += sa) {
    const float4 p = A.C.pos[a0 + i];
    for (uint32_t j = 0; j < nb; j += sb)
      if (linked(A, p, A.C.pos[b0 + j])) {
        rsd::uf_unite(A.C.parent, a, b);
        return;
      }
  }
  if (small) return;
  const uint32_t larger = max(na, nb);
  if (larger > kSmallPair) {
    const uint32_t chunks = (larger + kPairChunk - 1) / kPairChunk;
    const unsigned long long k = A.cap + atomicAdd(A.n_items + 1, (unsigned long long)chunks);
    for (uint32_t c = 0; c < chunks; ++c) A.items[k + c] = na < nb ? PairItem{b, a, c} : PairItem{a, b, c};
    return;
  }
  const unsigned long long k = atomicAdd(A.n_items, 1ull);
  if (k < A.cap) {
    A.items[k] = na < nb ? PairItem{b, a, 0} : PairItem{a, b, 0};
    return;
  }
  for (uint32_t i = 0; i < na; ++i) {
    const float4 p = A.C.pos[a0 + i];
    for (uint32_t j = 0; j < nb; ++j)
      if (linked(A, p, A.C.pos[b0 + j])) {
        rsd::uf_unite(A.C.parent, a, b);
        return;
      }
  }
}

// Candidate pairs of cells found by a warp's lanes, tested 32 at a time: a dense cell has a dozen
// occupied neighbours and most cells none, so testing them where they are found left three lanes in
// four idle.
struct PairQueue {
  uint32_t a[64], b[64];
  int n;
};

__device__ __forceinline__ void test_roots(const LinkArgs& A, uint32_t a, uint32_t b) {
  if (rsd::uf_find(A.C.parent, a) != rsd::uf_find(A.C.parent, b)) test_cells(A, a, b);
}

// Tests queued pairs while more than `keep` are left. Every lane of the warp takes part, with the
// length that one lane read: no lane goes on to queue its next row's pairs before all know it.
__device__ __forceinline__ void flush_pairs(const LinkArgs& A, PairQueue& Q, int keep, int lane) {
  __syncwarp();
  const int queued = __shfl_sync(0xffffffffu, min(Q.n, 64), 0);  // the pairs beyond were tested at once
  if (queued <= keep) return;
  int n = queued;
  while (n > keep) {
    const int k = max(n - 32, 0);
    if (k + lane < n) test_roots(A, Q.a[k + lane], Q.b[k + lane]);
    n = k;
  }
  __syncwarp();
  if (lane == 0) Q.n = n;
  __syncwarp();
}

// The occupied cells with x in [x0, x1] of a row against cell c. kFar: cells within one of x (kx) in a
// row of adjacent cells (`near_row`) are done, and parents are compressed, so equal parents mean one
// component (pc: c's).
template <bool kFar>
__device__ __forceinline__ void scan_cells(const LinkArgs& A, uint32_t c, uint32_t pc, uint32_t row, int x0, int x1,
                                           bool near_row, int kx, PairQueue& Q) {
  uint32_t lo = A.C.row_cell[row], hi = A.C.row_cell[row + 1];
  const uint32_t end = hi;
  while (lo < hi) {
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if (int(A.C.x[mid]) < x0) lo = mid + 1; else hi = mid;
  }
  for (; lo < end; ++lo) {
    const int x = int(A.C.x[lo]);
    if (x > x1) break;
    if (kFar) {
      const int dx = abs(x - kx);
      if ((near_row && (dx <= 1 || dx == A.ns - 1)) || __ldcg(A.C.parent + lo) == pc) continue;
    }
    const int k = atomicAdd(&Q.n, 1);
    if (k < 64) {
      Q.a[k] = c;
      Q.b[k] = lo;
    } else {
      test_roots(A, c, lo);
    }
  }
}

// One thread per occupied cell over half of its stencil: the adjacent cells (kFar = false), then the
// other cells within R.
template <bool kFar>
__global__ void __launch_bounds__(kThreads) k_link_cells(LinkArgs A) {
  __shared__ PairQueue queues[kThreads / 32];
  PairQueue& Q = queues[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31, ns = A.ns;
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool valid = t < *A.C.count;
  if (!__any_sync(0xffffffffu, valid)) return;
  const uint32_t c = uint32_t(t);
  if (A.full) {  // a box of a few cells: every pair once
    if (!valid) return;
    for (uint32_t o = c + 1; o < uint32_t(*A.C.count); ++o) test_roots(A, c, o);
    return;
  }
  if (lane == 0) Q.n = 0;
  __syncwarp();
  const uint32_t row = valid ? A.C.row[c] : 0u;
  const uint32_t pc = kFar && valid ? __ldcg(A.C.parent + c) : 0u;
  const int kz = int(row / uint32_t(ns)), ky = int(row) - kz * ns, kx = valid ? int(A.C.x[c]) : 0;
  const int R = kFar ? A.R : 1;
  for (int dz = 0; dz <= R; ++dz)
    for (int dy = dz == 0 ? 0 : -R; dy <= R; ++dy) {
      if (valid) {
        const bool own = dz == 0 && dy == 0, near_row = dz <= 1 && dy >= -1 && dy <= 1;
        // periodic wrap of offsets within one box length (|offset| <= R < ns): a compare and an add
        // instead of an integer division
        int zz = kz + dz, yy = ky + dy;
        zz -= zz >= ns ? ns : 0;
        yy += yy < 0 ? ns : (yy >= ns ? -ns : 0);
        const uint32_t r = uint32_t(zz) * uint32_t(ns) + uint32_t(yy);
        const int xa = own ? kx + (kFar ? 2 : 1) : kx - R, xb = kx + R;
        if (xa < ns) scan_cells<kFar>(A, c, pc, r, max(xa, 0), min(xb, ns - 1), near_row, kx, Q);
        if (xa < 0) scan_cells<kFar>(A, c, pc, r, xa + ns, ns - 1, near_row, kx, Q);
        if (xb >= ns) scan_cells<kFar>(A, c, pc, r, max(xa - ns, 0), xb - ns, near_row, kx, Q);
      }
      flush_pairs(A, Q, 31, lane);
    }
  flush_pairs(A, Q, 0, lane);
}

// Listed pairs of cells: a block per item, skipped when the cells have come to share a root.
__global__ void __launch_bounds__(kThreads) k_link_pairs(LinkArgs A) {
  __shared__ float4 tile[kThreads];
  __shared__ int skip;
  const unsigned long long few = min(A.n_items[0], A.cap), total = few + A.n_items[1];
  for (unsigned long long w = blockIdx.x; w < total; w += gridDim.x) {
    const PairItem it = A.items[w < few ? w : A.cap + (w - few)];
    __syncthreads();
    if (threadIdx.x == 0) skip = rsd::uf_find(A.C.parent, it.a) == rsd::uf_find(A.C.parent, it.b);
    __syncthreads();
    if (skip) continue;
    const uint32_t a0 = A.C.start[it.a] + it.chunk * kPairChunk, a1 = min(a0 + kPairChunk, A.C.start[it.a + 1]);
    const uint32_t b0 = A.C.start[it.b], b1 = A.C.start[it.b + 1];
    for (uint32_t j0 = b0; j0 < b1; j0 += kThreads) {
      const uint32_t jn = min(b1 - j0, uint32_t(kThreads));
      if (threadIdx.x < jn) tile[threadIdx.x] = A.C.pos[j0 + threadIdx.x];
      __syncthreads();
      bool hit = false;
      for (uint32_t i = a0 + threadIdx.x; i < a1 && !hit; i += kThreads) {
        const float4 p = A.C.pos[i];
        for (uint32_t j = 0; j < jn && !hit; ++j) hit = linked(A, p, tile[j]);
      }
      if (__syncthreads_or(hit)) {
        if (threadIdx.x == 0) rsd::uf_unite(A.C.parent, it.a, it.b);
        break;
      }
    }
  }
}

__global__ void __launch_bounds__(kThreads) k_fof_compress(Cells C) {
  const int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (c < *C.count) C.parent[c] = rsd::uf_find_ro(C.parent, uint32_t(c));
}

// Smallest id of every cell (minid starts at ~0): a plain store where the cell's particles lie within
// one warp (most cells hold one particle), an atomic minimum otherwise.
__global__ void __launch_bounds__(kThreads)
k_cell_min(int64_t n, const uint32_t* __restrict__ cell_of, const uint32_t* __restrict__ idx,
           const int64_t* __restrict__ ids, Cells C, unsigned long long* __restrict__ minid) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  const bool valid = i < n;  // every lane stays for the run reduction
  const uint32_t c = valid ? cell_of[i] : 0xffffffffu;
  unsigned long long v = valid ? (unsigned long long)ids[idx[i]] : ~0ull;
  bool head;
  const uint32_t rid = rsd::run_id(c, valid, head);
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const unsigned long long o = __shfl_down_sync(0xffffffffu, v, off);
    const uint32_t ro = __shfl_down_sync(0xffffffffu, rid, off);
    if (lane + off < 32 && ro == rid && o < v) v = o;
  }
  if (!head) return;
  if (int64_t(C.start[c]) == i && int64_t(C.start[c + 1]) <= i - lane + 32)
    minid[c] = v;
  else
    atomicMin(minid + c, v);
}

// Every other cell of a group lowers its root's id; roots are counted, one atomic per block of a grid
// that strides over the cells (one per warp of a full grid queued at that one address: 0.36 ms for
// 2^24 particles).
__global__ void __launch_bounds__(kThreads)
k_group_min(Cells C, unsigned long long* __restrict__ minid, unsigned long long* __restrict__ groups) {
  __shared__ unsigned long long wsum[kThreads / 32];
  const int64_t n = *C.count, step = int64_t(gridDim.x) * kThreads;
  unsigned long long roots = 0;
  for (int64_t c0 = int64_t(blockIdx.x) * kThreads; c0 < n; c0 += step) {
    const int64_t c = c0 + threadIdx.x;
    const bool in = c < n;  // every lane stays for the run reduction
    const uint32_t r = in ? C.parent[c] : 0u;
    const bool root = in && r == uint32_t(c);
    roots += __popc(__ballot_sync(0xffffffffu, root));
    rsd::warp_run_min(minid, r, in && !root, in && !root ? minid[c] : ~0ull);
  }
  if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = roots;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < kThreads / 32; ++w) roots += wsum[w];
    if (roots) atomicAdd(groups, roots);
  }
}

__global__ void __launch_bounds__(kThreads)
k_fof_labels(int64_t n, const uint32_t* __restrict__ cell_of, const uint32_t* __restrict__ idx, Cells C,
             const unsigned long long* __restrict__ minid, int64_t* __restrict__ label_out) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  label_out[idx[i]] = int64_t(minid[C.parent[cell_of[i]]]);
}

}  // namespace

namespace {
__global__ void k_ids_as_keys(int64_t n, const int64_t* __restrict__ ids, uint64_t* __restrict__ keys,
                              uint32_t* __restrict__ vals) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  keys[i] = uint64_t(ids[i]);
  vals[i] = uint32_t(i);
}

// Invalid ids among the sorted ids: a repeated value, or a negative one (sorted last as uint64).
__global__ void k_bad_ids(int64_t n, const uint64_t* __restrict__ keys, unsigned long long* __restrict__ bad) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const bool b = (i > 0 && keys[i] == keys[i - 1]) || (keys[i] >> 63) != 0;
  rsd::warp_count(bad, b);
}
}  // namespace

// The optional check that ids are unique and non-negative (rs_config.check_ids): a 64-bit radix
// sort of the ids and a comparison of neighbours.
static int check_ids(rs_ctx* ctx, int64_t n, const int64_t* ids, cudaStream_t st) {
  using namespace rs;
  uint64_t* ka = scratch_t<uint64_t>(ctx, S_KEY_A, n);
  uint64_t* kb = scratch_t<uint64_t>(ctx, S_KEY_B, n);
  uint32_t* va = scratch_t<uint32_t>(ctx, S_VAL_A, n);
  uint32_t* vb = scratch_t<uint32_t>(ctx, S_VAL_B, n);
  unsigned long long* bad = scratch_t<unsigned long long>(ctx, S_COUNTER, 8);
  if (!ka || !kb || !va || !vb || !bad) return RS_ERR_OOM;
  k_ids_as_keys<<<grid_for(n, 256), 256, 0, st>>>(n, ids, ka, va);
  RS_LAUNCHED(ctx, "k_ids_as_keys");
  uint64_t* ks;
  uint32_t* vs;
  RS_TRY(radix_sort_u64(ctx, n, 64, ka, va, kb, vb, &ks, &vs, st));
  RS_CUDA(ctx, cudaMemsetAsync(bad, 0, 8, st));
  k_bad_ids<<<grid_for(n, 256), 256, 0, st>>>(n, ks, bad);
  RS_LAUNCHED(ctx, "k_bad_ids");
  RS_TRY(read_back(ctx, bad, 8, st));
  if (ctx->host_box[0] != 0)
    return set_error(ctx, RS_ERR_INVALID_ARG, "%lld repeated or negative ids",
                     (long long)ctx->host_box[0]);
  return RS_OK;
}

extern "C" int rs_fof3d(rs_ctx* ctx, int64_t n, const float* pos, const int64_t* ids,
                        int64_t* label_out, int64_t* n_groups_out, void* stream) {
  if (!ctx) return RS_ERR_INVALID_ARG;
  ctx->err[0] = 0;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (n < 0 || n >= (int64_t(1) << 32) - 1)
    return rs::set_error(ctx, RS_ERR_INVALID_ARG, "n = %lld out of range", (long long)n);
  if (n > 0 && (!pos || !ids || !label_out))
    return rs::set_error(ctx, RS_ERR_INVALID_ARG, "null device pointer");
  RS_CUDA(ctx, cudaSetDevice(ctx->device));
  if (n == 0) {
    if (n_groups_out) *n_groups_out = 0;
    return RS_OK;
  }
  if (ctx->cfg.check_ids) RS_TRY(check_ids(ctx, n, ids, st));
  Grid3 g;
  RS_TRY(make_grid(ctx, ctx->cfg.box_L, ctx->cfg.link_len, &g));
  using namespace rs;
  uint64_t* ka = scratch_t<uint64_t>(ctx, S_KEY_A, n);
  uint64_t* kb = scratch_t<uint64_t>(ctx, S_KEY_B, n);
  uint32_t* va = scratch_t<uint32_t>(ctx, S_VAL_A, n);
  uint32_t* vb = scratch_t<uint32_t>(ctx, S_VAL_B, n);
  float4* posS = scratch_t<float4>(ctx, S_POS_SORTED, n);
  const int64_t rows = int64_t(g.ns) * g.ns, tiles = (n + kHeadTile - 1) / kHeadTile;
  uint32_t* row_cell = scratch_t<uint32_t>(ctx, S_ROW_CELL, size_t(rows) + 1);
  int64_t* tile_off = scratch_t<int64_t>(ctx, S_CELL_TILES, size_t(tiles) + 1);
  unsigned long long* counter = scratch_t<unsigned long long>(ctx, S_COUNTER, 8);
  const int64_t cap = n / 8 + 4096;
  PairItem* items = scratch_t<PairItem>(ctx, S_CELL_PAIRS, size_t(cap + pair_items(n, g.ns, g.R)));
  Cells C;
  C.count = tile_off + tiles;
  C.start = scratch_t<uint32_t>(ctx, S_CELL_START, size_t(n) + 1);
  C.x = scratch_t<uint16_t>(ctx, S_CELL_X, n);
  C.row_cell = row_cell;
  C.pos = posS;
  if (!ka || !kb || !va || !vb || !posS || !row_cell || !tile_off || !counter || !items || !C.start || !C.x)
    return RS_ERR_OOM;
  const unsigned grid = grid_for(n, kThreads);
  k_cell_keys<<<grid, kThreads, 0, st>>>(n, pos, g.inv_sc, g.ns, ka, va);
  RS_LAUNCHED(ctx, "k_cell_keys");
  uint64_t* keys;
  uint32_t* idx;
  const uint64_t ns3 = uint64_t(g.ns) * uint64_t(g.ns) * uint64_t(g.ns);
  int kbits = 1;
  while (kbits < 64 && ((ns3 - 1) >> kbits) != 0) ++kbits;
  RS_TRY(radix_sort_u64(ctx, n, kbits, ka, va, kb, vb, &keys, &idx, st));
  // the sort's other buffers: 51 bytes a particle in all instead of 67
  uint32_t* cell_of = idx == va ? vb : va;
  C.row = reinterpret_cast<uint32_t*>(keys == ka ? kb : ka);
  C.parent = C.row + n;
  k_cell_heads<<<unsigned(tiles), kThreads, 0, st>>>(n, keys, tile_off);
  RS_LAUNCHED(ctx, "k_cell_heads");
  RS_TRY(exclusive_scan_i64(ctx, tiles, tile_off, tile_off + tiles, st));
  k_cells<<<unsigned(tiles), kThreads, 0, st>>>(n, keys, idx, pos, g.ns, tile_off, C, posS, cell_of);
  RS_LAUNCHED(ctx, "k_cells");
  k_row_cells<<<grid_for(rows + 1, kThreads), kThreads, 0, st>>>(C, rows, row_cell);
  RS_LAUNCHED(ctx, "k_row_cells");
  RS_CUDA(ctx, cudaMemsetAsync(counter, 0, 5 * sizeof(unsigned long long), st));
  unsigned long long* minid = reinterpret_cast<unsigned long long*>(keys);  // the cells hold what the keys told
  RS_CUDA(ctx, cudaMemsetAsync(minid, 0xff, sizeof(unsigned long long) * size_t(n), st));
  // counter[0]: groups, [1, 2] and [3, 4]: items of the two link passes (every launch below covers n
  // cells, the most there can be)
  for (const bool far : {false, true}) {
    if (far && g.full) break;
    const LinkArgs A{C, g.ns, g.R, g.full, ctx->cfg.box_L, 0.5f * ctx->cfg.box_L, ctx->cfg.link_len * ctx->cfg.link_len,
                     items, counter + (far ? 3 : 1), (unsigned long long)cap};
    {
      ProfScope prof_(ctx, "k_fof_link", st);
      (far ? k_link_cells<true> : k_link_cells<false>)<<<grid, kThreads, 0, st>>>(A);
      RS_LAUNCHED(ctx, "k_link_cells");
      k_link_pairs<<<152 * 4, kThreads, 0, st>>>(A);
    }
    RS_LAUNCHED(ctx, "k_link_pairs");
    k_fof_compress<<<grid, kThreads, 0, st>>>(C);
    RS_LAUNCHED(ctx, "k_fof_compress");
  }
  k_cell_min<<<grid, kThreads, 0, st>>>(n, cell_of, idx, ids, C, minid);
  RS_LAUNCHED(ctx, "k_cell_min");
  k_group_min<<<std::min(grid, 152u * 8u), kThreads, 0, st>>>(C, minid, counter);
  RS_LAUNCHED(ctx, "k_group_min");
  k_fof_labels<<<grid, kThreads, 0, st>>>(n, cell_of, idx, C, minid, label_out);
  RS_LAUNCHED(ctx, "k_fof_labels");
  if (n_groups_out) {
    RS_TRY(read_back(ctx, counter, sizeof(int64_t), st));
    *n_groups_out = ctx->host_box[0];
  }
  return RS_OK;
}
