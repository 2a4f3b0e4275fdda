// Certified far-field bounds of the potential for large nodes (batched form of rs_unbind).
//
// A member's flag depends only on the sign of E_i = KE_i - G m S_i, S_i = sum_{j != i}
// (|u_j - u_i|^2 + eps^2)^(-1/2) (the float64 canonical-order sum). For most members of a large
// node |E_i| is a sizeable fraction of G m S_i, so an interval [S_lo, S_hi] that certainly holds
// S_i decides the flag without the O(g) sum; only members whose interval straddles the sign
// change take the exact path (blocked float32 list sum with its certified bound, then the
// float64 canonical-order potential). The flags are therefore identical to the direct sum's.
//
// Interval (a Barnes-Hut walk with a rigorous truncation bound):
//   tree    the node's members sorted by a 30-bit Hilbert key of their offset u inside the
//           node's bounding box; leaf cells are runs of 32 consecutive members, every level up
//           groups 8 consecutive cells; per cell: centre c (the member mean, rounded to float32),
//           count n, dipole p = sum (x_j - c) (small: c is rounded), second moments
//           Q = sum (x_j - c)(x_j - c)^T (all from float64 sums), a >= max |x_j - c| and
//           b >= sum |x_j - c|^3 (over the cell's members, rounded up);
//   expand  with D = t - c, R'^2 = |D|^2 + eps^2, h_j = |x_j - c| / R' and
//           x = (D.(x_j - c)) / (R' |x_j - c|), the softened kernel is
//           (1/R') (1 - 2 h_j x + h_j^2)^(-1/2) = (1/R') sum_l h_j^l P_l(x)
//           (the Legendre generating function; |x| <= |D| / R' <= 1), so summing l <= 2 over
//           the cell gives n/R' + p.D/R'^3 + (3 D^T Q D - tr(Q) R'^2) / (2 R'^5), and since
//           |P_l| <= 1 on [-1, 1] the rest is at most (1/R') sum_j h_j^3 / (1 - h_j)
//           <= (b / R'^4) / (1 - h), h = a / R' <= theta, with 1 / (1 - h) <= 1 + h / (1 - theta)
//           (the chord of a convex function);
//   walk    one warp per 32 consecutive target members (in tree order); a cell is taken as its
//           expansion when a <= theta R' for the distance to the warp's target box and it holds none
//           of the warp's targets, a leaf is summed directly (self excluded), otherwise its children
//           are visited;
//   slack   u = 2^-24, A = n/R', q^2 = tr(Q)/(n R'^2) <= h^2. A cell's R'^2 is within 6u (differences, three
//           FMAs, eps^2), 1/R' within 5.2u (rsqrt.approx 2^-22.9), so n/R' is within 5.2u A and the
//           quadrupole part, at most q^2 A, within 72u q^2 A (sum of the absolute values of its terms
//           <= 2 q^2 A, its R'^-5 the most part); 32-cell blocks add at most 32 terms in each packed half, Kahan
//           across blocks and the slices' sums 4u: at most 42u A + 109u q^2 A a cell. A <= (1 + q) S_cell
//           (every member's kernel is at least (1/R')/(1 + h_j)), so the first part is below 80u of the
//           cell's sum for theta <= 0.9. Direct terms: 8u each, 31u in a block, 2u Kahan; the target's own
//           term is left out. All of it is below 81u < 5e-6 relative, half of the slack of 1e-5. The
//           quadrupole part is covered by widening the truncation bound by 0.1%: that is at least
//           0.001 q^3 A (power means: b >= n (tr(Q)/n)^(3/2)), half of which exceeds 109u q^2 A from
//           q = 0.013 on, and below that it is under 0.02u A. The other half covers the bound's own
//           rounding, 30u a cell and 18u for its sums (16 adds a half of a block, Kahan across blocks):
//           S_lo = S~ (1 - 1e-5) - 1.001 B, S_hi = S~ (1 + 1e-5) + 1.001 B;
//           the float64 sum differs from the exact one by < g 2^-53 relative.
//   decide  bound iff KE - G m S_lo < -tol, unbound iff KE - G m S_hi > tol (tol = 1e-12 G m
//           S_hi covers the rounding of E itself); otherwise the member is walked again with a
//           smaller angle, and if that leaves it open too, listed for the exact path.
// The paper's implementation computes the exact potential (Rockstar's unbinding); this bound is
// the O(g log g) potential the build adds for nodes of 10^5 - 10^6 members, compared against the
// exact flags in the tests.
#include "rs_exact.cuh"

namespace rs {
int unbind_fallback(rs_ctx* ctx, const unsigned long long* n_ambig, const uint32_t* ambig,
                    const double* vbulk, uint8_t* bound, cudaStream_t st, float* phi_out = nullptr);
int tree_build(rs_ctx* ctx, cudaStream_t st);
int tree_decide(rs_ctx* ctx, const int* only, const uint8_t* want, const double* vbulk,
                uint8_t* bound, unsigned long long* counters, cudaStream_t st);
}  // namespace rs

using namespace rs;

namespace {

constexpr int kT = 256;
constexpr int kLeafBits = 5;   // 32 members per leaf cell
constexpr int kBrBits = 3;     // 8 children per cell
constexpr int kMaxLevels = 10;  // enough for g < 2^32
// Pending cells of a walk: entries lie by level, highest first, four are opened a step, and their up
// to 32 children are all the entries of their level then: at most 35 a level (rounded up).
constexpr int kStack = 35 * kMaxLevels;
// Angle of the second walk, in units of the first's, over the members that leaves undecided (about 1%
// at theta = 0.8 against 0.05% after it; the exact sums it saves cost 1e5 - 1e6 pairs a member). 0.35
// and 0.6 are within 2%.
constexpr float kRefine = 0.45f;
// Its warps take 8 members each, their lanes 4 slices of the interactions: the undecided members are
// few and scattered, so 32 a warp make few warps with long walks (12 nodes of up to 1e5 members:
// 1.3 -> 0.6 ms; 9 ms either way on the 2^27 snapshot).
constexpr int kRefineSlices = 4;
constexpr double kSlack = 1e-5;
constexpr double kBoundWiden = 1.001;

struct Cell {
  float4 ca;  // centre (x, y, z) and radius bound a (negative: no member left in the cell)
  float4 np;  // count n, dipole (px, py, pz)
  float4 q0;  // Qxx, Qyy, Qzz, Qxy
  float4 q1;  // Qxz, Qyz, tr Q, b (third-moment bound)
};

__host__ __device__ __forceinline__ int64_t cells_at(int64_t g, int lev) {
  const int sh = kLeafBits + kBrBits * lev;
  return (g + (int64_t(1) << sh) - 1) >> sh;
}

__host__ __device__ __forceinline__ int levels_of(int64_t g) {
  int l = 0;
  while (cells_at(g, l) > 1) ++l;
  return l + 1;
}

__host__ __device__ __forceinline__ int64_t level_off(int64_t g, int lev) {
  int64_t o = 0;
  for (int l = 0; l < lev; ++l) o += cells_at(g, l);
  return o;
}

// Order-preserving map of a float to uint32 (for atomic min / max of floats).
__device__ __forceinline__ uint32_t ord(float f) {
  const uint32_t b = __float_as_uint(f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float unord(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7fffffffu) : ~o);
}

// Tree nodes: g >= tmin. Per node q: member count, selection flag and cell count (scanned into
// member offsets, ranks and cell offsets).
__global__ void k_tree_sel(int64_t nn, const int64_t* __restrict__ node_size, int64_t tmin,
                           int64_t* __restrict__ tsz, int64_t* __restrict__ tflag,
                           int64_t* __restrict__ tcells) {
  const int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (q >= nn) return;
  const int64_t g = node_size[q];
  const bool sel = g >= tmin;
  tsz[q] = sel ? g : 0;
  tflag[q] = sel ? 1 : 0;
  tcells[q] = sel ? level_off(g, levels_of(g)) : 0;
}

// Per tree node b (rank order): node index, size, member offset in the tree arrays, cell offset.
__global__ void k_tree_list(int64_t nn, const int64_t* __restrict__ node_size, int64_t tmin,
                            const int64_t* __restrict__ toff, const int64_t* __restrict__ rank,
                            const int64_t* __restrict__ coff, int64_t* __restrict__ tnode,
                            int64_t* __restrict__ tg, int64_t* __restrict__ ttoff,
                            int64_t* __restrict__ tcoff) {
  const int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (q >= nn || node_size[q] < tmin) return;
  const int64_t b = rank[q];
  tnode[b] = q;
  tg[b] = node_size[q];
  ttoff[b] = toff[q];
  tcoff[b] = coff[q];
}

// Bounding box of every tree node's members: warp-aggregated atomic min of the ordered
// encodings (max as the min of the complement). box[6 q + d]: min x, y, z, ~max x, y, z.
__global__ void k_tree_bbox(int64_t m, const uint32_t* __restrict__ mnode, const int64_t* __restrict__ node_size,
                            int64_t tmin, const float4* __restrict__ U, unsigned long long* __restrict__ box) {
  const int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool in = p < m;
  const uint32_t q = in ? mnode[p] : 0u;
  const float4 u = in ? U[p] : make_float4(0, 0, 0, 0);
  // members moved to +inf (removed by an earlier unbinding pass) take no part in the tree
  const bool valid = in && node_size[q] >= tmin && isfinite(u.x);
  const float c[3] = {u.x, u.y, u.z};
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    rsd::warp_run_min(box, uint32_t(6u * q + d), valid, (unsigned long long)ord(c[d]));
    rsd::warp_run_min(box, uint32_t(6u * q + 3 + d), valid, (unsigned long long)(~ord(c[d])));
  }
}

// Sort keys of the tree members: tree rank above a 30-bit Hilbert key of the position inside
// the node's bounding cube (10 bits per axis; runs of the curve make compact cells).
__global__ void k_tree_keys(int64_t m, const uint32_t* __restrict__ mnode, const int64_t* __restrict__ node_off,
                            const int64_t* __restrict__ node_size, int64_t tmin,
                            const int64_t* __restrict__ toff, const int64_t* __restrict__ rank,
                            const float4* __restrict__ U, const unsigned long long* __restrict__ box,
                            uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  const int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (p >= m) return;
  const uint32_t q = mnode[p];
  if (node_size[q] < tmin) return;
  const unsigned long long* B = box + 6 * int64_t(q);
  const float lo[3] = {unord(uint32_t(B[0])), unord(uint32_t(B[1])), unord(uint32_t(B[2]))};
  const float hi[3] = {unord(~uint32_t(B[3])), unord(~uint32_t(B[4])), unord(~uint32_t(B[5]))};
  const float ext = fmaxf(fmaxf(hi[0] - lo[0], hi[1] - lo[1]), fmaxf(hi[2] - lo[2], 1e-30f));
  const float sc = 1023.0f / ext;
  const float4 u = U[p];
  const float c[3] = {u.x, u.y, u.z};
  uint32_t qc[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) qc[d] = uint32_t(fminf(fmaxf((c[d] - lo[d]) * sc, 0.f), 1023.f));
  const uint32_t code = rsd::hilbert3<10>(qc[0], qc[1], qc[2]);
  const int64_t k = toff[q] + (p - node_off[q]);
  keys[k] = (uint64_t(rank[q]) << 30) | uint64_t(code);
  vals[k] = uint32_t(p);
}

__global__ void k_tree_gather(int64_t T, const uint32_t* __restrict__ vals, const float4* __restrict__ U,
                              float4* __restrict__ TX, uint32_t* __restrict__ tpos) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= T) return;
  const uint32_t p = vals[s];
  const float4 u = U[p];
  TX[s] = make_float4(u.x, u.y, u.z, 0.f);
  tpos[s] = p;
}

// (tree rank b, level, index j in the level) of global cell c.
__device__ __forceinline__ void cell_decode(int64_t c, int64_t nt, const int64_t* __restrict__ tcoff,
                                            const int64_t* __restrict__ tg, int64_t& b, int& lev,
                                            int64_t& j) {
  b = rsd::upper_bound_i64(tcoff, nt, c) - 1;
  const int64_t g = tg[b];
  int64_t i = c - tcoff[b];
  lev = 0;
  while (i >= cells_at(g, lev)) {
    i -= cells_at(g, lev);
    ++lev;
  }
  j = i;
}

// An upper bound of |(x, y, z)| for offsets with at most a float32 rounding each.
__device__ __forceinline__ float radius_up(float x, float y, float z) {
  return sqrtf(x * x + y * y + z * z) * (1.0f + 1e-6f);
}

__device__ __forceinline__ Cell empty_cell() {
  return Cell{make_float4(0, 0, 0, -1.f), make_float4(0, 0, 0, 0), make_float4(0, 0, 0, 0), make_float4(0, 0, 0, 0)};
}

// Leaf cells (level 0): a block takes kLeafCells consecutive cells of the cell array, one warp each
// (cells of other levels are skipped). The float64 pipe runs two lanes a clock, so the lane sums go
// through shared memory, one thread per (cell, quantity) adding 32 values: 25 float64 warp
// instructions a leaf instead of about 90 with butterflies (12.1 -> 5.6 ms for 4.9e7 members,
// the third-moment bound included).
constexpr int kLeafCells = kT / 32;
constexpr int kLeafSums = 9;  // dx, dy, dz, then xx, yy, zz, xy, xz, yz

__global__ void __launch_bounds__(kT)
k_tree_leaves(int64_t C, int64_t nt, const int64_t* __restrict__ tcoff, const int64_t* __restrict__ tg,
              const int64_t* __restrict__ ttoff, const float4* __restrict__ TX, Cell* __restrict__ cells) {
  __shared__ double val[kLeafCells][kLeafSums][33];
  __shared__ double sum[kLeafCells][kLeafSums];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t c = int64_t(blockIdx.x) * kLeafCells + w;
  int64_t b = 0, j = 0;
  int lev = -1;
  if (c < C) cell_decode(c, nt, tcoff, tg, b, lev, j);
  const bool leaf = lev == 0;
  const int64_t s0 = leaf ? ttoff[b] + (j << kLeafBits) : 0;
  const int cnt = leaf ? int(rsd::min64(32, tg[b] - (j << kLeafBits))) : 0;
  const float4 xr = lane < cnt ? TX[s0 + lane] : make_float4(0, 0, 0, 0);
  // members moved to +inf (removed by an earlier unbinding pass) are left out of the moments
  const bool valid = lane < cnt && isfinite(xr.x);
  const int nv = __popc(__ballot_sync(0xffffffffu, valid));
  const double x = valid ? rsd::f2d(xr.x) : 0.0, y = valid ? rsd::f2d(xr.y) : 0.0, z = valid ? rsd::f2d(xr.z) : 0.0;
  auto block_sums = [&](int per) {  // sum[cell][t] of val[cell][t][0..32) for t < per
    __syncthreads();
    if (int(threadIdx.x) < kLeafCells * per) {
      const double* v = val[threadIdx.x / per][threadIdx.x % per];
      double a0 = 0.0, a1 = 0.0;
#pragma unroll
      for (int k = 0; k < 32; k += 2) {
        a0 += v[k];
        a1 += v[k + 1];
      }
      sum[threadIdx.x / per][threadIdx.x % per] = a0 + a1;
    }
    __syncthreads();
  };
  val[w][0][lane] = x;
  val[w][1][lane] = y;
  val[w][2][lane] = z;
  block_sums(3);
  const double inv = nv ? 1.0 / double(nv) : 0.0;
  const float cx = float(sum[w][0] * inv), cy = float(sum[w][1] * inv), cz = float(sum[w][2] * inv);
  // offsets from the float32 centre are exact in float64
  const double dx = valid ? x - rsd::f2d(cx) : 0.0, dy = valid ? y - rsd::f2d(cy) : 0.0,
               dz = valid ? z - rsd::f2d(cz) : 0.0;
  __syncthreads();  // the means are read
  const double v[kLeafSums] = {dx, dy, dz, dx * dx, dy * dy, dz * dz, dx * dy, dx * dz, dy * dz};
#pragma unroll
  for (int t = 0; t < kLeafSums; ++t) val[w][t][lane] = v[t];
  block_sums(kLeafSums);
  const float fx = float(dx), fy = float(dy), fz = float(dz);
  const float r = valid ? radius_up(fx, fy, fz) : 0.f;
  float a = r, r3 = r * r * r;
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, off));
    r3 += __shfl_xor_sync(0xffffffffu, r3, off);
  }
  if (leaf && lane == 0) {
    if (nv == 0) {
      cells[c] = empty_cell();
      return;
    }
    const double* S = sum[w];
    Cell cl;
    cl.ca = make_float4(cx, cy, cz, a);
    cl.np = make_float4(float(nv), float(S[0]), float(S[1]), float(S[2]));
    cl.q0 = make_float4(float(S[3]), float(S[4]), float(S[5]), float(S[6]));
    cl.q1 = make_float4(float(S[7]), float(S[8]), float(S[3] + S[4] + S[5]), r3 * (1.0f + 4e-6f));
    cells[c] = cl;
  }
}

// Cells of level `lev` >= 1 from their (up to 8) children, moments shifted to the parent's
// float32 centre in float64 (a and b are left to k_tree_radius).
__global__ void k_tree_up(int64_t C, int lev, int64_t nt, const int64_t* __restrict__ tcoff,
                          const int64_t* __restrict__ tg, Cell* __restrict__ cells) {
  const int64_t c = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (c >= C) return;
  int64_t b, j;
  int lv;
  cell_decode(c, nt, tcoff, tg, b, lv, j);
  if (lv != lev) return;
  const int64_t g = tg[b];
  const int64_t c0 = tcoff[b] + level_off(g, lev - 1) + (j << kBrBits);
  const int nch = int(rsd::min64(int64_t(1) << kBrBits, cells_at(g, lev - 1) - (j << kBrBits)));
  double n = 0.0, mx = 0.0, my = 0.0, mz = 0.0;
  for (int k = 0; k < nch; ++k) {
    const Cell ch = cells[c0 + k];
    if (ch.np.x == 0.f) continue;  // empty child
    n += ch.np.x;
    mx += double(ch.np.x) * ch.ca.x + ch.np.y;  // sum of x_j = n c + p
    my += double(ch.np.x) * ch.ca.y + ch.np.z;
    mz += double(ch.np.x) * ch.ca.z + ch.np.w;
  }
  if (n == 0.0) {
    cells[c] = empty_cell();
    return;
  }
  const float cx = float(mx / n), cy = float(my / n), cz = float(mz / n);
  double P[3] = {0.0, 0.0, 0.0}, Q[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int k = 0; k < nch; ++k) {
    const Cell ch = cells[c0 + k];
    if (ch.np.x == 0.f) continue;
    const double d[3] = {double(ch.ca.x) - cx, double(ch.ca.y) - cy, double(ch.ca.z) - cz};
    const double nc = ch.np.x;
    const double pc[3] = {ch.np.y, ch.np.z, ch.np.w};
    for (int e = 0; e < 3; ++e) P[e] += pc[e] + nc * d[e];
    // sum (y + d)(y + d)^T over the child's members, y = x - c_child: Q_c + p d^T + d p^T + n d d^T
    const double qc[6] = {ch.q0.x, ch.q0.y, ch.q0.z, ch.q0.w, ch.q1.x, ch.q1.y};
    const int ia[6] = {0, 1, 2, 0, 0, 1}, ib[6] = {0, 1, 2, 1, 2, 2};
    for (int t = 0; t < 6; ++t)
      Q[t] += qc[t] + pc[ia[t]] * d[ib[t]] + d[ia[t]] * pc[ib[t]] + nc * d[ia[t]] * d[ib[t]];
  }
  const float inf = __int_as_float(0x7f800000);
  Cell cl;
  cl.ca = make_float4(cx, cy, cz, inf);
  cl.np = make_float4(float(n), float(P[0]), float(P[1]), float(P[2]));
  cl.q0 = make_float4(float(Q[0]), float(Q[1]), float(Q[2]), float(Q[3]));
  cl.q1 = make_float4(float(Q[4]), float(Q[5]), float(Q[0] + Q[1] + Q[2]), inf);
  cells[c] = cl;
}

// a and b of the cells of level >= 1 over their members (a node's root keeps a = inf: it holds every
// target). Bounds through the children (a_child + |c_child - c|, and the same for b by the triangle
// inequality of the 3-norm) lose 10-20% a level in a, which costs 1.5 times the expansions and twice
// the undecided members at theta = 0.7. A block takes 32 consecutive cells of the cell array, the
// upper ones among them one by one.
__global__ void __launch_bounds__(kT)
k_tree_radius(int64_t C, int64_t nt, const int64_t* __restrict__ tcoff, const int64_t* __restrict__ tg,
              const int64_t* __restrict__ ttoff, const float4* __restrict__ TX, Cell* __restrict__ cells) {
  __shared__ float wa[kT / 32];
  __shared__ double wb[kT / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t cb = int64_t(blockIdx.x) * 32;
  int64_t b = 0, j = 0;
  int lev = 0;
  if (cb + lane < C) cell_decode(cb + lane, nt, tcoff, tg, b, lev, j);
  unsigned upper = __ballot_sync(0xffffffffu, lev > 0 && cells_at(tg[b], lev) > 1);  // every warp alike
  const int64_t first = ttoff[b] + (j << (kLeafBits + kBrBits * lev));
  const int64_t count = rsd::min64(int64_t(1) << (kLeafBits + kBrBits * lev),
                                   tg[b] - (j << (kLeafBits + kBrBits * lev)));
  while (upper) {
    const int l = __ffs(upper) - 1;
    upper &= upper - 1u;
    const int64_t f = __shfl_sync(0xffffffffu, first, l), n = __shfl_sync(0xffffffffu, count, l);
    const float4 ca = cells[cb + l].ca;
    float a = 0.f;
    double r3 = 0.0;
    if (ca.w >= 0.f)
      for (int64_t i = threadIdx.x; i < n; i += kT) {
        const float4 x = TX[f + i];
        if (!isfinite(x.x)) continue;
        const float r = radius_up(x.x - ca.x, x.y - ca.y, x.z - ca.z);
        a = fmaxf(a, r);
        r3 += rsd::f2d(r * r * r);
      }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      a = fmaxf(a, __shfl_xor_sync(0xffffffffu, a, off));
      r3 += __shfl_xor_sync(0xffffffffu, r3, off);
    }
    if (lane == 0) {
      wa[w] = a;
      wb[w] = r3;
    }
    __syncthreads();
    if (threadIdx.x == 0 && ca.w >= 0.f) {
      for (int k = 1; k < kT / 32; ++k) {
        a = fmaxf(a, wa[k]);
        r3 += wb[k];
      }
      cells[cb + l].ca.w = a;
      cells[cb + l].q1.w = __double2float_ru(r3 * (1.0 + 1e-6));
    }
    __syncthreads();
  }
}

// Walk order of the tree nodes: largest size class first (stable within a class).
__global__ void k_tree_okeys(int64_t nt, const int64_t* __restrict__ tg, uint64_t* __restrict__ keys,
                             uint32_t* __restrict__ vals) {
  const int64_t b = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (b >= nt) return;
  keys[b] = 255u - rsd::size_class(tg[b]);
  vals[b] = uint32_t(b);
}

// Wanted flag of every tree member (sorted position s): want[p] if given, else only[q] if given,
// else 1.
__global__ void k_tree_want(int64_t T, const uint32_t* __restrict__ tpos, const uint32_t* __restrict__ mnode,
                            const int* __restrict__ only, const uint8_t* __restrict__ want,
                            int64_t* __restrict__ wf) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= T) return;
  const uint32_t p = tpos[s];
  wf[s] = want ? int64_t(want[p] != 0) : (only ? int64_t(only[mnode[p]] != 0) : 1);
}

__global__ void k_tree_wlist(int64_t T, const int64_t* __restrict__ wf, uint32_t* __restrict__ wl) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= T) return;
  if (wf[s + 1] != wf[s]) wl[wf[s]] = uint32_t(s);
}

// Per node (walk order r): wanted range [wlo, wlo + wcnt) of the wanted list and its warp count at
// `targets` members a warp.
__global__ void k_tree_items(int64_t nt, const uint32_t* __restrict__ worder, const int64_t* __restrict__ ttoff,
                             const int64_t* __restrict__ tg, const int64_t* __restrict__ wf, int targets,
                             int64_t* __restrict__ wlo, int64_t* __restrict__ wcnt,
                             int64_t* __restrict__ items) {
  const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r >= nt) return;
  const int64_t b = worder[r];
  const int64_t a = wf[ttoff[b]], e = wf[ttoff[b] + tg[b]];
  wlo[r] = a;
  wcnt[r] = e - a;
  items[r] = (e - a + targets - 1) / targets;
}

struct WalkArgs {
  int64_t nt;
  const int64_t* item_off;  // [nt + 1], walk order
  const uint32_t* worder;   // walk order -> tree rank
  const int64_t* wlo;       // walk order
  const int64_t* wcnt;      // walk order
  const uint32_t* wl;       // wanted sorted positions
  const float4* TX;
  const uint32_t* tpos;
  const int64_t* ttoff;
  const int64_t* tcoff;
  const int64_t* tg;
  const int64_t* tnode;
  const Cell* cells;
  const float4* V;
  const double* vbulk;
  float eps2, theta2, chord;  // chord = 1 / (1 - theta)
  bool last;                  // the last walk: its undecided members go to the exact path
  double Gm;
  uint8_t* bound;
  int64_t* und;             // per sorted position: 1 = undecided
  double* rec_lo;           // per member position (optional record of the interval)
  double* rec_hi;
  unsigned long long* counters;  // [0] decided, [1] undecided, [2] expansions, [3] direct pairs
};

// Shared memory of one walking warp: pending cells to open (level << 28 | index in the level), lists
// of accepted cells and of leaves to sum (node-relative indices), 32 staged cells as 16 pairs for the
// packed arithmetic, and a leaf's members in x / y / z rows.
struct __align__(16) WalkShared {
  float4 st[8][16];
  float leaf[3][32];
  uint32_t stack[kStack];
  uint32_t acc[64];
  uint32_t dir[64];
};

// Sum and truncation bound of one target over the tree, for the warp's lanes: Kahan sums over blocks.
struct WalkSum {
  float S = 0.f, C = 0.f;
  float B = 0.f, D = 0.f;
  static __device__ __forceinline__ void add(float& sum, float& carry, float blk) {
    const float y = __fsub_rn(blk, carry);
    const float t = __fadd_rn(sum, y);
    carry = __fsub_rn(__fsub_rn(t, sum), y);
    sum = t;
  }
  __device__ __forceinline__ void add(float blk) { add(S, C, blk); }
  __device__ __forceinline__ void add_bound(float blk) { add(B, D, blk); }
};

// Quadrupole expansions of `cnt` (1..32) accepted cells: lane = cell while they are staged (as pairs,
// with the factors 3/2, 2 and -1/2 folded in and the centre negated), then lane = target, two cells a
// packed step. Explicit FMAs: the evaluation only has to stay inside the slack, and the library is
// compiled without contraction. A missing cell of the last pair has no members and lies far away.
template <bool kNormal, int kSlices>
__device__ __forceinline__ void walk_cells(const Cell* __restrict__ ncell, const uint32_t* idx, int cnt, float4 t,
                                           float eps2, float chord, int lane, WalkShared& W, WalkSum& R) {
  Cell cl{make_float4(1e18f, 1e18f, 1e18f, 0.f), make_float4(0, 0, 0, 0), make_float4(0, 0, 0, 0),
          make_float4(0, 0, 0, 0)};
  if (lane < cnt) cl = ncell[idx[lane]];
  const float v[16] = {-cl.ca.x, -cl.ca.y, -cl.ca.z, cl.ca.w, cl.np.x, cl.np.y, cl.np.z, cl.np.w,
                       1.5f * cl.q0.x, 1.5f * cl.q0.y, 1.5f * cl.q0.z, 3.0f * cl.q0.w,
                       3.0f * cl.q1.x, 3.0f * cl.q1.y, -0.5f * cl.q1.z, cl.q1.w};
  __syncwarp();
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    float* p = reinterpret_cast<float*>(&W.st[k][lane >> 1]) + (lane & 1);
    p[0] = v[2 * k];
    p[2] = v[2 * k + 1];
  }
  __syncwarp();
  const float2 tx = make_float2(t.x, t.x), ty = make_float2(t.y, t.y), tz = make_float2(t.z, t.z);
  const float2 e2 = make_float2(eps2, eps2), kc = make_float2(chord, chord), one = make_float2(1.f, 1.f);
  float2 blk = make_float2(0.f, 0.f), bnd = make_float2(0.f, 0.f);
  auto lo = [](float4 a) { return make_float2(a.x, a.y); };
  auto hi = [](float4 a) { return make_float2(a.z, a.w); };
  for (int k = lane / (32 / kSlices); 2 * k < cnt; k += kSlices) {
    const float4 a0 = W.st[0][k], a1 = W.st[1][k], a2 = W.st[2][k], a3 = W.st[3][k];
    const float2 dx = __fadd2_rn(tx, lo(a0)), dy = __fadd2_rn(ty, hi(a0)), dz = __fadd2_rn(tz, lo(a1));
    const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
    const float2 ri = make_float2(rsd::inv_sqrt<kNormal>(r2.x), rsd::inv_sqrt<kNormal>(r2.y));
    const float4 a4 = W.st[4][k], a5 = W.st[5][k], a6 = W.st[6][k], a7 = W.st[7][k];
    const float2 ri2 = __fmul2_rn(ri, ri);
    const float2 qx = __ffma2_rn(lo(a6), dz, __ffma2_rn(hi(a5), dy, __fmul2_rn(lo(a4), dx)));
    const float2 qy = __ffma2_rn(hi(a6), dz, __fmul2_rn(hi(a4), dy));
    const float2 dqd = __ffma2_rn(qx, dx, __ffma2_rn(qy, dy, __fmul2_rn(__fmul2_rn(lo(a5), dz), dz)));
    const float2 pd = __ffma2_rn(hi(a2), dx, __ffma2_rn(lo(a3), dy, __ffma2_rn(hi(a3), dz, lo(a7))));
    const float2 quad = __ffma2_rn(dqd, ri2, pd);
    blk = __ffma2_rn(lo(a2), ri, blk);
    blk = __ffma2_rn(__fmul2_rn(ri2, ri), quad, blk);
    const float2 f = __ffma2_rn(__fmul2_rn(hi(a1), ri), kc, one);
    bnd = __ffma2_rn(__fmul2_rn(hi(a7), __fmul2_rn(ri2, ri2)), f, bnd);
  }
  R.add(__fadd_rn(blk.x, blk.y));
  R.add_bound(__fadd_rn(bnd.x, bnd.y));
}

// Direct sums over `cnt` leaves, two members per packed float32x2 step; slots past a leaf's count
// hold +inf, whose term is exactly 0. The target's own term 1 / eps never enters: it would leave its
// rounding behind, which no multiple of the other terms bounds. The leaves that hold a target of the
// warp (one or a few of hundreds) test for it per pair.
template <bool kNormal, int kSlices>
__device__ __forceinline__ void walk_leaves(const float4* __restrict__ nx, const uint32_t* leaves, int cnt, uint32_t g,
                                            float4 t, uint32_t self_rel, float eps2, int lane, WalkShared& W,
                                            WalkSum& R, uint32_t& n_dir) {
  const float inf = __int_as_float(0x7f800000);
  auto load = [&](int k) {
    const uint32_t i = (leaves[k] << kLeafBits) + lane;
    return i < g ? nx[i] : make_float4(inf, inf, inf, 0.f);
  };
  float4 next = load(0);
  for (int l = 0; l < cnt; ++l) {
    const uint32_t j = leaves[l], c0 = j << kLeafBits;
    const int n = int(min(32u, g - c0));
    __syncwarp();
    W.leaf[0][lane] = next.x;
    W.leaf[1][lane] = next.y;
    W.leaf[2][lane] = next.z;
    __syncwarp();
    if (l + 1 < cnt) next = load(l + 1);
    float blk;
    if (kNormal) {
      const float2 ntx = make_float2(-t.x, -t.x), nty = make_float2(-t.y, -t.y), ntz = make_float2(-t.z, -t.z),
                   e2 = make_float2(eps2, eps2);
      float2 acc2 = make_float2(0.f, 0.f);
      const int slice = lane / (32 / kSlices);
      auto pair = [&](int k) {
        const float2 ex = __fadd2_rn(*reinterpret_cast<const float2*>(&W.leaf[0][k]), ntx);
        const float2 ey = __fadd2_rn(*reinterpret_cast<const float2*>(&W.leaf[1][k]), nty);
        const float2 ez = __fadd2_rn(*reinterpret_cast<const float2*>(&W.leaf[2][k]), ntz);
        const float2 r2 = __ffma2_rn(ex, ex, __ffma2_rn(ey, ey, __ffma2_rn(ez, ez, e2)));
        return make_float2(rsd::inv_sqrt<true>(r2.x), rsd::inv_sqrt<true>(r2.y));
      };
      const bool own = self_rel >> kLeafBits == j;
      if (__any_sync(0xffffffffu, own)) {
        const int self = own ? int(self_rel & 31u) : -1;
#pragma unroll 8
        for (int i = 0; i < 32 / kSlices; i += 2) {
          const int k = 2 * slice + kSlices * i;
          const float2 w = pair(k);
          acc2 = __fadd2_rn(acc2, make_float2(k == self ? 0.f : w.x, k + 1 == self ? 0.f : w.y));
        }
      } else {
#pragma unroll 8
        for (int i = 0; i < 32 / kSlices; i += 2) acc2 = __fadd2_rn(acc2, pair(2 * slice + kSlices * i));
      }
      blk = __fadd_rn(acc2.x, acc2.y);
    } else {
      blk = 0.f;
      for (int k = lane / (32 / kSlices); k < n; k += kSlices) {
        const float ex = __fsub_rn(W.leaf[0][k], t.x), ey = __fsub_rn(W.leaf[1][k], t.y),
                    ez = __fsub_rn(W.leaf[2][k], t.z);
        const float wv = rsqrtf(__fmaf_rn(ex, ex, __fmaf_rn(ey, ey, __fmaf_rn(ez, ez, eps2))));
        blk = __fadd_rn(blk, c0 + uint32_t(k) == self_rel ? 0.f : wv);
      }
    }
    R.add(blk);
    n_dir += uint32_t(n);
  }
}

// One warp per 32 wanted targets of one node: the certified walk, then the decision. A step opens up
// to four pending cells and tests their children side by side (lane = child) against the box of the
// warp's targets; accepted cells and leaves to sum are listed and evaluated 32 at a time with lane =
// target. In a 2^24-particle pass (ncu) the issue slots are busy 64% of the cycles, the float32 pipe 35%, the
// special-function unit 24%; warps wait for shared memory and for the units' queues (2.6 and 1.5 cycles
// an instruction). Testing one cell a step with every lane spent most of the walk on loads and stack
// traffic. On the 2^27 snapshot (4.9e7 members) the walk went from 295 to 58 ms: 2.5 times fewer
// interactions from the exact a and b at theta = 0.7, the rest from the form of the walk.
// Indices inside the walk are 32-bit and relative to the node (its members are [tb, tb + g) of the
// sorted arrays, its cells [cb, cb + cells) of the cell array).
template <bool kNormal, int kSlices>
__global__ void __launch_bounds__(kT, 4)
k_tree_walk(WalkArgs A) {
  constexpr int kTargets = 32 / kSlices;
  __shared__ WalkShared sh[kT / 32];
  const int lane = threadIdx.x & 31;
  WalkShared& W = sh[threadIdx.x >> 5];
  const int64_t items = A.item_off[A.nt], warps = int64_t(gridDim.x) * (kT / 32);
  for (int64_t w = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; w < items; w += warps) {
    const int64_t r = rsd::upper_bound_i64(A.item_off, A.nt, w) - 1;
    const int64_t b = A.worder[r];
    const int64_t i0 = kTargets * (w - A.item_off[r]);
    const bool valid = i0 + lane % kTargets < A.wcnt[r];
    // lane 0's entry is always valid
    const uint32_t s_self = A.wl[A.wlo[r] + i0 + (valid ? lane % kTargets : 0)];
    const float4 t = A.TX[s_self];
    const int64_t g = A.tg[b], tb = A.ttoff[b], cb = A.tcoff[b];
    const int nlev = levels_of(g);
    // per-level cell offsets inside the node, lane l holds level l's
    const uint32_t my_lvoff = lane < nlev ? uint32_t(level_off(g, lane)) : 0u;
    const uint32_t g32 = uint32_t(g), self_rel = s_self - uint32_t(tb);
    // the warp's targets as a range of node-relative positions (a cell holds one of them iff its
    // index at its level lies in [lo_rel >> sh, hi_rel >> sh]) and their box
    uint32_t lo_rel = self_rel, hi_rel = self_rel;
    float bl[3] = {t.x, t.y, t.z}, bh[3] = {t.x, t.y, t.z};
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
      lo_rel = min(lo_rel, __shfl_xor_sync(0xffffffffu, lo_rel, off));
      hi_rel = max(hi_rel, __shfl_xor_sync(0xffffffffu, hi_rel, off));
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        bl[d] = fminf(bl[d], __shfl_xor_sync(0xffffffffu, bl[d], off));
        bh[d] = fmaxf(bh[d], __shfl_xor_sync(0xffffffffu, bh[d], off));
      }
    }
    const Cell* __restrict__ ncell = A.cells + cb;
    const float4* __restrict__ nx = A.TX + tb;
    const unsigned below = (1u << lane) - 1u;
    WalkSum R;
    uint32_t n_exp = 0, n_dir = 0;
    int sp = 0, na = 0, nd = 0;
    if (nlev == 1) {
      nd = 1;
      if (lane == 0) W.dir[0] = 0u;
    } else {
      sp = 1;
      if (lane == 0) W.stack[0] = uint32_t(nlev - 1) << 28;
    }
    __syncwarp();
    while (sp > 0) {
      const int np = min(sp, 4);
      const int p = lane >> 3;
      const uint32_t e = p < np ? W.stack[sp - np + p] : 0u;
      sp -= np;
      const int lc = max(int(e >> 28) - 1, 0);  // the children's level
      const uint32_t jc = ((e & 0x0fffffffu) << kBrBits) + uint32_t(lane & 7);
      const int sh_c = kLeafBits + kBrBits * lc;
      const uint32_t nchild = uint32_t((uint64_t(g32) + (1ull << sh_c) - 1) >> sh_c);
      const uint32_t idx = __shfl_sync(0xffffffffu, my_lvoff, lc) + jc;
      bool acc = false, opn = false;
      if (p < np && jc < nchild) {
        const float4 ca = ncell[idx].ca;
        const float dx = fmaxf(fmaxf(bl[0] - ca.x, ca.x - bh[0]), 0.f), dy = fmaxf(fmaxf(bl[1] - ca.y, ca.y - bh[1]), 0.f),
                    dz = fmaxf(fmaxf(bl[2] - ca.z, ca.z - bh[2]), 0.f);
        const float r2 = __fmaf_rn(dx, dx, __fmaf_rn(dy, dy, __fmaf_rn(dz, dz, A.eps2)));
        const bool overlap = jc >= (lo_rel >> sh_c) && jc <= (hi_rel >> sh_c);
        const bool some = ca.w >= 0.f;  // a member is left in the cell (iterative unbinding)
        acc = some && !overlap && ca.w * ca.w <= A.theta2 * r2;
        opn = some && !acc;
      }
      const unsigned ba = __ballot_sync(0xffffffffu, acc), bd = __ballot_sync(0xffffffffu, opn && lc == 0),
                     bs = __ballot_sync(0xffffffffu, opn && lc > 0);
      if (acc) W.acc[na + __popc(ba & below)] = idx;
      if (opn && lc == 0) W.dir[nd + __popc(bd & below)] = jc;
      if (opn && lc > 0) W.stack[sp + __popc(bs & below)] = (uint32_t(lc) << 28) | jc;
      na += __popc(ba);
      nd += __popc(bd);
      sp += __popc(bs);
      __syncwarp();
      if (na >= 32) {
        na -= 32;
        n_exp += 32;
        walk_cells<kNormal, kSlices>(ncell, W.acc + na, 32, t, A.eps2, A.chord, lane, W, R);
      }
      if (nd >= 32) {
        walk_leaves<kNormal, kSlices>(nx, W.dir, nd, g32, t, self_rel, A.eps2, lane, W, R, n_dir);
        nd = 0;
        __syncwarp();
      }
    }
    if (na > 0) {
      n_exp += uint32_t(na);
      walk_cells<kNormal, kSlices>(ncell, W.acc, na, t, A.eps2, A.chord, lane, W, R);
    }
    if (nd > 0) walk_leaves<kNormal, kSlices>(nx, W.dir, nd, g32, t, self_rel, A.eps2, lane, W, R, n_dir);
    float S = R.S, Bt = R.B;
#pragma unroll
    for (int off = kTargets; off < 32; off <<= 1) {  // the slices of a target
      S = __fadd_rn(S, __shfl_xor_sync(0xffffffffu, S, off));
      Bt = __fadd_rn(Bt, __shfl_xor_sync(0xffffffffu, Bt, off));
    }
    const bool mine = valid && lane < kTargets;
    bool decided = false;
    if (mine) {
      const uint32_t p = A.tpos[s_self];
      const int64_t q = A.tnode[b];
      const double Sd = double(S), Bd = kBoundWiden * double(Bt);
      const double slo = Sd * (1.0 - kSlack) - Bd, shi = Sd * (1.0 + kSlack) + Bd;
      const double ke = kinetic(A.V[p], A.vbulk + 3 * q);
      const double tol = 1e-12 * A.Gm * fabs(shi);
      const double e_hi = ke - A.Gm * slo, e_lo = ke - A.Gm * shi;
      if (slo > 0.0 && e_hi < -tol) {
        A.bound[p] = 1;
        decided = true;
      } else if (e_lo > tol) {
        A.bound[p] = 0;
        decided = true;
      } else {
        A.und[s_self] = 1;
      }
      if (A.rec_lo) {
        A.rec_lo[p] = slo;
        A.rec_hi[p] = shi;
      }
    }
    const unsigned dec = __ballot_sync(0xffffffffu, mine && decided);
    const unsigned und = __ballot_sync(0xffffffffu, mine && !decided);
    if (lane == 0) {
      if (dec) atomicAdd(A.counters + 0, (unsigned long long)__popc(dec));
      if (und && A.last) atomicAdd(A.counters + 1, (unsigned long long)__popc(und));
      atomicAdd(A.counters + 2, (unsigned long long)n_exp * kTargets);
      atomicAdd(A.counters + 3, (unsigned long long)n_dir * kTargets);
    }
    __syncwarp();
  }
}

__global__ void k_tree_ulist(int64_t T, const int64_t* __restrict__ uf, uint32_t* __restrict__ list,
                             unsigned long long* __restrict__ count) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s == 0) *count = (unsigned long long)uf[T];
  if (s >= T) return;
  if (uf[s + 1] != uf[s]) list[uf[s]] = uint32_t(s);
}

__global__ void k_tree_lranges(int64_t nt, const int64_t* __restrict__ ttoff, const int64_t* __restrict__ tg,
                               const int64_t* __restrict__ uf, int tile, int64_t* __restrict__ lofs,
                               int64_t* __restrict__ lend, int64_t* __restrict__ tiles,
                               unsigned long long* __restrict__ list_pairs) {
  const int64_t b = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (b >= nt) return;
  const int64_t a = uf[ttoff[b]], e = uf[ttoff[b] + tg[b]];
  lofs[b] = a;
  lend[b] = e;
  tiles[b] = list_items(e - a, tg[b], tile);
  if (e > a) atomicAdd(list_pairs, (unsigned long long)((e - a) * tg[b]));
}

__global__ void k_tree_acc(unsigned long long* __restrict__ c, int from, int to) {
  c[to] += c[from];
  c[from] = 0;
}

int bits_for(uint64_t v) {
  int b = 1;
  while (b < 64 && (v >> b) != 0) ++b;
  return b;
}

}  // namespace

// Build the cells of every node with at least ctx->tree_min members (device state kept in the
// context's scratch until the next rs_unbind).
int rs::tree_build(rs_ctx* ctx, cudaStream_t st) {
  ctx->tree_nt = 0;
  ctx->tree_T = 0;
  ctx->tree_C = 0;
  const int64_t tmin = ctx->tree_min;
  if (tmin <= 0) return RS_OK;
  Hier h = hier_of(ctx);
  const int64_t nn = ctx->n_nodes, m = ctx->n_members;
  if (nn == 0) return RS_OK;
  int64_t* tsz = scratch_t<int64_t>(ctx, S_T_OFF, size_t(nn) + 1);
  int64_t* trank = scratch_t<int64_t>(ctx, S_T_RANK, size_t(nn) + 1);
  int64_t* tcells = scratch_t<int64_t>(ctx, S_T_COFF, size_t(nn) + 1);
  if (!tsz || !trank || !tcells) return RS_ERR_OOM;
  k_tree_sel<<<grid_for(nn, kT), kT, 0, st>>>(nn, h.node_size, tmin, tsz, trank, tcells);
  RS_LAUNCHED(ctx, "k_tree_sel");
  RS_TRY(exclusive_scans(ctx, nn, ScanJobs{{{tsz, tsz, tsz + nn}, {trank, trank, trank + nn},
                                            {tcells, tcells, tcells + nn}}}, st));
  RS_CUDA(ctx, cudaMemcpyAsync(ctx->host_box, tsz + nn, 8, cudaMemcpyDeviceToHost, st));
  RS_CUDA(ctx, cudaMemcpyAsync(ctx->host_box + 1, trank + nn, 8, cudaMemcpyDeviceToHost, st));
  RS_CUDA(ctx, cudaMemcpyAsync(ctx->host_box + 2, tcells + nn, 8, cudaMemcpyDeviceToHost, st));
  RS_CUDA(ctx, cudaStreamSynchronize(st));
  const int64_t T = ctx->host_box[0], nt = ctx->host_box[1], C = ctx->host_box[2];
  if (nt == 0) return RS_OK;
  int64_t* tn = scratch_t<int64_t>(ctx, S_T_NODES, size_t(nt) * 4 + 4);
  unsigned long long* box = scratch_t<unsigned long long>(ctx, S_T_BOX, size_t(nn) * 6);
  uint64_t* ka = scratch_t<uint64_t>(ctx, S_T_KA, size_t(T));
  uint64_t* kb = scratch_t<uint64_t>(ctx, S_T_KB, size_t(T));
  uint32_t* va = scratch_t<uint32_t>(ctx, S_T_VA, size_t(T));
  uint32_t* vb = scratch_t<uint32_t>(ctx, S_T_VB, size_t(T));
  float4* TX = scratch_t<float4>(ctx, S_T_X, size_t(T));
  uint32_t* tpos = scratch_t<uint32_t>(ctx, S_T_POS, size_t(T));
  Cell* cells = static_cast<Cell*>(scratch(ctx, S_T_CELL, size_t(C) * sizeof(Cell)));
  uint32_t* worder = scratch_t<uint32_t>(ctx, S_T_ORDER, size_t(nt));
  if (!tn || !box || !ka || !kb || !va || !vb || !TX || !tpos || !cells || !worder) return RS_ERR_OOM;
  int64_t *tnode = tn, *tg = tn + nt, *ttoff = tn + 2 * nt, *tcoff = tn + 3 * nt;
  k_tree_list<<<grid_for(nn, kT), kT, 0, st>>>(nn, h.node_size, tmin, tsz, trank, tcells, tnode, tg, ttoff,
                                              tcoff);
  RS_LAUNCHED(ctx, "k_tree_list");
  RS_CUDA(ctx, cudaMemsetAsync(box, 0xff, sizeof(unsigned long long) * 6 * nn, st));
  k_tree_bbox<<<grid_for(m, kT), kT, 0, st>>>(m, h.mnode, h.node_size, tmin, h.U, box);
  RS_LAUNCHED(ctx, "k_tree_bbox");
  k_tree_keys<<<grid_for(m, kT), kT, 0, st>>>(m, h.mnode, h.node_off, h.node_size, tmin, tsz, trank, h.U,
                                             box, ka, va);
  RS_LAUNCHED(ctx, "k_tree_keys");
  uint64_t* ko;
  uint32_t* vo;
  RS_TRY(radix_sort_u64(ctx, T, 30 + bits_for(uint64_t(nt)), ka, va, kb, vb, &ko, &vo, st));
  k_tree_gather<<<grid_for(T, kT), kT, 0, st>>>(T, vo, h.U, TX, tpos);
  RS_LAUNCHED(ctx, "k_tree_gather");
  {
    ProfScope prof_(ctx, "k_tree_build", st);
    k_tree_leaves<<<grid_for(C, kLeafCells), kT, 0, st>>>(C, nt, tcoff, tg, ttoff, TX, cells);
    RS_LAUNCHED(ctx, "k_tree_leaves");
    const int levels = levels_of(T);  // no node is larger than all of them together
    for (int lev = 1; lev < levels; ++lev) {
      k_tree_up<<<grid_for(C, kT), kT, 0, st>>>(C, lev, nt, tcoff, tg, cells);
      RS_LAUNCHED(ctx, "k_tree_up");
    }
    k_tree_radius<<<grid_for(C, 32), kT, 0, st>>>(C, nt, tcoff, tg, ttoff, TX, cells);
    RS_LAUNCHED(ctx, "k_tree_radius");
  }
  // walk order of the nodes (largest first)
  {
    uint64_t* oka = scratch_t<uint64_t>(ctx, S_U_OKEY_A, size_t(nt));
    uint64_t* okb = scratch_t<uint64_t>(ctx, S_U_OKEY_B, size_t(nt));
    uint32_t* ova = scratch_t<uint32_t>(ctx, S_U_OVAL_A, size_t(nt));
    uint32_t* ovb = scratch_t<uint32_t>(ctx, S_U_OVAL_B, size_t(nt));
    if (!oka || !okb || !ova || !ovb) return RS_ERR_OOM;
    k_tree_okeys<<<grid_for(nt, kT), kT, 0, st>>>(nt, tg, oka, ova);
    RS_LAUNCHED(ctx, "k_tree_okeys");
    uint64_t* oko;
    uint32_t* ovo;
    RS_TRY(radix_sort_u64(ctx, nt, 8, oka, ova, okb, ovb, &oko, &ovo, st));
    RS_CUDA(ctx, cudaMemcpyAsync(worder, ovo, 4 * size_t(nt), cudaMemcpyDeviceToDevice, st));
  }
  ctx->tree_nt = nt;
  ctx->tree_T = T;
  ctx->tree_C = C;
  return RS_OK;
}

// Decide the flags of the wanted members of the tree nodes (want[p] != 0 when `want` is given,
// else the members of the nodes with only[q] != 0 when `only` is given, else every member):
// certified interval walks, then the exact list path (blocked float32 list sums with their
// certified bound, float64 canonical-order potential) for the undecided ones.
// counters: [16] float64 queue of this call, [7] float64 total of the direct sums,
// [12..15] decided by the bound, listed for the exact path, expansions, direct pairs,
// [18] pair terms of the exact list sums.
int rs::tree_decide(rs_ctx* ctx, const int* only, const uint8_t* want, const double* vbulk,
                    uint8_t* bound, unsigned long long* counters, cudaStream_t st) {
  const int64_t nt = ctx->tree_nt, T = ctx->tree_T;
  if (nt == 0 || T == 0) return RS_OK;
  Hier h = hier_of(ctx);
  int64_t* tn = static_cast<int64_t*>(ctx->buf[S_T_NODES].ptr);
  int64_t *tnode = tn, *tg = tn + nt, *ttoff = tn + 2 * nt, *tcoff = tn + 3 * nt;
  const float4* TX = static_cast<const float4*>(ctx->buf[S_T_X].ptr);
  const uint32_t* tpos = static_cast<const uint32_t*>(ctx->buf[S_T_POS].ptr);
  const Cell* cells = static_cast<const Cell*>(ctx->buf[S_T_CELL].ptr);
  const uint32_t* worder = static_cast<const uint32_t*>(ctx->buf[S_T_ORDER].ptr);
  int64_t* wf = scratch_t<int64_t>(ctx, S_T_WF, size_t(T) + 1);
  uint32_t* wl = scratch_t<uint32_t>(ctx, S_T_WL, size_t(T));
  int64_t* wr = scratch_t<int64_t>(ctx, S_T_WR, size_t(nt) * 3 + 3);
  int64_t* uf = scratch_t<int64_t>(ctx, S_T_UF, size_t(T) + 1);
  uint32_t* ulist = scratch_t<uint32_t>(ctx, S_T_LIST, size_t(T));
  int64_t* lr = scratch_t<int64_t>(ctx, S_T_LR, size_t(nt) * 3 + 3);
  double* Sd = scratch_t<double>(ctx, S_T_SX, size_t(T));
  uint32_t* ambig = scratch_t<uint32_t>(ctx, S_U_AMBIG, size_t(ctx->n_members) + 1);
  if (!wf || !wl || !wr || !uf || !ulist || !lr || !Sd || !ambig) return RS_ERR_OOM;
  int64_t *wlo = wr, *wcnt = wr + nt, *items = wr + 2 * nt;
  k_tree_want<<<grid_for(T, kT), kT, 0, st>>>(T, tpos, h.mnode, only, want, wf);
  RS_LAUNCHED(ctx, "k_tree_want");
  RS_TRY(exclusive_scan_i64(ctx, T, wf, wf + T, st));
  k_tree_wlist<<<grid_for(T, kT), kT, 0, st>>>(T, wf, wl);
  RS_LAUNCHED(ctx, "k_tree_wlist");
  // an upper bound of the warps (items): T / 32 + nt
  const int64_t warps_ub = T / 32 + nt + 1;
  WalkArgs A;
  A.nt = nt;
  A.item_off = items;
  A.worder = worder;
  A.wlo = wlo;
  A.wcnt = wcnt;
  A.TX = TX;
  A.tpos = tpos;
  A.ttoff = ttoff;
  A.tcoff = tcoff;
  A.tg = tg;
  A.tnode = tnode;
  A.cells = cells;
  A.V = h.V;
  A.vbulk = vbulk;
  A.eps2 = ctx->cfg.softening * ctx->cfg.softening;
  A.Gm = ctx->cfg.G * ctx->cfg.particle_mass;
  A.bound = bound;
  A.rec_lo = ctx->tree_record ? static_cast<double*>(ctx->buf[S_T_REC].ptr) : nullptr;
  A.rec_hi = A.rec_lo ? A.rec_lo + ctx->n_members : nullptr;
  A.counters = counters + 12;
  // the wanted members at the opening angle, then the undecided ones at a smaller one
  unsigned long long* ucount = counters + 17;
  for (const bool last : {false, true}) {
    const float theta = last ? kRefine * ctx->tree_theta : ctx->tree_theta;
    const int targets = last ? 32 / kRefineSlices : 32;
    k_tree_items<<<grid_for(nt, kT), kT, 0, st>>>(nt, worder, ttoff, tg, wf, targets, wlo, wcnt, items);
    RS_LAUNCHED(ctx, "k_tree_items");
    RS_TRY(exclusive_scan_i64(ctx, nt, items, items + nt, st));
    RS_CUDA(ctx, cudaMemsetAsync(uf, 0, sizeof(int64_t) * (size_t(T) + 1), st));
    A.theta2 = theta * theta;
    A.chord = 1.0f / (1.0f - theta);
    A.last = last;
    A.wl = wl;
    A.und = uf;
    {
      ProfScope prof_(ctx, "k_tree_walk", st);
      const bool normal = normal_eps2(A.eps2);
      if (last) {  // few warps: a grid of one wave strides over them
        auto* kernel = normal ? k_tree_walk<true, kRefineSlices> : k_tree_walk<false, kRefineSlices>;
        kernel<<<std::min(grid_for(warps_ub * kRefineSlices * 32, kT), 152u * 4u), kT, 0, st>>>(A);
      } else {
        auto* kernel = normal ? k_tree_walk<true, 1> : k_tree_walk<false, 1>;
        kernel<<<grid_for(warps_ub * 32, kT), kT, 0, st>>>(A);
      }
    }
    RS_LAUNCHED(ctx, "k_tree_walk");
    RS_TRY(exclusive_scan_i64(ctx, T, uf, uf + T, st));
    k_tree_ulist<<<grid_for(T, kT), kT, 0, st>>>(T, uf, ulist, ucount);
    RS_LAUNCHED(ctx, "k_tree_ulist");
    std::swap(wf, uf);  // the undecided members are the next walk's targets, then the exact list
    std::swap(wl, ulist);
  }
  std::swap(wf, uf);
  std::swap(wl, ulist);
  // exact path for the undecided members
  constexpr int R = 2;  // the lists are short: few lanes of a tile are filled
  int64_t *lofs = lr, *lend = lr + nt, *ltiles = lr + 2 * nt;
  k_tree_lranges<<<grid_for(nt, kT), kT, 0, st>>>(nt, ttoff, tg, uf, kListThreads * R, lofs, lend, ltiles,
                                                  counters + 18);
  RS_LAUNCHED(ctx, "k_tree_lranges");
  RS_TRY(exclusive_scan_i64(ctx, nt, ltiles, ltiles + nt, st));
  const float eps2 = ctx->cfg.softening * ctx->cfg.softening;
  {
    ProfScope prof_(ctx, "k_potential_list", st);
    RS_TRY(launch_potential_list(ctx, R, eps2, T, Sd, st, nt, ltiles, tnode, lofs, lend, ulist, tpos,
                                 h.node_off, h.node_size, h.U));
  }
  const double Gm = ctx->cfg.G * ctx->cfg.particle_mass;
  auto* flags = normal_eps2(eps2) ? k_flags_list<true> : k_flags_list<false>;
  flags<<<grid_for(T, kT), kT, 0, st>>>(ucount, ulist, tpos, h.mnode, h.V, vbulk, eps2, Gm, Sd, bound, ambig,
                                       counters + 16);
  RS_LAUNCHED(ctx, "k_flags_list");
  RS_TRY(unbind_fallback(ctx, counters + 16, ambig, vbulk, bound, st));
  k_tree_acc<<<1, 1, 0, st>>>(counters, 16, 7);
  RS_LAUNCHED(ctx, "k_tree_acc");
  return RS_OK;
}

extern "C" int rs_tree_record(rs_ctx* ctx, int enable) {
  if (!ctx) return RS_ERR_INVALID_ARG;
  ctx->err[0] = 0;
  ctx->tree_record = enable != 0;
  return RS_OK;
}

extern "C" int rs_tree_bounds(rs_ctx* ctx, double* lo_out, double* hi_out, void* stream) {
  if (!ctx) return RS_ERR_INVALID_ARG;
  ctx->err[0] = 0;
  if (!ctx->have_unbind || !ctx->tree_recorded)
    return set_error(ctx, RS_ERR_STATE, "no recorded rs_unbind (rs_tree_record(ctx, 1) first)");
  const int64_t m = ctx->n_members;
  if (m > 0 && (!lo_out || !hi_out)) return set_error(ctx, RS_ERR_INVALID_ARG, "null output");
  RS_CUDA(ctx, cudaSetDevice(ctx->device));
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const double* rec = static_cast<const double*>(ctx->buf[S_T_REC].ptr);
  if (m > 0) {
    RS_CUDA(ctx, cudaMemcpyAsync(lo_out, rec, 8 * size_t(m), cudaMemcpyDeviceToDevice, st));
    RS_CUDA(ctx, cudaMemcpyAsync(hi_out, rec + m, 8 * size_t(m), cudaMemcpyDeviceToDevice, st));
  }
  return RS_OK;
}

extern "C" int rs_tree_stats(rs_ctx* ctx, int64_t* stats_out) {
  if (!ctx || !stats_out) return RS_ERR_INVALID_ARG;
  for (int i = 0; i < 8; ++i) stats_out[i] = ctx->tree_stats[i];
  return RS_OK;
}
