// Pruned 6D nearest-neighbour and link searches for the batched form of rs_fof6d.
//
// The plain form evaluates d6 for every pair of a node. Here the members of every node of a
// level are ordered by a 6D Hilbert key of their scaled position and velocity offsets and cut
// into buckets of 32 consecutive members; each bucket has a 6D bounding box, and every 32
// consecutive buckets of a node form a superbucket (1024 members) with its own box. Ordering by
// all six coordinates keeps a bucket small in velocity too: in a node of 7e5 members a search
// evaluates about a sixth of the pairs that buckets of a 3D position curve need.
//
// Persistent warps pull query buckets from a queue ordered by node size (largest first). A
// search tests 32 boxes at a time against the box of the warp's open queries (lane = box), then
// each surviving bucket box against every query (lane = query); a bucket that some queries need
// is loaded with lane = target, and the warp loops over those queries (about 3 of 32 lanes need a
// given bucket, so lane = query would idle most of the warp). Distances and bounds use packed
// float32x2 arithmetic over (position, velocity) pairs, each half rounded like the scalar
// operation. Lower bounds are computed with the same round-to-nearest float32 operations as d6
// on the per-axis gaps to the box: every step is monotone, so the bound never exceeds the
// computed d6 of any member inside the box, and pruning cannot change the minimum or the set of
// links. Results are therefore bit-identical to the brute-force kernels (and to the definition).
//
// Nearest neighbours: every member inside its own superbucket first (k_nn_near; complete for
// nodes of one superbucket). The k-th smallest of those values bounds l2 from above, so the rest
// of the search (k_nn_far) goes no further than that; nodes of 4096 members or more also get a
// lower bound from an exactly searched sample of their buckets and search only their members at
// or above it (a device check after the selection re-searches any node whose l2 falls outside).
//
// Links: only members with a friend (nn2 <= l2) can be linked; they are compacted in the same
// order and bucketed again, and each is first united with its nearest neighbour. k_link_near
// unites inside each superbucket, skipping targets that already share the query's root;
// k_link_far then searches the rest of the node for the members outside the node's largest
// component only (every remaining link has such an end), skipping buckets and targets that
// already share the query's root. Few distances are left to evaluate and few unions are made
// (about 0.3 a member instead of 17).
//
// Measured on the 2^27-particle snapshot (12 levels, 1.2e8 members), before and after this form:
// nearest-neighbour kernels 382 -> 99 ms, link kernels 266 -> 89 ms (3D Hilbert buckets with
// sub-boxes, lane = query). In a pass over 2^24 particles (ncu, level 0) the issue slots are busy 78% of
// the cycles in the nearest-neighbour kernels (ALU 40-52%, FMA 33%) and 69% in k_link_far: box tests and
// distances. k_link_near has them busy 53%: a warp waits 6 cycles an instruction for parents of the
// union-find. None moves more than 0.2 TB/s from memory.
#include "rs_cro.cuh"

namespace rs {
int prune6d_prepare(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t mb, int64_t m,
                    const double* sums, cudaStream_t st);
int prune6d_near(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t mb, int64_t m, float* nn2,
                 cudaStream_t st);
int prune6d_far(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t mb, int64_t m, float* nn2,
                cudaStream_t st);
int prune6d_check(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t m, float* nn2, const int** failed_out,
                  cudaStream_t st);
int prune6d_link(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t mb, int64_t m, const float* nn2,
                 uint32_t* uf, cudaStream_t st);
}  // namespace rs

using namespace rs;

namespace {

constexpr int kT = 256;
constexpr int kWarpsPerBlock = 8;
constexpr unsigned kFull = 0xffffffffu;

struct Bucket {
  uint32_t start;    // level-local sorted position of the first member
  uint32_t count;    // 1..32
  uint32_t node;     // global node index
  uint32_t first;    // index of the node's first bucket
  uint32_t last;     // index of the node's last bucket
  uint32_t sbfirst;  // index of the node's first superbucket
  uint32_t sbcount;  // superbuckets of the node
  uint32_t pad;
};

// 6D box, stored for the packed float32x2 bounds: (position, velocity) pairs per axis, the
// lower corner and the NEGATED upper corner (so both gaps are additions).
struct __align__(16) Box {
  float4 lo01;   // (x, vx, y, vy)
  float4 nhi01;  // -(x, vx, y, vy) of the upper corner
  float2 lo2;    // (z, vz)
  float2 nhi2;
};

// 4 bits an axis: 24 key bits (three sort passes below the node index); in a CPU model of a
// 7e5-member node a fifth bit saves 1% of the searches' work.
constexpr int kAxisBits = 4;
constexpr int kKeyBits = 6 * kAxisBits;

// Scaled offset c (units of the node's total sigma) to 0 .. 2^kAxisBits - 1 through c / (0.5 + |c|),
// which spends most cells on the node's dense middle (12% fewer box tests than a linear map).
__device__ __forceinline__ uint32_t quant_axis(float c) {
  constexpr float half = float(1 << (kAxisBits - 1));
  const float t = half + half * (c / (0.5f + fabsf(c)));
  return uint32_t(fminf(fmaxf(t, 0.0f), 2.0f * half - 1.0f));
}

// 6D Hilbert index of quantised coordinates by Skilling's transform (J. Skilling, "Programming
// the Hilbert curve", AIP Conf. Proc. 707, 2004), axis 0 leading.
__device__ __forceinline__ uint32_t hilbert6(uint32_t (&X)[6]) {
#pragma unroll
  for (uint32_t q = 1u << (kAxisBits - 1); q > 1; q >>= 1) {
    const uint32_t p = q - 1;
#pragma unroll
    for (int i = 0; i < 6; ++i) {
      if (X[i] & q) {
        X[0] ^= p;
      } else {
        const uint32_t t = (X[0] ^ X[i]) & p;
        X[0] ^= t;
        X[i] ^= t;
      }
    }
  }
#pragma unroll
  for (int i = 1; i < 6; ++i) X[i] ^= X[i - 1];
  uint32_t t = 0;
#pragma unroll
  for (uint32_t q = 1u << (kAxisBits - 1); q > 1; q >>= 1)
    if (X[5] & q) t ^= q - 1;
  uint32_t key = 0;
#pragma unroll
  for (int b = kAxisBits - 1; b >= 0; --b)
#pragma unroll
    for (int i = 0; i < 6; ++i) key = (key << 1) | (((X[i] ^ t) >> b) & 1u);
  return key;
}

// 6D Hilbert key of each member's offset from the node mean (scaled by the node's sigmas),
// prefixed by the node index.
__global__ void k_hilbert6(int64_t mb, int64_t m, int64_t nb, const uint32_t* __restrict__ mnode,
                           const float4* __restrict__ U, const float4* __restrict__ V,
                           const float4* __restrict__ inv, const float4* __restrict__ mean_u,
                           const float4* __restrict__ mean_v, uint64_t* __restrict__ keys,
                           uint32_t* __restrict__ vals) {
  const int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (p >= m) return;
  const uint32_t q = mnode[mb + p];
  const float4 iv = inv[q];
  const float sx = sqrtf(iv.x), sv = sqrtf(iv.y);
  const float4 u = U[mb + p], mu = mean_u[q], v = V[mb + p], mv = mean_v[q];
  uint32_t X[6] = {quant_axis((u.x - mu.x) * sx), quant_axis((u.y - mu.y) * sx), quant_axis((u.z - mu.z) * sx),
                   quant_axis((v.x - mv.x) * sv), quant_axis((v.y - mv.y) * sv), quant_axis((v.z - mv.z) * sv)};
  keys[p] = (uint64_t(q - nb) << kKeyBits) | uint64_t(hilbert6(X));
  vals[p] = uint32_t(p);
}

// Node means (float) from the canonical-order moment sums, for the quantisation only.
__global__ void k_node_means(int64_t nb, int64_t nn, const int64_t* __restrict__ node_size,
                             const double* __restrict__ sums, float4* __restrict__ mean_u,
                             float4* __restrict__ mean_v) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= nn) return;
  const double g = double(node_size[nb + k]);
  const double* S = sums + 12 * k;
  mean_u[nb + k] = make_float4(float(S[0] / g), float(S[1] / g), float(S[2] / g), 0.f);
  mean_v[nb + k] = make_float4(float(S[6] / g), float(S[7] / g), float(S[8] / g), 0.f);
}

// Members in sorted order as (position, velocity) pairs: XY = (x, vx, y, vy), Z = (z, vz).
__global__ void k_gather_sorted(int64_t mb, int64_t m, const uint32_t* __restrict__ order,
                                const float4* __restrict__ U, const float4* __restrict__ V,
                                float4* __restrict__ XY, float2* __restrict__ Z, uint32_t* __restrict__ sp) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= m) return;
  const uint32_t p = order[s];
  const float4 u = U[mb + p], v = V[mb + p];
  XY[s] = make_float4(u.x, v.x, u.y, v.y);
  Z[s] = make_float2(u.z, v.z);
  sp[s] = p;
}

// Members of each node of the level in the bucketed arrays: start (level-local sorted
// position) and count; all members for the NN pass, the members with a friend for the link pass.
__global__ void k_node_ranges(int64_t nb, int64_t nn, int64_t mb, const int64_t* __restrict__ node_off,
                              const int64_t* __restrict__ node_size, int64_t* __restrict__ start,
                              int64_t* __restrict__ cnt) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= nn) return;
  start[k] = node_off[nb + k] - mb;
  cnt[k] = node_size[nb + k];
}

__global__ void k_bucket_counts(int64_t nn, const int64_t* __restrict__ cnt, int64_t* __restrict__ bcnt,
                                int64_t* __restrict__ sbcnt) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= nn) return;
  const int64_t c = (cnt[k] + 31) / 32;
  bcnt[k] = c;
  sbcnt[k] = (c + 31) / 32;
}

// Link pass: the members with a friend (nn2 <= l2 of their node), compacted in sorted order.
__global__ void k_active_flags(int64_t m, int64_t mb, const uint32_t* __restrict__ sp,
                               const uint32_t* __restrict__ mnode, const float4* __restrict__ inv,
                               const float* __restrict__ nn2, int64_t* __restrict__ flag) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= m) return;
  flag[s] = nn2[s] <= inv[mnode[mb + sp[s]]].z ? 1 : 0;
}

__global__ void k_compact_active(int64_t m, const int64_t* __restrict__ pos, const float4* __restrict__ XY,
                                 const float2* __restrict__ Z, const uint32_t* __restrict__ sp,
                                 float4* __restrict__ XYA, float2* __restrict__ ZA,
                                 uint32_t* __restrict__ spA, uint32_t* __restrict__ ufA) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= m || pos[s + 1] == pos[s]) return;
  const int64_t a = pos[s];
  XYA[a] = XY[s];
  ZA[a] = Z[s];
  spA[a] = sp[s];
  ufA[a] = uint32_t(a);
}

// Each compacted member united with the neighbour that gave its nn2: their d6 is at most l2, so
// that neighbour has a friend too.
__global__ void k_link_friends(int64_t m, const int64_t* __restrict__ pos, const uint32_t* __restrict__ friend_of,
                               uint32_t* __restrict__ ufA) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= m || pos[s + 1] == pos[s]) return;
  const uint32_t f = friend_of[s];
  if (int64_t(f) != s && pos[f + 1] != pos[f]) rsd::uf_unite(ufA, uint32_t(pos[s]), uint32_t(pos[f]));
}

__global__ void k_active_ranges(int64_t nb, int64_t nn, int64_t mb, const int64_t* __restrict__ node_off,
                                const int64_t* __restrict__ node_size, const int64_t* __restrict__ pos,
                                int64_t* __restrict__ start, int64_t* __restrict__ cnt) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= nn) return;
  const int64_t s0 = node_off[nb + k] - mb;
  start[k] = pos[s0];
  cnt[k] = pos[s0 + node_size[nb + k]] - pos[s0];
}

// Box of the warp's valid lanes' points (lane = point; a = x, y, z, vx, vy, vz); every lane gets it.
__device__ __forceinline__ void warp_box(const float (&a)[6], bool valid, float (&lo)[6], float (&hi)[6]) {
  const float inf = __int_as_float(0x7f800000);
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    lo[d] = valid ? a[d] : inf;
    hi[d] = valid ? a[d] : -inf;
#pragma unroll
    for (int off = 1; off <= 16; off <<= 1) {
      lo[d] = fminf(lo[d], __shfl_xor_sync(kFull, lo[d], off));
      hi[d] = fmaxf(hi[d], __shfl_xor_sync(kFull, hi[d], off));
    }
  }
}

// lo, hi indexed (x, y, z, vx, vy, vz).
__device__ __forceinline__ Box make_box(const float (&lo)[6], const float (&hi)[6]) {
  return Box{make_float4(lo[0], lo[3], lo[1], lo[4]), make_float4(-hi[0], -hi[3], -hi[1], -hi[4]),
             make_float2(lo[2], lo[5]), make_float2(-hi[2], -hi[5])};
}

__device__ __forceinline__ Box query_box(const float (&c)[6], bool open) {
  float lo[6], hi[6];
  warp_box(c, open, lo, hi);
  return make_box(lo, hi);
}

// The warp's query box again once half of the queries it was made for are closed.
__device__ __forceinline__ void refresh_box(Box& QB, int& boxed, const float (&c)[6], bool open) {
  const int n = __popc(__ballot_sync(kFull, open));
  if (n == 0 || 2 * n > boxed) return;
  QB = query_box(c, open);
  boxed = n;
}

// Takes the set bit of a non-empty mask nearest to position `own`: near stretches of the curve first.
__device__ __forceinline__ int next_outward(unsigned& mask, int own) {
  const unsigned up = mask & ~((1u << own) - 1u), dn = mask & ((1u << own) - 1u);
  const int iu = up ? __ffs(up) - 1 : 64, id = dn ? 31 - __clz(dn) : -64;
  const int i = iu - own <= own - id ? iu : id;
  mask &= ~(1u << i);
  return i;
}

// One warp per bucket (padding warps write a queue key that sorts last): bucket table entry, box,
// and the work-queue key (largest node first).
__global__ void __launch_bounds__(kT)
k_buckets(int64_t nb, int64_t nn, int64_t nbk_ub, const int64_t* __restrict__ bucket_off,
          const int64_t* __restrict__ sb_off, const int64_t* __restrict__ nstart,
          const int64_t* __restrict__ ncnt, const float4* __restrict__ XY,
          const float2* __restrict__ Z, Bucket* __restrict__ bk, Box* __restrict__ box,
          uint64_t* __restrict__ qkey, uint32_t* __restrict__ qval) {
  const int64_t w = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= nbk_ub) return;
  if (w >= bucket_off[nn]) {
    if (lane == 0) {
      qkey[w] = 255u;  // the largest key: after every real bucket (stable sort, higher indices)
      qval[w] = uint32_t(w);
    }
    return;
  }
  const int64_t k = rsd::upper_bound_i64(bucket_off, nn, w) - 1;
  const int64_t q = nb + k;
  const int64_t kb = w - bucket_off[k];
  const int64_t start = nstart[k] + 32 * kb;
  const int cnt = int(rsd::min64(32, ncnt[k] - 32 * kb));
  const bool valid = lane < cnt;
  const float4 xy = XY[start + (valid ? lane : 0)];
  const float2 z = Z[start + (valid ? lane : 0)];
  const float a[6] = {xy.x, xy.z, z.x, xy.y, xy.w, z.y};
  float lo[6], hi[6];
  warp_box(a, valid, lo, hi);
  if (lane == 0) {
    Bucket b;
    b.start = uint32_t(start);
    b.count = uint32_t(cnt);
    b.node = uint32_t(q);
    b.first = uint32_t(bucket_off[k]);
    b.last = uint32_t(bucket_off[k + 1] - 1);
    b.sbfirst = uint32_t(sb_off[k]);
    b.sbcount = uint32_t(sb_off[k + 1] - sb_off[k]);
    b.pad = 0;
    bk[w] = b;
    box[w] = make_box(lo, hi);
    qkey[w] = 255u - rsd::size_class(ncnt[k]);
    qval[w] = uint32_t(w);
  }
}

// One warp per superbucket: the box of its (up to 32) bucket boxes.
__global__ void __launch_bounds__(kT)
k_superboxes(int64_t nn, const int64_t* __restrict__ bucket_off, const int64_t* __restrict__ sb_off,
             const Box* __restrict__ box, Box* __restrict__ sbox) {
  const int64_t w = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= sb_off[nn]) return;
  const int64_t k = rsd::upper_bound_i64(sb_off, nn, w) - 1;
  const int64_t b0 = bucket_off[k] + 32 * (w - sb_off[k]);
  const int64_t b1 = rsd::min64(b0 + 32, bucket_off[k + 1]);
  const bool valid = b0 + lane < b1;
  const Box B = box[valid ? b0 + lane : b0];
  const float inf = __int_as_float(0x7f800000);
  float lo[6] = {B.lo01.x, B.lo01.z, B.lo2.x, B.lo01.y, B.lo01.w, B.lo2.y};
  float hi[6] = {-B.nhi01.x, -B.nhi01.z, -B.nhi2.x, -B.nhi01.y, -B.nhi01.w, -B.nhi2.y};
#pragma unroll
  for (int d = 0; d < 6; ++d) {
    lo[d] = valid ? lo[d] : inf;
    hi[d] = valid ? hi[d] : -inf;
#pragma unroll
    for (int off = 1; off <= 16; off <<= 1) {
      lo[d] = fminf(lo[d], __shfl_xor_sync(0xffffffffu, lo[d], off));
      hi[d] = fmaxf(hi[d], __shfl_xor_sync(0xffffffffu, hi[d], off));
    }
  }
  if (lane == 0) sbox[w] = make_box(lo, hi);
}

// Packed float32x2 add and multiply, each half rounded exactly like __fadd_rn / __fmul_rn. The
// float2 intrinsics let the compiler fuse a multiply into a following add (an FMA: one rounding
// instead of two, which changes d6 in the last bit); inline PTX with the product taken as an
// fma with a +0 addend keeps every rounding (fl(a b + 0) = fl(a b) for the non-negative
// products used here).
__device__ __forceinline__ float2 padd(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "add.rn.f32x2 rd, ra, rb;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

__device__ __forceinline__ float2 pmul(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 ra, rb, rz, rd;\n\tmov.b64 ra, {%2, %3};\n\tmov.b64 rb, {%4, %5};\n\t"
      "mov.b64 rz, 0;\n\tfma.rn.f32x2 rd, ra, rb, rz;\n\tmov.b64 {%0, %1}, rd;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

__device__ __forceinline__ float2 max0(float2 a, float2 b) {
  return make_float2(fmaxf(fmaxf(a.x, b.x), 0.f), fmaxf(fmaxf(a.y, b.y), 0.f));
}

// Per-axis gap from q to [lo, hi]: max(fl(lo - q), fl(q - hi), 0). When q < lo this is
// fl(lo - q) (the other difference is negative), when q > hi it is fl(q - hi), otherwise 0:
// rounded like the d6 differences, hence never above |fl(y - q)| for any y in the interval.
__device__ __forceinline__ float2 gap_pt(float2 lo, float2 nhi, float2 q, float2 nq) {
  return max0(padd(lo, nq), padd(q, nhi));
}

// Gap between two intervals: max(fl(blo - ahi), fl(alo - bhi), 0).
__device__ __forceinline__ float2 gap_bb(float2 alo, float2 anhi, float2 blo, float2 bnhi) {
  return max0(padd(blo, anhi), padd(alo, bnhi));
}

// fl(fl(rx * inv_sx2) + fl(rv * inv_sv2)) with (rx, rv) = ((ga^2 + gb^2) + gc^2) per half:
// the operation order of d6.
__device__ __forceinline__ float metric(float2 ga, float2 gb, float2 gc, float2 s) {
  const float2 r = padd(padd(pmul(ga, ga), pmul(gb, gb)), pmul(gc, gc));
  const float2 t = pmul(r, s);
  return __fadd_rn(t.x, t.y);
}

__device__ __forceinline__ float lb_box_box(const Box& a, const Box& b, float2 s) {
  return metric(gap_bb(make_float2(a.lo01.x, a.lo01.y), make_float2(a.nhi01.x, a.nhi01.y),
                       make_float2(b.lo01.x, b.lo01.y), make_float2(b.nhi01.x, b.nhi01.y)),
                gap_bb(make_float2(a.lo01.z, a.lo01.w), make_float2(a.nhi01.z, a.nhi01.w),
                       make_float2(b.lo01.z, b.lo01.w), make_float2(b.nhi01.z, b.nhi01.w)),
                gap_bb(a.lo2, a.nhi2, b.lo2, b.nhi2), s);
}

// A query lane's own coordinates as (position, velocity) pairs per axis, with their negations.
struct Query {
  float2 a, b, c, na, nb, nc;
};

__device__ __forceinline__ Query make_query(float4 xy, float2 z) {
  Query Q;
  Q.a = make_float2(xy.x, xy.y);
  Q.b = make_float2(xy.z, xy.w);
  Q.c = z;
  Q.na = make_float2(-xy.x, -xy.y);
  Q.nb = make_float2(-xy.z, -xy.w);
  Q.nc = make_float2(-z.x, -z.y);
  return Q;
}

__device__ __forceinline__ float lb_point_box(const Query& Q, const Box& b, float2 s) {
  return metric(gap_pt(make_float2(b.lo01.x, b.lo01.y), make_float2(b.nhi01.x, b.nhi01.y), Q.a, Q.na),
                gap_pt(make_float2(b.lo01.z, b.lo01.w), make_float2(b.nhi01.z, b.nhi01.w), Q.b, Q.nb),
                gap_pt(b.lo2, b.nhi2, Q.c, Q.nc), s);
}

// d6 of target (xy, z) to the query with negated coordinates (nxy, nz): the differences formed as
// u_j + (-u_i) = fl(u_j - u_i), then d6's order of operations.
__device__ __forceinline__ float d6_pair(float4 xy, float2 z, float4 nxy, float2 nz, float2 s) {
  return metric(padd(make_float2(xy.x, xy.y), make_float2(nxy.x, nxy.y)),
                padd(make_float2(xy.z, xy.w), make_float2(nxy.z, nxy.w)), padd(z, nz), s);
}

// Shared memory of one warp: its queries' negated coordinates and roots, and 32 staged boxes.
struct __align__(16) WarpShared {
  Box box[32];
  float4 nxy[32];
  float2 nz[32];
  uint32_t root[32];   // link: root of each query
  uint32_t uni[32];    // link, far: root shared by all members of the staged box's bucket
};

// Target coordinates of a bucket, lane = member; lanes past its count hold NaN, whose distance is
// NaN: as an unsigned value above every distance, and it passes no <= test.
__device__ __forceinline__ void load_targets(const float4* __restrict__ XY, const float2* __restrict__ Z,
                                             uint32_t start, int cnt, int lane, float4& xy, float2& z) {
  const float nan = __int_as_float(0x7fc00000);
  xy = make_float4(nan, nan, nan, nan);
  z = make_float2(nan, nan);
  if (lane < cnt) {
    xy = XY[start + lane];
    z = Z[start + lane];
  }
}

// Next query bucket from the size-ordered queue (one atomic per warp).
__device__ __forceinline__ int64_t next_work(unsigned long long* counter, int lane) {
  unsigned long long w = 0;
  if (lane == 0) w = atomicAdd(counter, 1ull);
  return int64_t(__shfl_sync(kFull, w, 0));
}

struct SearchArgs {
  const int64_t* nbuckets;
  const Bucket* bk;
  const Box* box;
  const Box* sbox;
  const uint32_t* order;
  const float4* XY;
  const float2* Z;
  const float4* inv;
  unsigned long long* counter;
  unsigned long long* work;  // [4]: NN d6, NN box tests, link d6, link box tests (counting variant)
  int64_t nb;
};

// Per-lane tallies of the counting variant (evaluated d6 and box tests).
struct Tally {
  unsigned long long d6 = 0, box = 0;
};

template <bool kCount>
__device__ __forceinline__ void flush_tally(const Tally& T, unsigned long long* work, int lane) {
  if (!kCount) return;
  unsigned long long d = T.d6, b = T.box;
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    d += __shfl_xor_sync(kFull, d, off);
    b += __shfl_xor_sync(kFull, b, off);
  }
  if (lane == 0) {
    atomicAdd(work, d);
    atomicAdd(work + 1, b);
  }
}

// ---- Nearest neighbours -----------------------------------------------------------------------

// Minimum over bucket b's members for every query in the mask `need`: the lane of each such query
// lowers its best (float bits) and neighbour. kSelf: b is the query bucket itself.
template <bool kCount, bool kSelf>
__device__ __forceinline__ void nn_eval(const SearchArgs& A, uint32_t start, int cnt, unsigned need, float2 s,
                                        uint32_t& best, uint32_t& nbr, int lane, const WarpShared& W, Tally& T) {
  float4 xy;
  float2 z;
  load_targets(A.XY, A.Z, start, cnt, lane, xy, z);
  if (kCount && lane < cnt) T.d6 += __popc(need) - ((kSelf && ((need >> lane) & 1u)) ? 1 : 0);
  while (need) {
    const int l0 = __ffs(need) - 1;
    need &= need - 1u;
    const int l1 = need ? __ffs(need) - 1 : l0;  // two queries side by side
    need &= need - 1u;
    uint32_t d0 = __float_as_uint(d6_pair(xy, z, W.nxy[l0], W.nz[l0], s));
    uint32_t d1 = __float_as_uint(d6_pair(xy, z, W.nxy[l1], W.nz[l1], s));
    if (kSelf) {
      d0 = lane == l0 ? 0xffffffffu : d0;
      d1 = lane == l1 ? 0xffffffffu : d1;
    }
    const uint32_t m0 = __reduce_min_sync(kFull, d0), m1 = __reduce_min_sync(kFull, d1);
    const int j0 = __ffs(__ballot_sync(kFull, d0 == m0)) - 1, j1 = __ffs(__ballot_sync(kFull, d1 == m1)) - 1;
    if (lane == l0 && m0 < best) {
      best = m0;
      nbr = start + j0;
    }
    if (lane == l1 && m1 < best) {
      best = m1;
      nbr = start + j1;
    }
  }
}

// Candidate buckets of one superbucket, [b_lo, b_hi) (at most 32): boxes staged in shared memory
// by lane = box, those within `limit` (float bits) of the query box returned as a mask.
template <bool kCount>
__device__ __forceinline__ unsigned stage_boxes(const SearchArgs& A, int64_t b_lo, int64_t b_hi, const Box& Q,
                                                float limit, float2 s, int lane, WarpShared& W, Tally& T) {
  const bool in = b_lo + lane < b_hi;
  bool near = false;
  __syncwarp();
  if (in) {
    const Box B = A.box[b_lo + lane];
    W.box[lane] = B;
    near = lb_box_box(Q, B, s) <= limit;
    if (kCount) T.box += 1;
  }
  __syncwarp();
  return __ballot_sync(kFull, near);
}

// Exact nearest neighbour of every member inside its own superbucket -> nn2 (sorted order) and
// neighbour (sorted position).
template <bool kCount>
__global__ void __launch_bounds__(kT, 4)
k_nn_near(SearchArgs A, float* __restrict__ nn2, uint32_t* __restrict__ friend_of) {
  __shared__ WarpShared sh[kWarpsPerBlock];
  const int lane = threadIdx.x & 31;
  WarpShared& W = sh[threadIdx.x >> 5];
  const int64_t nbk = *A.nbuckets;
  Tally T;
  while (true) {
    const int64_t w = next_work(A.counter, lane);
    if (w >= nbk) break;
    const int64_t a = A.order[w];
    const Bucket Aq = A.bk[a];
    const float4 iv = A.inv[Aq.node];
    const float2 s = make_float2(iv.x, iv.y);
    const bool valid = lane < int(Aq.count);
    const uint32_t si = Aq.start + (valid ? lane : 0);
    const Query Q = make_query(A.XY[si], A.Z[si]);
    __syncwarp();
    W.nxy[lane] = make_float4(Q.na.x, Q.na.y, Q.nb.x, Q.nb.y);
    W.nz[lane] = Q.nc;
    __syncwarp();
    uint32_t best = 0x7f800000u, nbr = si;
    nn_eval<kCount, true>(A, Aq.start, int(Aq.count), Aq.count == 32 ? kFull : (1u << Aq.count) - 1u, s, best,
                          nbr, lane, W, T);
    const int64_t b_lo = int64_t(Aq.first) + ((a - int64_t(Aq.first)) & ~int64_t(31));
    const int64_t b_hi = rsd::min64(b_lo + 32, int64_t(Aq.last) + 1);
    if (b_hi - b_lo > 1) {
      const float lim = __uint_as_float(__reduce_max_sync(kFull, valid ? best : 0u));
      unsigned mask = stage_boxes<kCount>(A, b_lo, b_hi, A.box[a], lim, s, lane, W, T);
      const int own = int(a - b_lo);
      mask &= ~(1u << own);
      while (mask) {  // outward from the query bucket: near buckets lower the limit first
        const int i = next_outward(mask, own);
        const bool need = valid && lb_point_box(Q, W.box[i], s) <= __uint_as_float(best);
        if (kCount) T.box += valid;
        const unsigned nm = __ballot_sync(kFull, need);
        if (!nm) continue;
        const int64_t b = b_lo + i;
        const int cnt = b == int64_t(Aq.last) ? int(A.bk[b].count) : 32;
        nn_eval<kCount, false>(A, uint32_t(int64_t(Aq.start) + 32 * (b - a)), cnt, nm, s, best, nbr, lane, W, T);
      }
    }
    if (valid) {
      nn2[si] = __uint_as_float(best);
      friend_of[si] = nbr;
    }
  }
  flush_tally<kCount>(T, A.work, lane);
}

// Which query buckets a k_nn_far launch takes. The first launch: the sampled buckets of the nodes
// searched with bounds and every bucket of the other nodes; the second: the remaining buckets of the
// bounded nodes; the third: every bucket of the nodes that failed the check.
enum FarPass : int { kFarFirst, kFarRest, kFarFailed };

struct FarArgs {
  const float2* bounds;       // per node of the level: (lo, hi)
  const int64_t* node_size;
  const int* failed;          // third launch only
  int64_t min_members;        // smallest node searched with sampled bounds
  int pass;
};

constexpr int64_t kSampleBuckets = 48;

__device__ __forceinline__ int64_t sample_stride(int64_t nbk) {
  return nbk / kSampleBuckets > 1 ? nbk / kSampleBuckets : 1;
}

// The rest of the node for the members whose value is not yet known to be below lo: no further
// than min(best, hi) (a minimum above hi only needs to be known above hi). Members of nodes with
// one superbucket are complete.
template <bool kCount>
__global__ void __launch_bounds__(kT, 4)
k_nn_far(SearchArgs A, FarArgs F, float* __restrict__ nn2, uint32_t* __restrict__ friend_of) {
  __shared__ WarpShared sh[kWarpsPerBlock];
  const int lane = threadIdx.x & 31;
  WarpShared& W = sh[threadIdx.x >> 5];
  const int64_t nbk = *A.nbuckets;
  Tally T;
  while (true) {
    const int64_t w = next_work(A.counter, lane);
    if (w >= nbk) break;
    const int64_t a = A.order[w];
    const Bucket Aq = A.bk[a];
    const int64_t g = F.node_size[Aq.node];
    if (g < 1024) break;  // size-class order: only nodes of one superbucket follow
    if (Aq.sbcount == 1) continue;
    const int64_t k = int64_t(Aq.node) - A.nb;
    const int64_t own_rel = a - int64_t(Aq.first);
    if (F.pass == kFarFailed) {
      if (!F.failed[k]) continue;
    } else {
      const bool first = g < F.min_members ||
                         own_rel % sample_stride(int64_t(Aq.last) - int64_t(Aq.first) + 1) == 0;
      if (first != (F.pass == kFarFirst)) continue;
    }
    const float4 iv = A.inv[Aq.node];
    const float2 s = make_float2(iv.x, iv.y);
    const float2 bd = F.bounds[k];
    const bool valid = lane < int(Aq.count);
    const uint32_t si = Aq.start + (valid ? lane : 0);
    uint32_t best = __float_as_uint(nn2[si]), nbr = friend_of[si];
    bool open = valid && __uint_as_float(best) >= bd.x;
    if (!__any_sync(kFull, open)) continue;
    const float4 xy = A.XY[si];
    const float2 z = A.Z[si];
    const Query Q = make_query(xy, z);
    __syncwarp();
    W.nxy[lane] = make_float4(Q.na.x, Q.na.y, Q.nb.x, Q.nb.y);
    W.nz[lane] = Q.nc;
    __syncwarp();
    const float c[6] = {xy.x, xy.z, z.x, xy.y, xy.w, z.y};
    const Box QB = query_box(c, open);
    float lim = open ? fminf(__uint_as_float(best), bd.y) : -1.f;
    int wl = __reduce_max_sync(kFull, __float_as_int(lim));  // signed: a closed lane's -1 is below all
    const int64_t own = own_rel >> 5, nsb = Aq.sbcount;
    for (int64_t s0 = 0; s0 < nsb && wl >= 0; s0 += 32) {
      bool near = false;
      if (s0 + lane < nsb && s0 + lane != own) {
        near = lb_box_box(QB, A.sbox[Aq.sbfirst + s0 + lane], s) <= __int_as_float(wl);
        if (kCount) T.box += 1;
      }
      unsigned sm = __ballot_sync(kFull, near);
      while (sm && wl >= 0) {
        const int64_t sb = s0 + __ffs(sm) - 1;
        sm &= sm - 1u;
        const int64_t b_lo = int64_t(Aq.first) + 32 * sb;
        const int64_t b_hi = rsd::min64(b_lo + 32, int64_t(Aq.last) + 1);
        unsigned mask = stage_boxes<kCount>(A, b_lo, b_hi, QB, __int_as_float(wl), s, lane, W, T);
        while (mask) {
          const int i = __ffs(mask) - 1;
          mask &= mask - 1u;
          const bool need = open && lb_point_box(Q, W.box[i], s) <= lim;
          if (kCount) T.box += open;
          const unsigned nm = __ballot_sync(kFull, need);
          if (!nm) continue;
          const int64_t b = b_lo + i;
          const int cnt = b == int64_t(Aq.last) ? int(A.bk[b].count) : 32;
          nn_eval<kCount, false>(A, uint32_t(int64_t(Aq.start) + 32 * (b - a)), cnt, nm, s, best, nbr, lane, W, T);
          if (need) {
            open = __uint_as_float(best) >= bd.x;
            lim = open ? fminf(__uint_as_float(best), bd.y) : -1.f;
          }
        }
        wl = __reduce_max_sync(kFull, __float_as_int(lim));
      }
    }
    if (valid) {
      nn2[si] = __uint_as_float(best);
      friend_of[si] = nbr;
    }
  }
  flush_tally<kCount>(T, A.work, lane);
}

// ---- Links ------------------------------------------------------------------------------------

// Unite the queries in `need` with the members of one bucket that lie within l2 and do not share
// their root yet (returns whether there were any). rj: this lane's target's root. kSelf: the bucket is the query bucket itself
// (pairs j > l only).
template <bool kCount, bool kSelf>
__device__ __forceinline__ bool link_eval(const SearchArgs& A, uint32_t* uf, uint32_t start, int cnt, unsigned need,
                                          float2 s, float l2, uint32_t rj, int lane, WarpShared& W, Tally& T) {
  float4 xy;
  float2 z;
  load_targets(A.XY, A.Z, start, cnt, lane, xy, z);
  bool united = false;
  while (need) {
    const int l = __ffs(need) - 1;
    need &= need - 1u;
    const uint32_t rq = W.root[l];
    const bool cand = lane < cnt && rj != rq && (!kSelf || lane > l);
    if (!__any_sync(kFull, cand)) continue;
    if (kCount) T.d6 += cand;
    const bool hit = cand && d6_pair(xy, z, W.nxy[l], W.nz[l], s) <= l2;
    if (!__any_sync(kFull, hit)) continue;
    united = true;
    if (hit) rsd::uf_unite(uf, rq, rj);
    __syncwarp();
    const uint32_t r = rsd::uf_find(uf, rq);
    if (hit) rj = r;
    if (lane == 0) W.root[l] = r;
    if (kSelf && hit) W.root[lane] = r;
    __syncwarp();
  }
  return united;
}

// Links inside every superbucket (bucket pairs b >= a).
template <bool kCount>
__global__ void __launch_bounds__(kT, 4) k_link_near(SearchArgs A, uint32_t* __restrict__ uf) {
  __shared__ WarpShared sh[kWarpsPerBlock];
  const int lane = threadIdx.x & 31;
  WarpShared& W = sh[threadIdx.x >> 5];
  const int64_t nbk = *A.nbuckets;
  Tally T;
  while (true) {
    const int64_t w = next_work(A.counter, lane);
    if (w >= nbk) break;
    const int64_t a = A.order[w];
    const Bucket Aq = A.bk[a];
    const float4 iv = A.inv[Aq.node];
    const float2 s = make_float2(iv.x, iv.y);
    const float l2 = iv.z;
    const bool valid = lane < int(Aq.count);
    const uint32_t si = Aq.start + (valid ? lane : 0);
    const Query Q = make_query(A.XY[si], A.Z[si]);
    const uint32_t rl = rsd::uf_find(uf, si);
    __syncwarp();
    W.nxy[lane] = make_float4(Q.na.x, Q.na.y, Q.nb.x, Q.nb.y);
    W.nz[lane] = Q.nc;
    W.root[lane] = rl;
    __syncwarp();
    const unsigned all = Aq.count == 32 ? kFull : (1u << Aq.count) - 1u;
    link_eval<kCount, true>(A, uf, Aq.start, int(Aq.count), all, s, l2, rl, lane, W, T);
    const int64_t b_lo = int64_t(Aq.first) + ((a - int64_t(Aq.first)) & ~int64_t(31));
    const int64_t b_hi = rsd::min64(b_lo + 32, int64_t(Aq.last) + 1);
    if (a + 1 >= b_hi) continue;
    unsigned mask = stage_boxes<kCount>(A, b_lo, b_hi, A.box[a], l2, s, lane, W, T);
    mask &= ~((2u << int(a - b_lo)) - 1u);
    while (mask) {
      const int i = __ffs(mask) - 1;
      mask &= mask - 1u;
      const unsigned nm = __ballot_sync(kFull, valid && lb_point_box(Q, W.box[i], s) <= l2);
      if (kCount) T.box += valid;
      if (!nm) continue;
      const int64_t b = b_lo + i;
      const int cnt = b == int64_t(Aq.last) ? int(A.bk[b].count) : 32;
      const uint32_t start = uint32_t(int64_t(Aq.start) + 32 * (b - a));
      const uint32_t rj = lane < cnt ? rsd::uf_find(uf, start + lane) : 0u;
      link_eval<kCount, false>(A, uf, start, cnt, nm, s, l2, rj, lane, W, T);
    }
  }
  flush_tally<kCount>(T, A.work + 2, lane);
}

// Full compression, component sizes by root.
__global__ void k_link_compress(const int64_t* __restrict__ na, uint32_t* __restrict__ uf,
                                uint32_t* __restrict__ cnt) {
  const int64_t a = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool valid = a < *na;  // every lane stays: lanes with the same root add once
  const uint32_t r = valid ? rsd::uf_find_ro(uf, uint32_t(a)) : 0xffffffffu;
  if (valid) uf[a] = r;
  const unsigned peers = __match_any_sync(kFull, r);
  if (valid && int(threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(cnt + r, uint32_t(__popc(peers)));
}

// One warp per bucket: the root all its members share (0xffffffff: several), and the node's
// largest component, as (size << 32 | root), from the roots among its members.
__global__ void __launch_bounds__(kT)
k_link_uniform(int64_t nb, const int64_t* __restrict__ nbk, const Bucket* __restrict__ bk,
               const uint32_t* __restrict__ uf, const uint32_t* __restrict__ cnt, uint32_t* __restrict__ uni,
               unsigned long long* __restrict__ big) {
  const int64_t w = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (w >= *nbk) return;
  const Bucket B = bk[w];
  if (B.sbcount == 1) return;  // such nodes have no far search
  const uint32_t r = uf[B.start + (lane < int(B.count) ? lane : 0)];
  int same;
  __match_all_sync(kFull, r, &same);
  if (lane == 0) uni[w] = same ? r : 0xffffffffu;
  if (lane < int(B.count) && r == B.start + lane)
    atomicMax(big + (int64_t(B.node) - nb), ((unsigned long long)cnt[r] << 32) | r);
}

// Links between superbuckets, for the members outside their node's largest component; members that
// have joined it meanwhile are done too (from the near stretches of the curve on, and with the query
// box made again as they go: 69 -> 58 ms on the 2^27 snapshot. The nearest-neighbour search gains
// nothing from that order: its limit is known from the start).
template <bool kCount>
__global__ void __launch_bounds__(kT, 4)
k_link_far(SearchArgs A, const uint32_t* __restrict__ uni, const unsigned long long* __restrict__ big,
           const int64_t* __restrict__ active, uint32_t* __restrict__ uf) {
  __shared__ WarpShared sh[kWarpsPerBlock];
  const int lane = threadIdx.x & 31;
  WarpShared& W = sh[threadIdx.x >> 5];
  const int64_t nbk = *A.nbuckets;
  Tally T;
  while (true) {
    const int64_t w = next_work(A.counter, lane);
    if (w >= nbk) break;
    const int64_t a = A.order[w];
    const Bucket Aq = A.bk[a];
    if (active[int64_t(Aq.node) - A.nb] < 1024) break;  // size-class order: one superbucket from here on
    if (Aq.sbcount == 1) continue;
    const float4 iv = A.inv[Aq.node];
    const float2 s = make_float2(iv.x, iv.y);
    const float l2 = iv.z;
    const bool valid = lane < int(Aq.count);
    const uint32_t si = Aq.start + (valid ? lane : 0);
    const uint32_t rl = rsd::uf_find(uf, si);
    bool open = valid && rl != uint32_t(big[int64_t(Aq.node) - A.nb]);
    if (!__any_sync(kFull, open)) continue;
    const float4 xy = A.XY[si];
    const float2 z = A.Z[si];
    const Query Q = make_query(xy, z);
    __syncwarp();
    W.nxy[lane] = make_float4(Q.na.x, Q.na.y, Q.nb.x, Q.nb.y);
    W.nz[lane] = Q.nc;
    W.root[lane] = rl;
    __syncwarp();
    const float c[6] = {xy.x, xy.z, z.x, xy.y, xy.w, z.y};
    Box QB = query_box(c, open);
    unsigned left = __ballot_sync(kFull, open);
    int boxed = __popc(left);
    const int64_t own = (a - int64_t(Aq.first)) >> 5, nsb = Aq.sbcount;
    const int64_t nchunk = (nsb + 31) >> 5, chunk0 = own >> 5;
    for (int64_t k = 0; k < nchunk && left; ++k) {  // from the query's own stretch of the curve on
      const int64_t s0 = 32 * (chunk0 + k < nchunk ? chunk0 + k : chunk0 + k - nchunk);
      bool near = false;
      if (s0 + lane < nsb && s0 + lane != own) {
        near = lb_box_box(QB, A.sbox[Aq.sbfirst + s0 + lane], s) <= l2;
        if (kCount) T.box += 1;
      }
      unsigned sm = __ballot_sync(kFull, near);
      while (sm && left) {
        const int64_t sb = s0 + next_outward(sm, k == 0 ? int(own & 31) : 0);
        const int64_t b_lo = int64_t(Aq.first) + 32 * sb;
        const int64_t b_hi = rsd::min64(b_lo + 32, int64_t(Aq.last) + 1);
        unsigned mask = stage_boxes<kCount>(A, b_lo, b_hi, QB, l2, s, lane, W, T);
        if (b_lo + lane < b_hi) W.uni[lane] = uni[b_lo + lane];
        __syncwarp();
        bool united = false;
        while (mask) {
          const int i = __ffs(mask) - 1;
          mask &= mask - 1u;
          const bool need = open && W.uni[i] != W.root[lane] && lb_point_box(Q, W.box[i], s) <= l2;
          if (kCount) T.box += open;
          const unsigned nm = __ballot_sync(kFull, need);
          if (!nm) continue;
          const int64_t b = b_lo + i;
          const int cnt = b == int64_t(Aq.last) ? int(A.bk[b].count) : 32;
          const uint32_t start = uint32_t(int64_t(Aq.start) + 32 * (b - a));
          const uint32_t rj = lane < cnt ? rsd::uf_find(uf, start + lane) : 0u;
          united |= link_eval<kCount, false>(A, uf, start, cnt, nm, s, l2, rj, lane, W, T);
        }
        if (united) {  // members that have joined the largest component are done, like its others
          const uint32_t rb = rsd::uf_find(uf, uint32_t(big[int64_t(Aq.node) - A.nb]));
          if (open) open = rsd::uf_find(uf, W.root[lane]) != rb;
          left = __ballot_sync(kFull, open);
          refresh_box(QB, boxed, c, open);
        }
      }
    }
  }
  flush_tally<kCount>(T, A.work + 2, lane);
}

// Components over the compacted members -> level-local member positions: the smallest position of
// each component (the root of the definition), then every member's root.
__global__ void k_link_min(const int64_t* __restrict__ na, const uint32_t* __restrict__ uf,
                           const uint32_t* __restrict__ spA, uint32_t* __restrict__ root,
                           uint32_t* __restrict__ minp) {
  const int64_t a = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool valid = a < *na;
  const uint32_t r = valid ? rsd::uf_find_ro(uf, uint32_t(a)) : 0xffffffffu;
  if (valid) root[a] = r;
  const unsigned peers = __match_any_sync(kFull, r);
  const uint32_t least = __reduce_min_sync(peers, valid ? spA[a] : 0xffffffffu);
  if (valid && int(threadIdx.x & 31) == __ffs(peers) - 1) atomicMin(minp + r, least);
}

__global__ void k_link_roots(const int64_t* __restrict__ na, const uint32_t* __restrict__ root,
                             const uint32_t* __restrict__ spA, const uint32_t* __restrict__ minp,
                             uint32_t* __restrict__ uf) {
  const int64_t a = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (a < *na) uf[spA[a]] = minp[root[a]];
}

int bits_for(uint64_t v) {
  int b = 1;
  while (b < 64 && (v >> b) != 0) ++b;
  return b;
}

SearchArgs search_args(rs_ctx* ctx, int64_t nb, int64_t nn) {
  Hier h = hier_of(ctx);
  SearchArgs A;
  A.nbuckets = static_cast<const int64_t*>(ctx->buf[S_P_BOFF].ptr) + nn;
  A.bk = static_cast<const Bucket*>(ctx->buf[S_P_BUCKET].ptr);
  A.box = static_cast<const Box*>(ctx->buf[S_P_BOX].ptr);
  A.sbox = static_cast<const Box*>(ctx->buf[S_P_SBOX].ptr);
  A.order = static_cast<const uint32_t*>(ctx->buf[S_P_ORDER].ptr);
  A.XY = static_cast<const float4*>(ctx->buf[S_P_XY].ptr);
  A.Z = static_cast<const float2*>(ctx->buf[S_P_Z].ptr);
  A.inv = h.inv;
  A.counter = static_cast<unsigned long long*>(ctx->buf[S_P_QCTR].ptr);
  A.work = static_cast<unsigned long long*>(ctx->buf[S_P_WORK].ptr);
  A.nb = nb;
  return A;
}

// Bucket tables of the level over the members [start[k], start[k] + cnt[k]) of each node k in
// the arrays XY, Z (m entries at most): buckets of 32, boxes, superboxes and the work queue
// ordered by node size class.
int build_buckets(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t m, const int64_t* start, const int64_t* cnt,
                  const float4* XY, const float2* Z, cudaStream_t st) {
  int64_t* boff = scratch_t<int64_t>(ctx, S_P_BOFF, size_t(nn) + 1);
  int64_t* sboff = scratch_t<int64_t>(ctx, S_P_SBOFF, size_t(nn) + 1);
  const int64_t nbk_ub = nn + m / 32 + 1;
  const int64_t nsb_ub = nn + nbk_ub / 32 + 1;
  Bucket* bk = scratch_t<Bucket>(ctx, S_P_BUCKET, size_t(nbk_ub));
  Box* box = scratch_t<Box>(ctx, S_P_BOX, size_t(nbk_ub));
  Box* sbox = scratch_t<Box>(ctx, S_P_SBOX, size_t(nsb_ub));
  uint64_t* qk = scratch_t<uint64_t>(ctx, S_P_QKEY_A, size_t(nbk_ub));
  uint64_t* qk2 = scratch_t<uint64_t>(ctx, S_P_QKEY_B, size_t(nbk_ub));
  uint32_t* qv = scratch_t<uint32_t>(ctx, S_P_QVAL_A, size_t(nbk_ub));
  uint32_t* qv2 = scratch_t<uint32_t>(ctx, S_P_QVAL_B, size_t(nbk_ub));
  uint32_t* qorder = scratch_t<uint32_t>(ctx, S_P_ORDER, size_t(nbk_ub));
  if (!boff || !sboff || !bk || !box || !sbox || !qk || !qk2 || !qv || !qv2 || !qorder) return RS_ERR_OOM;
  k_bucket_counts<<<grid_for(nn, kT), kT, 0, st>>>(nn, cnt, boff, sboff);
  RS_LAUNCHED(ctx, "k_bucket_counts");
  RS_TRY(exclusive_scans(ctx, nn, ScanJobs{{{boff, boff, boff + nn}, {sboff, sboff, sboff + nn}}}, st));
  k_buckets<<<grid_for(nbk_ub * 32, kT), kT, 0, st>>>(nb, nn, nbk_ub, boff, sboff, start, cnt, XY, Z, bk, box, qk,
                                                     qv);
  RS_LAUNCHED(ctx, "k_buckets");
  k_superboxes<<<grid_for(nsb_ub * 32, kT), kT, 0, st>>>(nn, boff, sboff, box, sbox);
  RS_LAUNCHED(ctx, "k_superboxes");
  uint64_t* qk_out;
  uint32_t* qv_out;
  RS_TRY(radix_sort_u64(ctx, nbk_ub, 8, qk, qv, qk2, qv2, &qk_out, &qv_out, st));
  RS_CUDA(ctx, cudaMemcpyAsync(qorder, qv_out, sizeof(uint32_t) * nbk_ub, cudaMemcpyDeviceToDevice, st));
  return RS_OK;
}

// ---- Bounds of l2 for the far searches ----------------------------------------------------------
// The split needs each member's nn2 exactly only near the k-th smallest value (the adaptive l2)
// and, elsewhere, only whether it lies below or above it (the selection and the link pass's member
// filter). hi: the k-th smallest of the near values, each at or above its member's nn2, so hi >= l2
// always. lo: for nodes of at least min_members (4096 by default) members a sample of buckets
// (every S-th of the node, about kSampleBuckets of them) is searched up to hi first, and the
// sample's order statistics below and above rank p s (p = (k + 1/2) / g) give lo and a lower hi;
// smaller nodes keep lo = -inf. A member below lo keeps some value below lo, one in [lo, hi] its
// exact nn2, one above hi some value above hi, so the k-th smallest stored value is the exact l2
// whenever it lies in [lo, hi]; k_bounds_check verifies that per node after the selection and sends
// every node that fails through the search without bounds.
constexpr int64_t kBoundMinDefault = 4096;

// Radix select (4 passes of 8 bits over non-negative float bit patterns) of rank k among the
// sample values of one node, read through `val(t)` for t < n (invalid entries return false).
template <class Val>
__device__ float block_select(Val val, int64_t n, uint32_t k, uint32_t* hist, uint32_t* s_prefix,
                              uint32_t* s_k) {
  if (threadIdx.x == 0) {
    *s_prefix = 0;
    *s_k = k;
  }
  uint32_t mask = 0;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int d = threadIdx.x; d < 256; d += blockDim.x) hist[d] = 0;
    __syncthreads();
    const uint32_t prefix = *s_prefix;
    for (int64_t t = threadIdx.x; t < n; t += blockDim.x) {
      float v;
      if (!val(t, v)) continue;
      const uint32_t bits = __float_as_uint(v);
      if ((bits & mask) == prefix) atomicAdd(&hist[(bits >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t kk = *s_k, cum = 0;
      int d = 0;
      for (; d < 255; ++d) {
        if (cum + hist[d] > kk) break;
        cum += hist[d];
      }
      *s_k = kk - cum;
      *s_prefix = prefix | (uint32_t(d) << shift);
    }
    mask |= 255u << shift;
    __syncthreads();
  }
  return __uint_as_float(*s_prefix);
}

// First bounds of every node of the level: (-inf, k-th smallest near value), which the selection
// left in inv.z.
__global__ void k_first_bounds(int64_t nb, int64_t nn, const float4* __restrict__ inv, float2* __restrict__ bounds) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k < nn) bounds[k] = make_float2(-__int_as_float(0x7f800000), inv[nb + k].z);
}

// One block per node of the level: bounds (lo, hi) from the sample of a node of at least
// min_members members, unchanged otherwise. The sample of a node is every S-th of its buckets;
// its size s and the target rank r = p s with p = (k + 1/2) / g; the bounds are the sample's order
// statistics at r -+ d, d = 6 sqrt(s p (1 - p)) + 8 (twice three binomial standard deviations:
// the sampled buckets are clusters of neighbours).
__global__ void __launch_bounds__(256)
k_sample_bounds(int64_t nb, int64_t nn, const int64_t* __restrict__ node_size, const int64_t* __restrict__ boff,
                const Bucket* __restrict__ bk, const float* __restrict__ nn2,
                int f_num, int f_den, float margin, int64_t min_members, float2* __restrict__ bounds) {
  __shared__ uint32_t hist[256];
  __shared__ uint32_t s_prefix, s_k;
  const int64_t k = blockIdx.x;
  if (k >= nn) return;
  const int64_t g = node_size[nb + k];
  if (g < min_members) return;
  const float inf = __int_as_float(0x7f800000);
  const int64_t b0 = boff[k], nbk = boff[k + 1] - b0;
  const int64_t S = sample_stride(nbk), ns = (nbk + S - 1) / S;
  // sample members: 32 per sampled bucket except possibly the node's last bucket
  const Bucket last = bk[b0 + nbk - 1];
  const bool last_sampled = ((nbk - 1) % S) == 0;
  const int64_t s = ns * 32 - (last_sampled ? 32 - int64_t(last.count) : 0);
  const int64_t kk = (int64_t(f_num) * g + f_den - 1) / f_den - 1;
  const double p = (double(kk) + 0.5) / double(g);
  const double r = p * double(s);
  const double d = double(margin) * (6.0 * sqrt(double(s) * p * (1.0 - p)) + 8.0);
  const int64_t r_lo = int64_t(floor(r - d)), r_hi = int64_t(ceil(r + d));
  if (r_lo > r_hi) {  // empty bounds (margin < 0: the exact fallback under test)
    if (threadIdx.x == 0) bounds[k] = make_float2(inf, -inf);
    return;
  }
  auto val = [&](int64_t t, float& v) -> bool {
    const Bucket B = bk[b0 + (t >> 5) * S];
    const uint32_t l = uint32_t(t & 31);
    if (l >= B.count) return false;
    v = nn2[B.start + l];
    return true;
  };
  const float lo = r_lo <= 0 ? -inf : block_select(val, ns * 32, uint32_t(r_lo), hist, &s_prefix, &s_k);
  __syncthreads();
  const float hi = r_hi >= s - 1 ? inf : block_select(val, ns * 32, uint32_t(r_hi), hist, &s_prefix, &s_k);
  if (threadIdx.x == 0) bounds[k] = make_float2(lo, fminf(hi, bounds[k].y));
}

// After the selection: a bounded node whose l2 lies outside its [lo, hi] failed (its stored
// values are not exact there): mark it and open its bounds for the search again.
// tally (counting variant, may be null): [0] nodes searched with sampled bounds, [1] failed.
__global__ void k_bounds_check(int64_t nb, int64_t nn, const float4* __restrict__ inv,
                               const int64_t* __restrict__ node_size, int64_t min_members,
                               float2* __restrict__ bounds, int* __restrict__ failed,
                               unsigned long long* __restrict__ tally) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k >= nn) return;
  const float inf = __int_as_float(0x7f800000);
  const bool sampled = node_size[nb + k] >= min_members;
  const float2 bd = bounds[k];
  const float l2 = inv[nb + k].z;
  const bool bad = sampled && !(bd.x <= l2 && l2 <= bd.y);
  failed[k] = bad ? 1 : 0;
  if (bad) bounds[k] = make_float2(-inf, inf);
  if (tally && sampled) {
    atomicAdd(tally, 1ull);
    if (bad) atomicAdd(tally + 1, 1ull);
  }
}

unsigned persistent_grid(int64_t nbk_ub) {
  return unsigned(std::min<int64_t>((nbk_ub + kWarpsPerBlock - 1) / kWarpsPerBlock, 152 * 4));
}

// One persistent launch of a search kernel over the level's queue.
template <class K, class... Args>
int run_search(rs_ctx* ctx, const char* name, K counting, K plain, SearchArgs A, int64_t nbk_ub, cudaStream_t st,
               Args... args) {
  RS_CUDA(ctx, cudaMemsetAsync(A.counter, 0, sizeof(unsigned long long), st));
  const unsigned grid = persistent_grid(nbk_ub);
  {
    ProfScope prof_(ctx, name, st);
    (ctx->count_work ? counting : plain)<<<grid, kT, 0, st>>>(A, args...);
  }
  RS_LAUNCHED(ctx, name);
  return RS_OK;
}

// Smallest node of the level's searches with sampled bounds.
int64_t bound_min(rs_ctx* ctx) { return ctx->nn_bound_min > 0 ? ctx->nn_bound_min : kBoundMinDefault; }

int run_far(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t m, FarPass pass, const int* failed, float* nn2,
            cudaStream_t st) {
  const FarArgs F{static_cast<const float2*>(ctx->buf[S_P_BOUNDS].ptr), hier_of(ctx).node_size, failed,
                  bound_min(ctx), pass};
  return run_search(ctx, "k_nn6d_pruned", k_nn_far<true>, k_nn_far<false>, search_args(ctx, nb, nn),
                    nn + m / 32 + 1, st, F, nn2, static_cast<uint32_t*>(ctx->buf[S_P_FRIEND].ptr));
}

}  // namespace

int rs::prune6d_prepare(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t mb, int64_t m,
                        const double* sums, cudaStream_t st) {
  Hier h = hier_of(ctx);
  float4* mean_u = scratch_t<float4>(ctx, S_P_MEANU, size_t(nb + nn));
  float4* mean_v = scratch_t<float4>(ctx, S_P_MEANV, size_t(nb + nn));
  uint64_t* ka = scratch_t<uint64_t>(ctx, S_KEY_A, size_t(m));
  uint64_t* kb = scratch_t<uint64_t>(ctx, S_KEY_B, size_t(m));
  uint32_t* va = scratch_t<uint32_t>(ctx, S_VAL_A, size_t(m));
  uint32_t* vb = scratch_t<uint32_t>(ctx, S_VAL_B, size_t(m));
  float4* XY = scratch_t<float4>(ctx, S_P_XY, size_t(m));
  float2* Z = scratch_t<float2>(ctx, S_P_Z, size_t(m));
  uint32_t* sp = scratch_t<uint32_t>(ctx, S_P_SP, size_t(m));
  int64_t* nstart = scratch_t<int64_t>(ctx, S_P_NSTART, size_t(nn));
  int64_t* ncnt = scratch_t<int64_t>(ctx, S_P_NCNT, size_t(nn));
  unsigned long long* qctr = scratch_t<unsigned long long>(ctx, S_P_QCTR, 2);
  if (!scratch_t<unsigned long long>(ctx, S_P_WORK, 6)) return RS_ERR_OOM;
  if (!mean_u || !mean_v || !ka || !kb || !va || !vb || !XY || !Z || !sp || !nstart || !ncnt || !qctr)
    return RS_ERR_OOM;
  k_node_means<<<grid_for(nn, kT), kT, 0, st>>>(nb, nn, h.node_size, sums, mean_u, mean_v);
  RS_LAUNCHED(ctx, "k_node_means");
  k_hilbert6<<<grid_for(m, kT), kT, 0, st>>>(mb, m, nb, h.mnode, h.U, h.V, h.inv, mean_u, mean_v, ka, va);
  RS_LAUNCHED(ctx, "k_hilbert6");
  uint64_t* keys;
  uint32_t* order;
  RS_TRY(radix_sort_u64(ctx, m, kKeyBits + bits_for(uint64_t(nn)), ka, va, kb, vb, &keys, &order, st));
  k_gather_sorted<<<grid_for(m, kT), kT, 0, st>>>(mb, m, order, h.U, h.V, XY, Z, sp);
  RS_LAUNCHED(ctx, "k_gather_sorted");
  k_node_ranges<<<grid_for(nn, kT), kT, 0, st>>>(nb, nn, mb, h.node_off, h.node_size, nstart, ncnt);
  RS_LAUNCHED(ctx, "k_node_ranges");
  return build_buckets(ctx, nb, nn, m, nstart, ncnt, XY, Z, st);
}

// Nearest neighbours inside the superbuckets -> nn2 [m] in sorted order (each node's members keep
// their range), upper bounds of the exact values.
int rs::prune6d_near(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t mb, int64_t m, float* nn2,
                     cudaStream_t st) {
  (void)mb;
  uint32_t* friend_of = scratch_t<uint32_t>(ctx, S_P_FRIEND, size_t(m));
  if (!friend_of) return RS_ERR_OOM;
  return run_search(ctx, "k_nn6d_pruned", k_nn_near<true>, k_nn_near<false>, search_args(ctx, nb, nn),
                    nn + m / 32 + 1, st, nn2, friend_of);
}

// The far searches, after a selection over the near values (left in inv.z). No host round trip.
int rs::prune6d_far(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t mb, int64_t m, float* nn2,
                    cudaStream_t st) {
  (void)mb;
  Hier h = hier_of(ctx);
  float2* bounds = scratch_t<float2>(ctx, S_P_BOUNDS, size_t(std::max<int64_t>(nn, 1)));
  if (!bounds) return RS_ERR_OOM;
  k_first_bounds<<<grid_for(nn, kT), kT, 0, st>>>(nb, nn, h.inv, bounds);
  RS_LAUNCHED(ctx, "k_first_bounds");
  RS_TRY(run_far(ctx, nb, nn, m, kFarFirst, nullptr, nn2, st));
  const int64_t bmin = bound_min(ctx);
  ctx->nn_bounded_level = m >= bmin;  // a node of bmin members needs that many at the level
  if (!ctx->nn_bounded_level) return RS_OK;
  const int64_t* boff = static_cast<const int64_t*>(ctx->buf[S_P_BOFF].ptr);
  k_sample_bounds<<<unsigned(std::max<int64_t>(nn, 1)), 256, 0, st>>>(
      nb, nn, h.node_size, boff, static_cast<const Bucket*>(ctx->buf[S_P_BUCKET].ptr), nn2, ctx->cfg.f_num,
      ctx->cfg.f_den, ctx->nn_bound_margin, bmin, bounds);
  RS_LAUNCHED(ctx, "k_sample_bounds");
  return run_far(ctx, nb, nn, m, kFarRest, nullptr, nn2, st);
}

// After the selection of l2: nodes whose l2 fell outside their bounds are searched again without
// (*failed_out: int [nn], 1 for those nodes, for the selection to be repeated there).
int rs::prune6d_check(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t m, float* nn2, const int** failed_out,
                      cudaStream_t st) {
  *failed_out = nullptr;
  if (!ctx->nn_bounded_level) return RS_OK;  // no node of the level was sampled
  Hier h = hier_of(ctx);
  float2* bounds = static_cast<float2*>(ctx->buf[S_P_BOUNDS].ptr);
  int* failed = scratch_t<int>(ctx, S_P_FAILED, size_t(std::max<int64_t>(nn, 1)));
  if (!failed) return RS_ERR_OOM;
  unsigned long long* work = static_cast<unsigned long long*>(ctx->buf[S_P_WORK].ptr);
  k_bounds_check<<<grid_for(nn, kT), kT, 0, st>>>(nb, nn, h.inv, h.node_size, bound_min(ctx), bounds, failed,
                                                  ctx->count_work ? work + 4 : nullptr);
  RS_LAUNCHED(ctx, "k_bounds_check");
  RS_TRY(run_far(ctx, nb, nn, m, kFarFailed, failed, nn2, st));
  *failed_out = failed;
  return RS_OK;
}

// Components of the level's links -> uf [m] (level-local positions; a member without friends stays
// its own root).
int rs::prune6d_link(rs_ctx* ctx, int64_t nb, int64_t nn, int64_t mb, int64_t m, const float* nn2,
                     uint32_t* uf, cudaStream_t st) {
  Hier h = hier_of(ctx);
  const float4* XY = static_cast<const float4*>(ctx->buf[S_P_XY].ptr);
  const float2* Z = static_cast<const float2*>(ctx->buf[S_P_Z].ptr);
  const uint32_t* sp = static_cast<const uint32_t*>(ctx->buf[S_P_SP].ptr);
  const uint32_t* friend_of = static_cast<const uint32_t*>(ctx->buf[S_P_FRIEND].ptr);
  const int64_t nbk_ub = nn + m / 32 + 1;
  int64_t* pos = scratch_t<int64_t>(ctx, S_P_APOS, size_t(m) + 1);
  float4* XYA = scratch_t<float4>(ctx, S_P_XYA, size_t(m));
  float2* ZA = scratch_t<float2>(ctx, S_P_ZA, size_t(m));
  uint32_t* spA = scratch_t<uint32_t>(ctx, S_P_SPA, size_t(m));
  uint32_t* ufA = scratch_t<uint32_t>(ctx, S_P_UFA, size_t(m));
  uint32_t* cnt = scratch_t<uint32_t>(ctx, S_P_CNT, size_t(m));
  uint32_t* uni = scratch_t<uint32_t>(ctx, S_P_UNI, size_t(nbk_ub));
  unsigned long long* big = scratch_t<unsigned long long>(ctx, S_P_BIG, size_t(nn));
  int64_t* nstart = scratch_t<int64_t>(ctx, S_P_NSTART, size_t(nn));
  int64_t* ncnt = scratch_t<int64_t>(ctx, S_P_NCNT, size_t(nn));
  if (!pos || !XYA || !ZA || !spA || !ufA || !cnt || !uni || !big || !nstart || !ncnt) return RS_ERR_OOM;
  const unsigned grid = grid_for(m, kT);
  k_active_flags<<<grid, kT, 0, st>>>(m, mb, sp, h.mnode, h.inv, nn2, pos);
  RS_LAUNCHED(ctx, "k_active_flags");
  RS_TRY(exclusive_scan_i64(ctx, m, pos, pos + m, st));
  const int64_t* na = pos + m;
  k_compact_active<<<grid, kT, 0, st>>>(m, pos, XY, Z, sp, XYA, ZA, spA, ufA);
  RS_LAUNCHED(ctx, "k_compact_active");
  k_link_friends<<<grid, kT, 0, st>>>(m, pos, friend_of, ufA);
  RS_LAUNCHED(ctx, "k_link_friends");
  k_active_ranges<<<grid_for(nn, kT), kT, 0, st>>>(nb, nn, mb, h.node_off, h.node_size, pos, nstart, ncnt);
  RS_LAUNCHED(ctx, "k_active_ranges");
  RS_TRY(build_buckets(ctx, nb, nn, m, nstart, ncnt, XYA, ZA, st));
  SearchArgs A = search_args(ctx, nb, nn);
  A.XY = XYA;
  A.Z = ZA;
  RS_TRY(run_search(ctx, "k_link6d_pruned", k_link_near<true>, k_link_near<false>, A, nbk_ub, st, ufA));
  RS_CUDA(ctx, cudaMemsetAsync(cnt, 0, sizeof(uint32_t) * m, st));
  RS_CUDA(ctx, cudaMemsetAsync(big, 0, sizeof(unsigned long long) * nn, st));
  k_link_compress<<<grid, kT, 0, st>>>(na, ufA, cnt);
  RS_LAUNCHED(ctx, "k_link_compress");
  k_link_uniform<<<grid_for(nbk_ub * 32, kT), kT, 0, st>>>(nb, A.nbuckets, A.bk, ufA, cnt, uni, big);
  RS_LAUNCHED(ctx, "k_link_uniform");
  RS_TRY(run_search(ctx, "k_link6d_pruned", k_link_far<true>, k_link_far<false>, A, nbk_ub, st,
                    static_cast<const uint32_t*>(uni), static_cast<const unsigned long long*>(big),
                    static_cast<const int64_t*>(ncnt), ufA));
  // back to member positions: cnt becomes each component's smallest position
  RS_CUDA(ctx, cudaMemsetAsync(cnt, 0xff, sizeof(uint32_t) * m, st));
  uint32_t* root = static_cast<uint32_t*>(ctx->buf[S_P_FRIEND].ptr);  // the neighbours are done with
  k_link_min<<<grid, kT, 0, st>>>(na, ufA, spA, root, cnt);
  RS_LAUNCHED(ctx, "k_link_min");
  k_link_roots<<<grid, kT, 0, st>>>(na, root, spA, cnt, uf);
  RS_LAUNCHED(ctx, "k_link_roots");
  return RS_OK;
}
