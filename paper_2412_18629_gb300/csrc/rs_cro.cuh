// Segmented float64 sums in the canonical reduction order (CRO), used for every FP64 sum of the
// path: node moments (sigma_x, sigma_v of the 6D metric), bulk velocities, the exact FP64
// potential and halo properties.
//
// CRO of a[0..m): chunks of 1024 consecutive terms; inside chunk c lane l (0..31) adds
// a[1024c + l + 32k], k = 0..31, in order starting from 0.0; the 32 lane sums combine by the
// halving tree s[l] += s[l + off], off = 16..1 (an xor butterfly gives lane 0 the same value);
// chunk totals combine by the level-by-level pairwise tree with an odd last element carried up.
// That tree equals "merge equal-height subtrees as chunks arrive, then fold the remaining stack
// right to left", which is how the device evaluates it in O(log m) registers.
#pragma once

#include "rs_common.cuh"

namespace rsd {

// Streaming evaluation of the pairwise tree over chunk totals.
struct CroTree {
  double stk[40];
  int hgt[40];
  int sp = 0;
  __device__ __forceinline__ void push(double v) {
    int h = 0;
    while (sp > 0 && hgt[sp - 1] == h) {
      v = __dadd_rn(stk[sp - 1], v);
      --sp;
      ++h;
    }
    stk[sp] = v;
    hgt[sp] = h;
    ++sp;
  }
  __device__ __forceinline__ double result() const {
    if (sp == 0) return 0.0;
    double v = stk[sp - 1];
    for (int k = sp - 2; k >= 0; --k) v = __dadd_rn(stk[k], v);
    return v;
  }
};

__device__ __forceinline__ int64_t upper_bound_i64(const int64_t* a, int64_t n, int64_t v) {
  int64_t lo = 0, hi = n;
  while (lo < hi) {
    const int64_t mid = lo + ((hi - lo) >> 1);
    if (a[mid] <= v) lo = mid + 1; else hi = mid;
  }
  return lo;
}

// Halving trees of NS sums at once: at every step a pair of sums shares one addition, each half of the
// lanes keeping one of the two (a step of the tree needs half of the lanes only, and a float64 warp
// instruction occupies the pipe for 16 cycles whatever its lanes do): 13 additions for 12 sums instead
// of 60, the same additions in each sum. Returns the lane's sum and its index in `which`.
template <int NS>
__device__ __forceinline__ double warp_cro_combine_all(const double (&acc)[NS], int lane, int& which) {
  double v[NS];
  int id[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) {
    v[s] = acc[s];
    id[s] = s;
  }
  int n = NS;
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    const bool upper = (lane & off) != 0;
#pragma unroll
    for (int i = 0; i < (NS + 1) / 2; ++i) {
      if (2 * i + 1 < n) {
        const double mine = upper ? v[2 * i + 1] : v[2 * i], other = upper ? v[2 * i] : v[2 * i + 1];
        v[i] = __dadd_rn(mine, __shfl_xor_sync(0xffffffffu, other, off));
        id[i] = upper ? id[2 * i + 1] : id[2 * i];
      } else if (2 * i < n) {
        v[i] = __dadd_rn(v[2 * i], __shfl_xor_sync(0xffffffffu, v[2 * i], off));
        id[i] = id[2 * i];
      }
    }
    n = (n + 1) / 2;
  }
  which = id[0];
  return v[0];
}

// One warp per chunk of 1024 terms of one segment. Term::load(p) reads element p (global member
// position), Term::add<first>(q, value, acc) adds its NS terms (first: the lane's first term, added to
// 0.0 by rsd::cro_add<true>). Elements are loaded kCroAhead at a time before they are added in order.
// The totals of a segment of one chunk are its sums. Bound by the float64 pipe (two lanes a clock and
// SM; busy 77% of the cycles for the 12 moments of 2^24 particles' groups): consecutive chunks go to different blocks, so that the chunks of a large node do not queue at
// one SM's pipe (2^18 particles: 312 -> 225 us over eight
// levels; 2^27: 8.3 -> 6.0 ms, properties 16.5 -> 10.6 ms).
// chunk_off has nseg + 1 entries (the last one is the total number of chunks).
constexpr int kCroAhead = 4;
static_assert(32 % kCroAhead == 0, "a chunk of 32 rounds is a whole number of batches");

constexpr int kCroThreads = 128;

template <int NS, class Term>
__global__ void __launch_bounds__(kCroThreads)
k_cro_chunks(int64_t nseg, const int64_t* __restrict__ chunk_off,
             const int64_t* __restrict__ seg_off, const int64_t* __restrict__ seg_size, Term term,
             double* __restrict__ out, double* __restrict__ seg_sums) {
  const int64_t w = int64_t(threadIdx.x >> 5) * gridDim.x + blockIdx.x;
  const int lane = threadIdx.x & 31;
  if (w >= chunk_off[nseg]) return;
  const int64_t q = upper_bound_i64(chunk_off, nseg, w) - 1;
  const int64_t cc = w - chunk_off[q];
  const int64_t base = seg_off[q], g = seg_size[q];
  double acc[NS];
#pragma unroll
  for (int s = 0; s < NS; ++s) acc[s] = 0.0;
  const int64_t i0 = cc * 1024 + lane;
  const int rounds = int((rsd::min64(1024, g - cc * 1024) + 31) / 32);
  for (int k0 = 0; k0 < rounds; k0 += kCroAhead) {
    typename Term::Value v[kCroAhead];
#pragma unroll
    for (int r = 0; r < kCroAhead; ++r)
      if (i0 + 32 * (k0 + r) < g) v[r] = term.load(base + i0 + 32 * (k0 + r));
#pragma unroll
    for (int r = 0; r < kCroAhead; ++r) {
      if (i0 + 32 * (k0 + r) >= g) continue;
      if (r == 0 && k0 == 0)
        term.template add<true>(q, v[r], acc);
      else
        term.template add<false>(q, v[r], acc);
    }
  }
  // (lanes without terms hold 0.0, which leaves a lane sum as it is: none is -0.0)
  int which;
  const double v = warp_cro_combine_all<NS>(acc, lane, which);
  (g <= 1024 ? seg_sums + q * NS : out + w * NS)[which] = v;
}

// Pairwise tree over the first n (1..32) lanes' values, an odd last element carried up: lane 0 ends
// with the root.
__device__ __forceinline__ double warp_pair_tree(double v, int n, int lane) {
#pragma unroll
  for (int off = 1; off < 32; off <<= 1) {
    const double o = __shfl_down_sync(0xffffffffu, v, off);
    if (off < n && (lane & (2 * off - 1)) == 0 && lane + off < n) v = __dadd_rn(v, o);
  }
  return v;
}

// Pairwise tree over the chunk totals of each segment of several chunks -> seg_sums[q][NS] (an empty
// segment's sums are 0.0). A block takes kTreeSegs segments and goes through the large ones among them,
// one warp per sum. 32 aligned totals are a complete subtree (the last group an
// odd-carry tree of its own), so a warp reduces groups of 32, then groups of 32 roots, and so on: the same
// additions as the level-by-level tree. One thread per segment walking all its totals took 17 ms per
// 2^27 pass (1450 totals x 12 sums for the largest node), this form under 3 ms.
constexpr int kTreeSegs = 4;
constexpr int kTreeLevels = 5;  // groups of 32^5 totals: segments of any size

template <int NS>
__global__ void __launch_bounds__(32 * NS)
k_cro_tree(int64_t nseg, const int64_t* __restrict__ chunk_off,
           const double* __restrict__ chunk_sums, double* __restrict__ seg_sums) {
  const int lane = threadIdx.x & 31, s = threadIdx.x >> 5;
  const int64_t mine = int64_t(blockIdx.x) * kTreeSegs + lane;
  const bool in = lane < kTreeSegs && mine < nseg;
  const int64_t my_c0 = in ? chunk_off[mine] : 0, my_nc = in ? chunk_off[mine + 1] - my_c0 : 1;
  if (my_nc == 0) seg_sums[mine * NS + s] = 0.0;
  unsigned large = __ballot_sync(0xffffffffu, my_nc > 1);
  while (large) {
    const int l = __ffs(large) - 1;
    large &= large - 1u;
    const int64_t q = int64_t(blockIdx.x) * kTreeSegs + l;
    const int64_t c0 = __shfl_sync(0xffffffffu, my_c0, l), nc = __shfl_sync(0xffffffffu, my_nc, l);
    double pend[kTreeLevels];  // lane i: i-th pending root of that height
    int n[kTreeLevels];
#pragma unroll
    for (int h = 0; h < kTreeLevels; ++h) {
      pend[h] = 0.0;
      n[h] = 0;
    }
    for (int64_t c = 0; c < nc; c += 32) {
      const int k = int(rsd::min64(32, nc - c));
      double v = warp_pair_tree(lane < k ? chunk_sums[(c0 + c + lane) * NS + s] : 0.0, k, lane);
      bool carry = true;
#pragma unroll
      for (int h = 0; h < kTreeLevels; ++h) {
        if (!carry) continue;
        const double root = __shfl_sync(0xffffffffu, v, 0);
        if (lane == n[h]) pend[h] = root;
        carry = ++n[h] == 32 && h + 1 < kTreeLevels;
        if (carry) {
          v = warp_pair_tree(pend[h], 32, lane);
          n[h] = 0;
        }
      }
    }
    double v = 0.0;
    bool have = false;
#pragma unroll
    for (int h = 0; h < kTreeLevels; ++h) {
      if (have) {  // the partial subtree below is the last root of this height
        const double root = __shfl_sync(0xffffffffu, v, 0);
        if (lane == n[h]) pend[h] = root;
        ++n[h];
      }
      if (n[h] > 0) {
        v = warp_pair_tree(pend[h], n[h], lane);
        have = true;
      }
    }
    if (lane == 0) seg_sums[q * NS + s] = v;
  }
}

}  // namespace rsd

namespace rs {

// Segmented CRO driver: segment q covers global positions [seg_off[q], seg_off[q] + seg_size[q]);
// `total` = sum of the sizes (bounds the chunk count without a host round trip).
// Writes seg_sums[q * NS + s]. Uses the S_CHUNK_OFF / S_CHUNK_SUM scratch slots.
// `also` is an independent scan over the segments (`out` null: none) that shares the launches of the
// chunk offsets' scan: chunk_off[q] = sum over earlier segments of ceil(size / 1024), chunk_off[nseg] =
// total chunks.
template <int NS, class Term>
int cro_segmented(rs_ctx* ctx, int64_t nseg, const int64_t* seg_off, const int64_t* seg_size,
                  int64_t total, Term term, double* seg_sums, cudaStream_t st, ScanJob also = {}) {
  if (nseg <= 0) return RS_OK;
  int64_t* chunk_off = scratch_t<int64_t>(ctx, S_CHUNK_OFF, size_t(nseg) + 1);
  if (!chunk_off) return RS_ERR_OOM;
  RS_TRY(exclusive_scans(ctx, nseg, ScanJobs{{{seg_size, chunk_off, chunk_off + nseg, 10, 0, 0}, also}}, st));
  const int64_t nchunks_ub = nseg + total / 1024 + 1;
  double* chunk_sums = scratch_t<double>(ctx, S_CHUNK_SUM, size_t(nchunks_ub) * NS);
  if (!chunk_sums) return RS_ERR_OOM;
  rsd::k_cro_chunks<NS, Term><<<grid_for(nchunks_ub * 32, rsd::kCroThreads), rsd::kCroThreads, 0, st>>>(
      nseg, chunk_off, seg_off, seg_size, term, chunk_sums, seg_sums);
  RS_LAUNCHED(ctx, "k_cro_chunks");
  rsd::k_cro_tree<NS><<<grid_for(nseg, rsd::kTreeSegs), 32 * NS, 0, st>>>(nseg, chunk_off, chunk_sums, seg_sums);
  RS_LAUNCHED(ctx, "k_cro_tree");
  return RS_OK;
}

}  // namespace rs
