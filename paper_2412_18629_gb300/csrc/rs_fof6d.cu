// Recursive 6D phase-space friends-of-friends inside every 3D FoF group (Section
// "Parallelization": subhalo finding for each FoF halo from 6D phase-space information;
// metric |dx|^2/sigma_x^2 + |dv|^2/sigma_v^2, linked fraction f and recursion from Rockstar).
//
// Level-synchronous: level 0 = FoF groups with >= min members (sorted by (label, id)); each
// level runs, over all of its nodes at once,
//   k_level_members owning node of every member position; u = wrapped offset from the node's
//                   smallest-id member, v, as float4
//   CRO moments     12 float64 sums per node -> inv_sx2, inv_sv2 (k_node_inv)
//   k_nn6d          brute-force nearest-neighbour d6 per member, j-tiles in shared memory
//   k_select_l2     exact k-th smallest nn2 per node (radix select on the float bit patterns)
//   k_link6d        union-find over pairs with d6 <= l2 (upper triangle of each node)
//   k_comp_count    roots and component sizes; k_child_flags marks children; k_children
//   compaction + stable radix sort by child index -> next level's member list (ascending id
//   inside each child because member positions ascend with id)
// Every float32 operation of d6 is rounded separately (no FMA), so the result equals the
// oracle's plain definition bit for bit.
#include "rs_cro.cuh"

namespace {

constexpr int kT = 256;
constexpr int kTile6Bits = 7, kTile6 = 1 << kTile6Bits;

// ---------------------------------------------------------------------------------------------
// Level 0 from FoF labels.

// out[0] = max id, out[1] = max label (~0 in both when any id or label is negative); no particle has
// a deepest node yet.
__global__ void __launch_bounds__(256)
k_max_id(int64_t n, const int64_t* __restrict__ ids, const int64_t* __restrict__ lab,
         unsigned long long* __restrict__ out, int64_t* __restrict__ deepest) {
  __shared__ unsigned long long wmax[2][8];
  unsigned long long mi = 0, ml = 0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t a = ids[i], b = lab[i];
    deepest[i] = -1;
    if (a < 0 || b < 0) {
      mi = ml = ~0ull;
    } else {
      mi = (unsigned long long)a > mi ? (unsigned long long)a : mi;
      ml = (unsigned long long)b > ml ? (unsigned long long)b : ml;
    }
  }
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    const unsigned long long oi = __shfl_xor_sync(0xffffffffu, mi, off);
    const unsigned long long ol = __shfl_xor_sync(0xffffffffu, ml, off);
    mi = oi > mi ? oi : mi;
    ml = ol > ml ? ol : ml;
  }
  if ((threadIdx.x & 31) == 0) {
    wmax[0][threadIdx.x >> 5] = mi;
    wmax[1][threadIdx.x >> 5] = ml;
  }
  __syncthreads();
  if (threadIdx.x == 0) {  // one atomic per block and value
    for (int w = 1; w < int(blockDim.x >> 5); ++w) {
      mi = wmax[0][w] > mi ? wmax[0][w] : mi;
      ml = wmax[1][w] > ml ? wmax[1][w] : ml;
    }
    atomicMax(out, mi);
    atomicMax(out + 1, ml);
  }
}

// Sizes of a level's nodes for the choice of its searches: stat[0] += sum of g^2, stat[1] = max g (one
// atomic each per warp that holds a node; every lane of the warp calls this).
__device__ __forceinline__ void level_stat(unsigned long long* __restrict__ stat, bool node, int64_t g) {
  if (!__any_sync(0xffffffffu, node)) return;
  unsigned long long sq = node ? (unsigned long long)(g * g) : 0ull;
  unsigned mx = node ? unsigned(g) : 0u;
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, off);
  mx = __reduce_max_sync(0xffffffffu, mx);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(stat, sq);
    atomicMax(stat + 1, (unsigned long long)mx);
  }
}

// ---- level 0 over a dense label range (max label < 2 n + 4096): per-label member counts, the
// kept labels' node indices and member offsets from two scans over the label range, then one
// sort of the kept particles only, by (node, id).
// Particles of one large group are all over the input, and additions to one counter queue (about 1 ns
// each). So a block first counts in a table of its own in shared memory: a label takes a free slot, and
// where another label holds the slot the addition goes to its counter (equal neighbours at once). A group
// of a fraction f of the particles gets its slot with a probability near f / (f + 1 / kCountSlots), and
// blocks mix the labels differently. 2^27 particles: 12.1 -> 4.4 ms.
constexpr int kCountThreads = 512, kCountPer = 4, kCountBits = 11, kCountSlots = 1 << kCountBits;

__global__ void __launch_bounds__(kCountThreads)
k_label_count(int64_t n, const int64_t* __restrict__ lab, uint32_t* __restrict__ cnt) {
  constexpr uint32_t kFree = 0xffffffffu;  // labels are below 2^31
  __shared__ uint32_t skey[kCountSlots], scnt[kCountSlots];
  for (int t = threadIdx.x; t < kCountSlots; t += kCountThreads) {
    skey[t] = kFree;
    scnt[t] = 0;
  }
  __syncthreads();
  const uint32_t salt = blockIdx.x * 0x85ebca6bu;
  const int64_t step = int64_t(gridDim.x) * kCountThreads * kCountPer;
  for (int64_t i0 = int64_t(blockIdx.x) * kCountThreads * kCountPer; i0 < n; i0 += step) {
    uint32_t l[kCountPer];
#pragma unroll
    for (int k = 0; k < kCountPer; ++k) {
      const int64_t i = i0 + k * kCountThreads + threadIdx.x;
      l[k] = i < n ? uint32_t(lab[i]) : kFree;
    }
#pragma unroll
    for (int k = 0; k < kCountPer; ++k) {
      bool miss = l[k] != kFree;
      if (miss) {
        const uint32_t slot = ((l[k] ^ salt) * 0x9e3779b1u) >> (32 - kCountBits);
        uint32_t key = skey[slot];
        if (key == kFree) {
          key = atomicCAS(skey + slot, kFree, l[k]);
          if (key == kFree) key = l[k];
        }
        if (key == l[k]) {
          atomicAdd(scnt + slot, 1u);
          miss = false;
        }
      }
      rsd::warp_run_add<uint32_t>(cnt, l[k], miss, 1u);  // every lane
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < kCountSlots; t += kCountThreads)
    if (scnt[t]) atomicAdd(cnt + skey[t], scnt[t]);
}

__global__ void k_label_keep(int64_t nl, const uint32_t* __restrict__ cnt, int min_size,
                             int64_t* __restrict__ knode, int64_t* __restrict__ ksize,
                             unsigned long long* __restrict__ stat) {
  const int64_t l = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool keep = l < nl && cnt[l] >= uint32_t(min_size);
  level_stat(stat, keep, keep ? int64_t(cnt[l]) : 0);
  if (l >= nl) return;
  knode[l] = keep ? 1 : 0;
  ksize[l] = keep ? int64_t(cnt[l]) : 0;
}

__global__ void k_label_nodes(int64_t nl, int64_t nodes, int64_t members, const uint32_t* __restrict__ cnt, int min_size,
                              const int64_t* __restrict__ knode, const int64_t* __restrict__ koff,
                              int64_t* __restrict__ node_off, int64_t* __restrict__ node_size,
                              int64_t* __restrict__ node_parent, int32_t* __restrict__ node_level) {
  const int64_t l = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (l == 0) node_off[nodes] = members;
  if (l >= nl || cnt[l] < uint32_t(min_size)) return;
  const int64_t q = knode[l];
  node_off[q] = koff[l];
  node_size[q] = cnt[l];
  node_parent[q] = -1;
  node_level[q] = 0;
}

// Keys (node << bid | id) of the particles of kept groups, appended with one addition to the counter a
// block (one a warp queued at it: 2^27 particles 6.9 -> 2.1 ms). A kept label is one whose node index the
// scan raised, so both come from the same 32 bytes.
constexpr int kKeysPer = 8;

__global__ void __launch_bounds__(kT)
k_label_keys(int64_t n, const int64_t* __restrict__ ids, const int64_t* __restrict__ lab, int64_t nl,
             int64_t nodes, const int64_t* __restrict__ knode, int bid, unsigned long long* __restrict__ ctr,
             uint64_t* __restrict__ keys, uint32_t* __restrict__ vals) {
  __shared__ unsigned wsum[kT / 32];
  __shared__ unsigned long long sbase;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i0 = int64_t(blockIdx.x) * (kT * kKeysPer) + threadIdx.x;
  int64_t node[kKeysPer];
  unsigned votes[kKeysPer], total = 0;
#pragma unroll
  for (int k = 0; k < kKeysPer; ++k) {
    const int64_t i = i0 + k * kT;
    node[k] = -1;
    if (i < n) {
      const int64_t l = lab[i], q = knode[l];
      if ((l + 1 < nl ? knode[l + 1] : nodes) != q) node[k] = q;
    }
  }
#pragma unroll
  for (int k = 0; k < kKeysPer; ++k) {
    votes[k] = __ballot_sync(0xffffffffu, node[k] >= 0);
    total += __popc(votes[k]);
  }
  if (lane == 0) wsum[warp] = total;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned all = 0;
    for (int w = 0; w < kT / 32; ++w) {
      const unsigned c = wsum[w];
      wsum[w] = all;
      all += c;
    }
    sbase = all ? atomicAdd(ctr, (unsigned long long)all) : 0ull;
  }
  __syncthreads();
  unsigned long long pos = sbase + wsum[warp];
#pragma unroll
  for (int k = 0; k < kKeysPer; ++k) {
    if (node[k] >= 0) {
      const int64_t i = i0 + k * kT;
      const unsigned long long at = pos + __popc(votes[k] & ((1u << lane) - 1u));
      keys[at] = (uint64_t(node[k]) << bid) | uint64_t(ids[i]);
      vals[at] = uint32_t(i);
    }
    pos += __popc(votes[k]);
  }
}

// Sparse labels: all particles ordered by (label, id) with two stable radix sorts, first by id
// (k_id_keys), then by label (k_label_of: the labels of the id-sorted particles).
__global__ void k_id_keys(int64_t n, const int64_t* __restrict__ ids, uint64_t* __restrict__ keys,
                          uint32_t* __restrict__ vals) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  keys[i] = uint64_t(ids[i]);
  vals[i] = uint32_t(i);
}

__global__ void k_label_of(int64_t n, const uint32_t* __restrict__ vals, const int64_t* __restrict__ lab,
                           uint64_t* __restrict__ keys) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (k < n) keys[k] = uint64_t(lab[vals[k]]);
}

// head flag per sorted position (1 where a new label starts); run index comes from a scan.
__global__ void k_run_heads(int64_t n, const uint64_t* __restrict__ keys, int b, int64_t* __restrict__ head) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  head[i] = (i == 0 || (keys[i] >> b) != (keys[i - 1] >> b)) ? 1 : 0;
}

// After the scan: run start positions and, at the end, run sizes; runs with >= min members
// become level-0 nodes.
__global__ void k_run_starts(int64_t n, const uint64_t* __restrict__ keys, int b,
                             const int64_t* __restrict__ run_idx, int64_t* __restrict__ run_start) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (i == 0 || (keys[i] >> b) != (keys[i - 1] >> b)) run_start[run_idx[i]] = i;
}

__global__ void k_run_keep(int64_t nruns, int64_t n, const int64_t* __restrict__ run_start,
                           int min_size, int64_t* __restrict__ keep, int64_t* __restrict__ size,
                           unsigned long long* __restrict__ stat) {
  const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool in = r < nruns;
  const int64_t s = in ? (r + 1 < nruns ? run_start[r + 1] : n) - run_start[r] : 0;
  level_stat(stat, in && s >= min_size, s);
  if (!in) return;
  size[r] = s;
  keep[r] = s >= min_size ? 1 : 0;
}

// Level-0 node table and member list (particle indices), from kept runs.
__global__ void k_level0_nodes(int64_t nruns, int64_t nodes, int64_t members,
                               const int64_t* __restrict__ size, const int64_t* __restrict__ keep,
                               const int64_t* __restrict__ node_of_run /*scan of keep*/,
                               const int64_t* __restrict__ mem_off /*scan of kept sizes*/,
                               int64_t* __restrict__ node_off, int64_t* __restrict__ node_size,
                               int64_t* __restrict__ node_parent, int32_t* __restrict__ node_level) {
  const int64_t r = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (r == 0) node_off[nodes] = members;
  if (r >= nruns || !keep[r]) return;
  const int64_t q = node_of_run[r];
  node_off[q] = mem_off[r];
  node_size[q] = size[r];
  node_parent[q] = -1;
  node_level[q] = 0;
}

// run_heads holds the exclusive scan of the head flags: a run start sees its own run index,
// any later element of run r sees r + 1.
__device__ __forceinline__ int64_t run_of(const uint64_t* keys, int b, const int64_t* run_heads,
                                          int64_t i) {
  const bool head = (i == 0 || (keys[i] >> b) != (keys[i - 1] >> b));
  return run_heads[i] - (head ? 0 : 1);
}

__global__ void k_level0_members(int64_t n, const uint64_t* __restrict__ keys, int b,
                                 const int64_t* __restrict__ run_heads,
                                 const int64_t* __restrict__ run_start, const int64_t* __restrict__ keep,
                                 const int64_t* __restrict__ mem_off, const uint32_t* __restrict__ vals,
                                 uint32_t* __restrict__ mem) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const int64_t r = run_of(keys, b, run_heads, i);
  if (!keep[r]) return;
  mem[mem_off[r] + (i - run_start[r])] = vals[i];
}

__global__ void k_fill_i64(int64_t* __restrict__ a, int64_t v) { *a = v; }

__global__ void k_size_mask(int64_t n, const int64_t* __restrict__ keep, const int64_t* __restrict__ size,
                            int64_t* __restrict__ out) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) out[i] = keep[i] ? size[i] : 0;
}

// ---------------------------------------------------------------------------------------------
// Per-level kernels. Member positions p are global (into the hierarchy's member list);
// level-local position = p - mb.

// U, V of the member at position p, relative to its node's first member r (the smallest id).
__device__ __forceinline__ void member_uv(int64_t p, int64_t i, int64_t r, const float* __restrict__ pos,
                                          const float* __restrict__ vel, float L, float4* __restrict__ U,
                                          float4* __restrict__ V) {
  const float hL = 0.5f * L;
  U[p] = make_float4(rsd::wrap_diff(pos[3 * r], pos[3 * i], L, hL),
                     rsd::wrap_diff(pos[3 * r + 1], pos[3 * i + 1], L, hL),
                     rsd::wrap_diff(pos[3 * r + 2], pos[3 * i + 2], L, hL), 0.f);
  V[p] = make_float4(vel[3 * i], vel[3 * i + 1], vel[3 * i + 2], 0.f);
}

// Start of a level, one thread a member: its node, U and V; itself as its root, no neighbour yet, no
// component member counted. The thread of a node's first member also writes the node's reference
// position and smallest id (members ascend by id). One launch: on a level of a few thousand members a
// launch takes longer than the whole pass.
__global__ void k_level_members(int64_t mb, int64_t me, int64_t nb, int64_t nn,
                                const uint32_t* __restrict__ mem, const int64_t* __restrict__ node_off,
                                const int64_t* __restrict__ ids, const float* __restrict__ pos,
                                const float* __restrict__ vel, float L, uint32_t* __restrict__ mnode,
                                float4* __restrict__ U, float4* __restrict__ V, float4* __restrict__ ref,
                                int64_t* __restrict__ node_minid, uint32_t* __restrict__ uf,
                                float* __restrict__ nn2, uint32_t* __restrict__ cnt,
                                unsigned long long* __restrict__ stat) {
  const int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, p = mb + k;
  if (k < 2) stat[k] = 0;
  if (p >= me) return;
  const int64_t q = nb + rsd::upper_bound_i64(node_off + nb, nn, p) - 1, first = node_off[q];
  const int64_t i = mem[p], r = mem[first];
  mnode[p] = uint32_t(q);
  member_uv(p, i, r, pos, vel, L, U, V);
  uf[k] = uint32_t(k);
  nn2[k] = __int_as_float(0x7f800000);
  cnt[k] = 0;
  if (p == first) {
    ref[q] = make_float4(pos[3 * r], pos[3 * r + 1], pos[3 * r + 2], 0.f);
    node_minid[q] = ids[r];
  }
}

__global__ void k_gather_uv(int64_t mb, int64_t me, const uint32_t* __restrict__ mem,
                            const uint32_t* __restrict__ mnode, const int64_t* __restrict__ node_off,
                            const float* __restrict__ pos, const float* __restrict__ vel, float L,
                            float4* __restrict__ U, float4* __restrict__ V) {
  const int64_t p = mb + int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (p >= me) return;
  member_uv(p, mem[p], mem[node_off[mnode[p]]], pos, vel, L, U, V);
}

__global__ void k_node_ref(int64_t nb, int64_t ne, const uint32_t* __restrict__ mem,
                           const int64_t* __restrict__ node_off, const float* __restrict__ pos,
                           float4* __restrict__ ref) {
  const int64_t q = nb + int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (q >= ne) return;
  const int64_t r = mem[node_off[q]];
  ref[q] = make_float4(pos[3 * r], pos[3 * r + 1], pos[3 * r + 2], 0.f);
}

struct MomentTerm {
  const float4* U;
  const float4* V;
  struct Value {
    float4 u, v;
  };
  __device__ __forceinline__ Value load(int64_t p) const { return {U[p], V[p]}; }
  template <bool kFirst>
  __device__ __forceinline__ void add(int64_t, const Value& t, double* acc) const {
    const float4 u = t.u, v = t.v;
    const double a[3] = {rsd::f2d(u.x), rsd::f2d(u.y), rsd::f2d(u.z)};
    const double b[3] = {rsd::f2d(v.x), rsd::f2d(v.y), rsd::f2d(v.z)};
    const float uc[3] = {u.x, u.y, u.z}, vc[3] = {v.x, v.y, v.z};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
      rsd::cro_add<kFirst>(acc[d], a[d]);
      rsd::cro_add<kFirst>(acc[3 + d], rsd::sq_f2d(uc[d]));  // == a[d] * a[d], exactly
      rsd::cro_add<kFirst>(acc[6 + d], b[d]);
      rsd::cro_add<kFirst>(acc[9 + d], rsd::sq_f2d(vc[d]));
    }
  }
};

// Metric scales of the node's split, and (mean u, sigma_v,1D) in float32 for the surrogate's
// features. Total variance ((Q0/g - m0^2) + (Q1/g - m1^2)) + (Q2/g - m2^2), m_d = S_d / g.
// Sixteen lanes a node, one division each: a thread of its own did the 12 divisions one after the other,
// 9 us however few the nodes.
__global__ void k_node_inv(int64_t nb, int64_t nn, const int64_t* __restrict__ node_size,
                           const double* __restrict__ sums, float4* __restrict__ inv,
                           float4* __restrict__ mom) {
  const int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x, k = t >> 4;
  const int l = int(t & 15);
  const bool in = k < nn && l < 12;  // every lane stays for the shuffles
  const double g = in ? double(node_size[nb + k]) : 1.0;
  const double x = __ddiv_rn(in ? sums[12 * k + l] : 0.0, g);  // m (0-2, 6-8) and Q / g (3-5, 9-11)
  const double y = __shfl_down_sync(0xffffffffu, x, 3, 16);
  const double v0 = __dsub_rn(y, __dmul_rn(x, x));
  const double v1 = __shfl_down_sync(0xffffffffu, v0, 1, 16), v2 = __shfl_down_sync(0xffffffffu, v0, 2, 16);
  const double var = __dadd_rn(__dadd_rn(v0, v1), v2);  // lane 0: of u, lane 6: of v
  const bool whole = in && (l == 0 || l == 6);
  const float scale = whole && var > 0.0 ? __double2float_rn(__ddiv_rn(1.0, var)) : 0.f;
  const float sig = whole ? float(sqrt(fmax(var, 0.0) / 3.0)) : 0.f;
  const float iv = __shfl_sync(0xffffffffu, scale, 6, 16), s1 = __shfl_sync(0xffffffffu, sig, 6, 16);
  const float mx = float(x), my = __shfl_sync(0xffffffffu, mx, 1, 16), mz = __shfl_sync(0xffffffffu, mx, 2, 16);
  if (in && l == 0) {
    inv[nb + k] = make_float4(scale, iv, 0.f, 0.f);
    mom[nb + k] = make_float4(mx, my, mz, s1);
  }
}

__device__ __forceinline__ float d6(float4 ui, float4 vi, float4 uj, float4 vj, float isx, float isv) {
  const float rx = rsd::sq3(__fsub_rn(uj.x, ui.x), __fsub_rn(uj.y, ui.y), __fsub_rn(uj.z, ui.z));
  const float rv = rsd::sq3(__fsub_rn(vj.x, vi.x), __fsub_rn(vj.y, vi.y), __fsub_rn(vj.z, vi.z));
  return __fadd_rn(__fmul_rn(rx, isx), __fmul_rn(rv, isv));
}

// All-pairs kernels: a block per (tile of kTile6 members, chunk of kChunk6 targets) of a node, so that a
// single large node of a small level still spreads over the GPU (one block per tile over all targets
// took as long as the largest node has members). The blocks stride over these items: a node of 2^24 members
// has 2^31 of them, one more than a grid can have blocks.
constexpr int kChunk6Bits = 10, kChunk6 = 1 << kChunk6Bits;
constexpr int64_t kMaxBlocks6 = 1 << 16;

// Nearest-neighbour d6 per member (nn2 starts at +inf): the chunk's j-tiles staged in shared memory;
// the chunks of a member combine by an atomic minimum of the float bits (distances are not negative).
__global__ void __launch_bounds__(kTile6)
k_nn6d(int64_t nb, int64_t nn, const int64_t* __restrict__ item_off, const int64_t* __restrict__ node_off,
       const int64_t* __restrict__ node_size, const float4* __restrict__ inv,
       const float4* __restrict__ U, const float4* __restrict__ V, float* __restrict__ nn2, int64_t mb) {
  __shared__ float4 su[kTile6], sv[kTile6];
  for (int64_t b = blockIdx.x, items = item_off[nn]; b < items; b += gridDim.x) {
    const int64_t k = rsd::upper_bound_i64(item_off, nn, b) - 1;
    const int64_t q = nb + k;
    const int64_t base = node_off[q], g = node_size[q];
    const int64_t chunks = (g + kChunk6 - 1) / kChunk6, t = (b - item_off[k]) / chunks,
                  c = (b - item_off[k]) - t * chunks;
    const float isx = inv[q].x, isv = inv[q].y;
    const int64_t i = t * kTile6 + threadIdx.x, j_end = rsd::min64(g, (c + 1) * kChunk6);
    const bool valid = i < g;
    const float4 ui = valid ? U[base + i] : make_float4(0, 0, 0, 0);
    const float4 vi = valid ? V[base + i] : make_float4(0, 0, 0, 0);
    float best = __int_as_float(0x7f800000);
    for (int64_t j0 = c * kChunk6; j0 < j_end; j0 += kTile6) {
      const int64_t j = j0 + threadIdx.x;
      if (j < j_end) {
        su[threadIdx.x] = U[base + j];
        sv[threadIdx.x] = V[base + j];
      }
      __syncthreads();
      const int jn = int(rsd::min64(kTile6, j_end - j0));
      if (j0 != t * kTile6) {
#pragma unroll 4
        for (int jj = 0; jj < jn; ++jj) best = fminf(best, d6(ui, vi, su[jj], sv[jj], isx, isv));
      } else {  // the members' own tile
        for (int jj = 0; jj < jn; ++jj) {
          if (jj == int(threadIdx.x)) continue;
          best = fminf(best, d6(ui, vi, su[jj], sv[jj], isx, isv));
        }
      }
      __syncthreads();
    }
    if (!valid) continue;
    if (chunks == 1)
      nn2[base + i - mb] = best;
    else
      atomicMin(reinterpret_cast<unsigned int*>(nn2 + (base + i - mb)), __float_as_uint(best));
  }
}

// Exact k-th smallest nn2 of each node, k = ceil(f_num g / f_den) - 1: radix select on the
// (non-negative) float bit patterns. Nodes up to kSelectWarpMax members take one
// warp each (k_select_l2_warp), larger ones a block (k_select_l2): on a level of few nodes the largest
// node's warp is all there is to wait for. 2^18 particles, both kernels: 170 us with the line at 4096
// members, 117 us at 1024; the pass over 2^27 particles takes the same within 0.1%.
constexpr int64_t kSelectWarpMax = 1024;
// Levels of more ordered pairs (sum of g^2) take the pruned searches of the batched form; below, the
// all-pairs kernels cost less than their set-up (about 40 launches; 4e7 pairs are 0.05 ms of work on the
// whole GPU). rs_fof6d with the line at 0 / 1e7 / 4e7 / 1.6e8 pairs: 2^16 particles 2.98 / 1.72 / 1.36 /
// 1.35 ms, 2^18 5.35 / 4.53 / 4.14 / 3.64 ms, 2^20 6.32 / 5.25 / 4.85 / 4.33 ms (groups of up to 1e5 members
// 6.63 / 5.58 / 5.17 / 5.18 ms), 2^22 9.67 / 8.60 / 8.28 / 7.83 ms. The tests of the pruned searches' tallies
// hold it below 4.6e7.
constexpr unsigned long long kPrunedMinPairs = 40000000ull;

// only (if given): int [nn], the nodes to select for (the others keep their l2).
__global__ void __launch_bounds__(kT)
k_select_l2_warp(int64_t nb, int64_t nn, const int64_t* __restrict__ node_off,
                 const int64_t* __restrict__ node_size, const float* __restrict__ nn2, int64_t mb,
                 int f_num, int f_den, float4* __restrict__ inv, const int* __restrict__ only) {
  __shared__ uint32_t hist[kT / 32][256];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t k = int64_t(blockIdx.x) * (kT / 32) + w;
  if (k >= nn) return;
  const int64_t q = nb + k;
  const int64_t base = node_off[q] - mb, g = node_size[q];
  if (g > kSelectWarpMax || (only && !only[k])) return;
  uint32_t kk = uint32_t((int64_t(f_num) * g + f_den - 1) / f_den - 1);
  uint32_t prefix = 0, mask = 0;
  uint32_t* h = hist[w];
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    for (int d = lane; d < 256; d += 32) h[d] = 0;
    __syncwarp();
    for (int64_t a = lane; a < g; a += 32) {
      const uint32_t bits = __float_as_uint(nn2[base + a]);
      if ((bits & mask) == prefix) atomicAdd(&h[(bits >> shift) & 255u], 1u);
    }
    __syncwarp();
    // digit d with cum(d) <= kk < cum(d) + h[d]: lane l owns bins 8l .. 8l + 7
    uint32_t c[8], sum = 0;
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      c[t] = h[8 * lane + t];
      sum += c[t];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, incl, off);
      if (lane >= off) incl += v;
    }
    const uint32_t excl = incl - sum;
    const unsigned owner = __ballot_sync(0xffffffffu, excl <= kk && kk < incl);
    const int L = __ffs(owner) - 1;
    uint32_t d = 0, cum = excl;
    if (lane == L) {
      for (int t = 0; t < 8; ++t) {
        if (cum + c[t] > kk) {
          d = 8 * lane + t;
          break;
        }
        cum += c[t];
      }
    }
    d = __shfl_sync(0xffffffffu, d, L);
    cum = __shfl_sync(0xffffffffu, cum, L);
    kk -= cum;
    prefix |= d << shift;
    mask |= 255u << shift;
    __syncwarp();
  }
  if (lane == 0) inv[q].z = __uint_as_float(prefix);
}

// Blocks of 1024 threads stride over the level's nodes and select in the large ones, 11, 11 and 9 bits a
// pass (31 value bits). Bound by the latency of one block's loads: 256 threads and four
// passes took 20.3 ms per 2^27 pass (33 launches, nodes up to 1.5e6 members), this form 3.1 ms.
// only (if given): int [nn], the nodes to select for (the others keep their l2).
constexpr int kSelThreads = 1024;
constexpr int kSelBits = 11;

__global__ void __launch_bounds__(kSelThreads)
k_select_l2(int64_t nb, int64_t nn, const int64_t* __restrict__ node_off, const int64_t* __restrict__ node_size,
            const float* __restrict__ nn2, int64_t mb, int f_num, int f_den, float4* __restrict__ inv,
            const int* __restrict__ only) {
  __shared__ uint32_t hist[1 << kSelBits];
  __shared__ uint32_t wsum[kSelThreads / 32];
  __shared__ uint32_t s_digit, s_k;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int64_t k = blockIdx.x; k < nn; k += gridDim.x) {
    const int64_t q = nb + k, g = node_size[q];
    if (g <= kSelectWarpMax || (only && !only[k])) continue;
    const float* __restrict__ v = nn2 + (node_off[q] - mb);
    uint32_t rank = uint32_t((int64_t(f_num) * g + f_den - 1) / f_den - 1), prefix = 0, mask = 0;
#pragma unroll
    for (int shift = 31 - kSelBits; shift >= 0; shift = shift == 0 ? -1 : max(shift - kSelBits, 0)) {
      const int bits = shift == 0 ? 31 - 2 * kSelBits : kSelBits;
      hist[2 * threadIdx.x] = 0;
      hist[2 * threadIdx.x + 1] = 0;
      __syncthreads();
#pragma unroll 8
      for (int64_t a = threadIdx.x; a < g; a += kSelThreads) {
        const uint32_t b = __float_as_uint(v[a]);
        if ((b & mask) == prefix) atomicAdd(&hist[(b >> shift) & ((1u << bits) - 1u)], 1u);
      }
      __syncthreads();
      const uint32_t h0 = hist[2 * threadIdx.x], h1 = hist[2 * threadIdx.x + 1];
      uint32_t incl = h0 + h1;
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const uint32_t t = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += t;
      }
      if (lane == 31) wsum[warp] = incl;
      __syncthreads();
      uint32_t before = incl - h0 - h1;
      for (int w = 0; w < warp; ++w) before += wsum[w];
      if (before <= rank && rank < before + h0 + h1) {
        const bool second = rank >= before + h0;
        s_digit = 2 * threadIdx.x + second;
        s_k = rank - before - (second ? h0 : 0u);
      }
      __syncthreads();
      rank = s_k;
      prefix |= s_digit << shift;
      mask |= ((1u << bits) - 1u) << shift;
      __syncthreads();
    }
    if (threadIdx.x == 0) inv[q].z = __uint_as_float(prefix);
  }
}

// Union-find over pairs with d6 <= l2: block = (node, i-tile, chunk of targets), pairs j > i. Targets
// carry the root they had when their tile was staged: those that share the member's root already are
// skipped, so most of the dense middle's links (dozens a member) cost no union. Roots that were equal
// once stay in one component.
constexpr uint32_t kNoRoot = 0xffffffffu;

__global__ void __launch_bounds__(kTile6)
k_link6d(int64_t nb, int64_t nn, const int64_t* __restrict__ item_off, const int64_t* __restrict__ node_off,
         const int64_t* __restrict__ node_size, const float4* __restrict__ inv,
         const float4* __restrict__ U, const float4* __restrict__ V, const float* __restrict__ nn2,
         uint32_t* __restrict__ uf, int64_t mb) {
  __shared__ float4 su[kTile6], sv[kTile6];
  __shared__ uint32_t sroot[kTile6];  // kNoRoot: no friend at all
  for (int64_t b = blockIdx.x, items = item_off[nn]; b < items; b += gridDim.x) {
    const int64_t k = rsd::upper_bound_i64(item_off, nn, b) - 1;
    const int64_t q = nb + k;
    const int64_t base = node_off[q], g = node_size[q];
    const int64_t chunks = (g + kChunk6 - 1) / kChunk6, t = (b - item_off[k]) / chunks,
                  c = (b - item_off[k]) - t * chunks;
    const int64_t j_end = rsd::min64(g, (c + 1) * kChunk6),
                  j_begin = max(c * int64_t(kChunk6), t * int64_t(kTile6));
    if (j_begin >= j_end) continue;  // below the diagonal
    const float4 iv = inv[q];
    const float isx = iv.x, isv = iv.y, l2 = iv.z;
    const int64_t i = t * kTile6 + threadIdx.x;
    const bool valid = i < g;
    const float4 ui = valid ? U[base + i] : make_float4(0, 0, 0, 0);
    const float4 vi = valid ? V[base + i] : make_float4(0, 0, 0, 0);
    const bool active = valid && nn2[base + i - mb] <= l2;  // others have no friend at all
    uint32_t root = active ? rsd::uf_find(uf, uint32_t(base + i - mb)) : kNoRoot;
    for (int64_t j0 = j_begin; j0 < j_end; j0 += kTile6) {
      const int64_t j = j0 + threadIdx.x;
      if (j < j_end) {
        su[threadIdx.x] = U[base + j];
        sv[threadIdx.x] = V[base + j];
        sroot[threadIdx.x] = nn2[base + j - mb] <= l2 ? rsd::uf_find(uf, uint32_t(base + j - mb)) : kNoRoot;
      }
      __syncthreads();
      const int jn = int(rsd::min64(kTile6, j_end - j0));
      const int first = j0 == t * kTile6 ? int(threadIdx.x) + 1 : 0;  // its own tile: j > i
      for (int jb = 0; jb < jn; jb += 32) {
        unsigned hits = 0;
        if (active) {
          for (int jj = max(jb, first); jj < min(jb + 32, jn); ++jj) {
            const uint32_t rj = sroot[jj];
            if (rj != root && rj != kNoRoot && d6(ui, vi, su[jj], sv[jj], isx, isv) <= l2) hits |= 1u << (jj - jb);
          }
        }
        while (__any_sync(0xffffffffu, hits)) {  // one union a lane and round, the lanes side by side
          if (hits) {
            const uint32_t rj = sroot[jb + __ffs(hits) - 1];
            hits &= hits - 1u;
            if (rj != root) {
              rsd::uf_unite(uf, root, rj);
              root = rsd::uf_find(uf, root);
            }
          }
        }
      }
      __syncthreads();
    }
  }
}

// Roots (full compression) and component sizes.
__global__ void k_comp_count(int64_t m, uint32_t* __restrict__ uf, uint32_t* __restrict__ cnt) {
  const int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool valid = p < m;  // every lane stays: lanes with the same root add once
  const uint32_t r = valid ? rsd::uf_find_ro(uf, uint32_t(p)) : 0xffffffffu;
  if (valid) uf[p] = r;
  const unsigned peers = __match_any_sync(0xffffffffu, r);
  if (valid && (threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(cnt + r, uint32_t(__popc(peers)));
}

// Does the component of root r (c members) of node q go on as a child?
__device__ __forceinline__ bool is_child(int64_t c, int min_size, int64_t g) { return c >= min_size && c < g; }

// Per member: cidx = 1 at each root that forms a child, mpos = 1 for the members of children (the two
// are scanned into child indices and member positions). A member that goes on into no child has its
// deepest node here: node and position are written once.
__global__ void k_child_flags(int64_t m, int64_t mb, const uint32_t* __restrict__ uf,
                              const uint32_t* __restrict__ cnt, const uint32_t* __restrict__ mem,
                              const uint32_t* __restrict__ mnode, const int64_t* __restrict__ node_size,
                              int min_size, int64_t* __restrict__ cidx, int64_t* __restrict__ mpos,
                              int64_t* __restrict__ deepest, uint32_t* __restrict__ deepest_pos,
                              unsigned long long* __restrict__ stat) {
  const int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  int64_t c = 0;
  bool child = false, root = false;
  if (p < m) {
    const uint32_t r = uf[p], q = mnode[mb + p];
    c = cnt[r];
    child = is_child(c, min_size, node_size[q]);
    root = child && r == uint32_t(p);
    cidx[p] = root ? 1 : 0;
    mpos[p] = child ? 1 : 0;
    if (!child) {
      const uint32_t i = mem[mb + p];
      deepest[i] = q;
      deepest_pos[i] = uint32_t(mb + p);
    }
  }
  level_stat(stat, root, c);
}

// (child index, particle index) of the children's members in compacted order, and the children's node
// table entries (global node index ne + child index) from their roots.
__global__ void k_children(int64_t m, int64_t mb, int64_t ne, const uint32_t* __restrict__ uf,
                           const uint32_t* __restrict__ cnt, const int64_t* __restrict__ cidx,
                           const int64_t* __restrict__ mpos, const uint32_t* __restrict__ mem,
                           const uint32_t* __restrict__ mnode, int min_size, uint64_t* __restrict__ keys,
                           uint32_t* __restrict__ vals, int64_t* node_size,
                           int64_t* __restrict__ node_parent, int32_t* node_level) {
  const int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (p >= m) return;
  const uint32_t r = uf[p], q = mnode[mb + p];
  const int64_t c = cnt[r];
  if (!is_child(c, min_size, node_size[q])) return;
  const int64_t ci = cidx[r], at = mpos[p];
  keys[at] = uint64_t(ci);
  vals[at] = mem[mb + p];
  if (r != uint32_t(p)) return;
  node_size[ne + ci] = c;
  node_parent[ne + ci] = q;
  node_level[ne + ci] = node_level[q] + 1;
}

// Grow a persistent hierarchy buffer, keeping its first `used` bytes.
int grow_keep(rs_ctx* ctx, int slot, size_t used, size_t need, cudaStream_t st) {
  rs::Buffer& b = ctx->buf[slot];
  if (b.bytes >= need) return RS_OK;
  size_t want = std::max(need, b.bytes * 3 / 2);
  want = (want + 255) & ~size_t(255);
  void* p = nullptr;
  if (cudaMalloc(&p, want) != cudaSuccess) {
    cudaGetLastError();
    return rs::set_error(ctx, RS_ERR_OOM, "cudaMalloc of %zu bytes failed (slot %d)", want, slot);
  }
  if (used && b.ptr) RS_CUDA(ctx, cudaMemcpyAsync(p, b.ptr, used, cudaMemcpyDeviceToDevice, st));
  RS_CUDA(ctx, cudaStreamSynchronize(st));
  if (b.ptr) cudaFree(b.ptr);
  b.ptr = p;
  b.bytes = want;
  return RS_OK;
}

int bits_for(uint64_t v) {
  int b = 1;
  while (b < 64 && (v >> b) != 0) ++b;
  return b;
}

}  // namespace

namespace rs {

Hier hier_of(rs_ctx* ctx) {
  Hier h;
  h.mem = static_cast<uint32_t*>(ctx->buf[S_H_MEM].ptr);
  h.mnode = static_cast<uint32_t*>(ctx->buf[S_H_MNODE].ptr);
  h.U = static_cast<float4*>(ctx->buf[S_H_U].ptr);
  h.V = static_cast<float4*>(ctx->buf[S_H_V].ptr);
  h.node_off = static_cast<int64_t*>(ctx->buf[S_H_NODE_OFF].ptr);
  h.node_size = static_cast<int64_t*>(ctx->buf[S_H_NODE_SIZE].ptr);
  h.node_parent = static_cast<int64_t*>(ctx->buf[S_H_NODE_PARENT].ptr);
  h.node_level = static_cast<int32_t*>(ctx->buf[S_H_NODE_LEVEL].ptr);
  h.node_minid = static_cast<int64_t*>(ctx->buf[S_H_NODE_MINID].ptr);
  h.inv = static_cast<float4*>(ctx->buf[S_H_NODE_INV].ptr);
  h.mom = static_cast<float4*>(ctx->buf[S_H_NODE_MOM].ptr);
  h.ref = static_cast<float4*>(ctx->buf[S_H_NODE_REF].ptr);
  h.deepest = static_cast<int64_t*>(ctx->buf[S_H_DEEPEST].ptr);
  h.deepest_pos = static_cast<uint32_t*>(ctx->buf[S_H_DEEPPOS].ptr);
  return h;
}

// Batched form: exactly pruned nearest-neighbour and link searches (rs_prune6d.cu).
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

// Gather U, V (and node reference positions) for member positions [mb, me) and nodes [nb, ne).
int gather_members(rs_ctx* ctx, int64_t mb, int64_t me, int64_t nb, int64_t ne, const float* pos,
                   const float* vel, cudaStream_t st);

}  // namespace rs

using namespace rs;

int rs::gather_members(rs_ctx* ctx, int64_t mb, int64_t me, int64_t nb, int64_t ne,
                       const float* pos, const float* vel, cudaStream_t st) {
  Hier h = hier_of(ctx);
  if (me > mb) {
    k_gather_uv<<<grid_for(me - mb, kT), kT, 0, st>>>(mb, me, h.mem, h.mnode, h.node_off, pos, vel,
                                                     ctx->cfg.box_L, h.U, h.V);
    RS_LAUNCHED(ctx, "k_gather_uv");
  }
  if (ne > nb) {
    k_node_ref<<<grid_for(ne - nb, kT), kT, 0, st>>>(nb, ne, h.mem, h.node_off, pos, h.ref);
    RS_LAUNCHED(ctx, "k_node_ref");
  }
  return RS_OK;
}

static int ensure_nodes(rs_ctx* ctx, int64_t used, int64_t need, cudaStream_t st) {
  RS_TRY(grow_keep(ctx, S_H_NODE_OFF, size_t(used + 1) * 8, size_t(need + 1) * 8, st));
  RS_TRY(grow_keep(ctx, S_H_NODE_SIZE, size_t(used) * 8, size_t(need) * 8, st));
  RS_TRY(grow_keep(ctx, S_H_NODE_PARENT, size_t(used) * 8, size_t(need) * 8, st));
  RS_TRY(grow_keep(ctx, S_H_NODE_LEVEL, size_t(used) * 4, size_t(need) * 4, st));
  RS_TRY(grow_keep(ctx, S_H_NODE_MINID, size_t(used) * 8, size_t(need) * 8, st));
  RS_TRY(grow_keep(ctx, S_H_NODE_INV, size_t(used) * 16, size_t(need) * 16, st));
  RS_TRY(grow_keep(ctx, S_H_NODE_MOM, size_t(used) * 16, size_t(need) * 16, st));
  RS_TRY(grow_keep(ctx, S_H_NODE_REF, size_t(used) * 16, size_t(need) * 16, st));
  return RS_OK;
}

static int ensure_members(rs_ctx* ctx, int64_t used, int64_t need, cudaStream_t st) {
  RS_TRY(grow_keep(ctx, S_H_MEM, size_t(used) * 4, size_t(need) * 4, st));
  RS_TRY(grow_keep(ctx, S_H_MNODE, size_t(used) * 4, size_t(need) * 4, st));
  RS_TRY(grow_keep(ctx, S_H_U, size_t(used) * 16, size_t(need) * 16, st));
  RS_TRY(grow_keep(ctx, S_H_V, size_t(used) * 16, size_t(need) * 16, st));
  return RS_OK;
}

extern "C" int rs_fof6d(rs_ctx* ctx, int64_t n, const float* pos, const float* vel,
                        const int64_t* ids, const int64_t* fof_label, int64_t* n_nodes_out,
                        int64_t* n_members_out, void* stream) {
  if (!ctx) return RS_ERR_INVALID_ARG;
  ctx->err[0] = 0;
  ctx->have_hier = false;
  ctx->have_unbind = false;
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  if (n < 0 || n >= (int64_t(1) << 32) - 1)
    return set_error(ctx, RS_ERR_INVALID_ARG, "n = %lld out of range", (long long)n);
  if (n > 0 && (!pos || !vel || !ids || !fof_label))
    return set_error(ctx, RS_ERR_INVALID_ARG, "null device pointer");
  RS_CUDA(ctx, cudaSetDevice(ctx->device));
  const int min_size = ctx->cfg.min_halo_particles;
  const float L = ctx->cfg.box_L;
  // ---------------- level 0 from the FoF labels
  int64_t* deep = scratch_t<int64_t>(ctx, S_H_DEEPEST, size_t(std::max<int64_t>(n, 1)));
  uint32_t* deep_pos = scratch_t<uint32_t>(ctx, S_H_DEEPPOS, size_t(std::max<int64_t>(n, 1)));
  if (!deep) return RS_ERR_OOM;
  int64_t nodes = 0, members = 0;
  uint64_t level_pairs = 0;  // sum of g^2 over the level's nodes
  int64_t level_max = 0;     // its largest node
  if (n == 0) {
    RS_TRY(ensure_nodes(ctx, 0, 1, st));
    RS_TRY(ensure_members(ctx, 0, 1, st));
  } else {
    if (!deep_pos) return RS_ERR_OOM;
    unsigned long long* mx = scratch_t<unsigned long long>(ctx, S_COUNTER, 16);
    if (!mx) return RS_ERR_OOM;
    // sum of g^2 and largest node of the level being built, then its nodes and members
    unsigned long long* stat = mx + 4;
    int64_t* totals = reinterpret_cast<int64_t*>(stat + 2);
    RS_CUDA(ctx, cudaMemsetAsync(mx, 0, 128, st));
    k_max_id<<<std::min(grid_for(n, kT), 152u * 8u), kT, 0, st>>>(n, ids, fof_label, mx, deep);
    RS_LAUNCHED(ctx, "k_max_id");
    RS_TRY(read_back(ctx, mx, 16, st));
    const uint64_t max_id = uint64_t(ctx->host_box[0]), max_lab = uint64_t(ctx->host_box[1]);
    if (max_id == ~0ull) return set_error(ctx, RS_ERR_INVALID_ARG, "negative id or label");
    // dense label range: (node << bid | id) keys of the kept particles; otherwise two sorts
    const int bid = bits_for(max_id);
    if (max_lab < std::min<uint64_t>(uint64_t(2 * n + 4096), uint64_t(1) << 31) &&
        bits_for(max_lab + 1) + bid <= 64) {
      // dense label range: count per label, keep, scan, sort the kept particles only
      const int64_t nl = int64_t(max_lab) + 1;
      uint32_t* cntl = scratch_t<uint32_t>(ctx, S_ROOT_CNT, size_t(nl));
      int64_t* knode = scratch_t<int64_t>(ctx, S_GKEY_A, size_t(nl) + 1);
      int64_t* koff = scratch_t<int64_t>(ctx, S_GKEY_B, size_t(nl) + 1);
      if (!cntl || !knode || !koff) return RS_ERR_OOM;
      RS_CUDA(ctx, cudaMemsetAsync(cntl, 0, sizeof(uint32_t) * nl, st));
      k_label_count<<<std::min(grid_for(n, kCountThreads * kCountPer), 152u * 4u), kCountThreads, 0, st>>>(n, fof_label, cntl);
      RS_LAUNCHED(ctx, "k_label_count");
      k_label_keep<<<grid_for(nl, kT), kT, 0, st>>>(nl, cntl, min_size, knode, koff, stat);
      RS_LAUNCHED(ctx, "k_label_keep");
      RS_TRY(exclusive_scans(ctx, nl, ScanJobs{{{knode, knode, totals}, {koff, koff, totals + 1}}}, st));
      RS_TRY(read_back(ctx, stat, 32, st));
      level_pairs = uint64_t(ctx->host_box[0]);
      level_max = ctx->host_box[1];
      nodes = ctx->host_box[2];
      members = ctx->host_box[3];
      RS_TRY(ensure_nodes(ctx, 0, std::max<int64_t>(nodes, 1) * 2, st));
      RS_TRY(ensure_members(ctx, 0, std::max<int64_t>(members, 1) * 2, st));
      Hier h = hier_of(ctx);
      if (members > 0) {
        uint64_t* ka = scratch_t<uint64_t>(ctx, S_KEY_A, size_t(members));
        uint64_t* kb = scratch_t<uint64_t>(ctx, S_KEY_B, size_t(members));
        uint32_t* va = scratch_t<uint32_t>(ctx, S_VAL_A, size_t(members));
        uint32_t* vb = scratch_t<uint32_t>(ctx, S_VAL_B, size_t(members));
        if (!ka || !kb || !va || !vb) return RS_ERR_OOM;
        k_label_nodes<<<grid_for(nl, kT), kT, 0, st>>>(nl, nodes, members, cntl, min_size, knode, koff, h.node_off,
                                                      h.node_size, h.node_parent, h.node_level);
        RS_LAUNCHED(ctx, "k_label_nodes");
        const int bits = bits_for(uint64_t(std::max<int64_t>(nodes - 1, 1))) + bid;
        (sort_ends_in_b(members, bits) ? vb : va) = h.mem;
        k_label_keys<<<grid_for(n, kT * kKeysPer), kT, 0, st>>>(n, ids, fof_label, nl, nodes, knode, bid, mx + 8, ka, va);
        RS_LAUNCHED(ctx, "k_label_keys");
        uint64_t* keys;
        uint32_t* vals;
        RS_TRY(radix_sort_u64(ctx, members, bits, ka, va, kb, vb, &keys, &vals, st));  // vals == h.mem
      }
    } else {
      uint64_t* ka = scratch_t<uint64_t>(ctx, S_KEY_A, n);
      uint64_t* kb = scratch_t<uint64_t>(ctx, S_KEY_B, n);
      uint32_t* va = scratch_t<uint32_t>(ctx, S_VAL_A, n);
      uint32_t* vb = scratch_t<uint32_t>(ctx, S_VAL_B, n);
      int64_t* head = scratch_t<int64_t>(ctx, S_GKEY_A, size_t(n) + 1);
      int64_t* run_start = scratch_t<int64_t>(ctx, S_GKEY_B, size_t(n) + 1);
      int64_t* rsize = scratch_t<int64_t>(ctx, S_GVAL_A, size_t(n) * 2 + 2);
      int64_t* keep = scratch_t<int64_t>(ctx, S_GVAL_B, size_t(n) * 2 + 2);
      if (!ka || !kb || !va || !vb || !head || !run_start || !rsize || !keep) return RS_ERR_OOM;
      int64_t* node_of_run = rsize + n + 1;
      int64_t* mem_off = keep + n + 1;
      k_id_keys<<<grid_for(n, kT), kT, 0, st>>>(n, ids, ka, va);
      RS_LAUNCHED(ctx, "k_id_keys");
      uint64_t* keys;
      uint32_t* vals;
      RS_TRY(radix_sort_u64(ctx, n, bid, ka, va, kb, vb, &keys, &vals, st));
      {
        uint64_t* lk = keys == ka ? kb : ka;  // labels of the id-sorted particles
        uint32_t* lv = vals == va ? vb : va;
        k_label_of<<<grid_for(n, kT), kT, 0, st>>>(n, vals, fof_label, lk);
        RS_LAUNCHED(ctx, "k_label_of");
        RS_TRY(radix_sort_u64(ctx, n, bits_for(max_lab), lk, vals, keys, lv, &keys, &vals, st));
      }
      const int b = 0;  // keys are the labels themselves
      k_run_heads<<<grid_for(n, kT), kT, 0, st>>>(n, keys, b, head);
      RS_LAUNCHED(ctx, "k_run_heads");
      RS_TRY(exclusive_scan_i64(ctx, n, head, head + n, st));
      RS_TRY(read_back(ctx, head + n, 8, st));
      const int64_t nruns = ctx->host_box[0];
      k_run_starts<<<grid_for(n, kT), kT, 0, st>>>(n, keys, b, head, run_start);
      RS_LAUNCHED(ctx, "k_run_starts");
      k_run_keep<<<grid_for(nruns, kT), kT, 0, st>>>(nruns, n, run_start, min_size, keep, rsize, stat);
      RS_LAUNCHED(ctx, "k_run_keep");
      k_size_mask<<<grid_for(nruns, kT), kT, 0, st>>>(nruns, keep, rsize, mem_off);
      RS_LAUNCHED(ctx, "k_size_mask");
      RS_TRY(exclusive_scans(ctx, nruns, ScanJobs{{{keep, node_of_run, totals}, {mem_off, mem_off, totals + 1}}}, st));
      RS_TRY(read_back(ctx, stat, 32, st));
      level_pairs = uint64_t(ctx->host_box[0]);
      level_max = ctx->host_box[1];
      nodes = ctx->host_box[2];
      members = ctx->host_box[3];
      RS_TRY(ensure_nodes(ctx, 0, std::max<int64_t>(nodes, 1) * 2, st));
      RS_TRY(ensure_members(ctx, 0, std::max<int64_t>(members, 1) * 2, st));
      Hier h = hier_of(ctx);
      if (nruns > 0) {
        k_level0_nodes<<<grid_for(nruns, kT), kT, 0, st>>>(nruns, nodes, members, rsize, keep, node_of_run,
                                                         mem_off, h.node_off, h.node_size, h.node_parent,
                                                         h.node_level);
        RS_LAUNCHED(ctx, "k_level0_nodes");
        k_level0_members<<<grid_for(n, kT), kT, 0, st>>>(n, keys, b, head, run_start, keep, mem_off,
                                                         vals, h.mem);
        RS_LAUNCHED(ctx, "k_level0_members");
      }
    }
  }
  if (members == 0) {
    k_fill_i64<<<1, 1, 0, st>>>(hier_of(ctx).node_off, 0);
    RS_LAUNCHED(ctx, "k_fill_i64");
  }
  // ---------------- levels
  int64_t nb = 0, ne = nodes, mb = 0, me = members;
  int32_t levels = 0;
  const int f_num = ctx->cfg.f_num, f_den = ctx->cfg.f_den;
  while (ne > nb) {
    const int64_t nn = ne - nb, m = me - mb;
    Hier h = hier_of(ctx);
    double* sums = scratch_t<double>(ctx, S_NODE_TMP, size_t(nn) * 12);
    int64_t* item_off = scratch_t<int64_t>(ctx, S_SELECT, size_t(nn) + 1);
    float* nn2 = scratch_t<float>(ctx, S_NN2, size_t(m));
    uint32_t* uf = scratch_t<uint32_t>(ctx, S_UF, size_t(m));
    uint32_t* cnt = scratch_t<uint32_t>(ctx, S_ROOT_CNT, size_t(m));
    int64_t* cidx = scratch_t<int64_t>(ctx, S_CHILD_IDX, size_t(m));
    int64_t* mpos = scratch_t<int64_t>(ctx, S_GKEY_A, size_t(m));
    // of the children: sum of g^2, largest g, number, members
    unsigned long long* stat = scratch_t<unsigned long long>(ctx, S_COUNTER, 16);
    if (!sums || !item_off || !nn2 || !uf || !cnt || !cidx || !mpos || !stat) return RS_ERR_OOM;
    stat += 4;
    int64_t* totals = reinterpret_cast<int64_t*>(stat + 2);
    k_level_members<<<grid_for(m, kT), kT, 0, st>>>(mb, me, nb, nn, h.mem, h.node_off, ids, pos, vel, L, h.mnode,
                                                   h.U, h.V, h.ref, h.node_minid, uf, nn2, cnt, stat);
    RS_LAUNCHED(ctx, "k_level_members");
    // batched form: pruned searches, except on levels of few pairs (unless a smallest node for the
    // bounded searches was asked for and the level has one)
    const bool batched = ctx->cfg.batched != 0 && (level_pairs > kPrunedMinPairs ||
                                                   (ctx->nn_bound_min > 0 && level_max >= ctx->nn_bound_min));
    // all pairs: ceil(g / kTile6) ceil(g / kChunk6) items a node, at most (g / 128 + 1) (g / 1024 + 1)
    const ScanJob items = batched ? ScanJob{}
                                  : ScanJob{h.node_size + nb, item_off, item_off + nn, kTile6Bits, kChunk6Bits, 0};
    const int64_t items_ub = int64_t(level_pairs / (uint64_t(kTile6) * kChunk6)) + m / kTile6 + m / kChunk6 + nn + 1;
    const unsigned blocks6 = unsigned(rsd::min64(items_ub, kMaxBlocks6));
    RS_TRY((cro_segmented<12, MomentTerm>(ctx, nn, h.node_off + nb, h.node_size + nb, m,
                                          MomentTerm{h.U, h.V}, sums, st, items)));
    k_node_inv<<<grid_for(nn * 16, kT), kT, 0, st>>>(nb, nn, h.node_size, sums, h.inv, h.mom);
    RS_LAUNCHED(ctx, "k_node_inv");
    // k-th smallest nn2 of the level's nodes (of those with only[k] != 0 when `only` is given); the
    // batched form's nn2 is in its sorted order, in which every node keeps its range
    auto select = [&](const int* only) -> int {
      Hier hs = hier_of(ctx);
      ProfScope prof_(ctx, "k_select_l2", st);
      k_select_l2_warp<<<grid_for(nn, kT / 32), kT, 0, st>>>(nb, nn, hs.node_off, hs.node_size, nn2, mb, f_num,
                                                            f_den, hs.inv, only);
      RS_LAUNCHED(ctx, "k_select_l2_warp");
      if (level_max > kSelectWarpMax) {
        k_select_l2<<<unsigned(std::min<int64_t>(nn, 152 * 2)), kSelThreads, 0, st>>>(
            nb, nn, hs.node_off, hs.node_size, nn2, mb, f_num, f_den, hs.inv, only);
        RS_LAUNCHED(ctx, "k_select_l2");
      }
      return RS_OK;
    };
    if (batched) {
      RS_TRY(prune6d_prepare(ctx, nb, nn, mb, m, sums, st));
      RS_TRY(prune6d_near(ctx, nb, nn, mb, m, nn2, st));
      RS_TRY(select(nullptr));  // of the near values: bounds the far searches
      RS_TRY(prune6d_far(ctx, nb, nn, mb, m, nn2, st));
      h = hier_of(ctx);
    } else {
      {
        ProfScope prof_(ctx, "k_nn6d", st);
        k_nn6d<<<blocks6, kTile6, 0, st>>>(nb, nn, item_off, h.node_off, h.node_size, h.inv,
                                                        h.U, h.V, nn2, mb);
      }
      RS_LAUNCHED(ctx, "k_nn6d");
    }
    RS_TRY(select(nullptr));
    if (batched) {  // bounded searches: nodes whose l2 fell outside their bounds, exactly again
      const int* failed = nullptr;
      RS_TRY(prune6d_check(ctx, nb, nn, m, nn2, &failed, st));
      if (failed) RS_TRY(select(failed));
      h = hier_of(ctx);
    }
    if (batched) {
      RS_TRY(prune6d_link(ctx, nb, nn, mb, m, nn2, uf, st));
    } else {
      {
        ProfScope prof_(ctx, "k_link6d", st);
        k_link6d<<<blocks6, kTile6, 0, st>>>(nb, nn, item_off, h.node_off, h.node_size,
                                                          h.inv, h.U, h.V, nn2, uf, mb);
      }
      RS_LAUNCHED(ctx, "k_link6d");
    }
    k_comp_count<<<grid_for(m, kT), kT, 0, st>>>(m, uf, cnt);
    RS_LAUNCHED(ctx, "k_comp_count");
    k_child_flags<<<grid_for(m, kT), kT, 0, st>>>(m, mb, uf, cnt, h.mem, h.mnode, h.node_size, min_size, cidx,
                                                 mpos, deep, deep_pos, stat);
    RS_LAUNCHED(ctx, "k_child_flags");
    RS_TRY(exclusive_scans(ctx, m, ScanJobs{{{cidx, cidx, totals}, {mpos, mpos, totals + 1}}}, st));
    RS_TRY(read_back(ctx, stat, 32, st));
    level_pairs = uint64_t(ctx->host_box[0]);
    level_max = ctx->host_box[1];
    const int64_t nchild = ctx->host_box[2], mchild = ctx->host_box[3];
    ++levels;
    if (nchild == 0) {
      nb = ne;
      break;
    }
    RS_TRY(ensure_nodes(ctx, ne, ne + nchild, st));
    RS_TRY(ensure_members(ctx, me, me + mchild, st));
    h = hier_of(ctx);
    uint64_t* ka = scratch_t<uint64_t>(ctx, S_KEY_A, size_t(mchild));
    uint64_t* kb = scratch_t<uint64_t>(ctx, S_KEY_B, size_t(mchild));
    uint32_t* va = scratch_t<uint32_t>(ctx, S_VAL_A, size_t(mchild));
    uint32_t* vb = scratch_t<uint32_t>(ctx, S_VAL_B, size_t(mchild));
    if (!ka || !kb || !va || !vb) return RS_ERR_OOM;
    const int bits = bits_for(uint64_t(nchild));
    (sort_ends_in_b(mchild, bits) ? vb : va) = h.mem + me;  // the sorted members are the level's list
    k_children<<<grid_for(m, kT), kT, 0, st>>>(m, mb, ne, uf, cnt, cidx, mpos, h.mem, h.mnode, min_size, ka, va,
                                              h.node_size, h.node_parent, h.node_level);
    RS_LAUNCHED(ctx, "k_children");
    uint64_t* skeys;
    uint32_t* svals;
    RS_TRY(radix_sort_u64(ctx, mchild, bits, ka, va, kb, vb, &skeys, &svals, st));  // svals == h.mem + me
    RS_TRY(exclusive_scans(ctx, nchild, ScanJobs{{{h.node_size + ne, h.node_off + ne, h.node_off + ne + nchild,
                                                   0, 0, me}}}, st));
    nb = ne;
    ne += nchild;
    mb = me;
    me += mchild;
  }
  ctx->have_hier = true;
  ctx->h_pos = pos;
  ctx->h_vel = vel;
  ctx->n_particles = n;
  ctx->n_nodes = ne;
  ctx->n_members = me;
  ctx->n_level0 = members;
  ctx->n_levels = levels;
  if (n_nodes_out) *n_nodes_out = ne;
  if (n_members_out) *n_members_out = me;
  return RS_OK;
}

namespace {
__global__ void k_u32_to_i64(int64_t n, const uint32_t* __restrict__ a, int64_t* __restrict__ b) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) b[i] = a[i];
}
}  // namespace

extern "C" int rs_fof6d_copy(rs_ctx* ctx, int64_t* node_parent, int32_t* node_level,
                             int64_t* node_min_id, int64_t* node_size, int64_t* member_offsets,
                             int64_t* member_idx, int64_t* particle_deepest_node, void* stream) {
  if (!ctx) return RS_ERR_INVALID_ARG;
  ctx->err[0] = 0;
  if (!ctx->have_hier) return set_error(ctx, RS_ERR_STATE, "rs_fof6d has not run on this context");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  RS_CUDA(ctx, cudaSetDevice(ctx->device));
  Hier h = hier_of(ctx);
  const int64_t nn = ctx->n_nodes, nm = ctx->n_members;
  auto cp = [&](void* dst, const void* src, size_t bytes) -> int {
    if (dst && bytes) RS_CUDA(ctx, cudaMemcpyAsync(dst, src, bytes, cudaMemcpyDeviceToDevice, st));
    return RS_OK;
  };
  RS_TRY(cp(node_parent, h.node_parent, 8 * nn));
  RS_TRY(cp(node_level, h.node_level, 4 * nn));
  RS_TRY(cp(node_min_id, h.node_minid, 8 * nn));
  RS_TRY(cp(node_size, h.node_size, 8 * nn));
  RS_TRY(cp(member_offsets, h.node_off, 8 * (nn + 1)));
  RS_TRY(cp(particle_deepest_node, h.deepest, 8 * ctx->n_particles));
  if (member_idx && nm) {
    k_u32_to_i64<<<grid_for(nm, kT), kT, 0, st>>>(nm, h.mem, member_idx);
    RS_LAUNCHED(ctx, "k_u32_to_i64");
  }
  return RS_OK;
}

extern "C" int rs_fof6d_node_params(rs_ctx* ctx, float* params_out, void* stream) {
  if (!ctx) return RS_ERR_INVALID_ARG;
  ctx->err[0] = 0;
  if (!ctx->have_hier) return set_error(ctx, RS_ERR_STATE, "rs_fof6d has not run on this context");
  if (!params_out && ctx->n_nodes) return set_error(ctx, RS_ERR_INVALID_ARG, "params_out is NULL");
  RS_CUDA(ctx, cudaSetDevice(ctx->device));
  if (ctx->n_nodes)
    RS_CUDA(ctx, cudaMemcpyAsync(params_out, hier_of(ctx).inv, 16 * ctx->n_nodes,
                                 cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream)));
  return RS_OK;
}
