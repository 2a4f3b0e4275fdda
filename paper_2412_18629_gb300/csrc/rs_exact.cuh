// Exact float32 potential sums of a LIST of members (the members whose flag is still open after
// a gate), with certified flags; shared by the surrogate path and the certified tree bound.
//
// A list entry k indexes a member-position map (mem_of[k] = p, the member's position in the
// hierarchy's member CSR); the list is grouped by node, with per-node ranges [lofs, lend).
#pragma once

#include "rs_cro.cuh"

namespace {

constexpr double kU = 5.9604644775390625e-08;
// per-member warp sum: per term <= 8u, 32-term lane blocks <= 31u, Kahan <= 2u, 5-level warp
// tree <= 5u; 48u with slack.
constexpr double kCertB2 = 48.0 * kU + 1e-12;

// Blocked direct sum over a list: 128 threads x kListR members per tile (kListR: a template
// parameter the autotuner picks among 2, 4, 8 for the surrogate's lists) against chunks of
// kListChunk members of the node, so that a short list of a large node still fills the GPU.
constexpr int kListThreads = 128;
constexpr int64_t kListChunk = 2048;

// Work items of a list of `len` members of a node with g members: tiles x chunks.
__host__ __device__ __forceinline__ int64_t list_items(int64_t len, int64_t g, int tile) {
  return ((len + tile - 1) / tile) * ((g + kListChunk - 1) / kListChunk);
}

// 0.5 |v - v_bulk|^2 in float64, every operation rounded (the oracle's kinetic energy).
__device__ __forceinline__ double kinetic(float4 v, const double* vb) {
  const double dvx = __dsub_rn(rsd::f2d(v.x), vb[0]);
  const double dvy = __dsub_rn(rsd::f2d(v.y), vb[1]);
  const double dvz = __dsub_rn(rsd::f2d(v.z), vb[2]);
  const double s = __dadd_rn(__dadd_rn(__dmul_rn(dvx, dvx), __dmul_rn(dvy, dvy)), __dmul_rn(dvz, dvz));
  return __dmul_rn(0.5, s);
}

// Float32 sums S_all,i = sum over ALL members j of the node (self included) of
// (|u_j - u_i|^2 + eps^2)^(-1/2) for the members i of the exact-path list. A work item is one tile
// of one node's list against one chunk of its members: j-tiles of 128 members staged duplicated
// in shared memory, packed float32x2 arithmetic, 32-term sequential blocks added with Kahan
// compensation (the same summation as the direct-sum kernels, so a chunk's sum is within the same
// relative bound of its terms); the chunks of a member are added in float64 (Sd, zeroed before, by
// list position). Including the self term, whose computed value is exactly w0 = rsqrt(eps^2),
// removes every per-pair index test; k_flags_list subtracts it and widens the certified bound
// accordingly. Persistent blocks stride over the items. One block per tile over the whole node
// left most of the GPU idle: 2.7e3 listed members of 12 nodes of up to 1e5 members took
// 3.1 ms; the chunked form, with the second walk leaving 60 of them, takes 0.07 ms (2^27 snapshot:
// 82 -> 4.8 ms).
template <int kListR, bool kNormal>
__global__ void __launch_bounds__(kListThreads)
k_potential_list(int64_t nbig, const int64_t* __restrict__ item_off, const int64_t* __restrict__ nodes,
                 const int64_t* __restrict__ lofs, const int64_t* __restrict__ lend,
                 const uint32_t* __restrict__ list, const uint32_t* __restrict__ mem_of,
                 const int64_t* __restrict__ node_off, const int64_t* __restrict__ node_size,
                 const float4* __restrict__ U, float eps2, double* __restrict__ Sd) {
  __shared__ float4 sxy[kListThreads];
  __shared__ float2 sz[kListThreads];
  const int64_t items = item_off[nbig];
  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const int64_t bi = rsd::upper_bound_i64(item_off, nbig, item) - 1;
    const int64_t q = nodes[bi], it = item - item_off[bi];
    const int64_t base = node_off[q], g = node_size[q];
    const int64_t chunks = (g + kListChunk - 1) / kListChunk, t = it / chunks, c = it - t * chunks;
    const int64_t j_end = rsd::min64(g, (c + 1) * kListChunk);
    const int64_t l0 = lofs[bi] + t * (kListThreads * kListR), l1 = lend[bi];
    float2 nx[kListR / 2], ny[kListR / 2], nz[kListR / 2];
    float S[kListR], C[kListR];
#pragma unroll
    for (int pp = 0; pp < kListR / 2; ++pp) {
      const int64_t a0 = l0 + threadIdx.x + kListThreads * (2 * pp), a1 = a0 + kListThreads;
      const float4 u0 = a0 < l1 ? U[mem_of[list[a0]]] : make_float4(0, 0, 0, 0);
      const float4 u1 = a1 < l1 ? U[mem_of[list[a1]]] : make_float4(0, 0, 0, 0);
      nx[pp] = make_float2(-u0.x, -u1.x);
      ny[pp] = make_float2(-u0.y, -u1.y);
      nz[pp] = make_float2(-u0.z, -u1.z);
    }
#pragma unroll
    for (int k = 0; k < kListR; ++k) {
      S[k] = 0.f;
      C[k] = 0.f;
    }
    const float2 e2 = make_float2(eps2, eps2);
    for (int64_t j0 = c * kListChunk; j0 < j_end; j0 += kListThreads) {
      const int64_t j = j0 + threadIdx.x;
      if (j < j_end) {
        const float4 u = U[base + j];
        sxy[threadIdx.x] = make_float4(u.x, u.x, u.y, u.y);
        sz[threadIdx.x] = make_float2(u.z, u.z);
      }
      __syncthreads();
      const int jn = int(rsd::min64(kListThreads, j_end - j0));
      for (int jb = 0; jb < jn; jb += 32) {
        const int je = min(jb + 32, jn);
        float2 blk[kListR / 2];
#pragma unroll
        for (int pp = 0; pp < kListR / 2; ++pp) blk[pp] = make_float2(0.f, 0.f);
#pragma unroll 8
        for (int jj = jb; jj < je; ++jj) {
          const float4 a = sxy[jj];
          const float2 zz = sz[jj];
#pragma unroll
          for (int pp = 0; pp < kListR / 2; ++pp) {
            const float2 dx = __fadd2_rn(make_float2(a.x, a.y), nx[pp]);
            const float2 dy = __fadd2_rn(make_float2(a.z, a.w), ny[pp]);
            const float2 dz = __fadd2_rn(zz, nz[pp]);
            const float2 r2 = __ffma2_rn(dx, dx, __ffma2_rn(dy, dy, __ffma2_rn(dz, dz, e2)));
            blk[pp] = __fadd2_rn(blk[pp], make_float2(rsd::inv_sqrt<kNormal>(r2.x), rsd::inv_sqrt<kNormal>(r2.y)));
          }
        }
#pragma unroll
        for (int k = 0; k < kListR; ++k) {
          const float bk = (k & 1) ? blk[k >> 1].y : blk[k >> 1].x;
          const float y = __fsub_rn(bk, C[k]);
          const float tt = __fadd_rn(S[k], y);
          C[k] = __fsub_rn(__fsub_rn(tt, S[k]), y);
          S[k] = tt;
        }
      }
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < kListR; ++k) {
      const int64_t a = l0 + threadIdx.x + kListThreads * k;
      if (a < l1) atomicAdd(Sd + a, double(S[k]));
    }
  }
}

// The sums of a list of at most `len_ub` members with R members per thread (2, 4 or 8); Sd is zeroed
// first. Eight blocks an SM stride over the items, whose number only the device knows.
template <class... Args>
int launch_potential_list(rs_ctx* ctx, int R, float eps2, int64_t len_ub, double* Sd,
                          cudaStream_t st, Args... args) {
  RS_CUDA(ctx, cudaMemsetAsync(Sd, 0, sizeof(double) * size_t(len_ub), st));
  auto launch = [&](auto kernel) { kernel<<<152 * 8, kListThreads, 0, st>>>(args..., eps2, Sd); };
  if (rs::normal_eps2(eps2)) {
    if (R == 2) launch(k_potential_list<2, true>);
    else if (R == 8) launch(k_potential_list<8, true>);
    else launch(k_potential_list<4, true>);
  } else {
    if (R == 2) launch(k_potential_list<2, false>);
    else if (R == 8) launch(k_potential_list<8, false>);
    else launch(k_potential_list<4, false>);
  }
  RS_LAUNCHED(ctx, "k_potential_list");
  return RS_OK;
}

// Flags of the exact-path list from S_all: S = S_all - w0. With B = 41u the bound of the blocked
// sums relative to S_all = S + w0, |S - S_true| <= B (S + w0), so the member's relative bound is
// Bi = B (1 + w0 / S) (plus slack, which covers the float64 additions); the flag is certain when
// |KE + phi~| > 2 Bi |phi~|, otherwise the member is queued for the float64 potential. w0 is the value that
// the sums of the same kNormal hold.
template <bool kNormal>
__global__ void k_flags_list(const unsigned long long* __restrict__ count, const uint32_t* __restrict__ list,
                             const uint32_t* __restrict__ mem_of, const uint32_t* __restrict__ mnode,
                             const float4* __restrict__ V, const double* __restrict__ vbulk,
                             float eps2, double Gm, const double* __restrict__ Sd,
                             uint8_t* __restrict__ bound, uint32_t* __restrict__ ambig, unsigned long long* __restrict__ n_ambig) {
  const int64_t w = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (w >= int64_t(*count)) return;
  const uint32_t k = list[w];
  const uint32_t p = mem_of[k], q = mnode[p];
  const double w0 = double(rsd::inv_sqrt<kNormal>(eps2));
  const double S = Sd[w] - w0;
  const double ph = -__dmul_rn(Gm, S);
  const double e = __dadd_rn(kinetic(V[p], vbulk + 3 * int64_t(q)), ph);
  const double Bi = 41.0 * kU * (1.0 + w0 / fmax(S, 1e-30)) + 2.0 * kU + 1e-12;
  if (S > 0.0 && fabs(e) > 2.0 * Bi * fabs(ph)) {
    bound[p] = e < 0.0 ? 1 : 0;
  } else {
    ambig[atomicAdd(n_ambig, 1ull)] = p;
  }
}

}  // namespace
