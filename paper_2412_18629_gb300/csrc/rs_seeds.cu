// Seed halos, the assignment of every FoF-group particle to a seed, and the seeds' host
// relations: the step after the 6D hierarchy (Section "Parallelization": subhalo finding inside
// every FoF halo from 6D phase-space information). The paper gives no formulas for it; the
// reading implemented here:
//   seeds   the nodes without children (each level-0 node has at least one under it);
//   frame   u = wrapped offset from the level-0 node's reference member r0 (smallest id);
//   seed s  centre c_s = float(double(wrap(x_{r_s} - x_{r0})) + CRO(u^s) / g_s), u^s the
//           offsets from s's own reference member r_s, bulk velocity
//           w_s = float(CRO(v) / g_s), and the metric scales (inv_sx2, inv_sv2) of s's split;
//   metric  fl(|u - c_s|^2 inv_sx2_s) + fl(|v - w_s|^2 inv_sv2_s), float32 in d6's order;
//   particle  the seed holding it when its deepest node is a seed, otherwise the nearest seed
//           under its deepest node (ties: the smaller node index);
//   host    of a seed s: among the other seeds of the same level-0 node ranking above it (more
//           assigned particles; equal counts: the smaller node index), the nearest by the
//           candidate's metric at (c_s, w_s); -1 if none.
// Every comparison uses the same float32 operations as the CPU oracle, so the results are
// identical to it.
// Positions and velocities are read from the call's own arrays throughout: the hierarchy's U and V hold
// the contents that rs_fof6d or rs_unbind saw, and an address does not tell whether they still are.
#include "rs_cro.cuh"

using namespace rs;

namespace {

constexpr int kT = 256;

__global__ void k_seed_kids(int64_t nn, const int64_t* __restrict__ parent, int* __restrict__ nkids) {
  const int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (q < nn && parent[q] >= 0) atomicAdd(nkids + parent[q], 1);
}

// Per node the walk up its parents (as many steps as its level): its level-0 ancestor, and for a seed a
// count at each node of the walk and at itself. Also the position of its reference member, the segments of
// the seeds for the canonical-order sums (size 0 otherwise) and the number of seeds. The walk replaced
// seven pointer-jumping launches.
__global__ void k_seed_roots(int64_t nn, const int64_t* __restrict__ parent, const int* __restrict__ nkids,
                             const int64_t* __restrict__ node_size, int64_t* __restrict__ root,
                             unsigned long long* __restrict__ cnt, int64_t* __restrict__ seg_size,
                             unsigned long long* __restrict__ n_seeds, const int64_t* __restrict__ node_off,
                             const uint32_t* __restrict__ mem, const float* __restrict__ pos,
                             float4* __restrict__ ref) {
  const int64_t q = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool seed = q < nn && nkids[q] == 0;
  rsd::warp_count(n_seeds, seed);
  if (q >= nn) return;
  seg_size[q] = seed ? node_size[q] : 0;
  const int64_t i = mem[node_off[q]];
  ref[q] = make_float4(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], 0.f);
  int64_t r = q;
  for (int64_t p = q; p >= 0; p = parent[p]) {
    r = p;
    if (seed) atomicAdd(cnt + p, 1ull);
  }
  root[q] = r;
}

struct Particle {
  float3 x, v;
};

__device__ __forceinline__ Particle load_particle(const float* __restrict__ pos, const float* __restrict__ vel, int64_t i) {
  return {make_float3(pos[3 * i], pos[3 * i + 1], pos[3 * i + 2]), make_float3(vel[3 * i], vel[3 * i + 1], vel[3 * i + 2])};
}

// Wrapped offset of x from the reference position r.
__device__ __forceinline__ float3 offset_from(float4 r, float3 x, float L) {
  const float hL = 0.5f * L;
  return make_float3(rsd::wrap_diff(r.x, x.x, L, hL), rsd::wrap_diff(r.y, x.y, L, hL), rsd::wrap_diff(r.z, x.z, L, hL));
}

struct SeedTerm {  // u^s and v of a member of seed s
  const uint32_t* mem;
  const float4* ref;
  const float *pos, *vel;
  float L;
  using Value = Particle;
  __device__ __forceinline__ Value load(int64_t p) const { return load_particle(pos, vel, mem[p]); }
  template <bool kFirst>
  __device__ __forceinline__ void add(int64_t q, const Value& t, double* acc) const {
    const float3 u = offset_from(ref[q], t.x, L), v = t.v;
    rsd::cro_add<kFirst>(acc[0], rsd::f2d(u.x));
    rsd::cro_add<kFirst>(acc[1], rsd::f2d(u.y));
    rsd::cro_add<kFirst>(acc[2], rsd::f2d(u.z));
    rsd::cro_add<kFirst>(acc[3], rsd::f2d(v.x));
    rsd::cro_add<kFirst>(acc[4], rsd::f2d(v.y));
    rsd::cro_add<kFirst>(acc[5], rsd::f2d(v.z));
  }
};

// A seed as the searches read it, beside the others under the same node: centre and position scale, bulk
// velocity and velocity scale, its index. Read through a list of indices into four tables, the loads of
// one seed waited for the index; the records of a node are one run of memory.
struct SeedRec {
  float4 c, w;
};

// Seed centres (level-0 frame) and bulk velocities from the canonical-order sums.
__global__ void k_seed_stats(int64_t nn, const int* __restrict__ nkids, const int64_t* __restrict__ root,
                             const int64_t* __restrict__ node_size, const float4* __restrict__ ref, float L,
                             const double* __restrict__ sums, const float4* __restrict__ inv,
                             SeedRec* __restrict__ rec) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= nn || nkids[s] != 0) return;
  const float4 rs_ = ref[s];
  const float3 u = offset_from(ref[root[s]], make_float3(rs_.x, rs_.y, rs_.z), L);
  const double g = double(node_size[s]);
  const double* S = sums + 6 * s;
  const float o[3] = {u.x, u.y, u.z};
  float c[3], w[3];
#pragma unroll
  for (int d = 0; d < 3; ++d) {
    c[d] = __double2float_rn(__dadd_rn(double(o[d]), __ddiv_rn(S[d], g)));
    w[d] = __double2float_rn(__ddiv_rn(S[3 + d], g));
  }
  const float4 iv = inv[s];
  rec[s] = {make_float4(c[0], c[1], c[2], iv.x), make_float4(w[0], w[1], w[2], iv.y)};
}

__device__ __forceinline__ float seed_metric(float ax, float ay, float az, float vx, float vy, float vz,
                                             const SeedRec& s) {
  const float rx = rsd::sq3(__fsub_rn(ax, s.c.x), __fsub_rn(ay, s.c.y), __fsub_rn(az, s.c.z));
  const float rv = rsd::sq3(__fsub_rn(vx, s.w.x), __fsub_rn(vy, s.w.y), __fsub_rn(vz, s.w.z));
  return __fadd_rn(__fmul_rn(rx, s.c.w), __fmul_rn(rv, s.w.w));
}

// Every seed into the lists of its own node and of the nodes above it.
__global__ void k_seed_under_fill(int64_t nn, const int64_t* __restrict__ parent, const int* __restrict__ nkids,
                                  const int64_t* __restrict__ off, const SeedRec* __restrict__ rec,
                                  unsigned long long* __restrict__ fill, int64_t* __restrict__ list,
                                  SeedRec* __restrict__ lrec) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= nn || nkids[s] != 0) return;
  const SeedRec t = rec[s];
  for (int64_t q = s; q >= 0; q = parent[q]) {
    const int64_t at = off[q] + int64_t(atomicAdd(fill + q, 1ull));
    list[at] = s;
    lrec[at] = t;
  }
}

// One thread per member of a level-0 node, in the member list's order: its seed (argmin over the seeds
// under its deepest node). Neighbours share their group's list of seeds; in the order of the particles every
// lane walked another list (101 us for 2^21 particles in groups of up to 3e4 members, 36 us in this order;
// from the hierarchy's streamed U and V, which may be of another time, 27 us).
__global__ void k_seed_assign(int64_t m0, const uint32_t* __restrict__ mem, const uint32_t* __restrict__ mnode,
                              const float4* __restrict__ ref, const int64_t* __restrict__ deepest,
                              const int* __restrict__ nkids, const float* __restrict__ pos,
                              const float* __restrict__ vel, float L, const int64_t* __restrict__ uoff,
                              const int64_t* __restrict__ ulist, const SeedRec* __restrict__ lrec,
                              int64_t* __restrict__ seed, unsigned long long* __restrict__ count) {
  const int64_t p = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  const bool in = p < m0;  // every lane stays for the match
  const int64_t i = in ? mem[p] : 0, dq = in ? deepest[i] : -1;
  const Particle own = load_particle(pos, vel, i);  // beside the chain of loads to the node's list
  int64_t arg = dq;
  if (in && nkids[dq] != 0) {
    const float3 u = offset_from(ref[mnode[p]], own.x, L), v = own.v;
    float best = 0.f;
    arg = -1;
    const int64_t k1 = uoff[dq + 1];
#pragma unroll 4
    for (int64_t k = uoff[dq]; k < k1; ++k) {
      const SeedRec t = lrec[k];
      const int64_t s = ulist[k];
      const float d = seed_metric(u.x, u.y, u.z, v.x, v.y, v.z, t);
      if (arg < 0 || d < best || (d == best && s < arg)) {
        best = d;
        arg = s;
      }
    }
  }
  if (in) seed[i] = arg;
  // one addition per seed and warp
  const unsigned peers = __match_any_sync(0xffffffffu, arg);
  if (arg >= 0 && (threadIdx.x & 31) == __ffs(peers) - 1) atomicAdd(count + arg, (unsigned long long)__popc(peers));
}

// One thread per seed: its host among the seeds of its level-0 node ranking above it.
__global__ void k_seed_host(int64_t nn, const int* __restrict__ nkids, const int64_t* __restrict__ root,
                            const int64_t* __restrict__ uoff, const int64_t* __restrict__ ulist,
                            const SeedRec* __restrict__ rec, const SeedRec* __restrict__ lrec,
                            const unsigned long long* __restrict__ count,
                            int64_t* __restrict__ host, int64_t* __restrict__ count_out) {
  const int64_t s = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (s >= nn) return;
  if (nkids[s] != 0) {
    if (host) host[s] = -2;
    if (count_out) count_out[s] = 0;
    return;
  }
  const unsigned long long ns = count[s];
  const float4 c = rec[s].c, w = rec[s].w;
  const int64_t r = root[s], k1 = uoff[r + 1];
  float best = 0.f;
  int64_t arg = -1;
#pragma unroll 4
  for (int64_t k = uoff[r]; k < k1; ++k) {
    const int64_t h = ulist[k];
    const unsigned long long nh = count[h];
    const SeedRec t = lrec[k];
    if (h == s || !(nh > ns || (nh == ns && h < s))) continue;
    const float d = seed_metric(c.x, c.y, c.z, w.x, w.y, w.z, t);
    if (arg < 0 || d < best || (d == best && h < arg)) {
      best = d;
      arg = h;
    }
  }
  if (host) host[s] = arg;
  if (count_out) count_out[s] = int64_t(ns);
}

}  // namespace

extern "C" int rs_assign_seeds(rs_ctx* ctx, const float* pos, const float* vel, int64_t* particle_seed,
                               int64_t* node_host, int64_t* node_count, int64_t* n_seeds_out,
                               void* stream) {
  if (!ctx) return RS_ERR_INVALID_ARG;
  ctx->err[0] = 0;
  if (!ctx->have_hier) return set_error(ctx, RS_ERR_STATE, "rs_fof6d has not run on this context");
  const int64_t n = ctx->n_particles, nn = ctx->n_nodes, m = ctx->n_members;
  if (n > 0 && (!pos || !vel || !particle_seed))
    return set_error(ctx, RS_ERR_INVALID_ARG, "null device pointer");
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  RS_CUDA(ctx, cudaSetDevice(ctx->device));
  if (n_seeds_out) *n_seeds_out = 0;
  if (nn == 0) {
    if (n > 0) RS_CUDA(ctx, cudaMemsetAsync(particle_seed, 0xff, 8 * size_t(n), st));  // -1
    return RS_OK;
  }
  Hier h = hier_of(ctx);
  int* nkids = scratch_t<int>(ctx, S_SEED_KIDS, size_t(nn));
  int64_t* root = scratch_t<int64_t>(ctx, S_SEED_ROOT, size_t(nn));
  unsigned long long* ucnt = scratch_t<unsigned long long>(ctx, S_SEED_UCNT, 2 * size_t(nn) + 2);
  int64_t* uoff = scratch_t<int64_t>(ctx, S_SEED_UOFF, size_t(nn) + 1);
  SeedRec* rec = scratch_t<SeedRec>(ctx, S_SEED_CEN, size_t(nn));
  double* sums = scratch_t<double>(ctx, S_SEED_SUMS, 6 * size_t(nn));
  int64_t* segsz = scratch_t<int64_t>(ctx, S_SEED_SEG, size_t(nn));
  unsigned long long* count = scratch_t<unsigned long long>(ctx, S_SEED_COUNT, size_t(nn));
  float4* ref = scratch_t<float4>(ctx, S_SEED_REF, size_t(nn));
  if (!nkids || !root || !ucnt || !uoff || !rec || !sums || !segsz || !count || !ref) return RS_ERR_OOM;
  unsigned long long* fill = ucnt + nn + 1;
  RS_CUDA(ctx, cudaMemsetAsync(nkids, 0, 4 * size_t(nn), st));
  k_seed_kids<<<grid_for(nn, kT), kT, 0, st>>>(nn, h.node_parent, nkids);
  RS_LAUNCHED(ctx, "k_seed_kids");
  // level-0 ancestor of every node and the seeds under it: counts, offsets, lists
  RS_CUDA(ctx, cudaMemsetAsync(ucnt, 0, 8 * (2 * size_t(nn) + 2), st));
  unsigned long long* n_seeds = fill + nn;  // the spare last counter slot
  k_seed_roots<<<grid_for(nn, kT), kT, 0, st>>>(nn, h.node_parent, nkids, h.node_size, root, ucnt, segsz, n_seeds,
                                              h.node_off, h.mem, pos, ref);
  RS_LAUNCHED(ctx, "k_seed_roots");
  static_assert(sizeof(unsigned long long) == sizeof(int64_t), "counts scanned as int64");
  RS_TRY(exclusive_scans(ctx, nn, ScanJobs{{{reinterpret_cast<int64_t*>(ucnt), uoff, uoff + nn}}}, st));
  RS_CUDA(ctx, cudaMemcpyAsync(ctx->host_box + 1, n_seeds, 8, cudaMemcpyDeviceToHost, st));
  RS_TRY(read_back(ctx, uoff + nn, 8, st));
  const int64_t seeds = ctx->host_box[1];
  const int64_t total = ctx->host_box[0];
  int64_t* ulist = scratch_t<int64_t>(ctx, S_SEED_LIST, size_t(std::max<int64_t>(total, 1)));
  SeedRec* lrec = scratch_t<SeedRec>(ctx, S_SEED_REC, size_t(std::max<int64_t>(total, 1)));
  if (!ulist || !lrec) return RS_ERR_OOM;
  // seed centres and bulk velocities (canonical-order sums over the seeds' members)
  RS_TRY((cro_segmented<6, SeedTerm>(ctx, nn, h.node_off, segsz, m, SeedTerm{h.mem, ref, pos, vel, ctx->cfg.box_L},
                                     sums, st)));
  k_seed_stats<<<grid_for(nn, kT), kT, 0, st>>>(nn, nkids, root, h.node_size, ref, ctx->cfg.box_L, sums, h.inv, rec);
  RS_LAUNCHED(ctx, "k_seed_stats");
  k_seed_under_fill<<<grid_for(nn, kT), kT, 0, st>>>(nn, h.node_parent, nkids, uoff, rec, fill, ulist, lrec);
  RS_LAUNCHED(ctx, "k_seed_under_fill");
  RS_CUDA(ctx, cudaMemsetAsync(count, 0, 8 * size_t(nn), st));
  RS_CUDA(ctx, cudaMemsetAsync(particle_seed, 0xff, 8 * size_t(n), st));  // -1: in no group
  {
    ProfScope prof_(ctx, "k_seed_assign", st);
    k_seed_assign<<<grid_for(ctx->n_level0, kT), kT, 0, st>>>(ctx->n_level0, h.mem, h.mnode, ref, h.deepest,
                                                             nkids, pos, vel, ctx->cfg.box_L, uoff, ulist, lrec,
                                                             particle_seed, count);
  }
  RS_LAUNCHED(ctx, "k_seed_assign");
  k_seed_host<<<grid_for(nn, kT), kT, 0, st>>>(nn, nkids, root, uoff, ulist, rec, lrec, count,
                                              node_host, node_count);
  RS_LAUNCHED(ctx, "k_seed_host");
  if (n_seeds_out) {
    *n_seeds_out = seeds;
    RS_CUDA(ctx, cudaStreamSynchronize(st));
  }
  return RS_OK;
}
