// The inner BiCGstab of small batches as one launch: a thread-block cluster per
// (instance, group of right-hand sides) runs init, iterations and convergence
// checks of its systems, with cluster barriers where the launched form
// (krylov.cu) has kernel boundaries.
//
// The launched form is bound by its nine launches an iteration on small batches, and by
// one thread walking the eight directions of a site (5 us a hop however few sites there
// are).  Here the eight directions of 32 sites are eight warps: one load latency per hop
// step instead of eight, the links of a chunk serve the cluster's right-hand sides from
// registers, and the warps' loads of neighbouring sites meet in L1.  The half spinors are
// summed through shared memory.  What is left is latency on the smallest batches (8^4 x 4
// rhs: 15 us an iteration) and the issue rate on larger ones (about 2000
// warp instructions per step of a group).  Vectors stay in global memory (L2), in the
// layout and slots of the launched form.  Against the launched form, all else as now: 8^4 x 4 rhs
// whole solve 2206 -> 925 us.
#include <algorithm>
#include <cmath>
#include <type_traits>

#include "internal.h"
#include "spinor.cuh"

namespace dd {

namespace {

constexpr int CL_THREADS = 512;        // two groups of 8 warps
constexpr int CL_GROUPS = 2;
constexpr int CL_R = 4;                // most right-hand sides per cluster
constexpr int CL_DOTS = 7;
constexpr int CL_OWN = 192 + 1;        // threads of a group that own output pairs (6 warps), padded
constexpr int CL_UBUF = 8 * 6 * 32;    // half-spinor numbers of one 32-site chunk and rhs
// An inner product adds four numbers a lane and step in FP32.  After six steps the lane has added
// the 24 numbers that a site has in the launched form; the warp's sum of them (768 numbers, as
// there) is set aside, and everything above is FP64.  A lane has one step on 8^4, seven with framed
// 9^4 blocks and up to 34 on the largest frames taken; one FP32 sum over all of them was up to 72
// units of FP32 rounding off where these are at most 30.  A run's end costs a lane about 100
// instructions (16^4 x 4 rhs 4517 us a solve, without it 4417; 8^4 x 4 rhs has none).
constexpr int CL_FP32_STEPS = 6;
constexpr size_t CL_UBYTES = sizeof(float2) * CL_GROUPS * 2 * CL_UBUF;
// half spinors, the lanes' sums, the warps' sums of `runs` runs of steps
constexpr size_t cl_smem_bytes(int rb, int runs) {
  return CL_UBYTES + sizeof(float) * CL_DOTS * rb * (CL_GROUPS * CL_OWN + CL_THREADS / 32 * runs);
}
constexpr int CL_MAX_RUNS = 6;         // (see cluster_plan)
// runs of a lane with n steps
__host__ __device__ constexpr int cl_runs(int n) { return (n + CL_FP32_STEPS - 1) / CL_FP32_STEPS; }
// steps of a lane in a hop: its share of nq chunks
__host__ __device__ constexpr int cl_steps(int nq, int cs) { return (nq + CL_GROUPS * cs - 1) / (CL_GROUPS * cs); }

struct ClArgs {
  const void* rhs;
  void *x, *r, *p, *v, *s, *t, *tmp;
  SysState* st;
  double inner_tol2, floor_frac, k2;
  int maxiter, ngroups, rb;
  unsigned seed;
};

__device__ __forceinline__ unsigned cl_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cl_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// all threads of the cluster; what they wrote before (global and shared memory)
// is visible to all of them after
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ double cl_load(const double* p, unsigned rank) {
  unsigned a = (unsigned)__cvta_generic_to_shared(p), b;
  double v;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(b) : "r"(a), "r"(rank));
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(b) : "memory");
  return v;
}

// u = U h (forward) or U^+ h (backward) of the projected neighbour spinor
template <int MU, bool FWD>
__device__ __forceinline__ void half_hop(const float2 (&psi)[12], const float2 (&U)[9], float2 (&u)[6]) {
  float2 h[2][3];
  hop_project<MU, FWD>(psi, h);
#pragma unroll
  for (int s = 0; s < 2; ++s)
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      float2 w = make_float2(0.f, 0.f);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        if (FWD) cfma(w, U[a * 3 + b], h[s][b]);
        else cfmac(w, U[b * 3 + a], h[s][b]);
      }
      u[s * 3 + a] = w;
    }
}

// component K of the hop sum from the half spinors ub[dir][6][lane] of the eight
// directions: spins 0, 1 add up, spins 2, 3 are rebuilt as in hop_accum_row
template <int K>
__device__ __forceinline__ float2 hop_comp(const float2* ub) {
  float2 o = make_float2(0.f, 0.f);
  if constexpr (K < 6) {
#pragma unroll
    for (int d = 0; d < 8; ++d) o = cadd(o, ub[(d * 6 + K) * 32]);
  } else {
    constexpr int sp = (K - 6) / 3, a = (K - 6) % 3;
    constexpr int same = sp * 3 + a, other = (1 - sp) * 3 + a;
    o = csub(ub[same * 32], ub[(4 * 6 + same) * 32]);
    o = csubi(o, csub(ub[(6 + other) * 32], ub[(5 * 6 + other) * 32]));
    const float2 d2 = csub(ub[(12 + other) * 32], ub[(6 * 6 + other) * 32]);
    o = sp == 0 ? csub(o, d2) : cadd(o, d2);
    const float2 d3 = csub(ub[(18 + same) * 32], ub[(7 * 6 + same) * 32]);
    o = sp == 0 ? csubi(o, d3) : caddi(o, d3);
  }
  return o;
}

struct ClState {          // of one system, the same in every CTA of the cluster
  double2 rho, alpha, omega, beta;
  double rr, target2, outer2;
  int active, status, iters;
};

// the cluster's place in the batch
struct ClView {
  const DomInst* d;
  int n[2];
  int sys0, R;                 // first system and number of systems
  int q0[2], q1[2];            // this group's 32-site chunks of each parity
  int g, w, lane;              // group, warp in the group, lane
  int j0[2];                   // neighbour index of the first chunk per parity
  const long long* off;        // vector offsets [parity][CL_R]
};

template <class S>
__device__ __forceinline__ const unsigned char* cl_bundle(const DomInst& d) {
  if constexpr (std::is_same<S, float2>::value) return d.lb32;
  else return d.lb16;
}
// where a CTA's sum of a warp stands, [run][warp][system][number] (zero between the reductions)
__device__ __forceinline__ int cl_at(int R, int run, int warp, int rr, int k) {
  return ((run * (CL_THREADS / 32) + warp) * R + rr) * CL_DOTS + k;
}
__device__ __forceinline__ float cl_warp_sum(float v) {           // in lane 0
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}
// the same sum of 32 neighbouring numbers in shared memory, with the same tree
template <int N = 32>
__device__ __forceinline__ float cl_row_sum(const float* v) {
  if constexpr (N == 1) return v[0];
  else return cl_row_sum<N / 2>(v) + cl_row_sum<N / 2>(v + 32 / N);
}

// MODE 0: out = H in.  MODE 1: out = self - k2 H in with (r^, out).
// MODE 2: the same with (r^, out), (out, self), |out|^2, (r^, self).
// Warp w of a group takes direction w of the group's 32 sites, for each active rhs in turn
// with the link in registers; the half spinors meet in shared memory, and warps 0..5 form
// one component pair each.
template <class S, int MODE>
__device__ __forceinline__ void cl_hop(const ClView& V, const ClArgs& a, const ClState* st, int p, S* in, S* out,
                                       S* self, float2* ubuf, float* dacc, float* ps, unsigned& buf) {
  const int n_out = V.n[p], n_in = V.n[1 - p];
  const int w = V.w, lane = V.lane;
  constexpr int NK = MODE == 0 ? 0 : (MODE == 1 ? 2 : 7);
  float* row = dacc + (V.g * CL_DOTS * V.R) * CL_OWN + w * 32;     // number k of system rr at (k R + rr) CL_OWN
  float* my = row + lane;
  auto clear = [&]() {
#pragma unroll
    for (int k = 0; k < NK * CL_R; ++k)
      if (k < NK * V.R) my[k * CL_OWN] = 0.f;
  };
  if (w < 6) clear();
  const unsigned char* base = cl_bundle<S>(*V.d) + lb_quarter_base(p, V.n[0]) * lb_quarter_bytes<S>();
  const float mk2 = (float)-a.k2;
  // the neighbour index of the next chunk is read one chunk ahead (that of the first one
  // is kept through the whole solve), so only the spinor's latency is left in a step
  auto index = [&](int q) {
    return __ldg(reinterpret_cast<const int*>(base + (long long)q * lb_quarter_bytes<S>() + lb_link_bytes<S>()) +
                 w * LB_LANES + lane);
  };
  // a run is over: lane (k, rr) adds up its numbers of the warp's lanes
  int steps = 0, run = 0;
  auto fold = [&](bool last) {
    if (w >= 6) return;
    __syncwarp();
    if (lane < NK * V.R) ps[cl_at(V.R, run, threadIdx.x >> 5, lane % V.R, lane / V.R)] = cl_row_sum(row + lane * CL_OWN);
    if (last) return;
    __syncwarp();
    clear();
    ++run;
  };
  int jn = V.j0[p];
  for (int q = V.q0[p]; q < V.q1[p]; ++q) {
    const unsigned char* qb = base + (long long)q * lb_quarter_bytes<S>();
    const int j = jn;
    if (q + 1 < V.q1[p]) jn = index(q + 1);
    float2 U[9];
    {
      const S* lk = reinterpret_cast<const S*>(qb) + w * LB_DIR_S;
#pragma unroll
      for (int e = 0; e < 4; ++e) ld_pair(lk + (e * LB_LANES + lane) * 2, U[2 * e], U[2 * e + 1]);
      U[8] = ldc(lk + 4 * LB_LANES * 2 + lane);
    }
    const int i = q * 32 + lane;
    const bool live = i < n_out;
#pragma unroll 1
    for (int rr = 0; rr < V.R; ++rr) {
      if (!st[rr].active) continue;            // the same for the whole cluster
      float2* ub = ubuf + (V.g * 2 + buf) * CL_UBUF;
      float2 u[6];
      if (j >= 0) {
        float2 psi[12];
        S* src = in + V.off[(1 - p) * CL_R + rr];
#pragma unroll
        for (int e = 0; e < 6; ++e) ld_pair(src + ((long long)e * n_in + j) * 2, psi[2 * e], psi[2 * e + 1]);
        switch (w) {
          case 0: half_hop<0, true>(psi, U, u); break;
          case 1: half_hop<1, true>(psi, U, u); break;
          case 2: half_hop<2, true>(psi, U, u); break;
          case 3: half_hop<3, true>(psi, U, u); break;
          case 4: half_hop<0, false>(psi, U, u); break;
          case 5: half_hop<1, false>(psi, U, u); break;
          case 6: half_hop<2, false>(psi, U, u); break;
          default: half_hop<3, false>(psi, U, u); break;
        }
      } else {
#pragma unroll
        for (int c = 0; c < 6; ++c) u[c] = make_float2(0.f, 0.f);
      }
#pragma unroll
      for (int c = 0; c < 6; ++c) ub[(w * 6 + c) * 32 + lane] = u[c];
      __syncwarp();
      asm volatile("bar.sync %0, 256;" ::"r"(1 + V.g) : "memory");
      buf ^= 1;                                // the next step fills the other buffer
      if (w >= 6 || !live) continue;
      float2 o[2];
      const float2* ul = ub + lane;
      switch (w) {
        case 0: o[0] = hop_comp<0>(ul); o[1] = hop_comp<1>(ul); break;
        case 1: o[0] = hop_comp<2>(ul); o[1] = hop_comp<3>(ul); break;
        case 2: o[0] = hop_comp<4>(ul); o[1] = hop_comp<5>(ul); break;
        case 3: o[0] = hop_comp<6>(ul); o[1] = hop_comp<7>(ul); break;
        case 4: o[0] = hop_comp<8>(ul); o[1] = hop_comp<9>(ul); break;
        default: o[0] = hop_comp<10>(ul); o[1] = hop_comp<11>(ul); break;
      }
      const long long e = V.off[p * CL_R + rr] + ((long long)w * n_out + i) * 2;
      if constexpr (MODE > 0) {
        float2 sv[2], hv[2];
        ld_pair(self + e, sv[0], sv[1]);
        ld_rhat_pair<S>(a.seed, V.sys0 + rr, (const S*)nullptr, n_out, i, w, hv[0], hv[1]);
        float t[NK];
#pragma unroll
        for (int k = 0; k < NK; ++k) t[k] = my[(k * V.R + rr) * CL_OWN];
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
          o[h2].x = fmaf(mk2, o[h2].x, sv[h2].x);
          o[h2].y = fmaf(mk2, o[h2].y, sv[h2].y);
          const float2 O = o[h2], H = hv[h2], Z = sv[h2];
          t[0] = fmaf(H.x, O.x, fmaf(H.y, O.y, t[0]));
          t[1] = fmaf(H.x, O.y, fmaf(-H.y, O.x, t[1]));
          if constexpr (MODE == 2) {
            t[2] = fmaf(O.x, Z.x, fmaf(O.y, Z.y, t[2]));
            t[3] = fmaf(O.x, Z.y, fmaf(-O.y, Z.x, t[3]));
            t[4] = fmaf(O.x, O.x, fmaf(O.y, O.y, t[4]));
            t[5] = fmaf(H.x, Z.x, fmaf(H.y, Z.y, t[5]));
            t[6] = fmaf(H.x, Z.y, fmaf(-H.y, Z.x, t[6]));
          }
        }
#pragma unroll
        for (int k = 0; k < NK; ++k) my[(k * V.R + rr) * CL_OWN] = t[k];
      }
      st_pair(out + e, o[0], o[1]);
    }
    if constexpr (MODE > 0)
      if (++steps == CL_FP32_STEPS && q + 1 < V.q1[p]) {
        fold(false);
        steps = 0;
      }
  }
  if constexpr (MODE > 0) fold(true);
}

// sums over the cluster of NK numbers per system from the warps' sums ps (`runs` of them, zero where
// a warp has fewer): warps of the CTA and CTAs of the cluster in FP64, in a fixed order (trees of
// 16 and of the cluster's CTAs: an FP64 addition takes tens of cycles, so their chain is kept
// short).  slot: this CTA's sums, read by the others until the cluster barrier after the next one.
// On return sums[rr * NK + k] holds the result in every CTA, and ps is zero again.
template <int NK>
__device__ __forceinline__ void cl_reduce(const ClView& V, const ClState* st, float* ps, int runs, double* slot,
                                          double* sums) {
  constexpr int NW = CL_THREADS / 32;
  const int wi = threadIdx.x >> 5;
  __syncthreads();
  for (int e = wi; e < V.R * NK; e += NW) {
    if (!st[e / NK].active) continue;
    double v = 0.0;
    if (V.lane < NW) {
      float* at = ps + cl_at(V.R, 0, V.lane, e / NK, e % NK);
      v = widen(*at);
      *at = 0.f;
#pragma unroll 1
      for (int k = 1; k < runs; ++k) {
        at += cl_at(V.R, 1, 0, 0, 0);
        v += widen(*at);
        *at = 0.f;
      }
    }
#pragma unroll
    for (int o = NW / 2; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (V.lane == 0) slot[e] = v;
  }
  cl_sync();
  const unsigned nc = cl_size();
  for (int e = wi; e < V.R * NK; e += NW) {
    if (!st[e / NK].active) continue;
    double v = V.lane < (int)nc ? cl_load(slot + e, V.lane) : 0.0;
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (V.lane == 0) sums[e] = v;
  }
  __syncthreads();
}

__device__ __forceinline__ double2 zmul2(double2 a, double2 b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a / b with one division
__device__ __forceinline__ double2 zdiv2(double2 a, double2 b) {
  const double d = 1.0 / (b.x * b.x + b.y * b.y);
  return make_double2((a.x * b.x + a.y * b.y) * d, (a.y * b.x - a.x * b.y) * d);
}

template <class S>
__global__ void __launch_bounds__(CL_THREADS, 2) k_cl_bicgstab(BatchDev bd, ClArgs a) {
  extern __shared__ __align__(16) unsigned char cl_smem[];
  float2* ubuf = reinterpret_cast<float2*>(cl_smem);
  float* dacc = reinterpret_cast<float*>(cl_smem + CL_UBYTES);
  float* ps = dacc + CL_GROUPS * CL_DOTS * a.rb * CL_OWN;
  __shared__ double slots[3][CL_R * CL_DOTS];
  __shared__ double sums[CL_R * CL_DOTS];
  __shared__ ClState st[CL_R];
  __shared__ long long offs[2 * CL_R];
  const unsigned rank = cl_rank(), nc = cl_size();
  const int cid = blockIdx.x / nc;
  const int j = cid / a.ngroups, g0 = (cid % a.ngroups) * a.rb;
  ClView V;
  V.d = bd.inst_tab + bd.inst[j];
  V.n[0] = V.d->n[0];
  V.n[1] = V.d->n[1];
  V.sys0 = j * bd.nrhs + g0;
  V.R = min(a.rb, bd.nrhs - g0);
  V.w = (threadIdx.x >> 5) & 7;
  V.g = threadIdx.x >> 8;
  V.lane = threadIdx.x & 31;
  V.off = offs;
#pragma unroll
  for (int p = 0; p < 2; ++p) {
    const int nq = (V.n[p] + 31) / 32, ng = (int)nc * CL_GROUPS, me = (int)rank * CL_GROUPS + V.g;
    const int per = (nq + ng - 1) / ng;
    V.q0[p] = min(nq, me * per);
    V.q1[p] = min(nq, (me + 1) * per);
    V.j0[p] = -1;
    if (V.q0[p] < V.q1[p])
      V.j0[p] = __ldg(reinterpret_cast<const int*>(cl_bundle<S>(*V.d) +
                                                   (lb_quarter_base(p, V.n[0]) + V.q0[p]) * lb_quarter_bytes<S>() +
                                                   lb_link_bytes<S>()) +
                      V.w * LB_LANES + V.lane);
  }
  S *x = (S*)a.x, *r = (S*)a.r, *pv = (S*)a.p, *v = (S*)a.v, *s = (S*)a.s, *t = (S*)a.t, *tmp = (S*)a.tmp;
  const int n0 = V.n[0];
  const int ne = (V.q1[0] - V.q0[0]) * 6;          // (chunk, component pair) words of this group per rhs
  // lane's element of word e of rhs rr: chunk q0 + e / 6, pair e % 6
  auto elem = [&](int rr, int e, long long& at) -> bool {
    const int i = (V.q0[0] + e / 6) * 32 + V.lane;
    at = V.off[rr] + ((long long)(e % 6) * n0 + i) * 2;
    return i < n0;
  };
  // most runs of a warp, in a hop and in a pass over the vectors
  const int steps = cl_steps((V.n[0] + 31) / 32, (int)nc);
  const int hruns = cl_runs(steps), vruns = cl_runs((6 * steps + 7) / 8);
  unsigned buf = 0;

  for (int e = threadIdx.x; e < cl_at(V.R, hruns, 0, 0, 0); e += CL_THREADS) ps[e] = 0.f;
  // r = p = rhs, x = 0, (r^, r), |r|^2 and the targets
  if (threadIdx.x < V.R) {
    st[threadIdx.x] = ClState{};
    st[threadIdx.x].active = 1;
    offs[threadIdx.x] = bd.off[0][V.sys0 + threadIdx.x];
    offs[CL_R + threadIdx.x] = bd.off[1][V.sys0 + threadIdx.x];
  }
  __syncthreads();
  const int wi = threadIdx.x >> 5;
#pragma unroll 1
  for (int rr = 0; rr < V.R; ++rr) {
    float part[3] = {0.f, 0.f, 0.f};
    int run = 0;
    auto fold = [&]() {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const float v = cl_warp_sum(part[k]);
        if (V.lane == 0) ps[cl_at(V.R, run, wi, rr, k)] = v;
        part[k] = 0.f;
      }
      ++run;
    };
    int e = V.w;
#pragma unroll 1
    do {
      const int ee = min(ne, e + 8 * CL_FP32_STEPS);
      for (; e < ee; e += 8) {
        long long at;
        if (!elem(rr, e, at)) continue;
        float2 b[2], h[2];
        ld_pair((const S*)a.rhs + at, b[0], b[1]);
        st_pair(r + at, b[0], b[1]);
        st_pair(pv + at, b[0], b[1]);
        st_pair(x + at, make_float2(0.f, 0.f), make_float2(0.f, 0.f));
        ld_rhat_pair<S>(a.seed, V.sys0 + rr, (const S*)nullptr, n0, (V.q0[0] + e / 6) * 32 + V.lane, e % 6, h[0], h[1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          part[0] = fmaf(h[k].x, b[k].x, fmaf(h[k].y, b[k].y, part[0]));
          part[1] = fmaf(h[k].x, b[k].y, fmaf(-h[k].y, b[k].x, part[1]));
          part[2] = fmaf(b[k].x, b[k].x, fmaf(b[k].y, b[k].y, part[2]));
        }
      }
      fold();
    } while (e < ne);
  }
  cl_reduce<3>(V, st, ps, vruns, slots[0], sums);
  if (threadIdx.x < V.R) {
    ClState& z = st[threadIdx.x];
    const SysState& g = a.st[V.sys0 + threadIdx.x];
    const double* q = sums + threadIdx.x * 3;
    z.rho = make_double2(q[0], q[1]);
    z.rr = q[2];
    z.outer2 = g.outer2;
    z.target2 = fmax(a.inner_tol2 * z.rr, a.floor_frac * g.outer2);
    z.status = g.status == 2 ? 0 : g.status;
    z.iters = g.iters;
    z.active = g.outer_active && z.rr > z.target2;
  }
  __syncthreads();

  for (int it = 0; it < a.maxiter; ++it) {
    bool any = false;
    for (int rr = 0; rr < V.R; ++rr) any = any || st[rr].active;
    if (!any) break;                                  // the same decision in every CTA
    cl_hop<S, 0>(V, a, st, 1, pv, tmp, (S*)nullptr, ubuf, dacc, ps, buf);
    cl_sync();
    cl_hop<S, 1>(V, a, st, 0, tmp, v, pv, ubuf, dacc, ps, buf);
    cl_reduce<2>(V, st, ps, hruns, slots[0], sums);
    if (threadIdx.x < V.R && st[threadIdx.x].active) {
      ClState& z = st[threadIdx.x];
      z.iters += 1;
      const double2 den = make_double2(sums[threadIdx.x * 2], sums[threadIdx.x * 2 + 1]);
      if (den.x == 0.0 && den.y == 0.0) {             // breakdown
        z.active = 0;
        z.status = 2;
      } else {
        z.alpha = zdiv2(z.rho, den);
      }
    }
    __syncthreads();
    for (int rr = 0; rr < V.R; ++rr) {
      if (!st[rr].active) continue;
      const float2 al = make_float2((float)st[rr].alpha.x, (float)st[rr].alpha.y);
      for (int e = V.w; e < ne; e += 8) {
        long long at;
        if (!elem(rr, e, at)) continue;
        float2 rv[2], vv[2];
        ld_pair(r + at, rv[0], rv[1]);
        ld_pair(v + at, vv[0], vv[1]);
#pragma unroll
        for (int k = 0; k < 2; ++k) rv[k] = csub(rv[k], cmul(al, vv[k]));
        st_pair(s + at, rv[0], rv[1]);
      }
    }
    cl_sync();
    cl_hop<S, 0>(V, a, st, 1, s, tmp, (S*)nullptr, ubuf, dacc, ps, buf);
    cl_sync();
    cl_hop<S, 2>(V, a, st, 0, tmp, t, s, ubuf, dacc, ps, buf);
    cl_reduce<7>(V, st, ps, hruns, slots[1], sums);
    if (threadIdx.x < V.R && st[threadIdx.x].active) {
      ClState& z = st[threadIdx.x];
      const double* q = sums + threadIdx.x * 7;       // (r^, t), (t, s), |t|^2, (r^, s)
      const double inv = q[4] > 0.0 ? 1.0 / q[4] : 0.0;
      z.omega = make_double2(q[2] * inv, q[3] * inv);
      const double2 rn = make_double2(q[5] - (z.omega.x * q[0] - z.omega.y * q[1]),
                                      q[6] - (z.omega.x * q[1] + z.omega.y * q[0]));
      const bool rho0 = z.rho.x == 0.0 && z.rho.y == 0.0, rn0 = rn.x == 0.0 && rn.y == 0.0;
      z.beta = make_double2(0.0, 0.0);
      if (!rn0 && !rho0 && (z.omega.x != 0.0 || z.omega.y != 0.0))
        z.beta = zmul2(zdiv2(rn, z.rho), zdiv2(z.alpha, z.omega));
      if (rn0 || rho0) z.status = 2;
      z.rho = rn;
    }
    __syncthreads();
    // x += alpha p + omega s ; r = s - omega t ; p = r + beta (p - omega v) ; |r|^2
#pragma unroll
    for (int rr = 0; rr < CL_R; ++rr) {
      if (rr >= V.R || !st[rr].active) continue;
      float part = 0.f;
      int run = 0;
      auto fold = [&]() {
        const float v = cl_warp_sum(part);
        if (V.lane == 0) ps[cl_at(V.R, run, wi, rr, 0)] = v;
        part = 0.f;
        ++run;
      };
      const float2 al = make_float2((float)st[rr].alpha.x, (float)st[rr].alpha.y);
      const float2 om = make_float2((float)st[rr].omega.x, (float)st[rr].omega.y);
      const float2 be = make_float2((float)st[rr].beta.x, (float)st[rr].beta.y);
      int e = V.w;
#pragma unroll 1
      do {
        const int ee = min(ne, e + 8 * CL_FP32_STEPS);
        for (; e < ee; e += 8) {
          long long at;
          if (!elem(rr, e, at)) continue;
          float2 xv[2], pp[2], sv[2], tv[2], vv[2];
          ld_pair(x + at, xv[0], xv[1]);
          ld_pair(pv + at, pp[0], pp[1]);
          ld_pair(s + at, sv[0], sv[1]);
          ld_pair(t + at, tv[0], tv[1]);
          ld_pair(v + at, vv[0], vv[1]);
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            xv[k] = cadd(xv[k], cadd(cmul(al, pp[k]), cmul(om, sv[k])));
            const float2 q = csub(sv[k], cmul(om, tv[k]));
            part = fmaf(q.x, q.x, fmaf(q.y, q.y, part));
            pp[k] = cadd(q, cmul(be, csub(pp[k], cmul(om, vv[k]))));
            sv[k] = q;
          }
          st_pair(x + at, xv[0], xv[1]);
          st_pair(r + at, sv[0], sv[1]);
          st_pair(pv + at, pp[0], pp[1]);
        }
        fold();
      } while (e < ne);
    }
    cl_reduce<1>(V, st, ps, vruns, slots[2], sums);
    if (threadIdx.x < V.R && st[threadIdx.x].active) {
      ClState& z = st[threadIdx.x];
      z.rr = sums[threadIdx.x];
      // converged, broken down, or NaN (caught by the outer check)
      if (!(z.rr > z.target2) || z.status == 2) z.active = 0;
    }
    __syncthreads();
  }
  if (rank == 0 && threadIdx.x < V.R) {
    const ClState& z = st[threadIdx.x];
    SysState& g = a.st[V.sys0 + threadIdx.x];
    g.rr = z.rr;
    g.target2 = z.target2;
    g.rho = z.rho;
    g.alpha = z.alpha;
    g.omega = z.omega;
    g.status = z.status;
    g.iters = z.iters;
    g.active = z.active;
  }
  cl_sync();                 // no CTA leaves while another reads its sums
}

template <class S>
cudaError_t cl_launch(const BatchDev& bd, const ClArgs& a, int clusters, int cs, int runs, cudaStream_t s) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)(clusters * cs));
  cfg.blockDim = dim3(CL_THREADS);
  cfg.dynamicSmemBytes = cl_smem_bytes(a.rb, runs);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cs;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_cl_bicgstab<S>, bd, a);
}

}  // namespace

// once per device
void cluster_prepare() {
  static bool done[64] = {false};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64 || done[dev]) return;
  cudaFuncSetAttribute(k_cl_bicgstab<float2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cl_smem_bytes(CL_R, CL_MAX_RUNS));
  cudaFuncSetAttribute(k_cl_bicgstab<__nv_bfloat162>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)cl_smem_bytes(CL_R, CL_MAX_RUNS));
  done[dev] = true;
}

// Right-hand sides and CTAs per cluster of the one-launch inner solve for this batch;
// {0, 0} where it is not taken.
//
// A hop of a cluster takes steps of 32 sites x 1 rhs, one after the other in each group:
// ceil(chunks / groups) * rb of them, about 1 us each alone on an SM and 1.25 us with two CTAs
// per SM, in waves of 2 CTAs per SM.  On blocks of more than 8^4 sites neighbouring sites meet less
// often in L1 and a step takes longer, 1.1 us on 9^4 and 3 on 13^4; frames and frame pieces miss
// many of their hops and don't show that.  With one CTA per system a step takes 10 % longer (its
// barriers have nothing to overlap), with BF16 vectors too.  rb and cs are those with the least time
// by this count.  An iteration has four hops and about 12 us of barriers and reductions; the launched
// form takes 36 us + work / 2500 (work: even sites x rhs), and streams from DRAM once the vectors
// outgrow L2.  us an iteration, launched / one launch: blocks of 5^4 x 4 rhs 52 / 15, 7^4 x 4
// 67 / 37, 9^4 x 1 63 / 55, 9^4 x 4 121 / 103, frame of 12^4 with 12 rhs 55 / 35, 81 blocks of
// 7^4 x 2 113 / 94; launched are, among others, 10^4 x 1 70 / 76, 11^4 x 1 110 / 120, 13^4 x 1
// 176 / 241 (BF16 140 / 265), which a rule without the blocks' size gave to the one launch.  Over 140
// batches of 1 .. 81 systems with 1 .. 16 rhs the form taken is at most 1 % slower an iteration than
// the other (2 % in whole solves of uneven blocks, whose systems end at different times).
// From about 400 thousand even sites x rhs on the two meet, so the line lies at 300 thousand.
// Not taken with the clover term (its A^-1 is bulk-copied beside the link bundles, which has no place
// in this kernel), per-launch timing, a chosen launch form or the wait test, which concern the
// launched kernels.
ClusterPlan cluster_plan(dd_ctx* c, const Batch& b, dd_prec prec) {
  const ClusterPlan none{0, 0};
  if (prec != DD_F32 && prec != DD_BF16) return none;
  if (c->clover_active || c->timing || c->debug_wait_fault) return none;
  if (c->forced_variant[prec == DD_F32 ? 1 : 2] >= 0) return none;
  const double work = (double)b.tot[0] / 12.0;
  if (work > 3e5) return none;
  const int nq = (std::max(b.maxn[0], b.maxn[1]) + 31) / 32;
  // a step on whole blocks: their mean number of even sites against that of 9^4
  double big = 1.08 * std::pow(work / ((double)b.nrhs * b.nb) / 3281.0, 0.7);
  for (int j : b.inst)
    if (c->inst[j].d.kind != DD_DOMAIN_OMEGA && c->inst[j].d.kind != DD_DOMAIN_FULL) big = 0.0;
  ClusterPlan best = none;
  double tbest = 0.0;
  for (int rb = std::min(b.nrhs, CL_R); rb >= 1; --rb) {
    const long long ng = (b.nrhs + rb - 1) / rb;
    for (int cs = 1; cs <= 8; cs *= 2) {
      if (cl_runs(cl_steps(nq, cs)) > CL_MAX_RUNS) continue;   // 37 steps and more are never the faster form
      const long long ctas = b.nb * ng * cs;
      const double waves = (double)((ctas + 2LL * c->nsm - 1) / (2LL * c->nsm));
      const double step = std::max(ctas > c->nsm ? 1.25 : 1.0, big) * (cs == 1 ? 1.1 : 1.0);
      const double t = waves * (4.0 * cl_steps(nq, cs) * rb * step + 12.0) * (prec == DD_BF16 ? 1.1 : 1.0);
      if (best.cs == 0 || t < tbest) {
        best = {rb, cs};
        tbest = t;
      }
    }
  }
  return tbest < 36.0 + work / 2500.0 ? best : none;
}

dd_status run_cluster(dd_ctx* c, const Batch& b, dd_prec prec, ClusterPlan plan, const void* rhs, void* x, void* r,
                      void* p, void* v, void* s, void* t, void* tmp, SysState* st, double inner_tol2,
                      double floor_frac, int maxiter, unsigned seed, cudaStream_t q) {
  ClArgs a;
  a.rhs = rhs;
  a.x = x; a.r = r; a.p = p; a.v = v; a.s = s; a.t = t; a.tmp = tmp;
  a.st = st;
  a.inner_tol2 = inner_tol2;
  a.floor_frac = floor_frac;
  a.k2 = c->kappa * c->kappa;
  a.maxiter = maxiter;
  a.rb = plan.rb;
  a.ngroups = (b.nrhs + plan.rb - 1) / plan.rb;
  a.seed = seed;
  cluster_prepare();
  BatchDev bd = batch_view(c, b);
  DD_COUNT_LAUNCH();
  const int clusters = b.nb * a.ngroups, runs = std::max(1, cl_runs(cl_steps((b.maxn[0] + 31) / 32, plan.cs)));
  const cudaError_t e = prec == DD_F32 ? cl_launch<float2>(bd, a, clusters, plan.cs, runs, q)
                                       : cl_launch<__nv_bfloat162>(bd, a, clusters, plan.cs, runs, q);
  DD_CUDA(c, e);
  return DD_OK;
}

}  // namespace dd
