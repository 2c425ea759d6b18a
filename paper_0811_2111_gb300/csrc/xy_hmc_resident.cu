// xy_hmc_resident.cu -- many HMC trajectories of a small lattice in one launch:
// one thread-block cluster holds the lattice (strips of full rows, see
// xy_strip.cuh) and integrates, tests and records trajectory after trajectory.
//
// At these sides a leap-frog step is a few hundred cycles of dependent
// arithmetic; a launch per step (the per-site kernel: 26 us for the 13 launches
// of a ten-step trajectory at L = 64) or per trajectory costs more than the
// work, and a cluster's barrier and the dependent chain behind it (about 0.7 us
// a step) bound it here.  A thread owns the same pairs of adjacent sites throughout: angles,
// momenta and unit vectors in registers, the unit vectors published to shared
// memory (double-buffered by step, so one cluster barrier per step is enough)
// and to the neighbouring strips' halo rows.  Each warp's exact integer sums of
// a trajectory's two ends go to every CTA's shared memory, one barrier later
// every CTA forms the same dH and takes the same decision; a rejected
// trajectory takes its old angles back from registers.  The next momenta are
// drawn before that barrier is waited for.
//
// Per-site arithmetic and sums are the shared HMC device code's (packed where
// two sites allow it), so angles, momenta, sums and decisions are bit for bit
// those of the per-site, tiled and cluster kernels.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "xy_hmc_device.cuh"
#include "xy_internal.h"
#include "xy_strip.cuh"

namespace cg = cooperative_groups;

namespace xyk {

namespace {

using namespace xyh;

constexpr int kThreads = 512;                // at most; the launch takes what the pairs need
constexpr int kWarps = kThreads / 32;
constexpr int kMaxCtas = 16;
constexpr int kMaxPairs = 2;                 // pairs a thread owns
constexpr int kVals = 8;                     // a warp's integers of one end: HmcAcc

// The total of sum j (HmcAcc fields, see hmc_commit) over `n` warps' integers.
__device__ __forceinline__ long long acc_value(const int* v, int j) {
  switch (j) {
    case 0: return ((long long)v[0] << 21) + (long long)v[1];
    case 1: return ((long long)v[2] << 21) + (long long)v[3];
    default: return (long long)v[j + 2] << 9;
  }
}

// u < exp(-dH) for the uniform u on the 2^-24 grid: where FP32 decides it (its
// exp of a rounded dH is within 2^-20 of the exact one: |dH| 2^-24 + 2 ulp
// relative, and e^-x x <= 1/e), else in FP64 as hmc_decide.
__device__ __forceinline__ bool hmc_test(double dH, uint32_t w0) {
  const double u = (double)(w0 >> 8) * 0x1p-24;
  const float d = (float)(w0 >> 8) * 0x1p-24f - expf(-(float)dH);
  if (fabsf(d) > 0x1p-19f) return d < 0.f;
  return u < exp(-dH);
}

template <int MODE, int NP>
__global__ void __launch_bounds__(kThreads)
    k_hmc_resident(HmcArgs a, int C, int n_md, int n_traj, int draw, int mode, double beta,
                   double J) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ __align__(16) int s_acc[2][kMaxCtas * kWarps][kVals];  // [end][rank, warp]
  __shared__ int s_take;
  cg::cluster_group cluster = cg::this_cluster();
  const int rank = (int)cluster.block_rank();
  const int L = a.L;
  const xys::Strip st(L, L, C, rank);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = blockDim.x >> 5;
  float4* cs = reinterpret_cast<float4*>(smem);            // [2] planes, by step parity
  const int pvec = xys::plane_vec4(xys::strip_rows(L, C, 0), L);
  float4* up_cs = cluster.map_shared_rank(cs, st.up_rank);
  float4* dn_cs = cluster.map_shared_rank(cs, st.dn_rank);
  HmcCtl* ctl = a.ctl;
  float* state = hmc_buf(a, (int)ctl->cur);
  const uint32_t traj0 = (uint32_t)ctl->traj;
  auto meet = [&]() {
    __syncwarp();
    if (C > 1) {
      cluster.sync();
    } else {
      __syncthreads();
    }
  };

  xys::Pair pr[NP];
  float2 t[NP], p[NP], t_old[NP], p_new[NP];
  auto site_of = [&](int i) {
    return (uint32_t)(st.y0 + pr[i].r) * (uint32_t)L + (uint32_t)pr[i].k;
  };
  auto momenta = [&](int i, uint32_t traj) {
    const uint32_t s = site_of(i);
    return make_float2(hmc_momentum(s, traj, a.lattice_id, a.rk),
                       hmc_momentum(s + 1u, traj, a.lattice_id, a.rk));
  };
#pragma unroll
  for (int i = 0; i < NP; ++i) {
    pr[i].set(st, threadIdx.x + i * blockDim.x);
    t[i] = p_new[i] = make_float2(0.f, 0.f);
    if (!pr[i].on) continue;
    const uint32_t s = site_of(i);
    t[i].x = state[s];
    if (pr[i].two) t[i].y = state[s + 1u];
    if (draw) {
      p_new[i] = momenta(i, traj0);
    } else {
      p_new[i].x = a.p_in[s];
      if (pr[i].two) p_new[i].y = a.p_in[s + 1u];
    }
  }
  if (C > 1) cluster.sync();                // every CTA has started: its memory may be written

  const float half = 0.5f * a.eps;
  unsigned long long n_taken = 0;           // rank 0, thread 0
  for (int tr = 0; tr < n_traj; ++tr) {
    const uint32_t traj = traj0 + (uint32_t)tr;
#pragma unroll
    for (int i = 0; i < NP; ++i) {
      t_old[i] = t[i];
      p[i] = p_new[i];
    }
    for (int s = 0; s <= n_md; ++s) {
      float4* buf = cs + (s & 1) * pvec;
      float2 c[NP], sn[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        xyd::unit_vector2<MODE>(t[i], &sn[i], &c[i]);
        if (pr[i].on)
          xys::put(st, pr[i], buf, up_cs + (s & 1) * pvec, dn_cs + (s & 1) * pvec, c[i], sn[i]);
      }
      meet();
      const bool end = s == n_md, sums = s == 0 || end;
      const float coef = sums ? half : a.eps;
      HmcAcc acc;
      acc_zero(acc);
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        if (!pr[i].on) continue;
        const int at = pr[i].at;
        const float4 D = buf[at - st.pitch], U = buf[at + st.pitch];
        const float4 El = buf[at - 1], Er = buf[at + 1];
        float2 rc = make_float2(c[i].y, Er.x), rs = make_float2(sn[i].y, Er.z);
        if (!pr[i].two) {                   // the right neighbour is the copy of column 0
          rc.x = buf[at].y;
          rs.x = buf[at].w;
        }
        const float2 Sc = xyd::add2(xyd::add2(make_float2(El.y, c[i].x), rc),
                                    xyd::add2(make_float2(D.x, D.y), make_float2(U.x, U.y)));
        const float2 Ss = xyd::add2(xyd::add2(make_float2(El.w, sn[i].x), rs),
                                    xyd::add2(make_float2(D.z, D.w), make_float2(U.z, U.w)));
        const float2 F = hmc_force2(c[i], sn[i], Sc, Ss, a.K);
        auto terms = [&]() {
          hmc_terms(p[i].x, c[i].x, sn[i].x, rc.x, rs.x, U.x, U.z, acc);
          if (pr[i].two) hmc_terms(p[i].y, c[i].y, sn[i].y, rc.y, rs.y, U.y, U.w, acc);
        };
        if (s == 0) terms();
        p[i] = xyd::fma2(xyd::dup2(coef), F, p[i]);
        if (end) {
          terms();
        } else {
          const float2 d = xyd::fma2(xyd::dup2(a.eps), p[i], t[i]);
          t[i] = make_float2(hmc_wrap(d.x), hmc_wrap(d.y));
        }
      }
      if (sums) {
        // (n_md >= 1, so the two ends are different steps)
        int v[kVals] = {acc.kh, acc.kl, acc.ch, acc.cl, acc.ix, acc.iy, acc.mx, acc.my};
#pragma unroll
        for (int j = 0; j < kVals; ++j)
          v[j] = (int)__reduce_add_sync(0xffffffffu, (uint32_t)v[j]);
        if (lane < C) {
          int* to = cluster.map_shared_rank(&s_acc[end ? 1 : 0][rank * nwarps + warp][0], lane);
          reinterpret_cast<int4*>(to)[0] = make_int4(v[0], v[1], v[2], v[3]);
          reinterpret_cast<int4*>(to)[1] = make_int4(v[4], v[5], v[6], v[7]);
        }
      }
    }
    // every warp's sums of both ends reach every CTA
    __syncwarp();
    if (C > 1) cluster.barrier_arrive();
    if (draw && tr + 1 < n_traj) {
#pragma unroll
      for (int i = 0; i < NP; ++i)
        if (pr[i].on) p_new[i] = momenta(i, traj + 1u);
    }
    __syncwarp();
    if (C > 1) {
      cluster.barrier_wait();
    } else {
      __syncthreads();
    }
    // lanes walk the C x nwarps entries of an end
    const int entries = C * nwarps;
    if (warp == 0) {
      long long dK = 0, dC = 0;
      for (int e = lane; e < entries; e += 32) {
        dK += acc_value(s_acc[1][e], 0) - acc_value(s_acc[0][e], 0);
        dC += acc_value(s_acc[1][e], 1) - acc_value(s_acc[0][e], 1);
      }
      dK = warp_sum_ll(dK);
      dC = warp_sum_ll(dC);
      if (lane == 0) {
        bool take = true;
        if (mode == 0) {
          const uint4 w = xyd::philox4x32_10(make_uint4(0u, traj, a.lattice_id, 4u), a.rk);
          take = hmc_test(hmc_dH(dK, dC, beta, J), w.x);
        }
        s_take = take ? 1 : 0;
        if (rank == 0 && mode == 0) {
          xy_hmc_record* r = ctl->records + (ctl->rec + (unsigned long long)tr);
          r->dH = hmc_dH(dK, dC, beta, J);
          r->beta = beta;
          r->accepted = take ? 1ull : 0ull;
          n_taken += take ? 1ull : 0ull;
        }
      }
    }
    __syncthreads();
    const bool take = s_take != 0;
    if (rank == 0) {
      // the record's sums, one per warp
      for (int task = warp; task < 2 * kHmcSums; task += nwarps) {
        const int end = task / kHmcSums, j = task - end * kHmcSums;
        long long x = 0;
        for (int e = lane; e < entries; e += 32) x += acc_value(s_acc[end][e], j);
        x = warp_sum_ll(x);
        if (lane == 0) {
          if (mode == 0) {
            xy_hmc_record* r = ctl->records + (ctl->rec + (unsigned long long)tr);
            if (j == 0) r->kinetic[end] = x;
            if (j == 1) r->bonds[end] = x;
            if (j > 0 && end == (take ? 1 : 0)) r->sum[j - 1] = x;
          }
          if (tr + 1 == n_traj) ctl->last[end][j] = (unsigned long long)x;
        }
      }
    }
    if (!take) {
#pragma unroll
      for (int i = 0; i < NP; ++i) t[i] = t_old[i];
    }
  }

#pragma unroll
  for (int i = 0; i < NP; ++i) {
    if (!pr[i].on) continue;
    const uint32_t s = site_of(i);
    state[s] = t[i].x;
    a.p_out[s] = p[i].x;
    if (pr[i].two) {
      state[s + 1u] = t[i].y;
      a.p_out[s + 1u] = p[i].y;
    }
  }
  // every CTA has read the counters, and no CTA's memory is written any more
  meet();
  if (rank == 0 && threadIdx.x == 0 && mode == 0) {
    ctl->rec += (unsigned long long)n_traj;
    ctl->traj += (unsigned long long)n_traj;
    ctl->accepted += n_taken;
  }
}

// CTAs of the cluster for side L (0: not resident).  Measured, us per unit
// trajectory (eps = 0.1 (64 / L)^(1/2)) by cluster size, and the per-site
// kernel's graph of n_md + 3 launches:
//   L = 16   1: 5.2            16: 10.1   per site 16.6
//   L = 32   1: 8.0   8: 8.8   16: 11.3            18.6
//   L = 64   1: 25.7  8: 10.4  16: 10.5            23.0
//   L = 96            8: 17.3  16: 14.2            26.9
//   L = 128           8: 22.3  16: 17.6            29.6  (cluster kernel 39.3)
//   L = 160           8: 38.6  16: 23.8            33.7
//   L = 256                    16: 49.4            45.3  (cluster kernel 74.0)
// Above 176 a thread owns four pairs and sixteen SMs are slower than all of
// them at one launch a step.
int resident_ctas(int L) {
  if (L < 4 || L > 176) return 0;
  return L <= 32 ? 1 : L <= 64 ? 8 : 16;
}

struct Plan {
  int ctas, np, threads;
  size_t smem;
};

Plan plan_of(int L) {
  Plan p = {};
  p.ctas = resident_ctas(L);
  if (p.ctas == 0) return p;
  const int rows = xys::strip_rows(L, p.ctas, 0);
  const int pairs = rows * ((L + 1) / 2);
  p.np = (pairs + kThreads - 1) / kThreads;
  if (p.np > kMaxPairs) return Plan{};
  p.threads = ((pairs + p.np - 1) / p.np + 31) / 32 * 32;
  p.smem = sizeof(float4) * 2 * (size_t)xys::plane_vec4(rows, L);
  return p.smem <= kResidentSmem ? p : Plan{};
}

cudaLaunchConfig_t config_of(const Plan& p, cudaStream_t stream, cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.ctas);
  cfg.blockDim = dim3(p.threads);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = stream;
  attr->id = cudaLaunchAttributeClusterDimension;
  attr->val.clusterDim.x = p.ctas;
  attr->val.clusterDim.y = 1;
  attr->val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

template <int MODE, class F>
cudaError_t with_np(const Plan& p, const F& f) {
  return p.np == 1 ? f(k_hmc_resident<MODE, 1>) : f(k_hmc_resident<MODE, 2>);
}

template <class F>
cudaError_t with_kernel(int mode, const Plan& p, const F& f) {
  return mode == 0 ? with_np<0>(p, f) : mode == 1 ? with_np<1>(p, f) : with_np<2>(p, f);
}

}  // namespace

cudaError_t prepare_hmc_resident(int sincos_mode, int L, bool* fits) {
  *fits = false;
  const Plan p = plan_of(L);
  if (p.ctas == 0) return cudaSuccess;
  return with_kernel(sincos_mode, p, [&](auto* fn) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kResidentSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = config_of(p, nullptr, &attr);
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, fn, &cfg);
    *fits = e == cudaSuccess && n >= 1;
    return e;
  });
}

cudaError_t launch_hmc_resident(int sincos_mode, const HmcArgs& a, int n_md, int n_traj, int draw,
                                int mode, double beta, double J, cudaStream_t stream) {
  const Plan p = plan_of(a.L);
  if (p.ctas == 0 || n_md < 1 || n_traj < 1) return cudaErrorInvalidValue;
  return with_kernel(sincos_mode, p, [&](auto* fn) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = config_of(p, stream, &attr);
    return cudaLaunchKernelEx(&cfg, fn, a, p.ctas, n_md, n_traj, draw, mode, beta, J);
  });
}

}  // namespace xyk
