// xy_resident.cu -- all sweeps of a call of a small lattice in one launch, the
// lattice never leaving the chip: one thread-block cluster holds it, a strip of
// full rows per CTA.
//
// A sweep of a small lattice is two dependent half-sweeps of a few hundred
// cycles; with one launch per half-sweep (L = 32: 22 us per sweep) or one tile
// of 32 x 128 sites after the other through global memory (L = 128: 4.9 us) it
// is all latency.  Here every thread owns the same pairs of sites (plane
// columns 2m, 2m + 1 of a row: one Philox block) of both colours for the whole
// launch: their angles and unit vectors stay in its registers, and shared
// memory holds only what neighbours read, the unit vectors of both colours as
// (cos, cos, sin, sin) per pair, with the strip's two halo rows and the two
// halo columns as copies.  A half-sweep reads the other colour's unit vectors,
// updates its pairs (xyd::metropolis_pair, so every decision is bit for bit
// that of the other kernels), and stores the new unit vectors to its own
// strip, to the halo columns, and, from a strip's first and last row, to the
// neighbouring CTAs' halo rows through distributed shared memory; one cluster
// barrier (release / acquire) ends it.  The next half-sweep's Philox words
// depend on no state and are drawn between the barrier's arrive and wait.
//
// Why one barrier per half-sweep is enough: a half-sweep of colour c reads
// unit vectors of colour 1 - c only (its own pairs are in registers; the red
// spins of the magnetisation are read in the black half) and writes those of
// colour c only, here and in the neighbours' halo rows.
//
// Exact sums only: they do not depend on who adds what, while the compensated
// sums round by thread and warp and keep the kernels that define them.
// Any even side whose strips fit (L odd multiples of 2 included): rows have
// (W + 1) / 2 pairs, and where W = L / 2 is odd the last pair's second column
// is column W, the halo copy of column 0; its lane's results are dropped.
//
// What bounds it is the latency of a half-sweep's dependent chain (about a
// thousand cycles with its barrier), at 256 the SM's FMA pipes as well;
// resident_ctas has the times.
#include <cooperative_groups.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "xy_device.cuh"
#include "xy_internal.h"
#include "xy_strip.cuh"

namespace cg = cooperative_groups;

namespace xyk {

namespace {

constexpr int kRThreads = 512;               // at most; the launch takes what the pairs need
constexpr int kRWarps = kRThreads / 32;
constexpr int kRMaxPairs = 2;                // pairs per thread and colour

using xys::plane_vec4;
using xys::strip_rows;

// NP: pairs of each colour a thread owns, at most.  (Blocks of 1024 threads leave
// 64 registers a thread and spill the state: L = 256 4.6 against 3.5 us per
// sweep with 512 threads of two pairs.)
template <int MODE, int NP>
__global__ void __launch_bounds__(kRThreads) k_sweep_resident(ResidentArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint32_t s_part[kRWarps][5];
  __shared__ uint32_t s_cnt[kRWarps];
  cg::cluster_group cluster = cg::this_cluster();
  const int C = a.ctas, rank = (int)cluster.block_rank();
  const int L = a.L, W = L / 2;
  // the cluster's lattice: the only one, in place, or one of a batch, from the
  // buffer of the first sweep's parity to that behind the last's
  const float* src = a.theta;
  float* dst = a.theta;
  float K = a.K;
  double beta = a.beta;
  uint32_t lattice_id = a.lattice_id, sweep0 = a.sweep0;
  xy_record* rec = a.rec;
  if (a.lattices) {
    const int li = a.lattices[blockIdx.x / C];
    sweep0 = a.counters[0];
    const uint32_t last = sweep0 + (uint32_t)a.n_sweeps - 1u;
    src = ((sweep0 & 1u) ? a.theta2 : a.theta) + a.offset[li];
    dst = ((last & 1u) ? a.theta : a.theta2) + a.offset[li];
    beta = a.betas[li];
    K = (float)(beta * a.J);
    lattice_id = a.lattice_id + (uint32_t)li;
    rec = a.rec + (size_t)li * a.rec_stride + sweep0;
  }
  const xys::Strip st(L, W, C, rank);
  const int nthreads = blockDim.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nwarps = nthreads >> 5;
  const size_t plane = (size_t)L * (size_t)W;
  float4* cs = reinterpret_cast<float4*>(smem);            // [2] planes
  const int pvec = plane_vec4(strip_rows(L, C, 0), W);
  float4* up_cs = cluster.map_shared_rank(cs, st.up_rank);
  float4* dn_cs = cluster.map_shared_rank(cs, st.dn_rank);
  xys::Pair pr[NP];                                        // this thread's pairs
#pragma unroll
  for (int p = 0; p < NP; ++p) pr[p].set(st, threadIdx.x + p * nthreads);
  auto put = [&](int p, int c, float2 cv, float2 sv) {
    xys::put(st, pr[p], cs + c * pvec, up_cs + c * pvec, dn_cs + c * pvec, cv, sv);
  };

  float2 th[2][NP], cv[2][NP], sv[2][NP];
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      th[c][p] = make_float2(0.f, 0.f);
      if (pr[p].on) {
        const float* g = src + c * plane + (size_t)(st.y0 + pr[p].r) * W + pr[p].k;
        th[c][p].x = g[0];
        if (pr[p].two) th[c][p].y = g[1];
      }
      xyd::unit_vector2<MODE>(th[c][p], &sv[c][p], &cv[c][p]);
    }
  auto words = [&](int p, int c, uint32_t sweep) {
    const uint32_t y = (uint32_t)(st.y0 + pr[p].r);
    return xyd::philox_pair_words(
        y * (uint32_t)L + 2u * (uint32_t)pr[p].k + ((y + (uint32_t)c) & 1u), sweep, lattice_id,
        a.rk);
  };
  uint4 w[NP];
#pragma unroll
  for (int p = 0; p < NP; ++p) w[p] = words(p, 0, sweep0);
  cluster.sync();                          // every CTA has started: its memory may be written
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int p = 0; p < NP; ++p)
      if (pr[p].on) put(p, c, cv[c][p], sv[c][p]);
  cluster.sync();

  // The previous sweep's sums, left in s_part / s_cnt before the barrier: one
  // warp per sum adds the warps' values (16-bit halves, one lane per warp) and
  // issues the record's atomic.
  auto commit = [&](xy_record* r) {
    for (int task = warp; task < 6; task += nwarps) {
      const bool has = lane < nwarps;
      if (task == 5) {
        const uint32_t n = has ? s_cnt[lane] : 0u;
        const uint32_t total = __reduce_add_sync(0xffffffffu, n & 0x7fffffffu);
        const bool bad = __any_sync(0xffffffffu, (n & 0x80000000u) != 0u);
        if (lane == 0) {
          atomicAdd(reinterpret_cast<unsigned long long*>(&r->accepted),
                    (unsigned long long)total);
          if (bad) atomicOr(reinterpret_cast<unsigned long long*>(&r->flags), 1ull);
          if (rank == 0) r->beta = beta;
        }
      } else {
        const int32_t v = has ? (int32_t)s_part[lane][task] : 0;
        const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)v & 0xffffu);
        const int32_t hi = (int32_t)__reduce_add_sync(0xffffffffu, (uint32_t)(v >> 16));
        if (lane == 0)
          atomicAdd(reinterpret_cast<unsigned long long*>(&r->sum[task]),
                    (unsigned long long)((long long)hi * 65536ll + (long long)lo)
                        << (XY_FX_SHIFT - xyd::fx_term_shift(task)));
      }
    }
  };

  for (int s = 0; s < a.n_sweeps; ++s) {
    const uint32_t sweep = sweep0 + (uint32_t)s;
    unsigned int n_acc = 0;
    xyd::SweepSums<0> sums;                // at most 2 NP black sites per thread
    sums.init();
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const float4* nb = cs + (1 - c) * pvec;
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        if (!pr[p].on) continue;
        const int q = (st.y0 + pr[p].r + c) & 1;     // x = 2k + q
        const float4 P = nb[pr[p].at], D = nb[pr[p].at - st.pitch], U = nb[pr[p].at + st.pitch];
        const float4 E = nb[q ? pr[p].at + 1 : pr[p].at - 1];
        xyd::PairNeighbours n;
        n.lc = q ? make_float2(P.x, P.y) : make_float2(E.y, P.x);
        n.ls = q ? make_float2(P.z, P.w) : make_float2(E.w, P.z);
        n.rc = q ? make_float2(P.y, E.x) : make_float2(P.x, P.y);
        n.rs = q ? make_float2(P.w, E.z) : make_float2(P.z, P.w);
        n.dc = make_float2(D.x, D.y);
        n.ds = make_float2(D.z, D.w);
        n.uc = make_float2(U.x, U.y);
        n.us = make_float2(U.z, U.w);
        n.sum();
        const xyd::PairResult r = xyd::metropolis_pair<MODE>(th[c][p], cv[c][p], sv[c][p], n.Sc,
                                                             n.Ss, w[p], xyd::dup2(K), a.delta);
        th[c][p] = r.th;
        cv[c][p] = r.c;
        sv[c][p] = r.s;
        put(p, c, r.c, r.s);
        n_acc += (r.acc0 ? 1u : 0u) + (r.acc1 && pr[p].two ? 1u : 0u);
        if (c == 1) {
          // red sites with the same (y, k): their spins enter M once each
          float2 v[5];
          xyd::measure_terms2(r.c, r.s, n, make_float2(P.x, P.y), make_float2(P.z, P.w), v);
          if (pr[p].two) {
            sums.add2(v);
          } else {
            const float v0[5] = {v[0].x, v[1].x, v[2].x, v[3].x, v[4].x};
            sums.add(v0);
          }
        }
      }
      if (c == 0 && s > 0) commit(rec + (s - 1));
      if (c == 1) {
        const unsigned int acc = __reduce_add_sync(0xffffffffu, n_acc);
        const bool bad = __any_sync(0xffffffffu, xyd::fx_nonfinite(sums.fx));
        uint32_t t[5];
#pragma unroll
        for (int i = 0; i < 5; ++i)
          t[i] = __reduce_add_sync(0xffffffffu, (uint32_t)xyd::fx_value(sums.fx, i));
        if (lane == 0) {
          s_cnt[warp] = acc | (bad ? 0x80000000u : 0u);
#pragma unroll
          for (int i = 0; i < 5; ++i) s_part[warp][i] = t[i];
        }
      }
      __syncwarp();
      if (C > 1) cluster.barrier_arrive();
      // drawn for a sweep past the last too (never used)
#pragma unroll
      for (int p = 0; p < NP; ++p) w[p] = words(p, 1 - c, sweep + (c == 1 ? 1u : 0u));
      if (C > 1) {
        cluster.barrier_wait();
      } else {
        __syncthreads();
      }
    }
  }
  commit(rec + (a.n_sweeps - 1));
#pragma unroll
  for (int c = 0; c < 2; ++c)
#pragma unroll
    for (int p = 0; p < NP; ++p)
      if (pr[p].on) {
        float* g = dst + c * plane + (size_t)(st.y0 + pr[p].r) * W + pr[p].k;
        g[0] = th[c][p].x;
        if (pr[p].two) g[1] = th[c][p].y;
      }
}

// CTAs of the cluster for side L (0: not resident).  One CTA while a thread
// per pair keeps its barrier cheap, then enough of them that a strip is a
// pair or two per thread; the cluster barrier costs about 0.2 us a half-sweep,
// whatever the cluster's size.  Measured, us per sweep by cluster size:
//   L = 32   1: 1.00   4: 1.49   8: 1.82  16: 1.84   (two launches a sweep: 22)
//   L = 48   1: 2.16   4: 1.56   8: 1.39  16: 1.51
//   L = 64   1: 2.75   4: 1.49   8: 1.45  16: 1.50
//   L = 80             4: 1.93   8: 1.53  16: 1.45
//   L = 128            4: 3.50   8: 1.98  16: 1.52   (persistent tiles: 4.9)
//   L = 256                      8: 6.55  16: 3.1    (persistent tiles: 5.3)
// A single lattice above kClusterMaxL is spread over the whole chip instead
// (xy_grid.cu, L = 256 1.51); where it does not find room there, and in a batch,
// the clusters take sides up to 256, above which a thread would own more pairs
// than its registers hold (L = 320 with four each 5.9).
int resident_ctas(int L) {
  if (L < 4 || L > 256) return 0;
  return L <= 32 ? 1 : L <= 64 ? 8 : 16;
}

struct Plan {
  int ctas, np, threads;
  size_t smem;
};

Plan plan_of(int L, int ctas) {
  Plan p = {};
  p.ctas = ctas;
  if (p.ctas == 0 || p.ctas > L || (L & 1)) return Plan{};
  const int W = L / 2, rows = strip_rows(L, p.ctas, 0);
  const int pairs = rows * ((W + 1) / 2);
  p.np = (pairs + kRThreads - 1) / kRThreads;
  if (p.np > kRMaxPairs) return Plan{};
  p.threads = ((pairs + p.np - 1) / p.np + 31) / 32 * 32;
  p.smem = sizeof(float4) * 2 * (size_t)plane_vec4(rows, W);
  return p.smem <= kResidentSmem ? p : Plan{};
}

Plan plan_of(int L) { return plan_of(L, resident_ctas(L)); }

cudaLaunchConfig_t config_of(const Plan& p, int n_lattices, cudaStream_t stream,
                             cudaLaunchAttribute* attr) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.ctas * n_lattices);
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

// f(kernel) for the instantiation of a plan.
template <class F>
cudaError_t with_kernel(int mode, const Plan& p, const F& f) {
  switch (mode) {
    case 0: return p.np == 1 ? f(k_sweep_resident<0, 1>) : f(k_sweep_resident<0, 2>);
    case 1: return p.np == 1 ? f(k_sweep_resident<1, 1>) : f(k_sweep_resident<1, 2>);
    default: return p.np == 1 ? f(k_sweep_resident<2, 1>) : f(k_sweep_resident<2, 2>);
  }
}

}  // namespace

namespace {

// Sets the kernel's attributes and reports how many clusters of plan p the
// device runs at a time.
cudaError_t clusters_of(int mode, const Plan& p, int* n) {
  *n = 0;
  return with_kernel(mode, p, [&](auto* fn) {
    cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kResidentSmem);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = config_of(p, 1, nullptr, &attr);
    return cudaOccupancyMaxActiveClusters(n, fn, &cfg);
  });
}

}  // namespace

bool resident_supported(int L) { return plan_of(L).ctas > 0; }

cudaError_t prepare_resident(int sincos_mode, int L, bool* fits) {
  *fits = false;
  const Plan p = plan_of(L);
  if (p.ctas == 0) return cudaErrorInvalidValue;
  int n = 0;
  const cudaError_t e = clusters_of(sincos_mode, p, &n);
  *fits = e == cudaSuccess && n >= 1;
  return e;
}

// Time of a sweep of n lattices of side L by cluster size: a strip's latency
// (1.9 us for up to 64 pairs of a colour per CTA, whose two warps add up the six
// sums, 1.45 for 128, 1.5 for 256, 2.0 for 512, 3.5 for 1024, single lattices of
// L = 32 ... 256), once per wave of the
// clusters that run at a time, and a quarter more for each further CTA that
// shares an SM (L = 48 in clusters of 8: two lattices 1.55, 20 1.97, 30 2.04, 41
// 2.31).
cudaError_t prepare_resident_batch(int sincos_mode, int L, int n, int* ctas, double* us) {
  *ctas = 0;
  *us = 0.0;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  for (int c = 1; c <= 16; c *= 2) {
    const Plan p = plan_of(L, c);
    if (p.ctas == 0) continue;
    int at_a_time = 0;
    e = clusters_of(sincos_mode, p, &at_a_time);
    if (e != cudaSuccess) return e;
    if (at_a_time < 1) continue;
    const int pairs = strip_rows(L, c, 0) * ((L / 2 + 1) / 2);
    const double strip = pairs <= 64 ? 1.9 : pairs <= 256 ? 1.4 + 0.0004 * pairs
                         : 1.0 + 0.002 * pairs + (p.np > 1 ? 0.5 : 0.0);
    const int shared = ((n < at_a_time ? n : at_a_time) * c + sms - 1) / sms;
    const double t = strip * (1.0 + 0.25 * (shared - 1)) * (double)((n + at_a_time - 1) / at_a_time);
    if (*ctas == 0 || t < *us) {
      *ctas = c;
      *us = t;
    }
  }
  return cudaSuccess;
}

cudaError_t launch_resident(int sincos_mode, const ResidentArgs& args, cudaStream_t stream) {
  const Plan p = plan_of(args.L);
  if (p.ctas == 0 || args.n_sweeps < 1) return cudaErrorInvalidValue;
  ResidentArgs a = args;
  a.ctas = p.ctas;
  a.lattices = nullptr;
  return with_kernel(sincos_mode, p, [&](auto* fn) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = config_of(p, 1, stream, &attr);
    return cudaLaunchKernelEx(&cfg, fn, a);
  });
}

cudaError_t launch_resident_batch(int sincos_mode, const ResidentArgs& a, int n,
                                  cudaStream_t stream) {
  const Plan p = plan_of(a.L, a.ctas);
  if (p.ctas == 0 || a.n_sweeps < 1 || n < 1 || !a.lattices) return cudaErrorInvalidValue;
  return with_kernel(sincos_mode, p, [&](auto* fn) {
    cudaLaunchAttribute attr;
    const cudaLaunchConfig_t cfg = config_of(p, n, stream, &attr);
    return cudaLaunchKernelEx(&cfg, fn, a);
  });
}

}  // namespace xyk
