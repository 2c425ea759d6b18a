// xy_hmc.cu -- Hybrid Monte Carlo for the 2-d XY model (Sec. 1.2 of the
// paper): Gaussian momenta, the leap-frog integration of the equations of
// motion (the parallel core of the method) and the global Metropolis test.
//
//   H_hmc = sum_s p_s^2 / 2 + beta H(theta),  F_s = -beta J sum_nn sin(t_s - t_j)
//
// A trajectory of n_md steps is a chain of launches plus the test:
//   begin   draw p (Philox domain 3, Box-Muller), sums of (theta_0, p_0),
//           p += eps/2 F(theta_0), theta_1 = theta_0 + eps p
//   step    p += eps F(theta_k), theta_{k+1} = theta_k + eps p; on the tiled
//           path two such steps per launch (halo of two recomputed), one
//           single step for an odd remainder
//   final   p += eps/2 F(theta_n), sums of (theta_n, p_n)
//   accept  one thread: dH from the exact fixed-point sums, u < exp(-dH)
// Three angle buffers: the state stays untouched in buffer `cur` (restored on
// rejection for free), the integration ping-pongs between the other two, and
// the accept kernel moves `cur` on the device, so trajectories replay as one
// captured graph with no host round trip.  Sums are formed per site in FP32
// and converted to 64-bit fixed point before any addition: exact, and the
// same for every launch shape (the tiled and per-site kernels agree bit for
// bit in angles, momenta and sums).
#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>
#include <string.h>

#include "xy_hmc_device.cuh"
#include "xy_internal.h"
#include "xy_tma.cuh"

namespace xyk {

namespace {

using namespace xyh;

// ---------------------------------------------------------------------------
// Tiled kernel: a CTA of 256 threads owns 32 rows x 128 columns; a thread owns
// 4 rows x 4 columns (one float4 per row).  Horizontal neighbours come from
// the neighbouring lanes by shuffle (the warp's edge lanes read the tile's
// halo columns from shared memory); vertical neighbours from the thread's own
// rows, or from the edge rows that every warp leaves in shared memory (the
// tile's halo rows included).  Halo unit vectors are recomputed, not exchanged.
// ---------------------------------------------------------------------------
constexpr int kTileRows = 32;
constexpr int kTileCols = 128;
constexpr int kTileThreads = 256;
constexpr int kTileWarps = kTileThreads / 32;
constexpr int kRowsPerThread = kTileRows / kTileWarps;   // 4

template <int MODE, int KIND>
__global__ void __launch_bounds__(kTileThreads, KIND == kHmcStep ? 3 : 2) k_hmc_tile(HmcArgs a) {
  // cos / sin of tile rows -1 .. 32 (index row + 1); only each warp's first and
  // last row and the two halo rows are written and read
  __shared__ __align__(16) float sh_c[kTileRows + 2][kTileCols];
  __shared__ __align__(16) float sh_s[kTileRows + 2][kTileCols];
  __shared__ float side_c[2][kTileRows];   // [0] column -1, [1] column 128
  __shared__ float side_s[2][kTileRows];
  __shared__ long long red[kTileWarps][kHmcSums];

  const int L = a.L;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int x0 = blockIdx.x * kTileCols, y0 = blockIdx.y * kTileRows;
  const uint32_t cur = a.ctl->cur;
  int src, dst;
  hmc_buffers(a, cur, &src, &dst);
  const float* __restrict__ th_src = hmc_buf(a, src);

  // ---- loads: own 4 x 4 block, then halo sites ---------------------------
  const int xb = x0 + 4 * lane;
  const int yb = y0 + kRowsPerThread * warp;
  float4 t4[kRowsPerThread], p4[kRowsPerThread];
#pragma unroll
  for (int r = 0; r < kRowsPerThread; ++r)
    t4[r] = *reinterpret_cast<const float4*>(th_src + (size_t)(yb + r) * L + xb);
  if (KIND != kHmcBeginDraw) {
#pragma unroll
    for (int r = 0; r < kRowsPerThread; ++r)
      p4[r] = *reinterpret_cast<const float4*>(a.p_in + (size_t)(yb + r) * L + xb);
  }
  // halo: threads 0..127 row y0-1, 128..255 row y0+32; threads 0..31 column
  // x0-1 and 32..63 column x0+128 (rows y0..y0+31)
  const int tid = threadIdx.x;
  const int hy = tid < kTileCols ? (y0 == 0 ? L - 1 : y0 - 1)
                                 : (y0 + kTileRows == L ? 0 : y0 + kTileRows);
  const int hx = x0 + (tid & (kTileCols - 1));
  const float th_row = th_src[(size_t)hy * L + hx];
  float th_side = 0.f;
  const bool side = tid < 64;
  if (side) {
    const int sx = tid < 32 ? (x0 == 0 ? L - 1 : x0 - 1) : (x0 + kTileCols == L ? 0 : x0 + kTileCols);
    th_side = th_src[(size_t)(y0 + (tid & 31)) * L + sx];
  }

  // ---- momenta of the trajectory (begin with draw) -------------------------
  if (KIND == kHmcBeginDraw) {
    const uint32_t traj = (uint32_t)a.ctl->traj;
#pragma unroll
    for (int r = 0; r < kRowsPerThread; ++r) {
      const uint32_t s0 = (uint32_t)(yb + r) * (uint32_t)L + (uint32_t)xb;
      p4[r].x = hmc_momentum(s0 + 0u, traj, a.lattice_id, a.rk);
      p4[r].y = hmc_momentum(s0 + 1u, traj, a.lattice_id, a.rk);
      p4[r].z = hmc_momentum(s0 + 2u, traj, a.lattice_id, a.rk);
      p4[r].w = hmc_momentum(s0 + 3u, traj, a.lattice_id, a.rk);
    }
  }

  // ---- unit vectors -------------------------------------------------------
  float c[kRowsPerThread][4], s[kRowsPerThread][4];
#pragma unroll
  for (int r = 0; r < kRowsPerThread; ++r) {
    xyd::unit_vector<MODE>(t4[r].x, &s[r][0], &c[r][0]);
    xyd::unit_vector<MODE>(t4[r].y, &s[r][1], &c[r][1]);
    xyd::unit_vector<MODE>(t4[r].z, &s[r][2], &c[r][2]);
    xyd::unit_vector<MODE>(t4[r].w, &s[r][3], &c[r][3]);
  }
  {
    float hs, hc;
    xyd::unit_vector<MODE>(th_row, &hs, &hc);
    const int row = tid < kTileCols ? 0 : kTileRows + 1;
    sh_c[row][tid & (kTileCols - 1)] = hc;
    sh_s[row][tid & (kTileCols - 1)] = hs;
    if (side) {
      xyd::unit_vector<MODE>(th_side, &hs, &hc);
      side_c[tid >> 5][tid & 31] = hc;
      side_s[tid >> 5][tid & 31] = hs;
    }
  }
  // first and last row of this warp's band
  {
    const int rf = kRowsPerThread * warp + 1, rl = kRowsPerThread * warp + kRowsPerThread;
    *reinterpret_cast<float4*>(&sh_c[rf][4 * lane]) = make_float4(c[0][0], c[0][1], c[0][2], c[0][3]);
    *reinterpret_cast<float4*>(&sh_s[rf][4 * lane]) = make_float4(s[0][0], s[0][1], s[0][2], s[0][3]);
    *reinterpret_cast<float4*>(&sh_c[rl][4 * lane]) = make_float4(c[3][0], c[3][1], c[3][2], c[3][3]);
    *reinterpret_cast<float4*>(&sh_s[rl][4 * lane]) = make_float4(s[3][0], s[3][1], s[3][2], s[3][3]);
  }
  __syncthreads();

  // rows below (y - 1) and above (y + 4) the band
  const int rb = kRowsPerThread * warp;                  // index of row yb - 1
  const int ra = kRowsPerThread * warp + kRowsPerThread + 1;   // index of row yb + 4
  const float4 cdn = *reinterpret_cast<const float4*>(&sh_c[rb][4 * lane]);
  const float4 sdn = *reinterpret_cast<const float4*>(&sh_s[rb][4 * lane]);
  const float4 cup = *reinterpret_cast<const float4*>(&sh_c[ra][4 * lane]);
  const float4 sup = *reinterpret_cast<const float4*>(&sh_s[ra][4 * lane]);
  const float cdn_a[4] = {cdn.x, cdn.y, cdn.z, cdn.w}, sdn_a[4] = {sdn.x, sdn.y, sdn.z, sdn.w};
  const float cup_a[4] = {cup.x, cup.y, cup.z, cup.w}, sup_a[4] = {sup.x, sup.y, sup.z, sup.w};

  HmcAcc acc;
  acc_zero(acc);
  float4 tn[kRowsPerThread];
#pragma unroll
  for (int r = 0; r < kRowsPerThread; ++r) {
    // horizontal neighbours of the row's first and last column
    float cl = __shfl_up_sync(0xffffffffu, c[r][3], 1);
    float sl = __shfl_up_sync(0xffffffffu, s[r][3], 1);
    float cr = __shfl_down_sync(0xffffffffu, c[r][0], 1);
    float sr = __shfl_down_sync(0xffffffffu, s[r][0], 1);
    const int row = kRowsPerThread * warp + r;
    if (lane == 0) {
      cl = side_c[0][row];
      sl = side_s[0][row];
    }
    if (lane == 31) {
      cr = side_c[1][row];
      sr = side_s[1][row];
    }
    float pr[4] = {p4[r].x, p4[r].y, p4[r].z, p4[r].w};
    const float tr[4] = {t4[r].x, t4[r].y, t4[r].z, t4[r].w};
    float out[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float nlc = j == 0 ? cl : c[r][j - 1], nls = j == 0 ? sl : s[r][j - 1];
      const float nrc = j == 3 ? cr : c[r][j + 1], nrs = j == 3 ? sr : s[r][j + 1];
      const float ndc = r == 0 ? cdn_a[j] : c[r - 1][j], nds = r == 0 ? sdn_a[j] : s[r - 1][j];
      const float nuc = r == kRowsPerThread - 1 ? cup_a[j] : c[r + 1][j];
      const float nus = r == kRowsPerThread - 1 ? sup_a[j] : s[r + 1][j];
      const float Sc = xyd::nb_sum(nlc, nrc, ndc, nuc);
      const float Ss = xyd::nb_sum(nls, nrs, nds, nus);
      const float F = hmc_force(c[r][j], s[r][j], Sc, Ss, a.K);
      if (KIND == kHmcBeginDraw || KIND == kHmcBeginRead)
        hmc_terms(pr[j], c[r][j], s[r][j], nrc, nrs, nuc, nus, acc);
      pr[j] = __fmaf_rn(a.a, F, pr[j]);
      if (KIND == kHmcFinal) {
        hmc_terms(pr[j], c[r][j], s[r][j], nrc, nrs, nuc, nus, acc);
        out[j] = tr[j];
      } else {
        out[j] = hmc_wrap(__fmaf_rn(a.eps, pr[j], tr[j]));
      }
    }
    p4[r] = make_float4(pr[0], pr[1], pr[2], pr[3]);
    tn[r] = make_float4(out[0], out[1], out[2], out[3]);
  }

  // ---- stores -------------------------------------------------------------
#pragma unroll
  for (int r = 0; r < kRowsPerThread; ++r)
    *reinterpret_cast<float4*>(a.p_out + (size_t)(yb + r) * L + xb) = p4[r];
  if (KIND != kHmcFinal) {
    float* __restrict__ th_dst = hmc_buf(a, dst);
#pragma unroll
    for (int r = 0; r < kRowsPerThread; ++r)
      *reinterpret_cast<float4*>(th_dst + (size_t)(yb + r) * L + xb) = tn[r];
  }
  if (KIND == kHmcBeginDraw || KIND == kHmcBeginRead)
    hmc_commit<kTileWarps>(acc, a.ctl->acc[0], red);
  if (KIND == kHmcFinal) hmc_commit<kTileWarps>(acc, a.ctl->acc[1], red);
}

// ---------------------------------------------------------------------------
// Persistent TMA step kernel: the same step as k_hmc_tile<MODE, kHmcStep>, but
// a grid of about two CTAs per SM walks the tiles, and each CTA streams its
// next tiles' angles and momenta (two 32 x 128 boxes, 32 KB) into a
// double-buffered shared-memory stage with cp.async.bulk.tensor, completing on
// an mbarrier, while it computes the current tile.  The one-site halo (320
// floats) is read with plain loads issued before the wait.  Every wait is
// bounded: each thread polls the stage's barrier a fixed number of times; a
// thread that runs out flags HmcCtl::error and stops computing but keeps
// meeting the CTA's barriers, and thread 0 then issues no more loads and
// drains the ones in flight before the CTA exits.
// ---------------------------------------------------------------------------
// ROWS rows per thread: tiles of 8 ROWS x 128 sites.  ROWS = 4 (the tile of
// k_hmc_tile, two CTAs per SM) is the one launched: 16 x 128 tiles at four
// CTAs per SM measured slower (57.4 against 54.1 us per step at L = 4096; the
// halo grows from 8 % to 14 % of the sincos work and occupancy was not the
// limit).
template <int ROWS>
struct TmaGeom {
  static constexpr int kRows = 8 * ROWS;                               // tile rows
  static constexpr int kBox = kRows * kTileCols;                       // floats per box
  static constexpr uint32_t kStageBytes = 2u * kBox * sizeof(float);  // angles + momenta
  static constexpr size_t kSmem = 2 * (size_t)kStageBytes;             // two stages
  static constexpr int kMinBlocks = ROWS == 4 ? 2 : 4;
};
constexpr long long kSpinLimit = 1ll << 22;

template <int MODE, int ROWS>
__global__ void __launch_bounds__(kTileThreads, TmaGeom<ROWS>::kMinBlocks)
    k_hmc_step_tma(const __grid_constant__ CUtensorMap map0, const __grid_constant__ CUtensorMap map1,
                   const __grid_constant__ CUtensorMap map2, const __grid_constant__ CUtensorMap mapp,
                   HmcArgs a, int tiles_x, int n_tiles) {
  using G = TmaGeom<ROWS>;
  constexpr int TR = G::kRows;
  constexpr uint32_t kTmaStageBytes = G::kStageBytes;
  constexpr int kTmaBox = G::kBox;
  extern __shared__ __align__(128) unsigned char tma_smem[];
  // unit vectors (cos and sin planes) of the rows other warps read,
  // double-buffered by tile parity: lastrow[b][w + 1] = last row of warp w
  // (lastrow[b][0]: the halo row above the tile), firstrow[b][w] = first row of
  // warp w (firstrow[b][kTileWarps]: the halo row below); plus the halo columns
  __shared__ __align__(16) float lastrow_c[2][kTileWarps + 1][kTileCols];
  __shared__ __align__(16) float lastrow_s[2][kTileWarps + 1][kTileCols];
  __shared__ __align__(16) float firstrow_c[2][kTileWarps + 1][kTileCols];
  __shared__ __align__(16) float firstrow_s[2][kTileWarps + 1][kTileCols];
  __shared__ float2 side[2][2][TR];
  __shared__ __align__(8) uint64_t bar[2];

  const int L = a.L;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int src, dst;
  hmc_buffers(a, a.ctl->cur, &src, &dst);
  const CUtensorMap* mth = src == 0 ? &map0 : (src == 1 ? &map1 : &map2);
  const float* __restrict__ th_src = hmc_buf(a, src);
  float* __restrict__ th_dst = hmc_buf(a, dst);
  // stage s: angles [TR][128] then momenta [TR][128]
  auto stage_th = [&](int s) {
    return reinterpret_cast<float (*)[kTileCols]>(tma_smem + s * kTmaStageBytes);
  };
  auto stage_p = [&](int s) {
    return reinterpret_cast<float (*)[kTileCols]>(tma_smem + s * kTmaStageBytes +
                                                 kTmaBox * sizeof(float));
  };
  // Consecutive steps (buffer offsets 1, 2, 1, ...) walk the tiles in
  // opposite orders, so a step starts with the tiles the launch before it
  // wrote last, which are still in L2.  Every tile reads only the source
  // buffer and its own momenta, so the order changes no result.
  const bool rev = (a.src_off & 1) != 0;
  auto tile_at = [&](int t) { return rev ? n_tiles - 1 - t : t; };
  // thread 0's count of loads issued per stage (for the drain on a timeout)
  int issued[2] = {0, 0};
  auto issue = [&](int t, int s) {
    const int tt = tile_at(t);
    const int x0 = (tt % tiles_x) * kTileCols, y0 = (tt / tiles_x) * TR;
    xyt::mbar_arrive_expect_tx(&bar[s], kTmaStageBytes);
    xyt::tma_load_2d(stage_th(s), mth, x0, y0, &bar[s]);
    xyt::tma_load_2d(stage_p(s), &mapp, x0, y0, &bar[s]);
    ++issued[s];
  };
  auto bounded_wait = [&](int s, uint32_t parity) {
    return xyt::mbar_wait_bounded(&bar[s], parity, kSpinLimit);
  };

  if (tid == 0) {
    xyt::mbar_init(&bar[0], 1);
    xyt::mbar_init(&bar[1], 1);
    xyt::fence_mbarrier_init();
    xyt::fence_async_shared();
    for (int s = 0; s < 2; ++s) {
      const int t = blockIdx.x + s * gridDim.x;
      if (t < n_tiles) issue(t, s);
    }
  }
  __syncthreads();

  // A thread whose wait runs out flags the error and stops computing, but
  // keeps meeting the CTA's barriers (so no thread waits on one that left);
  // thread 0 then issues no more loads and drains the ones in flight.
  bool ok = true;
  int it = 0;
  for (int t = blockIdx.x; t < n_tiles; t += gridDim.x, ++it) {
    const int s = it & 1, b = it & 1;
    const uint32_t parity = (uint32_t)((it >> 1) & 1);
    const int tt = tile_at(t);
    const int x0 = (tt % tiles_x) * kTileCols, y0 = (tt / tiles_x) * TR;
    // halo loads first: rows y0-1, y0+TR (threads 0..127 / 128..255), columns
    // x0-1 and x0+128 (threads 0..TR-1 / TR..2TR-1)
    const int hy = tid < kTileCols ? (y0 == 0 ? L - 1 : y0 - 1) : (y0 + TR == L ? 0 : y0 + TR);
    const float th_row = th_src[(size_t)hy * L + x0 + (tid & (kTileCols - 1))];
    float th_side = 0.f;
    const bool is_side = tid < 2 * TR;
    if (is_side) {
      const int sx = tid < TR ? (x0 == 0 ? L - 1 : x0 - 1) : (x0 + kTileCols == L ? 0 : x0 + kTileCols);
      th_side = th_src[(size_t)(y0 + (tid % TR)) * L + sx];
    }
    if (ok && !bounded_wait(s, parity)) {
      ok = false;
      atomicOr(&a.ctl->error, 1u);
    }

    const int xb = 4 * lane, rb0 = ROWS * warp;
    float4 t4[ROWS], p4[ROWS];
    float c[ROWS][4], sn[ROWS][4];
    if (ok) {
      float (*sth)[kTileCols] = stage_th(s);
      float (*sp)[kTileCols] = stage_p(s);
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        t4[r] = *reinterpret_cast<const float4*>(&sth[rb0 + r][xb]);
        p4[r] = *reinterpret_cast<const float4*>(&sp[rb0 + r][xb]);
      }
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        xyd::unit_vector<MODE>(t4[r].x, &sn[r][0], &c[r][0]);
        xyd::unit_vector<MODE>(t4[r].y, &sn[r][1], &c[r][1]);
        xyd::unit_vector<MODE>(t4[r].z, &sn[r][2], &c[r][2]);
        xyd::unit_vector<MODE>(t4[r].w, &sn[r][3], &c[r][3]);
      }
      float hs, hc;
      xyd::unit_vector<MODE>(th_row, &hs, &hc);
      if (tid < kTileCols) {
        lastrow_c[b][0][tid] = hc;
        lastrow_s[b][0][tid] = hs;
      } else {
        firstrow_c[b][kTileWarps][tid - kTileCols] = hc;
        firstrow_s[b][kTileWarps][tid - kTileCols] = hs;
      }
      if (is_side) {
        xyd::unit_vector<MODE>(th_side, &hs, &hc);
        side[b][tid / TR][tid % TR] = make_float2(hc, hs);
      }
      *reinterpret_cast<float4*>(&firstrow_c[b][warp][xb]) = make_float4(c[0][0], c[0][1], c[0][2], c[0][3]);
      *reinterpret_cast<float4*>(&firstrow_s[b][warp][xb]) =
          make_float4(sn[0][0], sn[0][1], sn[0][2], sn[0][3]);
      *reinterpret_cast<float4*>(&lastrow_c[b][warp + 1][xb]) =
          make_float4(c[ROWS - 1][0], c[ROWS - 1][1], c[ROWS - 1][2], c[ROWS - 1][3]);
      *reinterpret_cast<float4*>(&lastrow_s[b][warp + 1][xb]) =
          make_float4(sn[ROWS - 1][0], sn[ROWS - 1][1], sn[ROWS - 1][2], sn[ROWS - 1][3]);
    }
    __syncthreads();   // stage s fully read; edges visible
    if (tid == 0 && ok) {
      const int tn = t + 2 * gridDim.x;
      if (tn < n_tiles) {
        xyt::fence_async_shared();
        issue(tn, s);
      }
    }
    if (!ok) continue;

    const float4 cdn = *reinterpret_cast<const float4*>(&lastrow_c[b][warp][xb]);
    const float4 sdn = *reinterpret_cast<const float4*>(&lastrow_s[b][warp][xb]);
    const float4 cup = *reinterpret_cast<const float4*>(&firstrow_c[b][warp + 1][xb]);
    const float4 sup = *reinterpret_cast<const float4*>(&firstrow_s[b][warp + 1][xb]);
    const float cdn_a[4] = {cdn.x, cdn.y, cdn.z, cdn.w}, sdn_a[4] = {sdn.x, sdn.y, sdn.z, sdn.w};
    const float cup_a[4] = {cup.x, cup.y, cup.z, cup.w}, sup_a[4] = {sup.x, sup.y, sup.z, sup.w};
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      float cl = __shfl_up_sync(0xffffffffu, c[r][3], 1);
      float sl = __shfl_up_sync(0xffffffffu, sn[r][3], 1);
      float cr = __shfl_down_sync(0xffffffffu, c[r][0], 1);
      float sr = __shfl_down_sync(0xffffffffu, sn[r][0], 1);
      const int row = rb0 + r;
      if (lane == 0) {
        const float2 v = side[b][0][row];
        cl = v.x;
        sl = v.y;
      }
      if (lane == 31) {
        const float2 v = side[b][1][row];
        cr = v.x;
        sr = v.y;
      }
      float pr[4] = {p4[r].x, p4[r].y, p4[r].z, p4[r].w};
      const float tr[4] = {t4[r].x, t4[r].y, t4[r].z, t4[r].w};
      float out[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float nlc = j == 0 ? cl : c[r][j - 1], nls = j == 0 ? sl : sn[r][j - 1];
        const float nrc = j == 3 ? cr : c[r][j + 1], nrs = j == 3 ? sr : sn[r][j + 1];
        const float ndc = r == 0 ? cdn_a[j] : c[r - 1][j], nds = r == 0 ? sdn_a[j] : sn[r - 1][j];
        const float nuc = r == ROWS - 1 ? cup_a[j] : c[r + 1][j];
        const float nus = r == ROWS - 1 ? sup_a[j] : sn[r + 1][j];
        const float Sc = xyd::nb_sum(nlc, nrc, ndc, nuc);
        const float Ss = xyd::nb_sum(nls, nrs, nds, nus);
        pr[j] = __fmaf_rn(a.a, hmc_force(c[r][j], sn[r][j], Sc, Ss, a.K), pr[j]);
        out[j] = hmc_wrap(__fmaf_rn(a.eps, pr[j], tr[j]));
      }
      const size_t g = (size_t)(y0 + row) * L + x0 + xb;
      *reinterpret_cast<float4*>(a.p_out + g) = make_float4(pr[0], pr[1], pr[2], pr[3]);
      *reinterpret_cast<float4*>(th_dst + g) = make_float4(out[0], out[1], out[2], out[3]);
    }
  }
  // loads still in flight after a timeout land in this CTA's shared memory:
  // wait for them (bounded) before the CTA exits
  if (tid == 0 && !ok) {
    for (int q = 0; q < 2; ++q)
      if (issued[q] > 0) (void)bounded_wait(q, (uint32_t)((issued[q] - 1) & 1));
  }
}

// ---------------------------------------------------------------------------
// All kick-drift steps of a trajectory in one cooperative launch (every CTA
// resident).  The work items (step j, tile) are ordered step-major, with the
// tile rows of a step visited folded (0, T-1, 1, T-2, ...) so that a tile's
// periodic neighbours are never more than two tile rows apart in that order;
// iteration i of CTA b takes item b + i * gridDim.x, so every CTA gets the
// same number of tiles to within one over the whole trajectory.  Step j of a
// tile reads the angles of the tile and of its one-site halo after step j - 1
// (its eight neighbours), its own momenta (updated in place by its step j - 1,
// which may have run on another CTA) and overwrites the angle buffer those
// nine tiles read during step j - 1, so it starts once the nine have published
// flags >= j.  A tile is published (j + 1) after the next tile's first CTA
// barrier, when its stores have long landed and the fence is cheap, or before
// that tile waits; either way without waiting on anything else.  Thread 0
// streams the next-but-one tile's angle and momentum boxes into the free TMA
// stage once that item's nine counters are found set (relaxed loads issued
// when the stage frees, looked at once the current tile is computed, then an
// acquire fence; at large L they are always set); otherwise the load is
// issued at the item's own turn, after a bounded wait.  Every wait is bounded
// (counters and stage barriers); a wait that runs out sets HmcCtl::error, the
// CTA drains its loads in flight (bounded) and ends, and CTAs waiting on it see
// the error word and end too.  Items wait only on items of the step before,
// and a finished item is published without waiting, so with every CTA
// resident every wait ends.  Per tile the arithmetic is k_hmc_step_tma's, so
// the trajectory is bit for bit that of one step launch per step.
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned int hmc_load_acquire(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ unsigned int hmc_load_relaxed(const unsigned int* p) {
  unsigned int v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void fence_acq_rel_gpu() {
  asm volatile("fence.acq_rel.gpu;" ::: "memory");
}

__device__ __forceinline__ void hmc_store_release(unsigned int* p, unsigned int v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}


__device__ __forceinline__ int hmc_wrap_tile(int v, int n) {
  v += (v < 0) ? n : 0;
  v -= (v >= n) ? n : 0;
  return v;
}

template <int MODE>
__global__ void __launch_bounds__(kTileThreads, TmaGeom<4>::kMinBlocks)
    k_hmc_steps_persist(const __grid_constant__ CUtensorMap map0,
                        const __grid_constant__ CUtensorMap map1,
                        const __grid_constant__ CUtensorMap map2,
                        const __grid_constant__ CUtensorMap mapp, HmcStepsArgs q, int tiles_x,
                        int n_tiles) {
  using G = TmaGeom<4>;
  constexpr int ROWS = 4;
  constexpr int TR = G::kRows;
  constexpr uint32_t kTmaStageBytes = G::kStageBytes;
  constexpr int kTmaBox = G::kBox;
  constexpr int kPublisher = kTileThreads - 32;   // lane 0 of the last warp
  extern __shared__ __align__(128) unsigned char tma_smem[];
  __shared__ __align__(16) float lastrow_c[2][kTileWarps + 1][kTileCols];
  __shared__ __align__(16) float lastrow_s[2][kTileWarps + 1][kTileCols];
  __shared__ __align__(16) float firstrow_c[2][kTileWarps + 1][kTileCols];
  __shared__ __align__(16) float firstrow_s[2][kTileWarps + 1][kTileCols];
  __shared__ float2 side[2][2][TR];
  __shared__ __align__(8) uint64_t bar[2];
  __shared__ int s_issued[2];        // the stage's load for its next item is in flight
  __shared__ int s_abort;

  const HmcArgs& a = q.a;
  const int L = a.L;
  const int tiles_y = L / TR;
  const int total = q.n_steps * n_tiles;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t cur = a.ctl->cur;
  auto stage_th = [&](int s) {
    return reinterpret_cast<float (*)[kTileCols]>(tma_smem + s * kTmaStageBytes);
  };
  auto stage_p = [&](int s) {
    return reinterpret_cast<float (*)[kTileCols]>(tma_smem + s * kTmaStageBytes +
                                                 kTmaBox * sizeof(float));
  };
  // item -> (step, tile x, tile y); iteration it of this CTA takes item
  // blockIdx.x + it * gridDim.x
  auto decode = [&](int item, int* j, int* tx, int* ty) {
    *j = item / n_tiles;
    const int k = item - *j * n_tiles;
    const int prow = k / tiles_x;
    *tx = k - prow * tiles_x;
    *ty = (prow & 1) ? tiles_y - 1 - (prow >> 1) : (prow >> 1);
  };
  // angle buffers of step j: read (cur + 1 or 2), written (cur + 2 or 1)
  auto src_of = [&](int j) { return (int)((cur + (j & 1 ? 2u : 1u)) % 3u); };
  auto dst_of = [&](int j) { return (int)((cur + (j & 1 ? 1u : 2u)) % 3u); };
  int issued[2] = {0, 0};            // thread 0: loads issued per stage (for the drain)
  auto issue = [&](int item, int s) {
    int j, tx, ty;
    decode(item, &j, &tx, &ty);
    const int sb = src_of(j);
    const CUtensorMap* mth = sb == 0 ? &map0 : (sb == 1 ? &map1 : &map2);
    xyt::fence_proxy_async_global();
    xyt::mbar_arrive_expect_tx(&bar[s], kTmaStageBytes);
    xyt::tma_load_2d(stage_th(s), mth, tx * kTileCols, ty * TR, &bar[s]);
    xyt::tma_load_2d(stage_p(s), &mapp, tx * kTileCols, ty * TR, &bar[s]);
    ++issued[s];
  };
  auto drain = [&]() {
    if (tid == 0)
      for (int s = 0; s < 2; ++s)
        if (issued[s] > 0) (void)xyt::mbar_wait_bounded(&bar[s], (uint32_t)((issued[s] - 1) & 1),
                                                   q.spin_limit);
  };
  // the previous tile, stored but not yet published (its counter slot and value)
  int pend_slot = -1;
  unsigned int pend_val = 0;
  // publish it: the caller has passed a CTA barrier after every thread's stores
  // of that tile; the GPU-scope release is cumulative over them
  auto publish = [&]() {
    if (tid == kPublisher && pend_slot >= 0) hmc_store_release(q.flags + pend_slot, pend_val);
    pend_slot = -1;
  };

  if (tid == 0) {
    s_abort = 0;
    xyt::mbar_init(&bar[0], 1);
    xyt::mbar_init(&bar[1], 1);
    xyt::fence_mbarrier_init();
    xyt::fence_async_shared();
    for (int s = 0; s < 2; ++s) {
      const int item = blockIdx.x + s * gridDim.x;
      s_issued[s] = 0;
      int j, tx, ty;
      if (item < total) {
        decode(item, &j, &tx, &ty);
        if (j == 0) {            // the first step reads the begin launch's output
          issue(item, s);
          s_issued[s] = 1;
        }
      }
    }
  }
  __syncthreads();

  for (int it = 0;; ++it) {
    const int item = blockIdx.x + it * gridDim.x;
    if (item >= total) break;
    const int s = it & 1, b = it & 1;
    const uint32_t parity = (uint32_t)((it >> 1) & 1);
    int j, tx, ty;
    decode(item, &j, &tx, &ty);
    const int x0 = tx * kTileCols, y0 = ty * TR;

    if (!s_issued[s]) {
      // its load was not issued ahead: publish the previous tile (this wait may
      // be for it), wait for the nine counters, then load
      __syncthreads();
      publish();
      if (j > 0 && tid < 9) {
        const int nx = hmc_wrap_tile(tx + tid % 3 - 1, tiles_x);
        const int ny = hmc_wrap_tile(ty + tid / 3 - 1, tiles_y);
        const unsigned int* f = q.flags + (ny * tiles_x + nx);
        long long n = 0;
        while (hmc_load_acquire(f) < (unsigned int)j) {
          if (++n > q.spin_limit ||
              ((n & 255) == 0 && *reinterpret_cast<volatile unsigned int*>(&a.ctl->error) != 0u)) {
            atomicOr(&a.ctl->error, 1u);
            s_abort = 1;
            break;
          }
          __nanosleep(128);
        }
      }
      __syncthreads();
      if (s_abort) {
        drain();
        return;
      }
      if (tid == 0) issue(item, s);
    }

    const float* __restrict__ th_src = hmc_buf(a, src_of(j));
    float* __restrict__ th_dst = hmc_buf(a, dst_of(j));
    // halo: rows y0-1, y0+TR (threads 0..127 / 128..255), columns x0-1 and
    // x0+128 (threads 0..TR-1 / TR..2TR-1), through L2 (written in this launch)
    const int hy = tid < kTileCols ? (y0 == 0 ? L - 1 : y0 - 1) : (y0 + TR == L ? 0 : y0 + TR);
    const float th_row = __ldcg(th_src + (size_t)hy * L + x0 + (tid & (kTileCols - 1)));
    float th_side = 0.f;
    const bool is_side = tid < 2 * TR;
    if (is_side) {
      const int sx = tid < TR ? (x0 == 0 ? L - 1 : x0 - 1) : (x0 + kTileCols == L ? 0 : x0 + kTileCols);
      th_side = __ldcg(th_src + (size_t)(y0 + (tid % TR)) * L + sx);
    }
    if (!xyt::mbar_wait_bounded(&bar[s], parity, q.spin_limit)) {
      atomicOr(&a.ctl->error, 1u);
      s_abort = 1;
    }

    const int xb = 4 * lane, rb0 = ROWS * warp;
    float4 t4[ROWS], p4[ROWS];
    float c[ROWS][4], sn[ROWS][4];
    {
      float (*sth)[kTileCols] = stage_th(s);
      float (*sp)[kTileCols] = stage_p(s);
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        t4[r] = *reinterpret_cast<const float4*>(&sth[rb0 + r][xb]);
        p4[r] = *reinterpret_cast<const float4*>(&sp[rb0 + r][xb]);
      }
#pragma unroll
      for (int r = 0; r < ROWS; ++r) {
        xyd::unit_vector<MODE>(t4[r].x, &sn[r][0], &c[r][0]);
        xyd::unit_vector<MODE>(t4[r].y, &sn[r][1], &c[r][1]);
        xyd::unit_vector<MODE>(t4[r].z, &sn[r][2], &c[r][2]);
        xyd::unit_vector<MODE>(t4[r].w, &sn[r][3], &c[r][3]);
      }
      float hs, hc;
      xyd::unit_vector<MODE>(th_row, &hs, &hc);
      if (tid < kTileCols) {
        lastrow_c[b][0][tid] = hc;
        lastrow_s[b][0][tid] = hs;
      } else {
        firstrow_c[b][kTileWarps][tid - kTileCols] = hc;
        firstrow_s[b][kTileWarps][tid - kTileCols] = hs;
      }
      if (is_side) {
        xyd::unit_vector<MODE>(th_side, &hs, &hc);
        side[b][tid / TR][tid % TR] = make_float2(hc, hs);
      }
      *reinterpret_cast<float4*>(&firstrow_c[b][warp][xb]) = make_float4(c[0][0], c[0][1], c[0][2], c[0][3]);
      *reinterpret_cast<float4*>(&firstrow_s[b][warp][xb]) =
          make_float4(sn[0][0], sn[0][1], sn[0][2], sn[0][3]);
      *reinterpret_cast<float4*>(&lastrow_c[b][warp + 1][xb]) =
          make_float4(c[ROWS - 1][0], c[ROWS - 1][1], c[ROWS - 1][2], c[ROWS - 1][3]);
      *reinterpret_cast<float4*>(&lastrow_s[b][warp + 1][xb]) =
          make_float4(sn[ROWS - 1][0], sn[ROWS - 1][1], sn[ROWS - 1][2], sn[ROWS - 1][3]);
    }
    __syncthreads();   // stage s fully read; edges visible; the previous tile's stores done
    if (s_abort) {
      drain();
      return;
    }
    publish();
    // the item after next: its nine counters are loaded now (relaxed, all in
    // flight together) and looked at once this tile is computed
    const int next = item + 2 * gridDim.x;
    unsigned int fl[9];
    int nj = 0;
    if (tid == 0) {
      s_issued[s] = 0;
      if (next < total) {
        int ntx, nty;
        decode(next, &nj, &ntx, &nty);
        if (nj > 0) {
#pragma unroll
          for (int d = 0; d < 9; ++d) {
            const int nx = hmc_wrap_tile(ntx + d % 3 - 1, tiles_x);
            const int ny = hmc_wrap_tile(nty + d / 3 - 1, tiles_y);
            fl[d] = hmc_load_relaxed(q.flags + (ny * tiles_x + nx));
          }
        }
      }
    }

    const float4 cdn = *reinterpret_cast<const float4*>(&lastrow_c[b][warp][xb]);
    const float4 sdn = *reinterpret_cast<const float4*>(&lastrow_s[b][warp][xb]);
    const float4 cup = *reinterpret_cast<const float4*>(&firstrow_c[b][warp + 1][xb]);
    const float4 sup = *reinterpret_cast<const float4*>(&firstrow_s[b][warp + 1][xb]);
    const float cdn_a[4] = {cdn.x, cdn.y, cdn.z, cdn.w}, sdn_a[4] = {sdn.x, sdn.y, sdn.z, sdn.w};
    const float cup_a[4] = {cup.x, cup.y, cup.z, cup.w}, sup_a[4] = {sup.x, sup.y, sup.z, sup.w};
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      float cl = __shfl_up_sync(0xffffffffu, c[r][3], 1);
      float sl = __shfl_up_sync(0xffffffffu, sn[r][3], 1);
      float cr = __shfl_down_sync(0xffffffffu, c[r][0], 1);
      float sr = __shfl_down_sync(0xffffffffu, sn[r][0], 1);
      const int row = rb0 + r;
      if (lane == 0) {
        const float2 v = side[b][0][row];
        cl = v.x;
        sl = v.y;
      }
      if (lane == 31) {
        const float2 v = side[b][1][row];
        cr = v.x;
        sr = v.y;
      }
      float pr[4] = {p4[r].x, p4[r].y, p4[r].z, p4[r].w};
      const float tr[4] = {t4[r].x, t4[r].y, t4[r].z, t4[r].w};
      float out[4];
#pragma unroll
      for (int jj = 0; jj < 4; ++jj) {
        const float nlc = jj == 0 ? cl : c[r][jj - 1], nls = jj == 0 ? sl : sn[r][jj - 1];
        const float nrc = jj == 3 ? cr : c[r][jj + 1], nrs = jj == 3 ? sr : sn[r][jj + 1];
        const float ndc = r == 0 ? cdn_a[jj] : c[r - 1][jj], nds = r == 0 ? sdn_a[jj] : sn[r - 1][jj];
        const float nuc = r == ROWS - 1 ? cup_a[jj] : c[r + 1][jj];
        const float nus = r == ROWS - 1 ? sup_a[jj] : sn[r + 1][jj];
        const float Sc = xyd::nb_sum(nlc, nrc, ndc, nuc);
        const float Ss = xyd::nb_sum(nls, nrs, nds, nus);
        pr[jj] = __fmaf_rn(a.a, hmc_force(c[r][jj], sn[r][jj], Sc, Ss, a.K), pr[jj]);
        out[jj] = hmc_wrap(__fmaf_rn(a.eps, pr[jj], tr[jj]));
      }
      p4[r] = make_float4(pr[0], pr[1], pr[2], pr[3]);
      t4[r] = make_float4(out[0], out[1], out[2], out[3]);
    }
    if (tid == 0 && next < total) {
      bool ready = true;
      if (nj > 0) {
#pragma unroll
        for (int d = 0; d < 9; ++d) ready = ready && fl[d] >= (unsigned int)nj;
      }
      if (ready) {
        // the relaxed loads saw every counter set: this acquire fence makes
        // the stores they publish visible to thread 0, and issue()'s proxy
        // fence to its TMA reads
        fence_acq_rel_gpu();
        xyt::fence_async_shared();
        issue(next, s);
        s_issued[s] = 1;
      }
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      const size_t g = (size_t)(y0 + rb0 + r) * L + x0 + xb;
      *reinterpret_cast<float4*>(a.p_out + g) = p4[r];
      *reinterpret_cast<float4*>(th_dst + g) = t4[r];
    }
    // published after the next tile's first barrier (its stores have landed
    // by then), or before that tile waits
    pend_slot = ty * tiles_x + tx;
    pend_val = (unsigned int)(j + 1);
  }
  __syncthreads();
  publish();
}

// ---------------------------------------------------------------------------
// Two full kick-drift steps per launch (temporal blocking).  A CTA of 256
// threads owns 32 rows x 128 columns, a thread 4 rows x 4 columns in
// registers as in k_hmc_tile.  The first step also updates the ring around
// the tile (rows -1 and 32, columns -1 and 128: 320 sites that belong to the
// neighbouring tiles, recomputed from the same inputs with the same
// arithmetic, so every copy agrees bit for bit); the second updates the tile
// and writes angles and momenta once: 8 bytes read and 8 written per site for
// two steps.  Shared memory holds one frame of unit vectors, rows -2 .. 33 and
// columns -4 .. 131 of the tile (cos and sin planes), of which only what
// crosses a warp is written: the halo of two (rows -2 and 33, columns -2 and
// 129, the four ring corners), the ring, each warp's first and last row and
// the tile's first and last column; after the first step the ring and the
// warps' edge rows are overwritten with their new values.  Horizontal
// neighbours inside a warp's rows come by shuffle.  Momenta are read from one
// buffer and written to another (the ring reads the neighbours' old momenta).
// ---------------------------------------------------------------------------
constexpr int kP2Rows = 32;
constexpr int kP2Cols = 128;
constexpr int kP2Threads = 256;
constexpr int kP2Warps = kP2Threads / 32;
constexpr int kP2Band = kP2Rows / kP2Warps;                  // 4 rows per warp
constexpr int kFrRows = kP2Rows + 4;                         // tile rows -2 .. 33
constexpr int kFrCols = kP2Cols + 8;                         // tile columns -4 .. 131
constexpr size_t kP2Smem = sizeof(float) * 2 * kFrRows * kFrCols;
__device__ __forceinline__ int wrap_near(int v, int n) { return v < 0 ? v + n : (v >= n ? v - n : v); }

// One leap-frog step of a site: kick by a F(unit vector, neighbour sums),
// drift by eps p, wrap (the per-site arithmetic of every HMC kernel).
__device__ __forceinline__ void hmc_site_step(float c, float s, float Sc, float Ss, float K,
                                              float a, float eps, float& p, float& t) {
  p = __fmaf_rn(a, hmc_force(c, s, Sc, Ss, K), p);
  t = hmc_wrap(__fmaf_rn(eps, p, t));
}

// The unit vectors of four adjacent sites as pairs of the even and of the odd
// ones, (c0, c2), (c1, c3): then an even pair's right neighbours are the odd
// pair and an odd pair's left neighbours the even one, as they stand in the
// registers, and of the packed sums' operands only (left lane's c3, c1) and
// (c2, right lane's c0) have to be put together.  The frame keeps its groups of
// four in the same order, frame_col(q) the place of column q.  46.7 issued
// instructions per site-step against 57.7 with scalar arithmetic; per unit
// trajectory L = 512 75.2 against 77.5 us, 1024 139 against 145, 2048 572
// against 610-648, 4096 3.20 against 3.21 ms (SFU sincos 2.67 against 2.84):
// the two CTAs of an SM wait on each other's barriers and on dependent packed
// instructions, not for issue slots or memory.  Measured and not kept: the
// wrap packed too (4096 3.25 ms), three CTAs per SM (140 bytes spilled, 512
// 94 us), consecutive launches walking the tiles in opposite orders (a tie),
// and the second step's stores after the band instead of row by row (4096
// 3.46 ms: the stores burst and stall the warp).
struct Quad4 {
  float2 cE, cO, sE, sO;
};

__device__ __forceinline__ int frame_col(int q) {
  return (q & ~3) | ((q & 1) << 1) | ((q >> 1) & 1);
}

template <int MODE>
__device__ __forceinline__ Quad4 quad_vectors(const float4& t) {
  float2 s01, c01, s23, c23;
  xyd::unit_vector2<MODE>(make_float2(t.x, t.y), &s01, &c01);
  xyd::unit_vector2<MODE>(make_float2(t.z, t.w), &s23, &c23);
  return Quad4{make_float2(c01.x, c23.x), make_float2(c01.y, c23.y), make_float2(s01.x, s23.x),
               make_float2(s01.y, s23.y)};
}

__device__ __forceinline__ void put_quad(float* c, float* s, const Quad4& v) {
  *reinterpret_cast<float4*>(c) = make_float4(v.cE.x, v.cE.y, v.cO.x, v.cO.y);
  *reinterpret_cast<float4*>(s) = make_float4(v.sE.x, v.sE.y, v.sO.x, v.sO.y);
}

__device__ __forceinline__ Quad4 get_quad(const float* c, const float* s) {
  const float4 a = *reinterpret_cast<const float4*>(c), b = *reinterpret_cast<const float4*>(s);
  return Quad4{make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y),
               make_float2(b.z, b.w)};
}

// One leap-frog step of four adjacent sites `o` (angles t, momenta p) with the
// rows below and above and the neighbouring lanes' sites (cl, sl), (cr, sr).
__device__ __forceinline__ void quad_step(const Quad4& o, const Quad4& dn, const Quad4& up,
                                          float cl, float sl, float cr, float sr, float K, float a,
                                          float eps, float4& p, float4& t) {
  using xyd::add2;
  const float2 ScE = add2(add2(make_float2(cl, o.cO.x), o.cO), add2(dn.cE, up.cE));
  const float2 SsE = add2(add2(make_float2(sl, o.sO.x), o.sO), add2(dn.sE, up.sE));
  const float2 ScO = add2(add2(o.cE, make_float2(o.cE.y, cr)), add2(dn.cO, up.cO));
  const float2 SsO = add2(add2(o.sE, make_float2(o.sE.y, sr)), add2(dn.sO, up.sO));
  const float2 FE = hmc_force2(o.cE, o.sE, ScE, SsE, K);
  const float2 FO = hmc_force2(o.cO, o.sO, ScO, SsO, K);
  p = make_float4(__fmaf_rn(a, FE.x, p.x), __fmaf_rn(a, FO.x, p.y), __fmaf_rn(a, FE.y, p.z),
                  __fmaf_rn(a, FO.y, p.w));
  t = make_float4(hmc_wrap(__fmaf_rn(eps, p.x, t.x)), hmc_wrap(__fmaf_rn(eps, p.y, t.y)),
                  hmc_wrap(__fmaf_rn(eps, p.z, t.z)), hmc_wrap(__fmaf_rn(eps, p.w, t.w)));
}

// RAG (any L >= 130): the last tiles of a side that is no multiple
// of the tile move back to end with the lattice and overlap the tiles before
// them.  A launch reads one angle and one momentum buffer and writes others,
// so the sites of an overlap are computed twice from the same inputs and
// stored twice with the same bits.  Rows are loaded and stored as wide as
// their alignment allows (16, 8 or 4 bytes for L % 4 = 0, 2, odd).
__device__ __forceinline__ float4 load_row4(const float* p, int L) {
  if ((L & 3) == 0) return *reinterpret_cast<const float4*>(p);
  if ((L & 1) == 0) {
    const float2 u = *reinterpret_cast<const float2*>(p), v = *reinterpret_cast<const float2*>(p + 2);
    return make_float4(u.x, u.y, v.x, v.y);
  }
  return make_float4(p[0], p[1], p[2], p[3]);
}

__device__ __forceinline__ void store_row4(float* p, const float4& v, int L) {
  if ((L & 3) == 0) {
    *reinterpret_cast<float4*>(p) = v;
  } else if ((L & 1) == 0) {
    *reinterpret_cast<float2*>(p) = make_float2(v.x, v.y);
    *reinterpret_cast<float2*>(p + 2) = make_float2(v.z, v.w);
  } else {
    p[0] = v.x;
    p[1] = v.y;
    p[2] = v.z;
    p[3] = v.w;
  }
}

template <int MODE, bool RAG>
__global__ void __launch_bounds__(kP2Threads, 2) k_hmc_tile2(HmcArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  float (*fc)[kFrCols] = reinterpret_cast<float (*)[kFrCols]>(smem);
  float (*fs)[kFrCols] = reinterpret_cast<float (*)[kFrCols]>(smem + sizeof(float) * kFrRows * kFrCols);

  const int L = a.L;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int src, dst;
  hmc_buffers(a, a.ctl->cur, &src, &dst);
  const float* __restrict__ th_src = hmc_buf(a, src);

  const int rb = kP2Band * warp;                             // first tile row of the band
  const int x0 = RAG ? min((int)blockIdx.x * kP2Cols, L - kP2Cols) : (int)blockIdx.x * kP2Cols;
  const int y0 = RAG ? min((int)blockIdx.y * kP2Rows, L - kP2Rows) : (int)blockIdx.y * kP2Rows;

  // ---- loads: own 4 x 4 block (angles and momenta), one site of the ring's
  // top or bottom row (threads 0..255), one of its side columns (0..63), one
  // halo-two site of rows -2 / 33 (0..255), of columns -2 / 129 (64..127) or a
  // ring corner (128..131); 
  const int xb = x0 + 4 * lane;
  float4 t4[kP2Band], p4[kP2Band];
#pragma unroll
  for (int r = 0; r < kP2Band; ++r) {
    const size_t g = (size_t)(y0 + rb + r) * L + xb;
    t4[r] = RAG ? load_row4(th_src + g, L) : *reinterpret_cast<const float4*>(th_src + g);
    p4[r] = RAG ? load_row4(a.p_in + g, L) : *reinterpret_cast<const float4*>(a.p_in + g);
  }
  // ring site A: row -1 (tid < 128) or 32, column tid & 127
  const int ay = tid < kP2Cols ? -1 : kP2Rows, ax = tid & (kP2Cols - 1);
  const size_t ga = (size_t)wrap_near(y0 + ay, L) * L + (x0 + ax);
  float ta = th_src[ga];
  float pa = a.p_in[ga];
  // ring site B: column -1 (tid < 32) or 128, row tid & 31
  const bool hasb = tid < 2 * kP2Rows;
  const int bx = tid < kP2Rows ? -1 : kP2Cols, by = tid & (kP2Rows - 1);
  float tb = 0.f, pb = 0.f;
  if (hasb) {
    const size_t gb = (size_t)(y0 + by) * L + wrap_near(x0 + bx, L);
    tb = th_src[gb];
    pb = a.p_in[gb];
  }
  // halo-two site H: rows -2 / 33; G: columns -2 / 129 or a corner
  const int hy = tid < kP2Cols ? -2 : kP2Rows + 1;
  const float th_h = th_src[(size_t)wrap_near(y0 + hy, L) * L + (x0 + ax)];
  const bool hasg = tid >= 64 && tid < 132;
  int gy = 0, gx = 0;
  float th_g = 0.f;
  if (hasg) {
    if (tid < 128) {
      gx = (tid - 64) < kP2Rows ? -2 : kP2Cols + 1;
      gy = (tid - 64) & (kP2Rows - 1);
    } else {
      gy = (tid & 2) ? kP2Rows : -1;
      gx = (tid & 1) ? kP2Cols : -1;
    }
    th_g = th_src[(size_t)wrap_near(y0 + gy, L) * L + wrap_near(x0 + gx, L)];
  }

  // ---- unit vectors of the old state; what crosses a warp goes to the frame
  Quad4 v[kP2Band];
#pragma unroll
  for (int r = 0; r < kP2Band; ++r) v[r] = quad_vectors<MODE>(t4[r]);
  // ring site A and halo-two site H, then ring site B or halo-two site G
  const int aq = frame_col(ax + 4), bq = frame_col(bx + 4), gq = frame_col(gx + 4);
  float ca, sa, cb = 0.f, sb = 0.f;
  {
    float2 s2, c2;
    xyd::unit_vector2<MODE>(make_float2(ta, th_h), &s2, &c2);
    ca = c2.x;
    sa = s2.x;
    fc[ay + 2][aq] = ca;
    fs[ay + 2][aq] = sa;
    fc[hy + 2][aq] = c2.y;
    fs[hy + 2][aq] = s2.y;
    if (hasb || hasg) {
      xyd::unit_vector<MODE>(hasb ? tb : th_g, &sb, &cb);
      fc[(hasb ? by : gy) + 2][hasb ? bq : gq] = cb;
      fs[(hasb ? by : gy) + 2][hasb ? bq : gq] = sb;
    }
  }
  // the band's first and last row, and the tile's first and last column
  put_quad(&fc[rb + 2][4 * lane + 4], &fs[rb + 2][4 * lane + 4], v[0]);
  put_quad(&fc[rb + kP2Band + 1][4 * lane + 4], &fs[rb + kP2Band + 1][4 * lane + 4],
           v[kP2Band - 1]);
  if (lane == 0 || lane == 31) {
    const int q = lane == 0 ? 4 : kP2Cols + 3;             // tile column 0 or 127
#pragma unroll
    for (int r = 1; r < kP2Band - 1; ++r) {
      fc[rb + r + 2][q] = lane == 0 ? v[r].cE.x : v[r].cO.y;
      fs[rb + r + 2][q] = lane == 0 ? v[r].sE.x : v[r].sO.y;
    }
  }
  __syncthreads();

  // ---- first step: the ring sites (from the frame), then the tile --------
  const float K = a.K, ka = a.a, eps = a.eps;
  auto ring_step = [&](int r, int q, float c0, float s0, float& p, float& t) {
    const int l = frame_col(q - 1), m = frame_col(q), n = frame_col(q + 1);
    const float Sc = xyd::nb_sum(fc[r][l], fc[r][n], fc[r - 1][m], fc[r + 1][m]);
    const float Ss = xyd::nb_sum(fs[r][l], fs[r][n], fs[r - 1][m], fs[r + 1][m]);
    hmc_site_step(c0, s0, Sc, Ss, K, ka, eps, p, t);
  };
  ring_step(ay + 2, ax + 4, ca, sa, pa, ta);
  if (hasb) ring_step(by + 2, bx + 4, cb, sb, pb, tb);
  // the ring's new unit vectors (its momenta and angles are not needed again)
  {
    float2 s2, c2;
    xyd::unit_vector2<MODE>(make_float2(ta, tb), &s2, &c2);
    ca = c2.x;
    sa = s2.x;
    cb = c2.y;
    sb = s2.y;
  }
  // a step of the band: vertical neighbours from its own rows or the frame's
  // rows below and above, horizontal ones from the neighbouring lanes (the
  // warp's edge lanes: the frame's ring columns)
  auto band_step = [&](auto&& done) {
    Quad4 dn = get_quad(&fc[rb + 1][4 * lane + 4], &fs[rb + 1][4 * lane + 4]);
    const Quad4 top = get_quad(&fc[rb + kP2Band + 2][4 * lane + 4], &fs[rb + kP2Band + 2][4 * lane + 4]);
#pragma unroll
    for (int r = 0; r < kP2Band; ++r) {
      float cl = __shfl_up_sync(0xffffffffu, v[r].cO.y, 1);
      float sl = __shfl_up_sync(0xffffffffu, v[r].sO.y, 1);
      float cr = __shfl_down_sync(0xffffffffu, v[r].cE.x, 1);
      float sr = __shfl_down_sync(0xffffffffu, v[r].sE.x, 1);
      if (lane == 0) {
        cl = fc[rb + r + 2][3];
        sl = fs[rb + r + 2][3];
      }
      if (lane == 31) {
        cr = fc[rb + r + 2][kP2Cols + 4];
        sr = fs[rb + r + 2][kP2Cols + 4];
      }
      quad_step(v[r], dn, r == kP2Band - 1 ? top : v[r == kP2Band - 1 ? r : r + 1], cl, sl, cr, sr,
                K, ka, eps, p4[r], t4[r]);
      dn = v[r];
      done(r);
    }
  };
  band_step([](int) {});
  // new unit vectors (the old ones are no longer read by this thread)
#pragma unroll
  for (int r = 0; r < kP2Band; ++r) v[r] = quad_vectors<MODE>(t4[r]);
  __syncthreads();   // every old frame value has been read
  fc[ay + 2][aq] = ca;
  fs[ay + 2][aq] = sa;
  if (hasb) {
    fc[by + 2][bq] = cb;
    fs[by + 2][bq] = sb;
  }
  put_quad(&fc[rb + 2][4 * lane + 4], &fs[rb + 2][4 * lane + 4], v[0]);
  put_quad(&fc[rb + kP2Band + 1][4 * lane + 4], &fs[rb + kP2Band + 1][4 * lane + 4],
           v[kP2Band - 1]);
  __syncthreads();

  // ---- second step: the tile, written out ----------------------------------
  float* __restrict__ th_dst = hmc_buf(a, dst);
  band_step([&](int r) {
    const size_t g = (size_t)(y0 + rb + r) * L + xb;
    if (RAG) {
      store_row4(a.p_out + g, p4[r], L);
      store_row4(th_dst + g, t4[r], L);
    } else {
      *reinterpret_cast<float4*>(a.p_out + g) = p4[r];
      *reinterpret_cast<float4*>(th_dst + g) = t4[r];
    }
  });
}

// ---------------------------------------------------------------------------
// Two full kick-drift steps per launch, each warp on its own.  A warp walks down
// the rows of a strip of 128 columns, four per lane, of which the outer lanes'
// are halo (the strips advance by 120 columns), and the unit vectors of both
// steps pass through its registers: with row r read it takes row r - 1 through
// the first step and row r - 2 through the second.  Horizontal neighbours come
// by shuffle; the rows arrive in the lane's own places in shared memory by
// cp.async, kRowsAhead rows ahead.  A warp's segment of rows starts two rows
// early and ends two rows late.  So there is no ring, no frame and no barrier:
// the tiles of k_hmc_tile2 spend a third of their time on those (their two CTAs
// per SM wait for each other and for dependent instructions, 51 % of the issue
// slots used).  The price is 128 columns computed for 120 and (rows + 3) rows for
// rows.  Here the FMA pipes are 64 % busy and 63 % of the issue slots used, DRAM
// at 4 TB/s; what is left is the tail of a launch (one wave: warps end at
// different times, 78 % resident on average) and the 16 warps per SM that the
// registers allow.
//
// us per unit trajectory, tiles and this: L = 1792 460 and 434, 2048 580 and 575
// (SFU sincos 520 and 413), 2560 1038 and 889, 3072 1740 and 1332, 4096 3343 and
// 2575, 8192 17360 and 12930; where the side is no multiple of 128 1500 384 and
// 367, 2000 706 and 612, 3000 2032 and 1438.  Below, a segment has too few rows
// for its early and late ones (1536 306 and 325, 1000 174 and 194).  With the
// next row's loads in registers instead of three rows ahead in shared memory
// 4096 2735; strips advancing by 124 with 8-byte accesses 2638; loops unrolled
// once 3449 (the rows' registers then move), twice 2916.
//
// VEC: columns that one access may take (the rows' alignment): 4, 2 or 1 where L
// is a multiple of 4, even or odd.
// ---------------------------------------------------------------------------
constexpr int kRowsThreads = 128;
constexpr int kRowsWarps = kRowsThreads / 32;
constexpr int kRowsPerSm = 4;              // CTAs per SM: 16 warps, 128 registers a thread
constexpr int kRowsAhead = 3;              // rows on their way to shared memory
constexpr int kRowsUnroll = 3;             // the rows' registers rotate with period three
constexpr int kStripCols = 120;
constexpr int kRowsMinTiled = 1792, kRowsMinRagged = 1500;

template <int V>
struct IntC {
  static constexpr int value = V;
};

template <int VEC>
__device__ __forceinline__ void hmc_cp_async(void* dst, const void* src) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  if (VEC == 4) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d), "l"(src) : "memory");
  } else {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(4 * VEC) : "memory");
  }
}

template <int MODE, int VEC>
__global__ void __launch_bounds__(kRowsThreads, kRowsPerSm)
    k_hmc_rows2(HmcArgs a, int strips, int rows) {
  __shared__ float4 s_rows[kRowsWarps][kRowsAhead][2][32];   // a lane reads its own places only
  constexpr int NV = 4 / VEC;
  const int L = a.L;
  const int lane = threadIdx.x & 31;
  const int w = blockIdx.x * kRowsWarps + (threadIdx.x >> 5);
  const int strip = w % strips, ys = (w / strips) * rows;
  if (ys >= L) return;
  const int ye = min(ys + rows, L);
  int src, dst;
  hmc_buffers(a, a.ctl->cur, &src, &dst);
  const float* __restrict__ th_src = hmc_buf(a, src);
  float* __restrict__ th_dst = hmc_buf(a, dst);
  const int xs = strip * kStripCols - 4 + 4 * lane;
  const bool inner = lane > 0 && lane < 31;
  uint32_t x[NV];                          // the lane's columns (a side may wrap between accesses)
#pragma unroll
  for (int i = 0; i < NV; ++i) x[i] = (uint32_t)wrap_near(xs + i * VEC, L);
  const float K = a.K, ka = a.a, eps = a.eps;
  float4 (*ahead)[2][32] = s_rows[threadIdx.x >> 5];
  auto fetch = [&](int r, int slot) {
    const uint32_t g = (uint32_t)wrap_near(min(r, ye + 1), L) * (uint32_t)L;
    float* t = reinterpret_cast<float*>(&ahead[slot][0][lane]);
    float* p = reinterpret_cast<float*>(&ahead[slot][1][lane]);
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      hmc_cp_async<VEC>(t + i * VEC, th_src + (g + x[i]));
      hmc_cp_async<VEC>(p + i * VEC, a.p_in + (g + x[i]));
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  auto step = [&](const Quad4& o, const Quad4& dn, const Quad4& up, float4& p, float4& t) {
    const float cl = __shfl_up_sync(0xffffffffu, o.cO.y, 1);
    const float sl = __shfl_up_sync(0xffffffffu, o.sO.y, 1);
    const float cr = __shfl_down_sync(0xffffffffu, o.cE.x, 1);
    const float sr = __shfl_down_sync(0xffffffffu, o.sE.x, 1);
    quad_step(o, dn, up, cl, sl, cr, sr, K, ka, eps, p, t);
  };
  auto store = [&](float* at, const float4& v, int i) {
    if (VEC == 4) {
      *reinterpret_cast<float4*>(at) = v;
    } else if (VEC == 2) {
      *reinterpret_cast<float2*>(at) = i ? make_float2(v.z, v.w) : make_float2(v.x, v.y);
    } else {
      *at = i == 0 ? v.x : i == 1 ? v.y : i == 2 ? v.z : v.w;
    }
  };
  int slot = 0;
#pragma unroll
  for (int i = 0; i < kRowsAhead; ++i) fetch(ys - 2 + i, i);
  float4 t0, p0, t1, p1;                   // row r - 1 as read, row r - 2 after one step
  Quad4 a0, a1;                            // rows r - 2 and r - 1 as read
  Quad4 w0, w1;                            // rows r - 3 and r - 2 after one step
  // row r: its unit vectors; STAGE >= 1: row r - 1's first step; 2: row r - 2's
  // second step, written out
  auto row = [&](auto stage, int r) {
    constexpr int STAGE = decltype(stage)::value;
    asm volatile("cp.async.wait_group %0;" ::"n"(kRowsAhead - 1) : "memory");
    const float4 tc = ahead[slot][0][lane], pc = ahead[slot][1][lane];
    fetch(r + kRowsAhead, slot);
    slot = slot + 1 == kRowsAhead ? 0 : slot + 1;
    const Quad4 n = quad_vectors<MODE>(tc);
    if (STAGE >= 1) {
      step(a1, a0, n, p0, t0);
      const Quad4 wn = quad_vectors<MODE>(t0);
      if (STAGE >= 2) {
        step(w1, w0, wn, p1, t1);
        const uint32_t g = (uint32_t)(r - 2) * (uint32_t)L;
#pragma unroll
        for (int i = 0; i < NV; ++i)
          if (inner && xs + i * VEC < L) {
            store(a.p_out + (g + x[i]), p1, i);
            store(th_dst + (g + x[i]), t1, i);
          }
      }
      w0 = w1;
      w1 = wn;
      t1 = t0;
      p1 = p0;
    }
    a0 = a1;
    a1 = n;
    t0 = tc;
    p0 = pc;
  };
  row(IntC<0>(), ys - 2);
  row(IntC<0>(), ys - 1);
  row(IntC<1>(), ys);
  row(IntC<1>(), ys + 1);
#pragma unroll kRowsUnroll
  for (int r = ys + 2; r < ye + 2; ++r) row(IntC<2>(), r);
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Per-site kernel (any L >= 2): one thread per site, the four neighbours' unit
// vectors recomputed from global memory.  Same per-site arithmetic as above.
// ---------------------------------------------------------------------------
constexpr int kSiteThreads = 256;

template <int MODE, int KIND>
__global__ void __launch_bounds__(kSiteThreads) k_hmc_site(HmcArgs a) {
  __shared__ long long red[kSiteThreads / 32][kHmcSums];
  const int L = a.L;
  const uint32_t N = (uint32_t)L * (uint32_t)L;
  const uint32_t cur = a.ctl->cur;
  int src, dst;
  hmc_buffers(a, cur, &src, &dst);
  const float* __restrict__ th_src = hmc_buf(a, src);
  HmcAcc acc;
  acc_zero(acc);
  const uint32_t site = blockIdx.x * kSiteThreads + threadIdx.x;
  if (site < N) {
    const int y = (int)(site / (uint32_t)L), x = (int)(site - (uint32_t)y * (uint32_t)L);
    const int xl = x == 0 ? L - 1 : x - 1, xr = x == L - 1 ? 0 : x + 1;
    const int yd = y == 0 ? L - 1 : y - 1, yu = y == L - 1 ? 0 : y + 1;
    const size_t row = (size_t)y * L;
    const float t = th_src[row + x];
    float cs[5], sn[5];
    xyd::unit_vector<MODE>(t, &sn[0], &cs[0]);
    xyd::unit_vector<MODE>(th_src[row + xl], &sn[1], &cs[1]);
    xyd::unit_vector<MODE>(th_src[row + xr], &sn[2], &cs[2]);
    xyd::unit_vector<MODE>(th_src[(size_t)yd * L + x], &sn[3], &cs[3]);
    xyd::unit_vector<MODE>(th_src[(size_t)yu * L + x], &sn[4], &cs[4]);
    float p = KIND == kHmcBeginDraw ? hmc_momentum(site, (uint32_t)a.ctl->traj, a.lattice_id, a.rk)
                                    : a.p_in[site];
    const float Sc = xyd::nb_sum(cs[1], cs[2], cs[3], cs[4]);
    const float Ss = xyd::nb_sum(sn[1], sn[2], sn[3], sn[4]);
    const float F = hmc_force(cs[0], sn[0], Sc, Ss, a.K);
    if (KIND == kHmcBeginDraw || KIND == kHmcBeginRead)
      hmc_terms(p, cs[0], sn[0], cs[2], sn[2], cs[4], sn[4], acc);
    p = __fmaf_rn(a.a, F, p);
    if (KIND == kHmcFinal) {
      hmc_terms(p, cs[0], sn[0], cs[2], sn[2], cs[4], sn[4], acc);
    } else {
      hmc_buf(a, dst)[site] = hmc_wrap(__fmaf_rn(a.eps, p, t));
    }
    a.p_out[site] = p;
  }
  if (KIND == kHmcBeginDraw || KIND == kHmcBeginRead)
    hmc_commit<kSiteThreads / 32>(acc, a.ctl->acc[0], red);
  if (KIND == kHmcFinal) hmc_commit<kSiteThreads / 32>(acc, a.ctl->acc[1], red);
}

// ---------------------------------------------------------------------------
// The test (mode 0) or the commit of a plain integration (mode 1).
// ---------------------------------------------------------------------------
__global__ void k_hmc_accept(HmcArgs a, int mode, double beta, double J) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  HmcCtl* c = a.ctl;
  int fin, unused;
  hmc_buffers(a, c->cur, &fin, &unused);
  if (xyh::hmc_decide(c, a.lattice_id, a.rk, mode, beta, J)) c->cur = (uint32_t)fin;
}

__global__ void k_hmc_draw(HmcArgs a) {
  const uint32_t N = (uint32_t)a.L * (uint32_t)a.L;
  const uint32_t traj = (uint32_t)a.ctl->traj;
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < N; s += gridDim.x * blockDim.x)
    a.p_out[s] = hmc_momentum(s, traj, a.lattice_id, a.rk);
}

__global__ void k_hmc_start(HmcArgs a, int hot) {
  const uint32_t N = (uint32_t)a.L * (uint32_t)a.L;
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < N; s += gridDim.x * blockDim.x) {
    float t = 0.f;
    if (hot) {
      const uint4 w = xyd::philox4x32_10(make_uint4(s, 0u, a.lattice_id, 0u), a.rk);
      t = (float)(w.x >> 8) * xyd::kHotScale;
    }
    a.th[0][s] = t;
    a.p_out[s] = 0.f;
  }
}

__global__ void k_hmc_canon_copy(HmcArgs a) {
  const uint32_t cur = a.ctl->cur;
  if (cur == 0u) return;
  const uint32_t N = (uint32_t)a.L * (uint32_t)a.L;
  const float* __restrict__ from = hmc_buf(a, (int)cur);
  float* __restrict__ to = a.th[0];
  for (uint32_t s = blockIdx.x * blockDim.x + threadIdx.x; s < N; s += gridDim.x * blockDim.x)
    to[s] = from[s];
}

__global__ void k_hmc_canon_reset(HmcCtl* ctl) {
  if (threadIdx.x == 0 && blockIdx.x == 0) ctl->cur = 0u;
}

}  // namespace

bool hmc_tiled_ok(int L) { return L >= kTileCols && L % kTileCols == 0; }

bool hmc_ragged_ok(int L) { return L > kTileCols && L % kTileCols != 0; }

namespace {

// Two full steps per launch: by rows where the segments are long enough (one
// wave of warps, so the longest that keep every SM full), else by tiles.
template <int MODE>
cudaError_t launch_step2(const HmcArgs& a, cudaStream_t stream) {
  if (!a.pairs || a.p_in == a.p_out) return cudaErrorInvalidValue;
  const bool tiled = hmc_tiled_ok(a.L);
  if (!tiled && !hmc_ragged_ok(a.L)) return cudaErrorInvalidValue;
  if (tiled && !a.tiled) return cudaErrorInvalidValue;
  if (a.L >= (tiled ? kRowsMinTiled : kRowsMinRagged)) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return e;
    const int strips = (a.L + kStripCols - 1) / kStripCols;
    const int fit = sms * kRowsPerSm * kRowsWarps / strips, segs = fit > 1 ? fit : 1;
    const int rows = (a.L + segs - 1) / segs;
    const int warps = strips * ((a.L + rows - 1) / rows);
    const int grid = (warps + kRowsWarps - 1) / kRowsWarps;
    switch (a.L % 4) {
      case 0: k_hmc_rows2<MODE, 4><<<grid, kRowsThreads, 0, stream>>>(a, strips, rows); break;
      case 2: k_hmc_rows2<MODE, 2><<<grid, kRowsThreads, 0, stream>>>(a, strips, rows); break;
      default: k_hmc_rows2<MODE, 1><<<grid, kRowsThreads, 0, stream>>>(a, strips, rows);
    }
  } else if (tiled) {
    k_hmc_tile2<MODE, false>
        <<<dim3(a.L / kP2Cols, a.L / kP2Rows), kP2Threads, kP2Smem, stream>>>(a);
  } else {
    const dim3 grid((a.L + kP2Cols - 1) / kP2Cols, (a.L + kP2Rows - 1) / kP2Rows);
    k_hmc_tile2<MODE, true><<<grid, kP2Threads, kP2Smem, stream>>>(a);
  }
  return cudaGetLastError();
}

template <int MODE>
cudaError_t launch_mode(int kind, const HmcArgs& a, cudaStream_t stream) {
  if (kind == kHmcStep2) return launch_step2<MODE>(a, stream);
  if (a.tiled) {
    const dim3 grid(a.L / kTileCols, a.L / kTileRows);
    switch (kind) {
      case kHmcBeginDraw: k_hmc_tile<MODE, kHmcBeginDraw><<<grid, kTileThreads, 0, stream>>>(a); break;
      case kHmcBeginRead: k_hmc_tile<MODE, kHmcBeginRead><<<grid, kTileThreads, 0, stream>>>(a); break;
      case kHmcStep: k_hmc_tile<MODE, kHmcStep><<<grid, kTileThreads, 0, stream>>>(a); break;
      default: k_hmc_tile<MODE, kHmcFinal><<<grid, kTileThreads, 0, stream>>>(a); break;
    }
  } else {
    const int64_t N = (int64_t)a.L * a.L;
    const int grid = (int)((N + kSiteThreads - 1) / kSiteThreads);
    switch (kind) {
      case kHmcBeginDraw: k_hmc_site<MODE, kHmcBeginDraw><<<grid, kSiteThreads, 0, stream>>>(a); break;
      case kHmcBeginRead: k_hmc_site<MODE, kHmcBeginRead><<<grid, kSiteThreads, 0, stream>>>(a); break;
      case kHmcStep: k_hmc_site<MODE, kHmcStep><<<grid, kSiteThreads, 0, stream>>>(a); break;
      default: k_hmc_site<MODE, kHmcFinal><<<grid, kSiteThreads, 0, stream>>>(a); break;
    }
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t hmc_prepare(int sincos_mode) {
  static bool done[3][64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const int m = sincos_mode < 0 || sincos_mode > 2 ? 0 : sincos_mode;
  if (dev >= 0 && dev < 64 && done[m][dev]) return cudaSuccess;
  const void* f = m == 0 ? (const void*)k_hmc_tile2<0, false>
                         : (m == 1 ? (const void*)k_hmc_tile2<1, false>
                                   : (const void*)k_hmc_tile2<2, false>);
  e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kP2Smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  const void* fr = m == 0 ? (const void*)k_hmc_tile2<0, true>
                          : (m == 1 ? (const void*)k_hmc_tile2<1, true>
                                    : (const void*)k_hmc_tile2<2, true>);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fr, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kP2Smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(fr, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  const void* g4 = m == 0 ? (const void*)k_hmc_step_tma<0, 4>
                          : (m == 1 ? (const void*)k_hmc_step_tma<1, 4> : (const void*)k_hmc_step_tma<2, 4>);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(g4, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TmaGeom<4>::kSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(g4, cudaFuncAttributePreferredSharedMemoryCarveout, 100);

  if (e == cudaSuccess && dev >= 0 && dev < 64) done[m][dev] = true;
  return e;
}

cudaError_t launch_hmc(int kind, int sincos_mode, const HmcArgs& a, cudaStream_t stream) {
  if (kind < kHmcBeginDraw || kind > kHmcStep2) return cudaErrorInvalidValue;
  if (a.tiled && !hmc_tiled_ok(a.L)) return cudaErrorInvalidValue;
  switch (sincos_mode) {
    case 0: return launch_mode<0>(kind, a, stream);
    case 1: return launch_mode<1>(kind, a, stream);
    default: return launch_mode<2>(kind, a, stream);
  }
}

template <int ROWS>
cudaError_t launch_tma_rows(int sincos_mode, const HmcArgs& a, const CUtensorMap* m, int ctas,
                            cudaStream_t stream) {
  const int tiles_x = a.L / kTileCols;
  const int n_tiles = tiles_x * (a.L / TmaGeom<ROWS>::kRows);
  const int grid = ctas < n_tiles ? ctas : n_tiles;
  const size_t smem = TmaGeom<ROWS>::kSmem;
  switch (sincos_mode) {
    case 0:
      k_hmc_step_tma<0, ROWS><<<grid, kTileThreads, smem, stream>>>(m[0], m[1], m[2], m[3], a, tiles_x, n_tiles);
      break;
    case 1:
      k_hmc_step_tma<1, ROWS><<<grid, kTileThreads, smem, stream>>>(m[0], m[1], m[2], m[3], a, tiles_x, n_tiles);
      break;
    default:
      k_hmc_step_tma<2, ROWS><<<grid, kTileThreads, smem, stream>>>(m[0], m[1], m[2], m[3], a, tiles_x, n_tiles);
      break;
  }
  return cudaGetLastError();
}

cudaError_t launch_hmc_step_tma(int sincos_mode, const HmcArgs& a, const void* maps4, int box_rows,
                                int ctas, cudaStream_t stream) {
  if (!a.tiled || a.p_in != a.p_out || !maps4 || ctas < 1) return cudaErrorInvalidValue;
  const CUtensorMap* m = static_cast<const CUtensorMap*>(maps4);
  if (box_rows == TmaGeom<4>::kRows) return launch_tma_rows<4>(sincos_mode, a, m, ctas, stream);
  return cudaErrorInvalidValue;
}

cudaError_t launch_hmc_steps_persist(int sincos_mode, const HmcStepsArgs& q, const void* maps4,
                                     cudaStream_t stream) {
  const HmcArgs& a = q.a;
  if (!a.tiled || a.p_in != a.p_out || !maps4 || q.n_steps < 1 || !q.flags ||
      q.spin_limit < 1 || (a.L % kTileCols) != 0 || (a.L % TmaGeom<4>::kRows) != 0)
    return cudaErrorInvalidValue;
  const int tiles_x = a.L / kTileCols;
  const int n_tiles = tiles_x * (a.L / TmaGeom<4>::kRows);
  if ((long long)q.n_steps * n_tiles > 0x7fffffffll - (1ll << 20)) return cudaErrorInvalidValue;
  const void* fn = sincos_mode == 0 ? (const void*)k_hmc_steps_persist<0>
                                    : (sincos_mode == 1 ? (const void*)k_hmc_steps_persist<1>
                                                        : (const void*)k_hmc_steps_persist<2>);
  const size_t smem = TmaGeom<4>::kSmem;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
  int per_sm = 0, dev = 0, sms = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, fn, kTileThreads, smem);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) return cudaErrorCooperativeLaunchTooLarge;
  const int grid = n_tiles < per_sm * sms ? n_tiles : per_sm * sms;
  e = cudaMemsetAsync(q.flags, 0, sizeof(unsigned int) * (size_t)n_tiles, stream);
  if (e != cudaSuccess) return e;
  const CUtensorMap* m = static_cast<const CUtensorMap*>(maps4);
  HmcStepsArgs qq = q;
  int tx = tiles_x, nt = n_tiles;
  void* args[] = {const_cast<CUtensorMap*>(&m[0]), const_cast<CUtensorMap*>(&m[1]),
                  const_cast<CUtensorMap*>(&m[2]), const_cast<CUtensorMap*>(&m[3]), &qq, &tx, &nt};
  return coop_launch(fn, grid, kTileThreads, args, smem, stream);
}

int hmc_persist_tiles(int L) {
  return (L % kTileCols == 0 && L % TmaGeom<4>::kRows == 0) ? (L / kTileCols) * (L / TmaGeom<4>::kRows)
                                                             : 0;
}

long long hmc_persist_spin_limit() { return kSpinLimit; }

namespace {
// The failure path of the bounded waits, exercised without a fault: wait on a
// barrier that nothing ever completes, exactly as the TMA kernel waits on its
// stage barriers, and set the error word when the bound runs out.
__global__ void k_selftest_wait(unsigned int* error, long long polls) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    xyt::mbar_init(&bar, 1);
    xyt::fence_mbarrier_init();
  }
  __syncthreads();
  const bool done = xyt::mbar_wait_bounded(&bar, 0u, polls);   // no arrival: must run out
  if (!done && threadIdx.x == 0) atomicOr(error, 1u);
}
}  // namespace

cudaError_t launch_selftest_wait(unsigned int* d_error, long long polls, cudaStream_t stream) {
  k_selftest_wait<<<1, 32, 0, stream>>>(d_error, polls);
  return cudaGetLastError();
}

cudaError_t launch_hmc_accept(int mode, const HmcArgs& a, double beta, double J,
                              cudaStream_t stream) {
  k_hmc_accept<<<1, 32, 0, stream>>>(a, mode, beta, J);
  return cudaGetLastError();
}

cudaError_t launch_hmc_draw(const HmcArgs& a, cudaStream_t stream) {
  k_hmc_draw<<<grid_for((int64_t)a.L * a.L, 256), 256, 0, stream>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_hmc_start(const HmcArgs& a, int hot, cudaStream_t stream) {
  k_hmc_start<<<grid_for((int64_t)a.L * a.L, 256), 256, 0, stream>>>(a, hot);
  return cudaGetLastError();
}

cudaError_t launch_hmc_canonical(const HmcArgs& a, cudaStream_t stream) {
  k_hmc_canon_copy<<<grid_for((int64_t)a.L * a.L, 256), 256, 0, stream>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  k_hmc_canon_reset<<<1, 32, 0, stream>>>(a.ctl);
  return cudaGetLastError();
}

}  // namespace xyk
