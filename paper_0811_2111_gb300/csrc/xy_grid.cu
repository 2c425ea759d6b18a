// xy_grid.cu -- all sweeps of a call of a middling lattice in one cooperative
// launch, every tile of the lattice staying with its CTA.
//
// Up to L = 1280 the lattice's angles and unit vectors fit the registers and
// shared memory of the chip.  The persistent tiles (xy_fused.cu) spend most of
// such a sweep on what this kernel does not do at all: each sweep a tile waits
// for its neighbours' counters, then for its rows, and stages them anew (4616
// unit vectors for 4096 sites); at L = 512 that is 5.8 us for work of 0.6 us.
// Here a CTA owns a tile of at most 64 plane columns and an even number of rows
// of both colours for the whole launch.  A lane of a tile warp owns one pair of
// columns (plane columns 2m, 2m + 1 of a row: one Philox block) in NR
// consecutive rows, their angles in registers; shared memory holds the unit
// vectors of both colours with the halo that the update reads.  A sweep:
//   the tile warps draw their next proposals (no neighbour enters them), while
//   the halo warps wait for the neighbours' edge sites and put their unit
//   vectors in place
//   -- barrier --
//   red accept tests; the halo warps update the ring of red sites around the
//   tile (recomputed from the same state and words as by its owners, so with
//   the same result)
//   -- barrier --
//   black accept tests, the sweep sums, the new edge sites to the neighbours.
// The red edge sites are sent from the red half already, so that the halo warps
// can draw the ring's proposals before the black ones arrive.
//
// The exchange: 64-bit words (angle, tag), one per edge site and sweep parity,
// written and polled with relaxed GPU-scope accesses.  A word itself says that
// it has arrived: no fence, no counter, no second round trip.  The tag counts
// exchanges over the lattice's lifetime (ctl[0], advanced by the last CTA to
// finish, so that captured launches replay).  A tile reads six of the tiles around
// it: left, right, above (row y0 - 1), below, and the corners at the upper right
// and the lower left (y0 and the heights are even: the red sites of the odd row
// y0 - 1 have a black neighbour right of the tile, those of the even row below it
// one left of it).  Those are the six that read it.  A slot is rewritten two
// exchanges later, when the writer has read the next exchange's words of all six,
// and they wrote those after reading the slot.  The first exchange carries the
// initial state, so the state buffer itself is touched by its owner only.  Every
// wait is bounded; one that runs out sets *error and ends the CTA, and those
// that wait for it see *error and end too.
//
// Up to four lattices run side by side in one launch: the replicas of a quad,
// whose angles lie `step` floats apart, each on its share of the SMs.
//
// Exact sums only: they do not depend on who adds what, while the compensated
// sums round by thread and warp and keep the kernels that define them.  Any even
// side: rows have (W + 1) / 2 pairs, and where W = L / 2 is odd (ODD) the last
// tile's last pair has its second column in the halo and drops that result.
//
// What bounds it: up to about L = 512 the chain of a sweep (the exchange, two
// barriers, two accept tests: about 1.5 us), above the SM's issue slots (57 %
// used at L = 1024, the heavy FMA pipe 56 %) and the barriers (a fifth of the
// warps' time).
#include <cuda_runtime.h>
#include <stdint.h>

#include "xy_device.cuh"
#include "xy_internal.h"
#include "xy_tile.cuh"

namespace xyk {

namespace {

typedef unsigned long long u64;

__device__ __forceinline__ void put_words(u64* at, float2 v, uint32_t tag) {
  const u64 t = (u64)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(at),
               "l"(t | __float_as_uint(v.x)), "l"(t | __float_as_uint(v.y))
               : "memory");
}
__device__ __forceinline__ void get_words(const u64* at, u64* x, u64* y) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(*x), "=l"(*y) : "l"(at) : "memory");
}
__device__ __forceinline__ u64 get_word(const u64* at) {
  u64 v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(at) : "memory");
  return v;
}
__device__ __forceinline__ float word_value(u64 w) { return __uint_as_float((uint32_t)w); }
__device__ __forceinline__ bool word_is(u64 w, uint32_t tag) { return (uint32_t)(w >> 32) == tag; }

constexpr size_t kGridSmem = 128 * 1024;    // unit vectors of a tile of 110 rows

// Polls before a wait gives up: about a second (the loops do not sleep, a word
// being on its way for less than that: a poll is a round trip to L2, 170 ns on an
// otherwise idle GPU).
constexpr long long kGridSpinLimit = 6ll << 20;

// Part i of n near-equal parts of `total`.
__host__ __device__ inline int part_size(int total, int n, int i) {
  return total / n + (i < total % n ? 1 : 0);
}
__host__ __device__ inline int part_first(int total, int n, int i) {
  return i * (total / n) + (i < total % n ? i : total % n);
}

// The whole CTA's barrier (warps of both kinds reach it at their own places).
__device__ __forceinline__ void cta_sync() {
  __syncwarp();
  asm volatile("bar.sync 0;" ::: "memory");
}

template <int MODE, int NR, int MAXT, bool ODD>
__global__ void __launch_bounds__(MAXT) k_sweep_grid(GridArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint32_t s_part[32][5];
  __shared__ uint32_t s_cnt[32];
  __shared__ int s_abort;
  const int L = a.L, W = L / 2, pitch = (W + 1) & ~1;
  const int tiles = a.nx * a.ny;
  const int rep = blockIdx.x / tiles, tile = blockIdx.x - rep * tiles;
  const int bx = tile % a.nx, by = tile / a.nx;
  const int np = part_size((W + 1) / 2, a.nx, bx), k0 = 2 * part_first((W + 1) / 2, a.nx, bx);
  const int H = 2 * part_size(L / 2, a.ny, by), y0 = 2 * part_first(L / 2, a.ny, by);
  const int width = min(2 * np, W - k0);
  const int rows = 2 * part_size(L / 2, a.ny, 0);          // the highest tile's
  CsRow* csr = reinterpret_cast<CsRow*>(smem);             // [rows + 2]: row r + 1 the tile's row r
  CsRow* csb = csr + rows + 2;                             // [rows + 4]: row r + 2
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pj = lane + 1, kp = k0 + 2 * lane;
  // the pair is the tile's; so is its second site (not the last of an odd W)
  const bool on = lane < np, both = ODD ? 2 * lane + 1 < width : on;
  const size_t plane = (size_t)L * (size_t)W;
  unsigned int* ctl = a.ctl + 2 * rep;
  const uint32_t base = __ldcg(ctl);
  const uint32_t lattice_id = a.lattice_id + (uint32_t)rep;
  xy_record* rec = a.rec + rep;
  if (threadIdx.x == 0) s_abort = 0;
  // where the lane's pair of row y of colour c is exchanged under tag t
  auto word_at = [&](uint32_t t, int c, int y) {
    return ((((uint32_t)rep * 2u + (t & 1u)) * 2u + (uint32_t)c) * (uint32_t)L + (uint32_t)y) *
               (uint32_t)pitch +
           (uint32_t)kp;
  };
  // lanes past the tile's pairs (fewer than 32) store to a row's last place,
  // which such a tile does not use; the half pair of an odd W leaves the halo
  // column in its second place alone
  const int pst = on ? pj : kCsPairs - 1;
  const bool half = ODD && on && !both;
  auto put_own = [&](CsRow& row, const xyd::PairResult& p) {
    if (!half) {
      put_pair(&row[pst], p.c, p.s);
    } else {
      put_one(row, 2 * pj, p.c.x, p.s.x);
    }
  };
  auto draw = [&](int y, int c, uint32_t sweep) {
    return xyd::philox_pair_words(
        (uint32_t)y * (uint32_t)L + 2u * (uint32_t)kp + (((uint32_t)y + (uint32_t)c) & 1u), sweep,
        lattice_id, a.rk);
  };
  const float2 K = xyd::dup2(a.K[rep]);

  if (warp >= a.tile_warps) {
    // ---- halo warps: 0 the row pairs above the tile, 1 those below, the rest
    // one row each (-1 .. H) of the two side columns ----
    const int e = warp - a.tile_warps;
    cta_sync();
    auto give_up = [&]() {
      atomicOr(a.error, 1u);
      s_abort = 1;
    };
    auto stop = [&](long long& it) {
      return ++it > a.spin_limit ||
             ((it & 255) == 0 && *reinterpret_cast<volatile unsigned int*>(a.error) != 0u);
    };
    if (e < 2) {
      // the rows above the tile (0) or below it: the black row beyond the
      // ring, the ring's black and red ones
      const int yr = e == 0 ? wrap_once(y0 - 1, L) : wrap_once(y0 + H, L);
      const int yb = e == 0 ? wrap_once(y0 - 2, L) : wrap_once(y0 + H + 1, L);
      const int ib = e == 0 ? 1 : H + 2;                   // csb row of the ring
      const int ob = e == 0 ? 0 : H + 3;                   // csb row beyond it
      const int q = yr & 1;
      for (int s = 0; s < a.n_sweeps; ++s) {
        const uint32_t sweep = a.sweep0 + (uint32_t)s, tag = base + (uint32_t)s;
        const uint4 w = draw(yr, 0, sweep);
        float2 o = make_float2(0.f, 0.f), n = o, r = o;
        // the red words were sent half a sweep before the black ones
        if (on) {
          const u64* p = a.words + word_at(tag, 0, yr);
          u64 v[2];
          for (long long it = 0;;) {
            get_words(p, &v[0], &v[1]);
            if (word_is(v[0], tag) && (!both || word_is(v[1], tag))) break;
            if (stop(it)) {
              give_up();
              break;
            }
          }
          r = make_float2(word_value(v[0]), both ? word_value(v[1]) : 0.f);
        }
        float2 c0, s0;
        xyd::unit_vector2<MODE>(r, &s0, &c0);
        const xyd::PairProposal pp = xyd::propose_pair<MODE>(r, w, a.delta);
        if (on) {
          const u64* pb = a.words + word_at(tag, 1, yb);
          const u64* pn = a.words + word_at(tag, 1, yr);
          u64 v[4];
          for (long long it = 0;;) {
            get_words(pb, &v[0], &v[1]);
            get_words(pn, &v[2], &v[3]);
            if (word_is(v[0], tag) && word_is(v[2], tag) &&
                (!both || (word_is(v[1], tag) && word_is(v[3], tag))))
              break;
            if (stop(it)) {
              give_up();
              break;
            }
          }
          o = make_float2(word_value(v[0]), both ? word_value(v[1]) : 0.f);
          n = make_float2(word_value(v[2]), both ? word_value(v[3]) : 0.f);
        }
        xyd::PairResult p;
        xyd::unit_vector2<MODE>(o, &p.s, &p.c);
        put_own(csb[ob], p);
        xyd::unit_vector2<MODE>(n, &p.s, &p.c);
        put_own(csb[ib], p);
        cta_sync();
        if (s_abort) break;
        xyd::PairNeighbours nb;
        float4 U;
        pair_neighbours(csb, ib, pj, q, csb[ib - 1][pj], csb[ib][pj], U, nb);
        put_own(csr[ib - 1], xyd::accept_pair<MODE>(pp, r, c0, s0, nb.Sc, nb.Ss, K));
        cta_sync();
      }
    } else {
      const int i = (e - 2) * 32 + lane - 1;               // row of the tile
      const bool here = i <= H, inner = i >= 0 && i < H;
      const int y = wrap_once(y0 + (here ? i : 0), L);
      const int q = y & 1;
      const int kl = wrap_once(k0 - 1, W), kr = wrap_once(k0 + width, W);
      const bool left = here && i >= 0, right = here && i < H;
      // the ring's red site: left of odd rows, right of even ones
      const int kc = q ? kl : kr, cc = (q ? -1 : width) + kCsOff;
      const uint32_t x = 2u * (uint32_t)kc + (uint32_t)q, site = (uint32_t)y * (uint32_t)L + x;
      for (int s = 0; s < a.n_sweeps; ++s) {
        const uint32_t sweep = a.sweep0 + (uint32_t)s, tag = base + (uint32_t)s;
        const uint4 w = xyd::philox4x32_10(
            make_uint4(xyd::metropolis_counter(site, x), sweep, lattice_id, 1u), a.rk);
        const uint2 uw = xyd::metropolis_words(w, x);
        auto wait_word = [&](const u64* p) {
          u64 v;
          for (long long it = 0;;) {
            v = get_word(p);
            if (word_is(v, tag)) break;
            if (stop(it)) {
              give_up();
              break;
            }
          }
          return word_value(v);
        };
        float t = 0.f, s0, c0;
        if (inner) t = wait_word(a.words + (word_at(tag, 0, y) + (uint32_t)(kc - kp)));
        xyd::unit_vector<MODE>(t, &s0, &c0);
        float2 b = make_float2(0.f, 0.f);
        if (here) {
          const u64* pl = a.words + (word_at(tag, 1, y) + (uint32_t)((left ? kl : kr) - kp));
          const u64* pr = a.words + (word_at(tag, 1, y) + (uint32_t)((right ? kr : kl) - kp));
          u64 v, u;
          for (long long it = 0;;) {
            v = get_word(pl);
            u = get_word(pr);
            if (word_is(v, tag) && word_is(u, tag)) break;
            if (stop(it)) {
              give_up();
              break;
            }
          }
          b = make_float2(word_value(v), word_value(u));
        }
        float2 bs, bc;
        xyd::unit_vector2<MODE>(b, &bs, &bc);
        if (left) put_one(csb[i + 2], kCsOff - 1, bc.x, bs.x);
        if (right) put_one(csb[i + 2], kCsOff + width, bc.y, bs.y);
        cta_sync();
        if (s_abort) break;
        if (inner) {
          const CsRow* nb = csb + i + 2;
          const float2 l = get_one(nb[0], cc + q - 1), r = get_one(nb[0], cc + q);
          const float2 d = get_one(nb[-1], cc), u = get_one(nb[1], cc);
          const xyd::SiteResult res = xyd::metropolis_step<MODE>(
              t, c0, s0, xyd::nb_sum(l.x, r.x, d.x, u.x), xyd::nb_sum(l.y, r.y, d.y, u.y), uw.x,
              uw.y, K.x, a.delta);
          put_one(csr[i + 1], cc, res.c, res.s);
        }
        cta_sync();
      }
    }
  } else {
    // ---- tile warps: NR rows each ----
    const int r0 = warp * NR;
    const bool edge = lane == 0 || lane == np - 1;
    auto publish = [&](int c, int rr, float2 v, uint32_t at, uint32_t tag) {
      const int deep = c == 0 ? 1 : 2, row = r0 + rr;      // rows that neighbours read
      if (on && (edge || row < deep || row >= H - deep))
        put_words(a.words + (at + (uint32_t)(rr * pitch)), v, tag);
    };
    float2 th[2][NR];
#pragma unroll
    for (int c = 0; c < 2; ++c)
#pragma unroll
      for (int rr = 0; rr < NR; ++rr) {
        th[c][rr] = make_float2(0.f, 0.f);
        const int row = r0 + rr;
        if (row < H) {
          if (on) {
            const float* g = a.theta + (c * plane + (size_t)(y0 + row) * W + kp) * a.step + rep;
            th[c][rr].x = g[0];
            if (both) th[c][rr].y = g[a.step];
          }
          publish(c, rr, th[c][rr], word_at(base, c, y0 + r0), base);
          xyd::PairResult p;
          xyd::unit_vector2<MODE>(th[c][rr], &p.s, &p.c);
          put_own(c ? csb[row + 2] : csr[row + 1], p);
        }
      }
    cta_sync();

    // The previous sweep's sums, left in s_part / s_cnt: one warp per sum adds
    // the warps' values (16-bit halves, one lane per warp).
    auto commit = [&](xy_record* r) {
      for (int task = warp; task < 6; task += a.tile_warps) {
        const bool has = lane < a.tile_warps;
        if (task == 5) {
          const uint32_t n = has ? s_cnt[lane] : 0u;
          const uint32_t total = __reduce_add_sync(0xffffffffu, n & 0x7fffffffu);
          const bool bad = __any_sync(0xffffffffu, (n & 0x80000000u) != 0u);
          if (lane == 0) {
            atomicAdd(reinterpret_cast<u64*>(&r->accepted), (u64)total);
            if (bad) atomicOr(reinterpret_cast<u64*>(&r->flags), 1ull);
            if (tile == 0) r->beta = a.beta[rep];
          }
        } else {
          const int32_t v = has ? (int32_t)s_part[lane][task] : 0;
          const uint32_t lo = __reduce_add_sync(0xffffffffu, (uint32_t)v & 0xffffu);
          const int32_t hi = (int32_t)__reduce_add_sync(0xffffffffu, (uint32_t)(v >> 16));
          if (lane == 0)
            atomicAdd(reinterpret_cast<u64*>(&r->sum[task]),
                      (u64)((long long)hi * 65536ll + (long long)lo)
                          << (XY_FX_SHIFT - xyd::fx_term_shift(task)));
        }
      }
    };

    auto propose = [&](int c, int rr, uint32_t sweep) {
      return xyd::propose_pair<MODE>(th[c][rr], draw(y0 + r0 + rr, c, sweep), a.delta);
    };
    bool aborted = false;
    for (int s = 0; s < a.n_sweeps; ++s) {
      const uint32_t sweep = a.sweep0 + (uint32_t)s, next = base + (uint32_t)s + 1u;
      const bool last = s + 1 == a.n_sweeps;
      // one proposal ahead; with one row a warp both colours' before the wait
      xyd::PairProposal ahead = propose(0, 0, sweep), early;
      if (NR == 1) early = propose(1, 0, sweep);
      cta_sync();
      if (s_abort) {
        aborted = true;
        break;
      }
      unsigned int n_acc = 0;
      uint32_t at = word_at(next, 0, y0 + r0);
      float4 D = csb[r0 + 1][pj], P = csb[r0 + 2][pj];
#pragma unroll
      for (int rr = 0; rr < NR; ++rr) {
        const int row = r0 + rr;
        const xyd::PairProposal pp = ahead;
        if (NR > 1) ahead = rr + 1 < NR ? propose(0, rr + 1, sweep) : propose(1, 0, sweep);
        if (row >= H) continue;
        xyd::PairNeighbours n;
        float4 U;
        pair_neighbours(csb, row + 2, pj, (y0 + row) & 1, D, P, U, n);
        D = P;
        P = U;
        const float4 o = csr[row + 1][pj];
        const xyd::PairResult p = xyd::accept_pair<MODE>(pp, th[0][rr], cosines(o), sines(o),
                                                         n.Sc, n.Ss, K);
        th[0][rr] = p.th;
        put_own(csr[row + 1], p);
        if (!last) publish(0, rr, p.th, at, next);
        n_acc += (p.acc0 ? 1u : 0u) + (p.acc1 && !half ? 1u : 0u);
      }
      if (s > 0) commit(rec + (size_t)(s - 1) * a.step);
      if (NR == 1) ahead = early;
      cta_sync();
      xyd::SweepSums<0> sums;
      sums.init();
      at = word_at(next, 1, y0 + r0);
      D = csr[r0][pj];
      P = csr[r0 + 1][pj];
#pragma unroll
      for (int rr = 0; rr < NR; ++rr) {
        const int row = r0 + rr;
        const xyd::PairProposal pp = ahead;
        if (rr + 1 < NR) ahead = propose(1, rr + 1, sweep);
        if (row >= H) continue;
        xyd::PairNeighbours n;
        float4 U;
        pair_neighbours(csr, row + 1, pj, (y0 + row + 1) & 1, D, P, U, n);
        const float4 m = P;                                // the red pair of the same row
        D = P;
        P = U;
        const float4 o = csb[row + 2][pj];
        const xyd::PairResult p = xyd::accept_pair<MODE>(pp, th[1][rr], cosines(o), sines(o),
                                                         n.Sc, n.Ss, K);
        th[1][rr] = p.th;
        put_own(csb[row + 2], p);
        if (!last) publish(1, rr, p.th, at, next);
        n_acc += (p.acc0 ? 1u : 0u) + (p.acc1 && !half ? 1u : 0u);
        // red sites with the same (y, k): their spins enter M once each
        float2 v[5];
        xyd::measure_terms2(p.c, p.s, n, cosines(m), sines(m), v);
        if (ODD) {                                         // a zero term adds nothing
#pragma unroll
          for (int i = 0; i < 5; ++i) v[i].y = half ? 0.f : v[i].y;
        }
        sums.add2(v);
      }
      if (!on) sums.init();
      const unsigned int acc = __reduce_add_sync(0xffffffffu, on ? n_acc : 0u);
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
    if (!aborted) {
      // the tile warps alone: the halo warps have left their loop
      asm volatile("bar.sync 1, %0;" ::"r"(a.tile_warps * 32) : "memory");
      commit(rec + (size_t)(a.n_sweeps - 1) * a.step);
#pragma unroll
      for (int c = 0; c < 2; ++c)
#pragma unroll
        for (int rr = 0; rr < NR; ++rr)
          if (on && r0 + rr < H) {
            float* g = a.theta + (c * plane + (size_t)(y0 + r0 + rr) * W + kp) * a.step + rep;
            g[0] = th[c][rr].x;
            if (both) g[a.step] = th[c][rr].y;
          }
    }
  }
  // the exchanges made: the next launch's tags go on from here.  Every thread of
  // the CTA read ctl[0] before its first barrier.
  if (threadIdx.x == 0 && atomicAdd(ctl + 1, 1u) == (unsigned int)tiles - 1u) {
    ctl[1] = 0u;
    ctl[0] = base + (uint32_t)a.n_sweeps;
  }
}

// Rows a tile warp owns and threads the kernel is compiled for, fewest rows
// first: a shape is taken where the tiles (152 CTAs: one per SM) fit it.  More
// warps of fewer rows hide each other's latency better until registers or
// threads run out; us per sweep:
//   L = 512 (tiles of 14 rows)   1 row, 640 threads 1.97   2 rows 2.6
//   L = 640 (22)                 1 row, 1024 threads 2.55  2 rows 3.13
//   L = 1024 (54)                2 rows 5.14   3 rows 5.64   4 rows 5.61
//   L = 1152 (72)                3 rows 8.24   4 rows 7.28   6 rows 7.81
// against the persistent tiles' 5.8, 6.2, 8.9 and 10.0 (1280: 8.33 against
// 11.0).  Two CTAs per SM of half the rows are slower (each has its own halo
// warps), and beyond 92 rows a tile (L > 1280) so are the shapes that fit (1536:
// 8 rows 13.6 against the tiles' 12.7).
struct Shape {
  int nr, maxt;
};
constexpr Shape kShapes[] = {{1, 640}, {1, 1024}, {2, 1024}, {4, 896}};
constexpr int kNumShapes = sizeof(kShapes) / sizeof(kShapes[0]);

struct Plan {
  int shape, nx, ny, tile_warps, threads;
  size_t smem;
};

// The tiles of a lattice of side L on `sms` multiprocessors (shape < 0: they fit none).  As
// many as there are SMs, of four rows at least: us per sweep by rows of a tile
//   L = 256   4: 1.51   8: 1.69   12: 1.91      (one cluster of 16 CTAs: 3.1)
//   L = 384   8: 1.70  12: 1.93   16: 2.09
Plan plan_of(int L, int sms) {
  Plan p = {};
  p.shape = -1;
  const int W = L / 2;
  if (L & 1) return p;
  p.nx = ((W + 1) / 2 + 31) / 32;
  p.ny = sms / p.nx < L / 4 ? sms / p.nx : L / 4;
  if (p.ny < 3) return p;
  const int rows = 2 * part_size(L / 2, p.ny, 0);
  p.smem = sizeof(CsRow) * (size_t)(2 * rows + 6);
  if (p.smem > kGridSmem) return p;
  for (int i = 0; i < kNumShapes; ++i) {
    p.tile_warps = (rows + kShapes[i].nr - 1) / kShapes[i].nr;
    p.threads = 32 * (p.tile_warps + 2 + (rows + 2 + 31) / 32);
    if (p.threads <= kShapes[i].maxt) {
      p.shape = i;
      break;
    }
  }
  return p;
}

// f(kernel) for the instantiation of a shape.
template <int MODE, bool ODD, class F>
cudaError_t with_shape(int shape, const F& f) {
  switch (shape) {
    case 0: return f(k_sweep_grid<MODE, 1, 640, ODD>);
    case 1: return f(k_sweep_grid<MODE, 1, 1024, ODD>);
    case 2: return f(k_sweep_grid<MODE, 2, 1024, ODD>);
    default: return f(k_sweep_grid<MODE, 4, 896, ODD>);
  }
}
template <class F>
cudaError_t with_kernel(int mode, int L, int shape, const F& f) {
  const bool odd = (L / 2) & 1;
  switch (mode) {
    case 0: return odd ? with_shape<0, true>(shape, f) : with_shape<0, false>(shape, f);
    case 1: return odd ? with_shape<1, true>(shape, f) : with_shape<1, false>(shape, f);
    default: return odd ? with_shape<2, true>(shape, f) : with_shape<2, false>(shape, f);
  }
}

}  // namespace

long long grid_spin_limit() { return kGridSpinLimit; }

size_t grid_words(int L) {
  return 4 * (size_t)L * (size_t)((L / 2 + 1) & ~1);
}

cudaError_t prepare_grid(int sincos_mode, int L, int sms, int replicas, bool* fits) {
  *fits = false;
  if (replicas < 1 || replicas > kGridReplicas) return cudaErrorInvalidValue;
  const Plan p = plan_of(L, sms / replicas);
  if (p.shape < 0) return cudaSuccess;
  int n = 0;
  const cudaError_t e = with_kernel(sincos_mode, L, p.shape, [&](auto* fn) {
    cudaError_t r = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)kGridSmem);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (r != cudaSuccess) return r;
    return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, fn, p.threads, p.smem);
  });
  *fits = e == cudaSuccess && n * sms >= replicas * p.nx * p.ny;
  return e;
}

cudaError_t launch_grid(int sincos_mode, const GridArgs& args, int sms, cudaStream_t stream) {
  if (args.replicas < 1 || args.replicas > kGridReplicas || args.n_sweeps < 1 || args.spin_limit < 1)
    return cudaErrorInvalidValue;
  const Plan p = plan_of(args.L, sms / args.replicas);
  if (p.shape < 0 || args.skip_tiles < 0 || args.skip_tiles >= p.nx * p.ny)
    return cudaErrorInvalidValue;
  GridArgs a = args;
  a.nx = p.nx;
  a.ny = p.ny;
  a.tile_warps = p.tile_warps;
  return with_kernel(sincos_mode, args.L, p.shape, [&](auto* fn) {
    void* params[] = {&a};
    return coop_launch(reinterpret_cast<const void*>(fn),
                       args.replicas * p.nx * p.ny - args.skip_tiles, p.threads, params, p.smem,
                       stream);
  });
}

}  // namespace xyk
