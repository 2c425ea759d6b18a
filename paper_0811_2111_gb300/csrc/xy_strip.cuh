// xy_strip.cuh -- strips of full lattice rows, one per CTA of a thread-block
// cluster: which rows a CTA holds, where a pair of sites' unit vectors lie in
// its shared memory, and how they are published to everyone that reads them.
// Shared by the resident Metropolis sweep and the resident HMC trajectory.
//
// A plane of unit vectors is (rows + 2) x (pairs + 2) float4: row r + 1 the
// strip's row r, float4 m + 1 the columns 2m, 2m + 1 as (cos, cos, sin, sin).
// Rows 0 and rows + 1 are the neighbouring strips' edge rows, column -1 (float4
// 0, second) and column `cols` the periodic copies of the last and the first
// column.  Where the number of columns is odd, column `cols` is the last pair's
// second place, and that lane's own results are dropped.
#pragma once

#include <cooperative_groups.h>
#include <cuda_runtime.h>

namespace xys {

__host__ __device__ inline int strip_rows(int L, int C, int rank) {
  return L / C + (rank < L % C ? 1 : 0);
}
__host__ __device__ inline int strip_first(int L, int C, int rank) {
  return rank * (L / C) + (rank < L % C ? rank : L % C);
}

// float4 of one plane.
__host__ __device__ inline int plane_vec4(int max_rows, int cols) {
  return (max_rows + 2) * ((cols + 1) / 2 + 2);
}

struct Strip {
  int cols, pairs, pitch;      // columns, pairs and float4 of a row
  int rows, y0;                // this CTA's rows
  int up_row, dn_row;          // float4 index of the neighbours' halo rows for this strip
  int up_rank, dn_rank;

  __device__ __forceinline__ Strip(int L, int columns, int C, int rank) {
    cols = columns;
    pairs = (columns + 1) / 2;
    pitch = pairs + 2;
    rows = strip_rows(L, C, rank);
    y0 = strip_first(L, C, rank);
    up_rank = rank + 1 == C ? 0 : rank + 1;          // holds row y0 + rows
    dn_rank = rank == 0 ? C - 1 : rank - 1;          // holds row y0 - 1
    up_row = 0;
    dn_row = (strip_rows(L, C, dn_rank) + 1) * pitch;
  }
};

// One pair of sites: its row in the strip, first column, float4 in a plane.
struct Pair {
  int r, k, at;
  bool on, two;                // owned by a thread; its second column exists
  __device__ __forceinline__ void set(const Strip& s, int i) {
    on = i < s.rows * s.pairs;
    r = on ? i / s.pairs : 0;
    const int m = on ? i - r * s.pairs : 0;
    k = 2 * m;
    at = (r + 1) * s.pitch + m + 1;
    two = k + 1 < s.cols;
  }
};

// Publishes a pair's unit vectors in plane `own` (up, dn: the same plane of
// the neighbouring CTAs, through distributed shared memory): the strip, its
// halo columns and, from the strip's edge rows, the neighbours' halo rows.
__device__ __forceinline__ void put(const Strip& s, const Pair& p, float4* own, float4* up,
                                    float4* dn, float2 c, float2 sn) {
  const float4 v = make_float4(c.x, c.y, sn.x, sn.y);
  if (p.two) {
    own[p.at] = v;
  } else {                                 // the halo copy in the second place stays
    float* f = reinterpret_cast<float*>(&own[p.at]);
    f[0] = v.x;
    f[2] = v.z;
  }
  float* row = reinterpret_cast<float*>(&own[(p.r + 1) * s.pitch]);
  if (p.k == 0) {                          // column 0 -> column `cols`
    float* f = row + 4 * ((s.cols + 2) >> 1) + (s.cols & 1);
    f[0] = v.x;
    f[2] = v.z;
  }
  if (p.k + 2 >= s.cols) {                 // the last column -> column -1
    row[1] = p.two ? v.y : v.x;
    row[3] = p.two ? v.w : v.z;
  }
  const int m = (p.k >> 1) + 1;
  if (p.r == 0) dn[s.dn_row + m] = v;
  if (p.r == s.rows - 1) up[s.up_row + m] = v;
}

}  // namespace xys
