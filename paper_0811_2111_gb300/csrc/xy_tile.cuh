// xy_tile.cuh -- rows of unit vectors in shared memory, 64 plane columns and one
// or two halo columns on either side: how a warp's lanes (a pair of columns
// each) read and write them, and a pair's four neighbours.  Shared by the fused
// sweeps (tiles staged from memory) and the sweep whose tiles stay on the chip.
#pragma once

#include <cuda_runtime.h>

#include "xy_device.cuh"

namespace xyk {

namespace {

constexpr int kTileK = 64;                   // plane columns (2 per lane)
// a row: column c is place c + kCsOff, two columns per float4 as (cos, cos,
// sin, sin), the operands of the packed FP32 instructions: lane l's pair is
// float4 l + 1
constexpr int kCsOff = 2;
constexpr int kCsPairs = kTileK / 2 + 2;
typedef float4 CsRow[kCsPairs];

__device__ __forceinline__ int wrap_once(int v, int n) {
  v += (v < 0) ? n : 0;
  v -= (v >= n) ? n : 0;
  return v;
}

// The cosine and sine pairs of a float4 of unit vectors.
__device__ __forceinline__ float2 cosines(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 sines(const float4& v) { return make_float2(v.z, v.w); }

__device__ __forceinline__ void put_pair(float4* at, const float2& c, const float2& s) {
  *at = make_float4(c.x, c.y, s.x, s.y);
}

// The unit vector (cos, sin) at unit-vector column c of a row.
__device__ __forceinline__ float2 get_one(const CsRow& row, int c) {
  const float* p = reinterpret_cast<const float*>(&row[c >> 1]) + (c & 1);
  return make_float2(p[0], p[2]);
}

__device__ __forceinline__ void put_one(CsRow& row, int c, float cv, float sv) {
  float* p = reinterpret_cast<float*>(&row[c >> 1]) + (c & 1);
  p[0] = cv;
  p[2] = sv;
}

// The four neighbour unit vectors of the two sites of pair j of row i of the
// other colour's unit vectors `nb`, where a site at column c has its same-row
// neighbours at c+q-1 and c+q.  The three same-row columns are the pair's own
// and one of the pair before (q = 0) or after (q = 1); q is a compile-time
// constant where the row loops are unrolled (rows alternate q), so no selects
// are issued.  Rows i-1 and i of the pair's columns come in as D and P (a warp
// walks its rows downwards, so they are the previous row's P and U); row i+1
// is loaded and returned in U.
__device__ __forceinline__ void pair_neighbours(const CsRow* nb, int i, int j, int q,
                                                const float4 D, const float4 P, float4& U,
                                                xyd::PairNeighbours& n) {
  const float4 E = nb[i][q ? j + 1 : j - 1];
  U = nb[i + 1][j];
  if (q) {
    n.lc = cosines(P);
    n.ls = sines(P);
    n.rc = make_float2(P.y, E.x);
    n.rs = make_float2(P.w, E.z);
  } else {
    n.lc = make_float2(E.y, P.x);
    n.ls = make_float2(E.w, P.z);
    n.rc = cosines(P);
    n.rs = sines(P);
  }
  n.dc = cosines(D);
  n.ds = sines(D);
  n.uc = cosines(U);
  n.us = sines(U);
  n.sum();
}

}  // namespace

}  // namespace xyk
