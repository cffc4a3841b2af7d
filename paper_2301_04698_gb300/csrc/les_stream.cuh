// les_stream.cuh -- tiles, runs of planes and sums of the persistent kernels that
// march any grid from memory (les_cg_stream.cu, les_jacobi.cu).
#pragma once

#include <algorithm>

#include "les_gridsync.cuh"

namespace les {

constexpr int kStreamThreads = 256;

// tile shapes: WX x WY columns, NO per thread (x = lane + 32 (m mod NWX),
// y = warp + 8 (m / NWX)), planes of (WY + 2) rows of SP elements
template <int WX_, int WY_>
struct StreamTile {
  static constexpr int WX = WX_, WY = WY_, NWX = WX / 32, NO = WX * WY / kStreamThreads;
  static constexpr int SP = WX + 2, SN = SP * (WY + 2);
  static_assert(2 * (WX + WY) <= kStreamThreads && 8 * (NO / NWX) == WY, "one ring node per thread");
};

__device__ __forceinline__ void stream_part(int n, int parts, int i, int& first, int& len) {
  const int base = n / parts, rem = n - base * parts;
  len = base + (i < rem ? 1 : 0);
  first = i * base + min(i, rem);
}
__device__ __forceinline__ int stream_wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }
__device__ __forceinline__ int stream_z(int k, int nz, int walls) {
  if (walls) return k < 0 ? -1 - k : (k >= nz ? 2 * nz - 1 - k : k);
  return k < 0 ? k + nz : (k >= nz ? k - nz : k);
}

// The ring node of thread tid around a tile of w x h nodes at (x0, y0): its
// offset in a plane of the grid (-1: none) and in a staged plane.
template <typename S>
__device__ __forceinline__ void stream_ring(int tid, int x0, int y0, int w, int h, int nx, int ny, int& gr, int& er) {
  gr = -1, er = 0;
  int ex, ey;
  if (tid < 2 * w) ex = tid < w ? tid : tid - w, ey = tid < w ? -1 : h;
  else if (tid < 2 * (w + h)) ex = tid - 2 * w < h ? -1 : w, ey = (tid - 2 * w) - (tid - 2 * w < h ? 0 : h);
  else return;
  gr = stream_wrap(y0 + ey, ny) * nx + stream_wrap(x0 + ex, nx);
  er = (ey + 1) * S::SP + ex + 1;
}

// Per-thread sums: the FP32 terms of one plane or 16-byte chunk (at most four) are
// added in FP32, all else in FP64
template <typename T>
struct StreamSum;
template <>
struct StreamSum<float> {
  double s = 0.0;
  float run = 0.f;
  __device__ __forceinline__ void add(float v) { run += v; }
  __device__ __forceinline__ void tick() {
    s += (double)run;
    run = 0.f;
  }
};
template <>
struct StreamSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ void tick() {}
};
template <int NV, typename T>
__device__ __forceinline__ bool stream_sum(const StreamSum<T> (&d)[NV], GridSync& gs, double (&tot)[NV]) {
  double v[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) v[q] = d[q].s;
  return grid_sum_t0<NV>(v, gs, tot);
}
// The same, of FP32 terms whose sum is about 2^e: the threads' sums, scaled so, are
// combined as FP32 pairs, whatever their range (an FP64 sum across the grid takes 1.9 us
// longer: 470 x 239 x 58 55.1 us per iteration against 52.9).
__device__ __forceinline__ double pow2(int e) { return __hiloint2double((1023 + max(-1022, min(1023, e))) << 20, 0); }
__device__ __forceinline__ bool stream_sum_scaled(const StreamSum<float>& d, int e, GridSync& gs, double& tot) {
  const double v = d.s * pow2(-e);
  const float hi = (float)v;
  F2 p[1] = {F2{hi, (float)(v - (double)hi)}}, t[1];
  const bool ok = grid_sum_t0_acc<1>(p, gs, t, NoWork{});
  if (threadIdx.x == 0) tot = f2_value(t[0]) * pow2(e);
  return ok;
}
__device__ __forceinline__ bool stream_sum_scaled(const StreamSum<double>& d, int, GridSync& gs, double& tot) {
  double v[1] = {d.s}, t[1];
  const bool ok = grid_sum_t0<1>(v, gs, t);
  if (threadIdx.x == 0) tot = t[0];
  return ok;
}

// nodes handled together in the streaming sweeps: 16 bytes
template <typename T>
struct StreamVec {
  static constexpr int N = 16 / (int)sizeof(T);
  T v[N];
};
template <typename T>
__device__ __forceinline__ StreamVec<T> svld(const T* p) {
  const uint4 u = __ldcg(reinterpret_cast<const uint4*>(p));
  StreamVec<T> r;
  memcpy(&r, &u, 16);
  return r;
}
template <typename T>
__device__ __forceinline__ void svst(T* p, const StreamVec<T>& r) {
  uint4 u;
  memcpy(&u, &r, 16);
  __stcg(reinterpret_cast<uint4*>(p), u);
}

using Tile64 = StreamTile<64, 16>;
using Tile32 = StreamTile<32, 32>;
using Tile32s = StreamTile<32, 16>;

// The work of a launch: units (a tile's run of planes) dealt to the blocks in turns,
// nchunk runs per tile; or (nchunk = 0) the planes of all tiles one after the other in
// equal shares, a share being the end of one tile's planes and the beginning of
// another's.
struct StreamPlan {
  int shape = 0, ntx = 0, nty = 0, nchunk = 1;
  long long units = 0;  // units, or planes
};
template <bool Shares>
struct StreamTurns {
  int u, end;  // a tile has 512 nodes or more: the planes of all tiles are an int
  __device__ __forceinline__ explicit StreamTurns(int units) {
    u = blockIdx.x;
    end = units;
    if (Shares) {
      int len;
      stream_part(units, gridDim.x, blockIdx.x, u, len);
      end = u + len;
    }
  }
  // the block's next tile and its planes k0 .. k0 + kn - 1
  __device__ __forceinline__ bool next(int nchunk, int nz, int& tile, int& k0, int& kn) {
    if (u >= end) return false;
    if (Shares) {
      tile = u / nz;
      k0 = u - tile * nz;
      kn = min(nz - k0, end - u);
      u += kn;
    } else {
      tile = u / nchunk;
      stream_part(nz, nchunk, u - tile * nchunk, k0, kn);
      u += gridDim.x;
    }
    return true;
  }
};
// The tile shape and the division of the planes with the least work of the busiest
// block, in node slots (every lane counts, with a node or without).  A run costs
// planes beyond its own -- one more of p and the fill of its loads -- and a plane
// costs slots beyond its nodes: its ring and, where arithmetic does not hide them
// (FP32), the barrier and the loop.  Fitted to timed plans: FP64 200 x 180 x 90
// prefers 32 x 16 tiles (100 us per iteration against 108 with 64 x 16), FP32 470 x
// 239 x 58 64 x 16 ones (56 us against 70).  Equal shares, for FP64 alone: 256 x 256 x
// 128 192 -> 187 us, 512 x 512 x 128 719 -> 678, 512 x 256 x 64 202 -> 188; their
// neighbours in the grid are at other planes at the time, and where memory bounds the
// march (FP32) their rings are then read twice: 470 x 239 x 58 54 us in runs, 59 in
// shares.
inline StreamPlan make_stream_plan(int nx, int ny, int nz, long long G, bool fp64) {
  static constexpr int shapes[3][2] = {{64, 16}, {32, 32}, {32, 16}};
  StreamPlan best;
  double cost = 0;
  for (int q = 0; q < 3; ++q) {
    const int wx = shapes[q][0], wy = shapes[q][1];
    const int ntx = (nx + wx - 1) / wx, nty = (ny + wy - 1) / wy;
    const long long tiles = (long long)ntx * nty;
    const double plane = fp64 ? wx * wy + 0.5 * (wx + wy) + 24.0 : wx * wy + (wx + wy) + (wx == 64 ? 200.0 : 240.0);
    const double fill = fp64 ? 0.7 : 2.0;
    auto offer = [&](double planes, int nchunk, long long units) {
      if (best.units == 0 || planes * plane < cost) {
        cost = planes * plane;
        best = {q, ntx, nty, nchunk, units};
      }
    };
    // for each number of turns as many runs of planes per tile as fill them
    for (int turns = 1; turns <= 8; ++turns) {
      const long long nchunk = std::max<long long>(1, std::min<long long>(nz, G * turns / tiles));
      const long long units = tiles * nchunk, per = (units + G - 1) / G;
      offer((double)per * ((double)((nz + nchunk - 1) / nchunk) + fill), (int)nchunk, units);
    }
    // a share of `per` planes touches at most (per - 2) / nz + 2 tiles
    const long long per = (tiles * nz + G - 1) / G;
    if (fp64) offer((double)per + 1.5 * (double)(per > 1 ? (per - 2) / nz + 2 : 1), 0, tiles * nz);
  }
  return best;
}

}  // namespace les
