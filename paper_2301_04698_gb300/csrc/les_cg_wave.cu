// les_cg_wave.cu -- conjugate-gradient Poisson solve in one persistent
// cooperative launch with one pass over memory and one grid-wide sum per
// iteration, for grids whose horizontal extents are multiples of 64 x 16 or
// 32 x 32 (Sec. 2.4: L_c psi = b, compact 7-point Laplacian, periodic in x, y,
// mirror or periodic in z; mean of b removed, psi returned with zero mean).
//
// The iterates are those of standard CG, formed as in the one-pass kernel of
// les_cg_roll.cu: with alpha_i and beta_i known, iteration i forms
//   p_i = r_i + beta_i p_{i-1},  q_i = L_c p_i,  x += alpha_i p_i,
//   r_{i+1} = r_i - alpha_i q_i,  w = L_c r_{i+1},
// and r'.r', r'.w, r'.q, p.q (r' = r_{i+1}) in one grid-wide sum; then
// alpha_{i+1} = r'.r' / (r'.w + 2 beta r'.q + beta^2 p.q) and
// beta_{i+1} = r'.r' / r_i.r_i (p_{i+1}.L_c p_{i+1} expanded with L_c
// symmetric), every vector formed from its definition.
//
// A block owns a column of 128 x 16, 64 x 16 or 32 x 32 nodes and marches a run of
// planes.  A thread holds a pair of nodes along x in two adjacent rows, and some
// threads one pair of the column's halo of two, for the whole run, so the z
// neighbours of both stencils are registers: per pair p on the planes f-2 .. f, r'
// on f-3 .. f-1 and r_i on f-1 .. f, where f is the plane that enters the march.
// The other row is a register too; the remaining in-plane neighbours pass through
// shared memory (one plane of p and one of r', each double-buffered).  The planes
// of r_i and p_{i-1} (halo two) arrive by TMA through rings filled five planes
// ahead, one mbarrier per ring slot, and x a plane ahead in registers.  Per plane
// step, after one block barrier:
//   A  p(f) = r(f) + beta p_old(f), stored; every other pass, x += alpha_{i-1}
//      p_old + alpha_i p
//   B  q(f-1) = L_c p, r'(f-1) = r(f-1) - alpha q(f-1) within the halo of one,
//      stored
//   C  w(f-2) = L_c r' at the owned nodes
// r and p are double-buffered by iteration parity (the pass reads the
// neighbours' r_i while writing r_{i+1}); the grid sum is the barrier
// between passes.  Per iteration each node's r_i and p_{i-1} are read and p_i and
// r_{i+1} written, and x is read and written every other one (an update of x
// needs nothing of q: both take place where p_{i-1} and p_i are at hand, in one
// pass out of two, which saves 4 of 24 bytes).  Every other pass takes the columns
// and their planes in reverse and so begins with what the last one left in L2.
//
// What bounds it: memory.  768 x 768 x 128 in FP32 takes 321 us an iteration, where
// its 20 bytes a node would take 222 us at the rate of a plain copy; without the
// arithmetic of B and C it takes 309 us, without the copies 232.  With one node per
// lane and position, windows that were moved each step and half the columns' planes
// fetched by every thread it was bound by instruction issue (132 a node, 393 us).
// What took it from there, in that order: pairs in packed FP32 arithmetic with a
// march unrolled by six (windows, ring slots and buffers known at compile time),
// the copies left to two threads, rows of 288 bytes instead of strips, byte
// pointers that follow the march (351 -> 325 us), the reverse passes (341 -> 322).
#include <cuda.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdint>
#include <mutex>
#include <string>

#include <type_traits>

#include "les_gridsync.cuh"
#include "les_internal.h"

namespace les {
namespace {

constexpr int WH = 2;  // halo of the staged planes
constexpr int D = 6;   // r_i / p_{i-1} rings: planes f .. f+5

// A column shape: WX x WY owned nodes in pairs along x.
// A thread owns a pair in two adjacent rows, and one of its threads each pair
// of the halo ring, those within the halo of one first (the rows and pairs next
// to the owned ones), then the two outer rows.
template <int WX_, int WY_>
struct Col {
  static constexpr int WX = WX_, WY = WY_, PX = WX / 2;
  static constexpr int NT = PX * WY / 2;                // threads
  static constexpr int NH1 = 2 * (PX + 2) + 2 * WY;     // pairs of the halo of one
  static constexpr int NH = NH1 + 2 * (PX + 2);         // and with the outer rows
  static constexpr int SP = WX + 4, SN = SP * (WY + 2 * WH);  // a plane of p or r' with its halo
  static_assert(NT % 256 == 0 && NH <= NT - 64 && WY % 8 == 0, "column shape and thread count");
};
using Col128 = Col<128, 16>;
using Col64 = Col<64, 16>;
using Col32 = Col<32, 32>;

// A staged plane of r_i or p_{i-1}.  A column inside the grid takes boxes of
// rows with 16 bytes of halo at either end; one at an x edge, whose halo wraps,
// takes the owned nodes and, as a strip of 16-byte rows each, the two ends (a
// strip costs the copy engine as many requests as the owned rows: with strips in
// every column 768 x 768 x 128 took 338 us an iteration).
// All rows come in one box; in a column at a y edge the two rows below, the WY
// owned and the two above come in three, each on a 128-byte boundary.
template <typename T, typename C>
struct Staged {
  static constexpr int SZ = (int)sizeof(T), SW = 16 / SZ;  // nodes of a strip's row
  static constexpr int ROWS = C::WY + 2 * WH;
  static constexpr int RW = C::WX + 2 * SW;                               // a row with its ends
  static constexpr int O1 = (WH * RW * SZ + 127) / 128 * 128;             // bytes: the owned rows of a y edge
  static constexpr int CB = C::WX * ROWS * SZ, SB = C::WY * 16 + 256;     // bytes: owned columns, a strip
  static constexpr int RB = CB + 2 * SB;                                  // bytes: the whole
  static constexpr unsigned TX = (unsigned)(RW * ROWS * SZ);              // bytes that arrive
  static_assert(CB % 128 == 0 && RB % 128 == 0 && WH * C::WX * SZ % 128 == 0 && C::WY * RW * SZ % 128 == 0 &&
                    C::WY * 16 % 128 == 0 && 16 * ROWS <= SB && O1 + (C::WY + WH) * RW * SZ <= RB,
                "box alignment");
};

template <typename T, typename C>
constexpr size_t wave_smem() {
  return (size_t)D * 2 * Staged<T, C>::RB + (size_t)4 * C::SN * sizeof(T);
}

// pairs of nodes: packed FP32 arithmetic (two results per instruction, each
// rounded as by the scalar one)
template <typename T>
struct Vec2;
template <>
struct Vec2<float> {
  using V = float2;
};
template <>
struct Vec2<double> {
  using V = double2;
};
__device__ __forceinline__ float2 vadd(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 vmul(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 vfma(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ double2 vadd(double2 a, double2 b) { return double2{a.x + b.x, a.y + b.y}; }
__device__ __forceinline__ double2 vmul(double2 a, double2 b) { return double2{a.x * b.x, a.y * b.y}; }
__device__ __forceinline__ double2 vfma(double2 a, double2 b, double2 c) {
  return double2{fma(a.x, b.x, c.x), fma(a.y, b.y, c.y)};
}

template <typename T>
struct WaveArgs {
  // TMA descriptors of r[0], r[1], p[0], p[1]: boxes of rows with their ends, of
  // the owned columns, of a strip, each WY + 4, WY and 2 rows high
  CUtensorMap tm[4][3][3];
  int nx, ny, nz, walls;
  T cx, cy, cz;  // 1/dx^2, 1/dy^2, 1/dz^2
  int ntx, nty, zrun, nchunk;
  // runs of a block: units (column, z-run of zrun planes) u = blockIdx.x,
  // + gridDim.x, ... below nunits; then an equal share (tail_per planes) of the
  // tail_planes of the columns left
  int nunits, tail_planes, tail_per;
  long long n;
  const T* b;
  T* x;
  T* r[2];  // r_i in r[i & 1]
  T* p[2];  // p_i in p[i & 1]
  double* partials;
  FusedBar* bar;
  SolverCtl* ctl;
  double tol;
  int maxit;
  long long spin_cycles;
  unsigned expected;
  int guard;
};

__device__ __forceinline__ int wrapw(int i, int n) {
  while (i < 0) i += n;
  while (i >= n) i -= n;
  return i;
}
// the stored plane that stands for plane k: mirror images across the walls
// (planes beyond one image: any valid plane, unused), or periodic
__device__ __forceinline__ int zmapw(int k, int nz, int walls) {
  if (walls) {
    k = k < 0 ? -1 - k : (k >= nz ? 2 * nz - 1 - k : k);
    return k < 0 ? 0 : (k >= nz ? nz - 1 : k);
  }
  return wrapw(k, nz);
}

// Long per-thread sums: FP32 within a run of 16 planes, compensated across
template <typename T>
struct WaveSum;
template <>
struct WaveSum<float> {
  F2 s{0.f, 0.f};
  float run = 0.f;
  __device__ __forceinline__ void add(float v) { run += v; }
  __device__ __forceinline__ void add(float2 v) {
    f2_acc(s, v.x);
    f2_acc(s, v.y);
  }
  __device__ __forceinline__ void flush() {
    f2_acc(s, run);
    run = 0.f;
  }
  __device__ __forceinline__ F2 acc() const { return s; }
};
template <>
struct WaveSum<double> {
  double s = 0.0;
  __device__ __forceinline__ void add(double v) { s += v; }
  __device__ __forceinline__ void add(double2 v) { s += v.x + v.y; }
  __device__ __forceinline__ void flush() {}
  __device__ __forceinline__ double acc() const { return s; }
};

template <int NV, typename T>
__device__ __forceinline__ bool wave_sum_t0(WaveSum<T> (&d)[NV], GridSync& gs, double (&tot)[NV]) {
  decltype(d[0].acc()) v[NV];
#pragma unroll
  for (int q = 0; q < NV; ++q) {
    d[q].flush();
    v[q] = d[q].acc();
  }
  return grid_sum_t0<NV, 2>(v, gs, tot);
}

// mbarrier and TMA (cp.async.bulk.tensor) helpers
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, unsigned parity) {
  unsigned ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, int x, int y, int z, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::
          "r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(smem_u32(bar))
      : "memory");
}

template <typename T, typename C>
__global__ void __launch_bounds__(C::NT, sizeof(T) == 4 ? 512 / C::NT : 1) k_cg_wave(const __grid_constant__ WaveArgs<T> f) {
  constexpr int WX = C::WX, WY = C::WY, PX = C::PX, NT = C::NT, SP = C::SP, SN = C::SN;
  using G = Staged<T, C>;
  using V = typename Vec2<T>::V;
  extern __shared__ __align__(128) unsigned char smraw[];
  unsigned char* const RINGR = smraw;                        // [D][RB] r_i as copied
  unsigned char* const RINGP = RINGR + D * G::RB;            // [D][RB] p_{i-1} as copied
  T* const PP = reinterpret_cast<T*>(RINGP + D * G::RB);     // [2][SN] p of a plane, alternating
  T* const RP = PP + 2 * SN;                                 // [2][SN] r' of a plane, alternating
  // one barrier per ring slot: the TMA copies of a plane (r_i, p_{i-1})
  // complete on it; bit s of phase is the parity this thread waits for next
  __shared__ __align__(8) uint64_t bars[D];
  __shared__ decltype(WaveSum<T>().acc()) sums[4][NT];
  __shared__ long long limit;  // of a wait for copies; -1: one has run out
  unsigned phase = 0;
  if (threadIdx.x == 0) {
    limit = f.spin_cycles;
    for (int q = 0; q < D; ++q) mbar_init(&bars[q], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  __shared__ struct {
    T ta, tb, mean;
    int status, restart;
  } sc;
  const int tid = threadIdx.x;
  const long long ncol = (long long)f.ntx * f.nty;
  const size_t plane = (size_t)f.nx * f.ny;
  const T cx = f.cx, cy = f.cy, cz = f.cz;
  GridSync gs{f.bar, f.partials, f.spin_cycles, f.expected, 0u};
  const long long gstride = (long long)gridDim.x * NT;
  const long long gtid = (long long)blockIdx.x * NT + tid;

  // the set-up and gauge sweeps in 16-byte chunks of VC nodes along x (nx is
  // a multiple of 32 and every vector 16-byte aligned here), chunks dealt to
  // the grid's threads in order
  constexpr int VC = 16 / (int)sizeof(T);
  using VQ = typename std::conditional<sizeof(T) == 4, float4, double2>::type;
  struct Ch {
    T e[VC];
  };
  auto ldch = [](const T* ptr) -> Ch {
    const VQ q = __ldcg(reinterpret_cast<const VQ*>(ptr));
    Ch c;
    if constexpr (sizeof(T) == 4) {
      c.e[0] = q.x, c.e[1] = q.y, c.e[2] = q.z, c.e[3] = q.w;
    } else {
      c.e[0] = q.x, c.e[1] = q.y;
    }
    return c;
  };
  auto stch = [](T* ptr, const Ch& c) {
    VQ q;
    if constexpr (sizeof(T) == 4) {
      q.x = c.e[0], q.y = c.e[1], q.z = c.e[2], q.w = c.e[3];
    } else {
      q.x = c.e[0], q.y = c.e[1];
    }
    __stcg(reinterpret_cast<VQ*>(ptr), q);
  };
  const long long nch = f.n / VC;
  const int cpr = f.nx / VC;  // chunks per row
  // a chunk's place (i / VC, j, k) and the grid's stride as one
  const int pi0 = (int)(gtid % cpr), si = (int)(gstride % cpr);
  const int pj0 = (int)(gtid / cpr % f.ny), sj = (int)(gstride / cpr % f.ny);
  const int pk0 = (int)(gtid / cpr / f.ny), sk = (int)(gstride / cpr / f.ny);
  auto each_chunk = [&](auto&& body) {
    int pi = pi0, pj = pj0, pk = pk0;
    for (long long c = gtid; c < nch; c += gstride) {
      body((size_t)c * VC, pi * VC, pj, pk);
      pi += si;
      pj += sj;
      pk += sk;
      if (pi >= cpr) pi -= cpr, ++pj;
      if (pj >= f.ny) pj -= f.ny, ++pk;
    }
  };
  // the 7-point operator at a chunk's nodes straight from global memory
  // (set-up sweeps only), and the chunk's own values
  auto lap_chunk = [&](const T* v, size_t m, int i0, int j, int k, Ch& lap, Ch& own) {
    const size_t row = (size_t)k * plane + (size_t)j * f.nx;
    own = ldch(v + m);
    const T xl = __ldcg(v + row + wrapw(i0 - 1, f.nx)), xr = __ldcg(v + row + wrapw(i0 + VC, f.nx));
    const Ch ym = ldch(v + (size_t)k * plane + (size_t)wrapw(j - 1, f.ny) * f.nx + i0);
    const Ch yp = ldch(v + (size_t)k * plane + (size_t)wrapw(j + 1, f.ny) * f.nx + i0);
    const Ch zm = ldch(v + (size_t)zmapw(k - 1, f.nz, f.walls) * plane + (size_t)j * f.nx + i0);
    const Ch zp = ldch(v + (size_t)zmapw(k + 1, f.nz, f.walls) * plane + (size_t)j * f.nx + i0);
#pragma unroll
    for (int q = 0; q < VC; ++q) {
      const T c2 = T(2) * own.e[q];
      const T xm = q == 0 ? xl : own.e[q - 1], xp = q == VC - 1 ? xr : own.e[q + 1];
      lap.e[q] = (xm + xp - c2) * cx + (ym.e[q] + yp.e[q] - c2) * cy + (zm.e[q] + zp.e[q] - c2) * cz;
    }
  };

  double rr = 0.0, bb = 0.0, rel = 0.0, pq = 0.0;  // meaningful in thread 0
  int status = 0;  // 0 running, 1 converged, 2 maxit, 3 breakdown, 4 zero rhs, 5 timeout

  // ---- set-up: mean of b ---------------------------------------------------------
  {
    WaveSum<T> s[1];
    int cnt = 0;
    for (long long c = gtid; c < nch; c += gstride) {
      const Ch bq = ldch(f.b + (size_t)c * VC);
#pragma unroll
      for (int q = 0; q < VC; ++q) s[0].add(bq.e[q]);
      if ((++cnt & 3) == 0) s[0].flush();
    }
    double t[1];
    const bool ok = wave_sum_t0<1>(s, gs, t);
    if (tid == 0) {
      sc.status = ok ? 0 : 5;
      sc.mean = (T)(t[0] / (double)f.n);
    }
    __syncthreads();
    status = sc.status;
  }
  const T mean = sc.mean;
  // ---- r_0 = (b - mean) - L_c x0 into r[0]; r.r and |b - mean|^2 ----------------
  if (!status) {
    WaveSum<T> s[2];
    int cnt = 0;
    each_chunk([&](size_t m, int i0, int j, int k) {
      Ch lap, xo;
      lap_chunk(f.x, m, i0, j, k, lap, xo);
      const Ch bq = ldch(f.b + m);
      Ch rq;
#pragma unroll
      for (int q = 0; q < VC; ++q) {
        const T bm = bq.e[q] - mean;
        const T rv = bm - lap.e[q];
        rq.e[q] = rv;
        s[0].add(rv * rv);
        s[1].add(bm * bm);
      }
      stch(f.r[0] + m, rq);
      if ((++cnt & 3) == 0) {
        s[0].flush();
        s[1].flush();
      }
    });
    double t[2];
    const bool ok = wave_sum_t0<2>(s, gs, t);
    if (tid == 0) {
      // the plain solver judges a learned first guess: if it leaves a larger
      // residual than x0 = 0, restart from zero (r = b - mean b, r.r = |b|^2)
      sc.status = ok ? 0 : 5;
      sc.restart = ok && f.guard && t[0] > t[1];
      rr = sc.restart ? t[1] : t[0];
      bb = t[1];
    }
    __syncthreads();
    status = sc.status;
    if (!status && sc.restart) {
      for (long long m = gtid; m < f.n; m += gstride) {
        __stcg(f.x + m, T(0));
        __stcg(f.r[0] + m, __ldcg(f.b + m) - mean);
      }
      WaveSum<T> none[1];
      double t1[1];
      const bool ok2 = wave_sum_t0<1>(none, gs, t1);  // a grid barrier: r_0 complete everywhere
      if (tid == 0) sc.status = ok2 ? 0 : 5;
      __syncthreads();
      status = sc.status;
    }
  }
  if (tid == 0) {
    if (!status) {
      if (bb == 0.0) status = 4;
      else {
        rel = sqrt(rr / bb);
        if (rel <= f.tol) status = 1;
        else if (f.maxit <= 0) status = 2;
      }
    }
    sc.status = status;
  }
  __syncthreads();
  status = sc.status;
  // ---- p_0 = r_0: r_0 . L_c r_0 gives alpha_0 --------------------------------------
  if (!status) {
    WaveSum<T> s[1];
    int cnt = 0;
    each_chunk([&](size_t m, int i0, int j, int k) {
      Ch lap, ro;
      lap_chunk(f.r[0], m, i0, j, k, lap, ro);
#pragma unroll
      for (int q = 0; q < VC; ++q) s[0].add(ro.e[q] * lap.e[q]);
      if ((++cnt & 3) == 0) s[0].flush();
    });
    double t[1];
    const bool ok = wave_sum_t0<1>(s, gs, t);
    if (tid == 0) {
      pq = t[0];
      if (!ok) status = 5;
      else if (pq == 0.0 || !isfinite(pq)) status = 3;
      else {
        sc.ta = (T)(rr / pq);
        sc.tb = T(0);
      }
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
  }

  // ---- iterations ----------------------------------------------------------------
  const V vcx{cx, cx}, vcy{cy, cy}, vcz{cz, cz}, m2{T(-2), T(-2)};
  // L_c at the pair c with its left and right nodes and its neighbours in y and z
  auto lap = [&](T l, V c, T r, V ym, V yp, V zm, V zp) -> V {
    const V sx = vfma(c, m2, V{l + c.y, c.x + r}), sy = vfma(c, m2, vadd(ym, yp)), sz = vfma(c, m2, vadd(zm, zp));
    return vfma(sz, vcz, vfma(sy, vcy, vmul(sx, vcx)));
  };
  auto ld2 = [](const T* q) -> V { return *reinterpret_cast<const V*>(q); };
  auto st2 = [](T* q, V v) { *reinterpret_cast<V*>(q) = v; };
  auto st2g = [](T* q, V v) { __stcg(reinterpret_cast<V*>(q), v); };
  int iter = 0;
  T ta = T(0);  // alpha of the last pass
  while (!status) {
    const T tp = ta;  // alpha_{i-1}
    ta = sc.ta;
    const T tb = sc.tb;
    const V vtp{tp, tp}, vta{ta, ta}, vna{-ta, -ta}, vtb{tb, tb};
    // x takes two updates every other pass: p_{i-1} is read anyway
    const bool upd = iter & 1;
    // every other pass takes the units and their planes in reverse: it begins
    // with what the last one left in L2
    const bool rev = upd;
    T* ro = f.r[(iter + 1) & 1];
    T* pw = f.p[iter & 1];
    // r'.r', r'.w, r'.q, p.q: of a run of planes, and in shared memory of the pass
    V run[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      run[q] = V{T(0), T(0)};
      sums[q][tid] = decltype(WaveSum<T>().acc()){};
    }
    auto flush = [&]() {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        WaveSum<T> a{sums[q][tid]};
        a.add(run[q]);
        sums[q][tid] = a.acc();
        run[q] = V{T(0), T(0)};
      }
    };
    // r and p of the last pass, written by plain stores, are read by TMA
    asm volatile("fence.proxy.async;" ::: "memory");
    const int nfull = f.nunits > (int)blockIdx.x ? (f.nunits - 1 - (int)blockIdx.x) / (int)gridDim.x + 1 : 0;
    const int ts = min((int)blockIdx.x * f.tail_per, f.tail_planes), te = min(ts + f.tail_per, f.tail_planes);
    int ui = 0, tt = ts;  // units done, next plane of the tail
    for (;;) {
      int col, k0, k1;
      if (ui < nfull && (!rev || tt >= te)) {
        const int u = (int)blockIdx.x + (rev ? nfull - 1 - ui : ui) * (int)gridDim.x;
        col = u % (int)ncol;
        k0 = (u / (int)ncol) * f.zrun;
        k1 = min(k0 + f.zrun, f.nz);
        ++ui;
      } else if (tt < te) {  // the units, if any, are whole columns here
        col = f.nunits + tt / f.nz;
        k0 = tt % f.nz;
        k1 = min(f.nz, k0 + (te - tt));
        tt += k1 - k0;
      } else {
        break;
      }
      if (rev) {  // planes counted from the top
        const int k = k0;
        k0 = f.nz - k1;
        k1 = f.nz - k;
      }
      auto stored = [&](int k) { return rev ? f.nz - 1 - k : k; };
      const int x0 = (col % f.ntx) * WX, y0 = (col / f.ntx) * WY;
      // this thread's pairs: owned rows py and py + 1, and one of the halo (formed
      // again for each unit: held across them they cost spills)
      int t = tid;
      asm volatile("" : "+r"(t));
      const int px = 2 * (t % PX), py = 2 * (t / PX);
      const int eo = (py + WH) * SP + px + 2;  // in a plane of p or r'; the halo pair's: eh
      int hrow, hpair;
      if (t < 2 * (PX + 2)) {
        hrow = t < PX + 2 ? -1 : WY;
        hpair = t % (PX + 2) - 1;
      } else if (t < C::NH1) {
        hrow = (t - 2 * (PX + 2)) >> 1;
        hpair = (t & 1) ? PX : -1;
      } else {
        const int j = min(t - C::NH1, 2 * (PX + 2) - 1);
        hrow = j < PX + 2 ? -2 : WY + 1;
        hpair = j % (PX + 2) - 1;
      }
      const bool halo2 = t < C::NH, halo1 = t < C::NH1;
      const int eh = (hrow + WH) * SP + 2 * hpair + 2;
      const int go = (y0 + py) * f.nx + x0 + px;  // in-plane global offset of the lower pair
      // an interior column's rows are one box, those of a y edge three
      const bool yin = y0 >= WH && y0 + WY + WH <= f.ny;
      const bool xin = x0 > 0 && x0 + WX < f.nx;
      // the pairs in a staged plane
      const int pitch = xin ? G::RW : WX;
      auto row_at = [&](int row, int p, int o1) {  // o1: bytes, of the owned rows of a y edge
        return yin ? (row + WH) * p : (row < 0 ? (row + WH) * p : o1 / G::SZ + row * p);
      };
      int so[2], ho;
      if (xin) {
        so[0] = row_at(py, G::RW, G::O1) + G::SW + px;
        ho = row_at(hrow, G::RW, G::O1) + G::SW + 2 * hpair;
      } else {
        so[0] = (py + WH) * WX + px;
        if (hpair >= 0 && hpair < PX) ho = (hrow + WH) * WX + 2 * hpair;
        else if (hpair < 0) ho = G::CB / G::SZ + row_at(hrow, G::SW, 128) + G::SW - 2;
        else ho = (G::CB + G::SB) / G::SZ + row_at(hrow, G::SW, 128);
      }
      so[1] = so[0] + pitch;
      const int xl = x0 == 0 ? f.nx - G::SW : x0 - G::SW, xr = x0 + WX == f.nx ? 0 : x0 + WX;
      // plane kk of r_i or (isp) p_{i-1} into ring slot sl, issued by one thread
      auto copy = [&](bool isp, int sl, int kk) {
        if (kk > k1 + 1) return;
        const int zs = stored(zmapw(kk, f.nz, f.walls));
        if (!isp) mbar_expect_tx(&bars[sl], 2 * G::TX);
        const CUtensorMap(*tm)[3] = f.tm[isp && iter ? 2 + ((iter + 1) & 1) : iter & 1];  // beta_0 = 0: r for p_{-1}
        unsigned char* at = (isp ? RINGP : RINGR) + sl * G::RB;
        // all rows at once; of a y edge the owned, those below, those above
#pragma unroll 1
        for (int seg = yin ? 0 : 1; seg < (yin ? 1 : 4); ++seg) {
          const int y = seg == 0 ? y0 - WH
                                 : (seg == 1 ? y0
                                             : (seg == 2 ? (y0 == 0 ? f.ny : y0) - WH : (y0 + WY == f.ny ? 0 : y0 + WY)));
          const int h = seg > 2 ? 2 : seg;
          // bytes down to these rows, where a row has rb bytes and the owned begin at o1
          auto down = [&](int rb, int o1) { return seg == 1 ? o1 : (seg == 3 ? o1 + WY * rb : 0); };
          if (xin) {
            tma_load_3d(at + down(G::RW * G::SZ, G::O1), &tm[0][h], x0 - G::SW, y, zs, &bars[sl]);
          } else {
            tma_load_3d(at + down(WX * G::SZ, WH * WX * G::SZ), &tm[1][h], x0, y, zs, &bars[sl]);
            at += G::CB + down(16, 128);
            tma_load_3d(at, &tm[2][h], xl, y, zs, &bars[sl]);
            tma_load_3d(at + G::SB, &tm[2][h], xr, y, zs, &bars[sl]);
            at -= G::CB + down(16, 128);
          }
        }
      };
      // in the march by a thread each of the last two warps, which have no halo pairs
      auto fetch = [&](int sl, int kk) {
        if (tid == NT - 64 || tid == NT - 32) copy(tid == NT - 32, sl, kk);
      };
      // wait (bounded) for the copies in a ring slot.  When one runs out, the block's
      // later ones do at once, and its sums are not numbers, so that the pass ends as a
      // timeout in every block.
      auto landed = [&](int sl) {
        if (!mbar_try_wait(&bars[sl], (phase >> sl) & 1u)) {
          const long long t0 = clock64();
          while (!mbar_try_wait(&bars[sl], (phase >> sl) & 1u)) {
            if (clock64() - t0 > *(volatile long long*)&limit) {
              atomicExch(&f.bar->fail.v, 1u);
              *(volatile long long*)&limit = -1;
              break;
            }
          }
        }
        phase ^= 1u << sl;
      };
      // register windows per pair, by plane mod 3: p on f-2 .. f, r' on
      // f-3 .. f-1, r_i on f-1 .. f; slot 2 is the halo pair
      V pv[3][3], rv[3][2], ra[3][3], xv[2];
#pragma unroll
      for (int q = 0; q < 3; ++q)
#pragma unroll
        for (int m = 0; m < 3; ++m) {
          pv[q][m] = ra[q][m] = V{T(0), T(0)};
          if (m < 2) rv[q][m] = xv[m] = V{T(0), T(0)};
        }
      __syncthreads();  // the previous unit's readers are done with every buffer
      if ((tid & 31) == 0)
#pragma unroll 1
        for (int q = tid >> 6; q < D - 1; q += NT / 64) copy((tid >> 5) & 1, q, k0 - 2 + q);
      int cnt = 0;
      // the owned pairs in global memory, as byte pointers that follow the march
      // (offsets formed from the plane each time cost 30 integer instructions a
      // step): p of plane fp, r' of fp - 1, x of fp
      const long long dg = (rev ? -(long long)plane : (long long)plane) * (long long)sizeof(T);
      const long long g0 = ((long long)stored(k0 - 2) * (long long)plane + go) * (long long)sizeof(T);
      const unsigned nxb = (unsigned)(f.nx * sizeof(T));
      char *gp = reinterpret_cast<char*>(pw) + g0, *gr = reinterpret_cast<char*>(ro) + (g0 - dg),
           *gx = reinterpret_cast<char*>(f.x) + g0;
      auto at2 = [&](char* q, int m) { return reinterpret_cast<T*>(m ? q + nxb : q); };
      // plane fp enters the march; PH = (fp - k0 + 2) mod 6, so that every ring
      // slot, buffer and window is known at compile time
      // FULL: planes fp .. fp - 2 are all of the run, so that a step is one block of
      // code but for the halo pairs and x
      auto step = [&](auto ph, auto full, int fp) {
        constexpr int PH = decltype(ph)::value;
        constexpr bool FULL = decltype(full)::value;
        constexpr int P0 = PH % 3, P1 = (PH + 2) % 3, P2 = (PH + 1) % 3;  // planes fp, fp-1, fp-2
        T* const pn = PP + (PH & 1) * SN;        // p of planes fp, fp-1
        T* const pc = PP + ((PH + 1) & 1) * SN;
        T* const rn = RP + ((PH + 1) & 1) * SN;  // r' of planes fp-1, fp-2
        T* const rc = RP + (PH & 1) * SN;
        landed(PH);
        __syncthreads();
        fetch((PH + D - 1) % D, fp + D - 1);  // into the slot of plane fp - 1, which A has read
        const T* sr = reinterpret_cast<const T*>(RINGR + PH * G::RB);
        const T* sp = reinterpret_cast<const T*>(RINGP + PH * G::RB);
        // A: p(fp) = r(fp) + beta p_old(fp)
        const V a0 = ld2(sr + so[0]), a1 = ld2(sr + so[1]), o0 = ld2(sp + so[0]), o1 = ld2(sp + so[1]);
        const V p0 = vfma(vtb, o0, a0), p1 = vfma(vtb, o1, a1);
        // neighbours of p(fp - 1), read before anything is written
        const V pym = ld2(pc + eo - SP), pyp = ld2(pc + eo + 2 * SP);
        const T pl0 = pc[eo - 1], pr0 = pc[eo + 2], pl1 = pc[eo + SP - 1], pr1 = pc[eo + SP + 2];
        ra[P0][0] = a0;
        ra[P0][1] = a1;
        pv[P0][0] = p0;
        pv[P0][1] = p1;
        xv[0] = vfma(vtp, o0, xv[0]);
        xv[1] = vfma(vtp, o1, xv[1]);
        st2(pn + eo, p0);
        st2(pn + eo + SP, p1);
        if (FULL || (fp >= k0 && fp < k1)) {
          st2g(at2(gp, 0), p0);
          st2g(at2(gp, 1), p1);
        }
        // B: q(fp-1), r'(fp-1) within the halo of one
        if (FULL || fp >= k0) {
          const V q0 = lap(pl0, pv[P1][0], pr0, pym, pv[P1][1], pv[P2][0], p0);
          const V q1 = lap(pl1, pv[P1][1], pr1, pv[P1][0], pyp, pv[P2][1], p1);
          const V r0 = vfma(vna, q0, ra[P1][0]), r1 = vfma(vna, q1, ra[P1][1]);
          rv[P1][0] = r0;
          rv[P1][1] = r1;
          st2(rn + eo, r0);
          st2(rn + eo + SP, r1);
          if (FULL || (fp > k0 && fp <= k1)) {
            run[2] = vfma(r1, q1, vfma(r0, q0, run[2]));
            run[3] = vfma(pv[P1][1], q1, vfma(pv[P1][0], q0, run[3]));
            st2g(at2(gr, 0), r0);
            st2g(at2(gr, 1), r1);
          }
        }
        // C: w(fp-2) at the owned nodes
        if (FULL || fp >= k0 + 2) {
          const V ylo = ld2(rc + eo - SP), yhi = ld2(rc + eo + 2 * SP);
          const V c0 = rv[P2][0], c1 = rv[P2][1];
          const V w0 = lap(rc[eo - 1], c0, rc[eo + 2], ylo, c1, rv[P0][0], rv[P1][0]);
          const V w1 = lap(rc[eo + SP - 1], c1, rc[eo + SP + 2], c0, yhi, rv[P0][1], rv[P1][1]);
          run[0] = vfma(c1, c1, vfma(c0, c0, run[0]));
          run[1] = vfma(c1, w1, vfma(c0, w0, run[1]));
        }
        // the halo pair
        if (halo2) {
          const V r = ld2(sr + ho), p = vfma(vtb, ld2(sp + ho), r);
          pv[P0][2] = p;
          ra[P0][2] = r;
          st2(pn + eh, p);
          if (halo1 && (FULL || fp >= k0)) {
            const V q = lap(pc[eh - 1], pv[P1][2], pc[eh + 2], ld2(pc + eh - SP), ld2(pc + eh + SP), pv[P2][2], p);
            st2(rn + eh, vfma(vna, q, ra[P1][2]));
          }
        }
        if (upd) {
          if (FULL || (fp >= k0 && fp < k1)) {
            st2g(at2(gx, 0), vfma(vta, p0, xv[0]));
            st2g(at2(gx, 1), vfma(vta, p1, xv[1]));
          }
          if (FULL ? fp + 1 < k1 : (fp + 1 >= k0 && fp + 1 < k1)) {
            xv[0] = __ldcg(reinterpret_cast<const V*>(at2(gx + dg, 0)));
            xv[1] = __ldcg(reinterpret_cast<const V*>(at2(gx + dg, 1)));
          }
        }
        if ((++cnt & 15) == 0) flush();
        gp += dg;
        gr += dg;
        gx += dg;
      };
      auto march = [&](auto ph, int fp) {
        if (fp >= k0 + 2 && fp < k1) step(ph, std::true_type{}, fp);
        else step(ph, std::false_type{}, fp);
        return fp <= k1;
      };
      for (int fp = k0 - 2;; fp += 6) {
        if (!march(std::integral_constant<int, 0>{}, fp)) break;
        if (!march(std::integral_constant<int, 1>{}, fp + 1)) break;
        if (!march(std::integral_constant<int, 2>{}, fp + 2)) break;
        if (!march(std::integral_constant<int, 3>{}, fp + 3)) break;
        if (!march(std::integral_constant<int, 4>{}, fp + 4)) break;
        if (!march(std::integral_constant<int, 5>{}, fp + 5)) break;
      }
    }
    flush();
    WaveSum<T> s[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) s[q] = WaveSum<T>{sums[q][tid]};
    if (*(volatile long long*)&limit < 0) s[0].add((T)NAN);
    double t[4];
    const bool ok = wave_sum_t0<4>(s, gs, t);
    iter += 1;
    if (tid == 0) {
      if (!ok) {
        status = 5;
      } else {
        const double rr_new = t[0];
        rel = sqrt(rr_new / bb);
        if (isnan(rr_new) && ld_volatile(&f.bar->fail.v) != 0u) status = 5;
        else if (rel <= f.tol) status = 1;
        else if (iter >= f.maxit) status = 2;
        else if (!isfinite(rr_new)) status = 3;
        else {
          const double beta = rr_new / rr;
          const double pq_new = t[1] + 2.0 * beta * t[2] + beta * beta * t[3];
          if (pq_new == 0.0 || !isfinite(pq_new)) status = 3;
          else {
            sc.ta = (T)(rr_new / pq_new);
            sc.tb = (T)beta;
          }
        }
        rr = rr_new;
      }
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
  }

  // ---- zero-mean gauge (or zero for a zero right side) ------------------------
  if (status != 5) {
    const bool pend = iter & 1;  // the last pass left alpha p to the next
    const T* pl = f.p[(iter + 1) & 1];
    WaveSum<T> s[1];
    int cnt = 0;
    for (long long c = gtid; c < nch; c += gstride) {
      Ch xq = ldch(f.x + (size_t)c * VC);
      if (pend) {
        const Ch pq2 = ldch(pl + (size_t)c * VC);
#pragma unroll
        for (int q = 0; q < VC; ++q) xq.e[q] += ta * pq2.e[q];
        stch(f.x + (size_t)c * VC, xq);
      }
#pragma unroll
      for (int q = 0; q < VC; ++q) s[0].add(xq.e[q]);
      if ((++cnt & 3) == 0) s[0].flush();
    }
    double t[1];
    const bool ok = wave_sum_t0<1>(s, gs, t);
    if (tid == 0) {
      if (!ok) status = 5;
      sc.mean = (T)(t[0] / (double)f.n);
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
    if (status != 5) {
      const T mx = sc.mean;
      for (long long c = gtid; c < nch; c += gstride) {
        Ch xq = ldch(f.x + (size_t)c * VC);
#pragma unroll
        for (int q = 0; q < VC; ++q) xq.e[q] = status == 4 ? T(0) : xq.e[q] - mx;
        stch(f.x + (size_t)c * VC, xq);
      }
    }
  }
  if (limit < 0) {  // copies that are still in flight may land before the block ends
    const long long t0 = clock64();
    while (clock64() - t0 < f.spin_cycles) {
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    f.ctl->iter = iter;
    f.ctl->rel = rel;
    f.ctl->done = status;
  }
}

}  // namespace

namespace {

bool col_fits(int nx, int ny, int wx, int wy) { return nx % wx == 0 && ny % wy == 0; }

// cuTensorMapEncodeTiled from the driver, looked up once
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static std::mutex mu;
  static bool tried = false;
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  std::lock_guard<std::mutex> lock(mu);
  if (!tried) {
    tried = true;
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) ==
            cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  }
  return fn;
}

// a 3-D map of an nx x ny x nz vector with bx x by x 1 boxes (no swizzle,
// no interleave; out-of-range elements are never requested)
template <typename T>
bool encode_map(CUtensorMap* m, const void* base, int nx, int ny, int nz, int bx, int by) {
  const auto enc = tensor_map_encoder();
  if (!enc) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)nx, (cuuint64_t)ny, (cuuint64_t)nz};
  const cuuint64_t strides[2] = {(cuuint64_t)nx * sizeof(T), (cuuint64_t)nx * ny * sizeof(T)};
  const cuuint32_t box[3] = {(cuuint32_t)bx, (cuuint32_t)by, 1u};
  const cuuint32_t estr[3] = {1u, 1u, 1u};
  return enc(m, sizeof(T) == 4 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_FLOAT64, 3,
             const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <typename T, typename C>
int solve_wave(const SolverArgs<T>& a, const FusedCfg& fc, const T* b, T* x, double tol, int maxit, int* iters,
               double* rel, std::string* err) {
  WaveArgs<T> f;
  f.nx = a.g.nx;
  f.ny = a.g.ny;
  f.nz = a.g.nz;
  f.walls = a.g.walls;
  f.cx = a.g.idx * a.g.idx;
  f.cy = a.g.idy * a.g.idy;
  f.cz = a.g.idz * a.g.idz;
  f.ntx = f.nx / C::WX;
  f.nty = f.ny / C::WY;
  f.n = (long long)f.nx * f.ny * f.nz;
  f.b = b;
  f.x = x;
  f.r[0] = a.r;
  f.r[1] = a.q;
  f.p[0] = a.p0;
  f.p[1] = a.p1;
  f.partials = a.partials;
  f.bar = a.bar;
  f.ctl = a.ctl;
  f.tol = tol;
  f.maxit = maxit;
  f.spin_cycles = fc.spin_cycles;
  f.guard = a.guard;
  const T* vec[4] = {a.r, a.q, a.p0, a.p1};
  bool maps = true;
  for (int v = 0; v < 4; ++v)
    for (int w = 0; w < 3; ++w)
      for (int h = 0; h < 3; ++h)
        maps = maps && encode_map<T>(&f.tm[v][w][h], vec[v], f.nx, f.ny, f.nz,
                                     w == 2 ? Staged<T, C>::SW : (w == 1 || f.nx < Staged<T, C>::RW ? C::WX : Staged<T, C>::RW),
                                     h == 2 ? WH : (h == 1 || f.ny < Staged<T, C>::ROWS ? C::WY : Staged<T, C>::ROWS));
  if (!maps) return poisson_solve_roll<T>(a, fc, b, x, tol, maxit, iters, rel, err);
  int per_sm = 0, dev = 0, nsm = 0;
  cudaError_t e;
  const void* kern = (const void*)k_cg_wave<T, C>;
  const size_t smem = wave_smem<T, C>();
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem)) != cudaSuccess ||
      (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, C::NT, smem)) != cudaSuccess) {
    if (err) *err = std::string("wave CG occupancy: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  if (per_sm < 1) {
    if (err) *err = "wave CG: no block fits on an SM";
    return LES_ERR_CUDA;
  }
  long long G = (long long)per_sm * nsm;
  G = std::min<long long>(G, fc.max_blocks);
  G = std::min<long long>(G, 8LL * nsm);  // the partials hold 2 x kSumSlot words of 8 blocks per SM
  // z-runs as long as possible (each run re-forms two planes of p and r'
  // below it)
  const long long ncol = (long long)f.ntx * f.nty;
  // the (column, run) units are dealt to the G persistent blocks in turns.
  // Fewer columns than blocks: at most G units, one turn (a G-th + 1 unit
  // would double the iteration for the rest).  More: whole columns in full
  // turns, then the planes of the columns left in equal shares, so that no
  // block takes a whole extra column (on 1536 x 1536 x 256: 2304 columns,
  // 7 turns of 304 and 148 planes each of the last 176 columns)
  if (ncol >= G) {
    f.zrun = f.nz;
    f.nchunk = 1;
    f.nunits = (int)((ncol / G) * G);
    f.tail_planes = (int)((ncol - f.nunits) * f.nz);
    f.tail_per = (int)((f.tail_planes + G - 1) / G);
  } else {
    const long long want = std::max<long long>(1, std::min<long long>((long long)f.nz, G / ncol));
    f.zrun = (int)((f.nz + want - 1) / want);
    f.nchunk = (f.nz + f.zrun - 1) / f.zrun;
    f.nunits = (int)(ncol * f.nchunk);
    f.tail_planes = 0;
    f.tail_per = 0;
    // or all planes in equal shares, when the second run of a block whose share
    // spans two columns (four planes more and a start, as long as another two)
    // costs less than the blocks that whole runs leave idle
    const long long per = (ncol * f.nz + G - 1) / G;
    if (per + 10 < f.zrun + 4) {
      f.nunits = 0;
      f.tail_planes = (int)(ncol * f.nz);
      f.tail_per = (int)per;
    }
    G = std::max<long long>(1, std::min<long long>(G, f.nunits ? f.nunits : (f.tail_planes + per - 1) / per));
  }
  f.expected = (unsigned)G + (unsigned)std::max(0, fc.missing);
  if ((e = cudaMemsetAsync(a.bar, 0, sizeof(FusedBar), a.st)) != cudaSuccess) {
    if (err) *err = std::string("wave CG barrier reset: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  void* args[] = {&f};
  {
    ProfScope ps(a.prof, KI_CG_WAVE, a.st);
    e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)G), dim3(C::NT), args, smem, a.st);
  }
  if (e != cudaSuccess) {
    if (err) *err = std::string("wave CG launch: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  if ((e = cudaMemcpyAsync(a.ctl_host, a.ctl, sizeof(SolverCtl), cudaMemcpyDeviceToHost, a.st)) != cudaSuccess ||
      (e = cudaStreamSynchronize(a.st)) != cudaSuccess) {
    if (err) *err = std::string("wave CG: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  const SolverCtl& c = *a.ctl_host;
  if (iters) *iters = c.iter;
  if (rel) *rel = c.rel;
  // algorithmic traffic of the solve, with one set-up sweep for alpha_0 (the kernel
  // also reads a third of r_i and p_{i-1} again for the halo)
  if (a.prof) a.prof->bytes[KI_CG_WAVE] += (kCgSetupFields + 1.0 + kCgWaveFields * c.iter) * (double)f.n * sizeof(T);
  switch (c.done) {
    case 1:
    case 4: return LES_OK;
    case 2: return LES_ERR_NOT_CONVERGED;
    case 3:
      if (err) *err = "poisson: breakdown (zero or non-finite p.Ap / residual)";
      return LES_ERR_NONFINITE;
    case 5:
      if (err) *err = "poisson: a grid barrier wait timed out";
      return LES_ERR_TIMEOUT;
    default:
      if (err) *err = "poisson: wave solver returned no status";
      return LES_ERR_CUDA;
  }
}

}  // namespace

bool wave_cg_eligible(int nx, int ny, int nz) {
  return (col_fits(nx, ny, Col64::WX, Col64::WY) || col_fits(nx, ny, Col32::WX, Col32::WY)) && nz >= 2 &&
         (long long)nx * ny < (1LL << 29);  // 32-bit byte offsets in a plane
}

template <typename T>
int poisson_solve_wave(const SolverArgs<T>& a, const FusedCfg& fc, const T* b, T* x, double tol, int maxit,
                       int* iters, double* rel, std::string* err) {
  // the staging copies move 16-byte chunks: every vector must start on a
  // 16-byte boundary (a caller's view at an odd offset takes the one-pass
  // kernel for any grid instead)
  auto aligned = [](const void* p) { return ((uintptr_t)p & 15u) == 0; };
  if (!wave_cg_eligible(a.g.nx, a.g.ny, a.g.nz) ||
      !(aligned(b) && aligned(x) && aligned(a.r) && aligned(a.q) && aligned(a.p0) && aligned(a.p1)))
    return poisson_solve_roll<T>(a, fc, b, x, tol, maxit, iters, rel, err);
  // the wider the column, the fewer lines its ends take: 105 -> 98 us an iteration
  // on 256 x 256 x 256, 61 -> 56 on 256 x 256 x 128, the same on 768 x 768 x 128
  if constexpr (sizeof(T) == 4)
    if (col_fits(a.g.nx, a.g.ny, Col128::WX, Col128::WY))
      return solve_wave<T, Col128>(a, fc, b, x, tol, maxit, iters, rel, err);
  if (col_fits(a.g.nx, a.g.ny, Col64::WX, Col64::WY))
    return solve_wave<T, Col64>(a, fc, b, x, tol, maxit, iters, rel, err);
  return solve_wave<T, Col32>(a, fc, b, x, tol, maxit, iters, rel, err);
}

template int poisson_solve_wave<float>(const SolverArgs<float>&, const FusedCfg&, const float*, float*, double, int,
                                       int*, double*, std::string*);
template int poisson_solve_wave<double>(const SolverArgs<double>&, const FusedCfg&, const double*, double*, double,
                                        int, int*, double*, std::string*);

}  // namespace les
