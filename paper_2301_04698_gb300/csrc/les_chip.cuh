// les_chip.cuh -- what the on-chip conjugate-gradient kernels of les_cg_chip.cu,
// les_cg_brick.cu and les_cg_regs.cu share: the bricks, and the grid-wide sum of an
// iteration's four dot products.
#pragma once

#include <type_traits>

#include "les_gridsync.cuh"
#include "les_internal.h"

namespace les {

constexpr int kChipThreads = 512;
constexpr int kChipWarps = kChipThreads / 32;
constexpr int kChipSpread = 8;      // counters of the blocks' arrivals
constexpr int kChipLine = 32;       // counters 128 bytes apart
constexpr int kChipGhosts = 4;      // ghost nodes per thread in registers

template <typename T>
struct ChipArgs {
  int nx, ny, nz, walls;
  // 1/dx^2, 1/dy^2, 1/dz^2; FP32: times 2^-k, so that no eigenvalue is above one and
  // none of the four sums above r.r, whatever the spacings (exact)
  T cx, cy, cz;
  T sc, isc;           // 2^k, 2^-k (FP64: 1)
  int px, py, pz, zs;  // bricks along x, y, z; runs of planes per brick
  int smem_p, smem_g;  // shared memory of P and (XS) of one ghost array, in elements (even)
  long long n;
  const T* b;
  T* x;
  T* rg;               // published faces of the first residual
  T* qg0;              // published faces of q, even iterations
  T* qg1;              // ... odd iterations
  // the same as tagged words, one per node of the grid: those of the first half of the
  // nodes at qt[0][parity], the others at qt[1][parity]
  char* qt[2][2];
  double* partials;    // two slots of kSumSlot words per block (the set-up and gauge sums)
  unsigned* counters;  // kChipSpread counters of the blocks' releases of their faces, kChipLine apart, zeroed
  void* spread;        // [2 slots][gridDim.x][4 values] partials of the iterations' sums, tagged words
  unsigned missing;    // test hook: arrivals that never come
  FusedBar* bar;
  SolverCtl* ctl;
  double tol;
  int maxit;
  long long spin_cycles;
  unsigned expected;
  int guard;
};

// packed FP32: two results per instruction, each rounded as by the scalar one
__device__ __forceinline__ float2 f32x2(float v) { return float2{v, v}; }
__device__ __forceinline__ float2 lo2(float4 v) { return float2{v.x, v.y}; }
__device__ __forceinline__ float2 hi2(float4 v) { return float2{v.z, v.w}; }
__device__ __forceinline__ float4 join2(float2 a, float2 b) { return float4{a.x, a.y, b.x, b.y}; }
// a v + b for four nodes
__device__ __forceinline__ float4 fma4(float a, float4 v, float4 b) {
  return join2(__ffma2_rn(f32x2(a), lo2(v), lo2(b)), __ffma2_rn(f32x2(a), hi2(v), hi2(b)));
}
__device__ __forceinline__ void dot4(float2& s, float4 a, float4 b) {
  s = __ffma2_rn(lo2(a), lo2(b), s);
  s = __ffma2_rn(hi2(a), hi2(b), s);
}

// part i of n nodes in `parts` parts whose sizes differ by at most one
__device__ __forceinline__ void chip_part(int n, int parts, int i, int& first, int& len) {
  const int base = n / parts, rem = n - base * parts;
  len = base + (i < rem ? 1 : 0);
  first = i * base + min(i, rem);
}
__device__ __forceinline__ int chip_wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }
__device__ __forceinline__ F2 acc_of(float v) { return F2{v, 0.f}; }
__device__ __forceinline__ F2 acc_of(F2 v) { return v; }
__device__ __forceinline__ double acc_of(double v) { return v; }
__device__ __forceinline__ float acc_add(float a, float b) { return a + b; }
__device__ __forceinline__ float acc_xor(float a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ F2 acc_xor(F2 a, int o) {
  return F2{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ double acc_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ F2 acc_from_lane(F2 a, int l) {
  return F2{__shfl_sync(0xffffffffu, a.hi, l), __shfl_sync(0xffffffffu, a.lo, l)};
}
__device__ __forceinline__ double acc_from_lane(double a, int l) { return __shfl_sync(0xffffffffu, a, l); }

// alpha and beta from the totals; false on a zero or non-finite p.q or r.r.  beta is
// |r - alpha q|^2 / r.r, expanded in the totals: where next to nothing is left of r the
// expansion may come out below zero, and is taken for none.
// FP32: from the totals as pairs, each product and addition with its rounding error, and
// rounded once (from FP64 totals in FP64 they would take thread 0 about a microsecond);
// a quotient from an approximate reciprocal ib of b and its remainder.
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float f2_quotient(F2 a, F2 b, float ib) {
  const float q = a.hi * ib;
  return q + (fmaf(-q, b.hi, a.hi) + fmaf(-q, b.lo, a.lo)) * ib;
}
__device__ __forceinline__ bool chip_scalars(const F2 (&t)[4], float& ta, float& tb) {
  const F2 pq = t[0], r2 = t[1], rq = t[2], q2 = t[3];
  if (!(pq.hi != 0.f) || !isfinite(pq.hi) || !isfinite(r2.hi)) return false;
  const float ir = rcp_approx(r2.hi);
  ta = f2_quotient(r2, pq, rcp_approx(pq.hi));
  const float m = -2.f * ta, a2 = ta * ta, u = m * rq.hi, v = a2 * q2.hi;
  F2 n = r2;
  f2_acc(n, u);
  f2_acc(n, v);
  n.lo += (fmaf(m, rq.hi, -u) + m * rq.lo) + (fmaf(a2, q2.hi, -v) + a2 * q2.lo) + fmaf(ta, ta, -a2) * q2.hi;
  tb = f2_quotient(n, r2, ir);
  if (!(isfinite(ta) && isfinite(tb))) {  // nothing left of r but subnormal squares
    ta = r2.hi / pq.hi;
    tb = fmaf(ta * ta, q2.hi, fmaf(-2.f * ta, rq.hi, r2.hi)) / r2.hi;
  }
  tb = tb < 0.f ? 0.f : tb;
  return true;
}
// FP64: called by the whole of warp 0, for both quotients take one division, a lane each.
// (One of 1 / (r.r p.q) for both would leave the range of FP64 where r.r is beyond
// 1e154 or below 1e-154.)
__device__ __forceinline__ bool chip_scalars(const double (&t)[4], double& ta, double& tb) {
  const double pq = t[0], r2 = t[1], rq = t[2], q2 = t[3];
  const bool odd = threadIdx.x & 1;
  const double quo = (odd ? 1.0 : r2) / (odd ? r2 : pq);
  const double alpha = __shfl_sync(0xffffffffu, quo, 0), ir2 = __shfl_sync(0xffffffffu, quo, 1);
  if (!(pq != 0.0) || !isfinite(pq) || !isfinite(r2)) return false;
  ta = alpha;
  const double beta = fma(alpha, fma(alpha, q2, -2.0 * rq), r2) * ir2;
  tb = beta < 0.0 ? 0.0 : beta;
  return true;
}

// A thread's sum over the planes 0 .. ZP - 1 of its run, in order: FP32 within 16
// planes, compensated across, as in the streaming kernels.
template <typename T, int ZP>
struct ChipRun;
template <int ZP>
struct ChipRun<float, ZP> {
  F2 s{0.f, 0.f};
  float run = 0.f;
  __device__ __forceinline__ void add(int j, float v) {
    if (j > 0 && j % 16 == 0) {
      f2_acc(s, run);
      run = 0.f;
    }
    run += v;
  }
  __device__ __forceinline__ F2 total() const {
    F2 t = s;
    if (ZP > 16) f2_acc(t, run);
    else t.hi = run;
    return t;
  }
};
template <int ZP>
struct ChipRun<double, ZP> {
  double s = 0.0;
  __device__ __forceinline__ void add(int, double v) { s += v; }
  __device__ __forceinline__ double total() const { return s; }
};

// FP32: the power of two that brings the right side and L_c x0 to the size of one, from
// |b|_1 and |x0|_1 (c0: L_c's centre coefficient), so that the solve's sums of squares
// stay in range.  It changes no rounding.
__device__ __forceinline__ float chip_scale(double b1, double x1, float c0, double n) {
  const double m = fmax(b1, x1 * (double)c0) / n;
  const int e = (__double2hiint(m) >> 20 & 0x7ff) - 1023;
  return m == 0.0 ? 1.f : __int_as_float((127 - max(-126, min(126, e))) << 23);
}

// a warp's four values by a transposing butterfly (six additions instead of twenty)
template <typename D>
__device__ __forceinline__ void chip_butterfly(D d0, D d1, D d2, D d3, D (&shv)[4][kChipWarps]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // after the butterfly lanes 8k .. 8k + 7 hold the warp's value k
  const bool up = lane & 16, odd = lane & 8;
  const D s0 = up ? d0 : d2, s1 = up ? d1 : d3;  // given to lane ^ 16
  const D a0 = acc_add(up ? d2 : d0, acc_xor(s0, 16)), a1 = acc_add(up ? d3 : d1, acc_xor(s1, 16));
  D v = acc_add(odd ? a1 : a0, acc_xor(odd ? a0 : a1, 8));
  v = acc_add(v, acc_xor(v, 4));
  v = acc_add(v, acc_xor(v, 2));
  v = acc_add(v, acc_xor(v, 1));
  if ((lane & 7) == 0) shv[lane >> 3][warp] = v;
}

// warps that fold; an FP64 addition takes a scheduler 64 cycles, so fewer warps with
// more of their own
template <typename Acc>
constexpr int kFoldWarps = 8;
template <>
constexpr int kFoldWarps<double> = 4;

// the fold's end: lane l holds the sum of value l mod 4 over some of the blocks of
// part id; the four totals, the same in every block, in the lanes of warp 0
template <typename Acc>
__device__ __forceinline__ void chip_fold_warp(Acc t, Acc (&part)[32], int id) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o >= 4; o >>= 1) t = acc_add(t, acc_xor(t, o));
  if (lane < 4) part[id * 4 + lane] = t;
}
template <typename Acc>
__device__ __forceinline__ void chip_fold(Acc (&part)[32], Acc (&tot)[4]) {
  constexpr int FW = kFoldWarps<Acc>;
  asm volatile("bar.sync 3, %0;" ::"r"(min((int)blockDim.x, 32 * FW)) : "memory");
  if (threadIdx.x < 32) {
    Acc t = part[threadIdx.x % (4 * FW)];
#pragma unroll
    for (int o = 2 * FW; o >= 4; o >>= 1) t = acc_add(t, acc_xor(t, o));
#pragma unroll
    for (int k = 0; k < 4; ++k) tot[k] = acc_from_lane(t, k);
  }
}

// ---- tagged words ------------------------------------------------------------
// A value that other blocks wait for travels with the number of its iteration: every
// 8 bytes hold 32 bits of it and a 32-bit tag, written and read whole, so a reader
// that finds the tag has the value, and neither side orders it against anything
// else.  A writer that released a flag would wait for its stores to reach L2, and a
// reader that had seen it would read the value by another trip.  The tags are NaN
// patterns, which no finite FP32 value left in the same memory can look like; as the
// upper half of an FP64 one they are beyond 1e305, whose square stops the solve first.
__device__ __forceinline__ unsigned chip_tag(int iter) { return 0xff800001u + ((unsigned)iter & 0x3fffffu); }
// FP32: 8 bytes; FP64: 16, each half of the value with the tag.  A compensated pair
// takes 8, its tag the last bit of lo (2^-48 of the value): the two values that share a
// slot are two iterations apart, so one bit of the iteration / 2 tells them apart.
template <typename V>
struct Tagged {
  static constexpr int BYTES = 8;
  unsigned long long w;
};
template <>
struct Tagged<double> {
  static constexpr int BYTES = 16;
  unsigned long long w, v;
};
template <typename V>
__device__ __forceinline__ void tagged_load(Tagged<V>& t, const char* at) {
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(t.w) : "l"(at));
}
__device__ __forceinline__ void tagged_load(Tagged<double>& t, const char* at) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(t.w), "=l"(t.v) : "l"(at));
}
__device__ __forceinline__ bool tagged_ok(const Tagged<float>& t, int iter) { return (unsigned)(t.w >> 32) == chip_tag(iter); }
__device__ __forceinline__ bool tagged_ok(const Tagged<F2>& t, int iter) { return ((unsigned)(t.w >> 32) & 1u) == ((unsigned)iter >> 1 & 1u); }
__device__ __forceinline__ bool tagged_ok(const Tagged<double>& t, int iter) {
  return (unsigned)(t.w >> 32) == chip_tag(iter) && (unsigned)(t.v >> 32) == chip_tag(iter);
}
__device__ __forceinline__ float tagged_value(const Tagged<float>& t) { return __uint_as_float((unsigned)t.w); }
__device__ __forceinline__ F2 tagged_value(const Tagged<F2>& t) {
  return F2{__uint_as_float((unsigned)t.w), __uint_as_float((unsigned)(t.w >> 32))};
}
__device__ __forceinline__ double tagged_value(const Tagged<double>& t) {
  return __hiloint2double((int)(unsigned)t.v, (int)(unsigned)t.w);
}
__device__ __forceinline__ void tagged_store8(char* at, unsigned lo, unsigned hi) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(at), "l"((unsigned long long)hi << 32 | lo) : "memory");
}
__device__ __forceinline__ void tagged_store(char* at, float v, int iter) {
  tagged_store8(at, __float_as_uint(v), chip_tag(iter));
}
__device__ __forceinline__ void tagged_store(char* at, F2 v, int iter) {
  tagged_store8(at, __float_as_uint(v.hi), (__float_as_uint(v.lo) & ~1u) | ((unsigned)iter >> 1 & 1u));
}
__device__ __forceinline__ void tagged_store(char* at, double v, int iter) {
  const unsigned long long tag = (unsigned long long)chip_tag(iter) << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(at), "l"(tag | (unsigned)__double2loint(v)),
               "l"(tag | (unsigned)__double2hiint(v))
               : "memory");
}
// a word that no reader takes for that of iteration 0 or 1.  Of an FP64 one both
// halves: a vector access is whole only per 8 bytes, and a half left with the tag of an
// earlier solve's iteration 0 or 1 would pass with the other half's new value.
template <typename V>
__device__ __forceinline__ void tagged_clear(char* at) {
  tagged_store8(at, 0u, std::is_same<V, F2>::value ? 1u : 0u);
  if constexpr (Tagged<V>::BYTES == 16) tagged_store8(at + 8, 0u, 0u);
}

// The words of a sum's partials: [2 slots][gridDim.x][4 values].  A block's four lie
// together, so that a line has few writers: with a value's words of
// all blocks together, and eight writers to a line that is being read, an iteration on
// 32^3 in FP32 took 3.1 us instead of 2.2.  Several copies do not help.  A block may
// write a slot again two sums later: it gets there only after every block has posted
// the sum between, and so has read this one.  Cleared by each block for itself before
// the set-up sums, which order that for everyone.
template <typename Acc>
__device__ __forceinline__ void chip_sum_clear(void* spread) {
  const int slot = threadIdx.x >> 2, k = threadIdx.x & 3;
  if (slot < 2)
    tagged_clear<Acc>(static_cast<char*>(spread) + (((size_t)slot * gridDim.x + blockIdx.x) * 4 + k) * Tagged<Acc>::BYTES);
}

// the warps from chip_ghost_warp<W0>() on issue() what comes counted
template <int W0>
__device__ __forceinline__ int chip_ghost_warp() {
  return (int)blockDim.x > 32 * W0 ? W0 : 0;
}

// The grid-wide sum of p.q, r.r, r.q and q.q at iteration `iter`: each warp's four
// values by a transposing butterfly (D: the threads' sums, FP64, compensated FP32 pairs,
// or plain FP32); warp 0 combines the warps' (FP32 ones as compensated pairs) and posts
// the block's; the first kFoldWarps warps read the words of a part of the blocks each,
// until all have come, and fold them in a fixed order, so every block obtains the same
// totals in tot (in warp 0).  Words of a lane's loads are in flight together (3 of 8
// warps or 5 of 4 read 160 blocks or more in one turn; fewer cost another trip, more
// registers).  meanwhile() runs in every warp but warp 0: before its wait, or after it
// where the warp folds or acquires and the neighbours' words are counted.
//   What a block awaits of its neighbours comes in one of two ways.  As tagged words
// (W0 < 0): when the sum has come, issue() starts the loads of what this thread awaits,
// check() takes what has come and tells whether that was all, and both are called
// again until it is (begun earlier, they disturb the lines that are being written: 64^3
// in FP32 then takes 3.05 us, not 2.97).  Or, where the words are many, as plain ones
// that the last warp releases on one of kChipSpread counters before the sum is posted
// and acquires beside the fold; issue() then runs once in the warps from W0 on (in a
// folding warp after its fold; 128 x 128 x 96 takes 5.0 us with W0 past them, 5.3 with
// W0 = 1), and check is not called.
//   fail (0 before the first sum) is set when a wait runs out, in warps other than the
// folding ones perhaps too late for this sum but in time for the next.
struct ChipNothing {
  __device__ __forceinline__ bool operator()() const { return true; }
};
template <int W0, int Words, typename Args, typename D, typename Acc, typename Meanwhile, typename Issue, typename Check>
__device__ __forceinline__ void chip_sum(const Args& f, int iter, D d0, D d1, D d2, D d3, D (&shv)[4][kChipWarps],
                                         Acc (&part)[32], Acc (&tot)[4], volatile int& fail, Meanwhile&& meanwhile,
                                         Issue&& issue, Check&& check) {
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
  constexpr bool Counted = W0 >= 0;
  constexpr int FW = kFoldWarps<Acc>, U = Words, W = Tagged<Acc>::BYTES;
  const unsigned G = gridDim.x;
  const long long t0 = clock64();
  chip_butterfly(d0, d1, d2, d3, shv);
  __syncthreads();
  // orders every thread's stores before the barrier; counter i takes blocks i, i + kChipSpread, ...
  if (Counted && tid == nthr - 32) red_release_add(f.counters + (blockIdx.x % kChipSpread) * kChipLine, 1u);
  char* slot = reinterpret_cast<char*>(f.spread) + (size_t)(iter & 1) * 4 * G * W;
  const bool late = Counted && (warp < FW || warp == nwarp - 1);
  if (warp == 0) {
    // lanes 8k .. 8k + 7: value k of the block
    const int k = lane >> 3, c = lane & 7;
    Acc a{};
    for (int w = c; w < nwarp; w += 8) a = acc_add(a, acc_of(shv[k][w]));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a = acc_add(a, acc_xor(a, o));
    if (c == 0) tagged_store(slot + ((size_t)blockIdx.x * 4 + k) * W, a, iter);
    // posted: the other warps may start their own work
    asm volatile("bar.arrive 2, %0;" ::"r"(nthr) : "memory");
  } else {
    asm volatile("bar.sync 2, %0;" ::"r"(nthr) : "memory");
    if (!late) meanwhile();
  }
  // every 64th turn: has another block given up, or has the time run out?
  auto over = [&](unsigned spins) {
    const bool quit = (spins & 63u) == 0u && (ld_volatile(&f.bar->fail.v) != 0u || clock64() - t0 > f.spin_cycles);
    if (!__any_sync(0xffffffffu, quit)) return false;
    if (lane == 0) {
      atomicExch(&f.bar->fail.v, 1u);
      fail = 1;
    }
    return true;
  };
  if (warp < FW) {
    for (int id = warp; id < FW; id += nwarp) {  // eight blocks at a time, a lane per value
      Acc t{};
      for (unsigned base = (unsigned)id * 8 + (lane >> 2); base - (lane >> 2) < G; base += 8 * FW * U) {
        const char* at = slot + ((size_t)base * 4 + (lane & 3)) * W;
        Tagged<Acc> w[U];
        unsigned miss = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) miss |= base + 8 * FW * u < G ? 1u << u : 0u;
        for (unsigned spins = 1;; ++spins) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (miss >> u & 1u) tagged_load(w[u], at + 32 * W * FW * u);
#pragma unroll
          for (int u = 0; u < U; ++u)
            if ((miss >> u & 1u) && tagged_ok(w[u], iter)) miss &= ~(1u << u);
          if (__all_sync(0xffffffffu, miss == 0u && f.missing == 0u) || over(spins)) break;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) t = acc_add(t, base + 8 * FW * u < G ? tagged_value(w[u]) : Acc{});
      }
      if (!Counted && id + nwarp >= FW) {
        if (nwarp > FW) asm volatile("bar.arrive 1, %0;" ::"r"(nthr) : "memory");
        issue();
      }
      chip_fold_warp(t, part, id);
    }
    chip_fold(part, tot);
  } else if (!Counted) {
    asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
    issue();
  }
  if constexpr (Counted) {
    const int w0 = chip_ghost_warp<W0>();
    if (warp < w0) {
      if (warp) meanwhile();
      return;
    }
    if (warp == nwarp - 1) {
      bool done = lane >= kChipSpread || lane >= (int)G;
      const unsigned target = ((unsigned)iter + 1u) * ((G - lane + kChipSpread - 1) / kChipSpread);
      for (unsigned spins = 1;; ++spins) {
        if (!done) done = (int)(ld_acquire(f.counters + lane * kChipLine) - target) >= 0;
        if (__all_sync(0xffffffffu, done) || over(spins)) break;
      }
      __syncwarp();  // orders the lanes' acquires before the barrier
    }
    asm volatile("bar.sync 1, %0;" ::"r"(nthr - 32 * w0) : "memory");
    issue();
    if (late && warp) meanwhile();
  } else {
    for (unsigned spins = 1;; ++spins) {
      if (__all_sync(0xffffffffu, check()) || over(spins)) break;
      issue();
    }
  }
}

// les_cg_brick.cu: a brick's columns and planes at most; the kernel for bricks of at
// most zp planes (a multiple of 8), its shared memory and the elements of its arrays
constexpr int kBrickX = 32, kBrickY = 16, kBrickPlanes = 64;
size_t brick_smem(int zp, int* np, int* ng);
const void* brick_kernel(int zp);

}  // namespace les
