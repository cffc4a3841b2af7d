// les_chip.cuh -- what the on-chip conjugate-gradient kernels of les_cg_chip.cu and
// les_cg_brick.cu share: their arguments, the bricks, and the grid-wide sum of an
// iteration's four dot products.
#pragma once

#include "les_gridsync.cuh"
#include "les_internal.h"

namespace les {

constexpr int kChipThreads = 512;
constexpr int kChipWarps = kChipThreads / 32;
constexpr int kChipSpread = 8;      // arrival counters and copies of the partials per sum
constexpr int kChipLine = 32;       // counters 128 bytes apart
constexpr int kChipGhosts = 4;      // ghost nodes per thread in registers
static_assert(kChipSpread * 4 == 32, "one lane of warp 0 per (copy, value) of the partials");

template <typename T>
struct ChipArgs {
  int nx, ny, nz, walls;
  T cx, cy, cz;        // 1/dx^2, 1/dy^2, 1/dz^2
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
  unsigned* counters;  // kChipSpread arrival counters of the iterations' sums, kChipLine apart, zeroed
  void* spread;        // [2 slots][kChipSpread copies][gridDim.x][4 values] partials of those sums, or tagged words
  unsigned missing;    // test hook: arrivals on counter 0 that never come
  FusedBar* bar;
  SolverCtl* ctl;
  double tol;
  int maxit;
  long long spin_cycles;
  unsigned expected;
  int guard;
};

// part i of n nodes in `parts` parts whose sizes differ by at most one
__device__ __forceinline__ void chip_part(int n, int parts, int i, int& first, int& len) {
  const int base = n / parts, rem = n - base * parts;
  len = base + (i < rem ? 1 : 0);
  first = i * base + min(i, rem);
}
__device__ __forceinline__ int chip_wrap(int i, int n) { return i < 0 ? i + n : (i >= n ? i - n : i); }
__device__ __forceinline__ F2 acc_of(float v) { return F2{v, 0.f}; }
__device__ __forceinline__ double acc_of(double v) { return v; }
__device__ __forceinline__ F2 acc_xor(F2 a, int o) {
  return F2{__shfl_xor_sync(0xffffffffu, a.hi, o), __shfl_xor_sync(0xffffffffu, a.lo, o)};
}
__device__ __forceinline__ double acc_xor(double a, int o) { return __shfl_xor_sync(0xffffffffu, a, o); }
__device__ __forceinline__ F2 acc_from_lane(F2 a, int l) {
  return F2{__shfl_sync(0xffffffffu, a.hi, l), __shfl_sync(0xffffffffu, a.lo, l)};
}
__device__ __forceinline__ double acc_from_lane(double a, int l) { return __shfl_sync(0xffffffffu, a, l); }

// alpha and beta from the totals; false on a zero or non-finite p.q or r.r.
// An FP32 solve takes them in FP32 from the high parts of the totals.
__device__ __forceinline__ bool chip_scalars(const F2 (&t)[4], float& ta, float& tb) {
  const float pq = t[0].hi, r2 = t[1].hi, rq = t[2].hi, q2 = t[3].hi;
  if (!(pq != 0.f) || !isfinite(pq) || !isfinite(r2)) return false;
  const float alpha = r2 / pq;
  ta = alpha;
  tb = fmaf(alpha * alpha, q2, fmaf(-2.f * alpha, rq, r2)) / r2;  // |r - alpha q|^2 / r.r
  return true;
}
__device__ __forceinline__ bool chip_scalars(const double (&t)[4], double& ta, double& tb) {
  const double pq = t[0], r2 = t[1], rq = t[2], q2 = t[3];
  if (!(pq != 0.0) || !isfinite(pq) || !isfinite(r2)) return false;
  const double inv = 1.0 / (r2 * pq);  // one FP64 division for both
  const double alpha = r2 * r2 * inv;
  ta = alpha;
  tb = fma(alpha * alpha, q2, fma(-2.0 * alpha, rq, r2)) * (pq * inv);
  return true;
}

// a warp's four values by a transposing butterfly (six additions instead of twenty)
template <typename T>
__device__ __forceinline__ void chip_butterfly(T d0, T d1, T d2, T d3, T (&shv)[4][kChipWarps]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // after the butterfly lanes 8k .. 8k + 7 hold the warp's value k
  const bool up = lane & 16, odd = lane & 8;
  T a0 = up ? d2 : d0, a1 = up ? d3 : d1;        // kept
  const T s0 = up ? d0 : d2, s1 = up ? d1 : d3;  // given to lane ^ 16
  a0 += __shfl_xor_sync(0xffffffffu, s0, 16);
  a1 += __shfl_xor_sync(0xffffffffu, s1, 16);
  T v = odd ? a1 : a0;
  v += __shfl_xor_sync(0xffffffffu, odd ? a0 : a1, 8);
  v += __shfl_xor_sync(0xffffffffu, v, 4);
  v += __shfl_xor_sync(0xffffffffu, v, 2);
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  if ((lane & 7) == 0) shv[lane >> 3][warp] = v;
}

// warps that fold and the words of a lane in flight (160 or 192 blocks in one turn): an
// FP64 addition takes a scheduler 64 cycles, so fewer warps with more of their own
template <typename Acc>
constexpr int kFoldWarps = 8;
template <>
constexpr int kFoldWarps<double> = 4;
template <typename Acc>
constexpr int kFoldWords = kFoldWarps<Acc> == 4 ? 5 : 3;

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

// The grid-wide sum of p.q, r.r, r.q and q.q at iteration `iter`: each warp's four
// values by a transposing butterfly; warp 0 combines the warps' (FP32 ones as
// compensated pairs), writes them into kChipSpread copies, arrives on one of
// kChipSpread counters and waits for all of them; the first kFoldWarps warps fold a
// part of the blocks each from the block's copy, in a fixed order, so every block
// obtains the same totals in tot (in warp 0).  A block's four values lie together: a line that eight
// blocks read has four writers, not sixteen.  meanwhile() runs in the other warps
// while warp 0 waits and must not depend on the sum; load() runs in every thread once
// all blocks have arrived and may read what they published before; in the folding warps
// its loads follow the fold's own, or with LoadFirst precede them, which takes fewer
// registers.  At the return tot and fail are valid in warp 0.
struct ChipNothing {
  __device__ __forceinline__ void operator()() const {}
};
template <bool LoadFirst, typename T, typename Acc, typename Meanwhile, typename Load>
__device__ __forceinline__ void chip_sum(const ChipArgs<T>& f, int iter, T d0, T d1, T d2, T d3, T (&shv)[4][kChipWarps],
                                         Acc (&part)[32], Acc (&tot)[4], int& fail, Meanwhile&& meanwhile,
                                         Load&& load) {
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
  const unsigned G = gridDim.x;
  chip_butterfly(d0, d1, d2, d3, shv);
  // also orders every thread's q-face stores before warp 0's release
  __syncthreads();
  // this sum's partials: kChipSpread copies, this block reads copy b mod kChipSpread
  Acc* slot = reinterpret_cast<Acc*>(f.spread) + (size_t)(iter & 1) * kChipSpread * 4 * G;
  if (warp == 0) {
    // lanes 8k .. 8k + 7: value k of the block
    const int k = lane >> 3;
    Acc a = acc_of(T(0));
    for (int w = lane & 7; w < nwarp; w += 8) a = acc_add(a, acc_of(shv[k][w]));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a = acc_add(a, acc_xor(a, o));
    // lane l writes value l mod 4 into copy l / 4
    const Acc mine = acc_from_lane(a, 8 * (lane & 3));
    acc_store(slot + ((size_t)(lane >> 2) * G + blockIdx.x) * 4 + (lane & 3), mine);
    __syncwarp();  // orders the lanes' stores before lane 0's release
    if (lane == 0) red_release_add(f.counters + (blockIdx.x % kChipSpread) * kChipLine, 1u);
    // posted: the other warps may start their own work
    asm volatile("bar.arrive 2, %0;" ::"r"(nthr) : "memory");
    // lanes 0 .. kChipSpread - 1 wait for one counter each (counter i takes
    // blocks i, i + kChipSpread, ...; counter 0 also the test hook's missing
    // arrivals)
    bool done = lane >= kChipSpread;
    const unsigned mine_n = lane < (int)G ? (G - lane + kChipSpread - 1) / kChipSpread : 0u;
    const unsigned target = done ? 0u : ((unsigned)iter + 1u) * (mine_n + (lane == 0 ? f.missing : 0u));
    const long long t0 = clock64();
    int gave_up = 0;
    for (unsigned spins = 1;; ++spins) {
      if (!done) done = (int)(ld_acquire(f.counters + lane * kChipLine) - target) >= 0;
      if (__all_sync(0xffffffffu, done)) break;
      const bool quit = (spins & 63u) == 0u && (ld_volatile(&f.bar->fail.v) != 0u || clock64() - t0 > f.spin_cycles);
      if (__any_sync(0xffffffffu, quit)) {
        if (lane == 0) atomicExch(&f.bar->fail.v, 1u);
        gave_up = 1;
        break;
      }
    }
    __syncwarp();  // orders the lanes' acquires before the reads of every lane
    if (lane == 0) fail = gave_up;
    // every block has arrived (or the wait gave up)
    asm volatile("bar.arrive 1, %0;" ::"r"(nthr) : "memory");
  } else {
    asm volatile("bar.sync 2, %0;" ::"r"(nthr) : "memory");
    meanwhile();
    asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
  }
  const Acc* mycopy = slot + (size_t)(blockIdx.x % kChipSpread) * 4 * G;
  constexpr int FW = kFoldWarps<Acc>, U = kFoldWords<Acc>;
  if (LoadFirst || warp >= FW) load();
  if (warp < FW) {
    for (int id = warp; id < FW; id += nwarp) {  // eight blocks at a time, a lane per value
      Acc t = acc_of(T(0));
      for (unsigned b0 = (unsigned)id * 8 + (lane >> 2); b0 - (lane >> 2) < G; b0 += 8 * FW * U) {
        Acc w[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          w[u] = b0 + 8 * FW * u < G ? acc_load(mycopy + (size_t)(b0 + 8 * FW * u) * 4 + (lane & 3)) : acc_of(T(0));
        if (!LoadFirst && id == warp && b0 == (unsigned)id * 8 + (lane >> 2)) load();
#pragma unroll
        for (int u = 0; u < U; ++u) t = acc_add(t, w[u]);
      }
      if (!LoadFirst && id == warp && (unsigned)id * 8 >= G) load();
      chip_fold_warp(t, part, id);
    }
    chip_fold(part, tot);
  }
}

// ---- tagged words ------------------------------------------------------------
// A value that other blocks wait for travels with the number of its iteration: every
// 8 bytes hold 32 bits of it and a 32-bit tag, written and read whole, so a reader
// that finds the tag has the value, and neither side orders it against anything
// else.  A writer that released a flag would wait for its stores to reach L2, and a
// reader that had seen it would read the value by another trip.  The tags are NaN
// patterns, which no finite value left in the same memory can look like.
__device__ __forceinline__ unsigned chip_tag(int iter) { return 0xff800001u + ((unsigned)iter & 0x3fffffu); }
template <typename V>
struct Tagged {  // F2 or double: 16 bytes
  unsigned long long w[2];
};
template <>
struct Tagged<float> {
  unsigned long long w[1];
};
__device__ __forceinline__ void tagged_load(Tagged<float>& t, const char* at) {
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(t.w[0]) : "l"(at));
}
template <typename V>
__device__ __forceinline__ void tagged_load(Tagged<V>& t, const char* at) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(t.w[0]), "=l"(t.w[1]) : "l"(at));
}
__device__ __forceinline__ bool tagged_ok(const Tagged<float>& t, unsigned tag) { return (unsigned)(t.w[0] >> 32) == tag; }
template <typename V>
__device__ __forceinline__ bool tagged_ok(const Tagged<V>& t, unsigned tag) {
  return (unsigned)(t.w[0] >> 32) == tag && (unsigned)(t.w[1] >> 32) == tag;
}
__device__ __forceinline__ float tagged_value(const Tagged<float>& t) { return __uint_as_float((unsigned)t.w[0]); }
__device__ __forceinline__ F2 tagged_value(const Tagged<F2>& t) {
  return F2{__uint_as_float((unsigned)t.w[0]), __uint_as_float((unsigned)t.w[1])};
}
__device__ __forceinline__ double tagged_value(const Tagged<double>& t) {
  return __hiloint2double((int)(unsigned)t.w[1], (int)(unsigned)t.w[0]);
}
__device__ __forceinline__ void tagged_store16(char* at, unsigned a, unsigned b, unsigned tag) {
  const unsigned long long hi = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(at), "l"(hi | a), "l"(hi | b) : "memory");
}
__device__ __forceinline__ void tagged_store(char* at, float v, unsigned tag) {
  const unsigned long long w = (unsigned long long)tag << 32 | __float_as_uint(v);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(at), "l"(w) : "memory");
}
__device__ __forceinline__ void tagged_store(char* at, F2 v, unsigned tag) {
  tagged_store16(at, __float_as_uint(v.hi), __float_as_uint(v.lo), tag);
}
__device__ __forceinline__ void tagged_store(char* at, double v, unsigned tag) {
  tagged_store16(at, (unsigned)__double2loint(v), (unsigned)__double2hiint(v), tag);
}

// The words of a sum's partials: [2 slots][gridDim.x][4 values] of 16 bytes.  A
// block's four lie together, so that a line has two writers: with a value's words of
// all blocks together, and eight writers to a line that is being read, an iteration on
// 32^3 in FP32 took 3.1 us instead of 2.2.  Several copies do not help.  A block may
// write a slot again two sums later: it gets there only after every block has posted
// the sum between, and so has read this one.  Cleared by each block for itself before
// the set-up sums, which order that for everyone.
__device__ __forceinline__ void chip_sum_clear(void* spread) {
  const int slot = threadIdx.x >> 2, k = threadIdx.x & 3;
  if (slot < 2)
    tagged_store16(static_cast<char*>(spread) + (((size_t)slot * gridDim.x + blockIdx.x) * 4 + k) * 16, 0u, 0u, 0u);
}

// The same sum by tagged words: warp 0 posts the block's four values; the first
// kFoldWarps warps read the words of a part of the blocks each, until all have come,
// and fold them in a fixed order, so every block obtains the same totals in tot (in
// warp 0).  meanwhile() runs in the other warps before they wait.  When the sum has
// come, issue() starts the loads of what this thread awaits of the neighbours; check()
// takes what has come and tells whether that was all, and both are called again until
// it is (begun earlier, they disturb the lines that are being written: 100 x 76 x 61
// FP32 takes 4.2 us, not 4.05).  fail (0 before the first sum) is set when a wait runs
// out, in other warps perhaps too late for this sum but in time for the next.
template <typename T, typename Acc, typename Meanwhile, typename Issue, typename Check>
__device__ __forceinline__ void chip_sum_tagged(const ChipArgs<T>& f, int iter, T d0, T d1, T d2, T d3, T (&shv)[4][kChipWarps],
                                         Acc (&part)[32], Acc (&tot)[4], volatile int& fail, Meanwhile&& meanwhile, Issue&& issue,
                                         Check&& check) {
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
  constexpr int FW = kFoldWarps<Acc>, U = kFoldWords<Acc>;
  const unsigned G = gridDim.x, tag = chip_tag(iter);
  chip_butterfly(d0, d1, d2, d3, shv);
  __syncthreads();
  char* slot = static_cast<char*>(f.spread) + (size_t)(iter & 1) * 4 * G * 16;
  if (warp == 0) {
    // lanes 8k .. 8k + 7: value k of the block
    const int k = lane >> 3, c = lane & 7;
    Acc a = acc_of(T(0));
    for (int w = c; w < nwarp; w += 8) a = acc_add(a, acc_of(shv[k][w]));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a = acc_add(a, acc_xor(a, o));
    if (c == 0) tagged_store(slot + ((size_t)blockIdx.x * 4 + k) * 16, a, tag);
    // posted: the other warps may start their own work
    asm volatile("bar.arrive 2, %0;" ::"r"(nthr) : "memory");
  } else {
    asm volatile("bar.sync 2, %0;" ::"r"(nthr) : "memory");
    meanwhile();
  }
  const long long t0 = clock64();
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
      Acc t = acc_of(T(0));
      for (unsigned base = (unsigned)id * 8 + (lane >> 2); base - (lane >> 2) < G; base += 8 * FW * U) {
        const char* at = slot + ((size_t)base * 4 + (lane & 3)) * 16;
        Tagged<Acc> w[U];
        unsigned miss = 0;
#pragma unroll
        for (int u = 0; u < U; ++u) miss |= base + 8 * FW * u < G ? 1u << u : 0u;
        const unsigned have = miss;
        for (unsigned spins = 1;; ++spins) {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (miss >> u & 1u) tagged_load(w[u], at + 512 * FW * u);
#pragma unroll
          for (int u = 0; u < U; ++u)
            if ((miss >> u & 1u) && tagged_ok(w[u], tag)) miss &= ~(1u << u);
          if (__all_sync(0xffffffffu, miss == 0u && f.missing == 0u) || over(spins)) break;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) t = acc_add(t, have >> u & 1u ? tagged_value(w[u]) : acc_of(T(0)));
      }
      if (id + nwarp >= FW) {
        if (nwarp > FW) asm volatile("bar.arrive 1, %0;" ::"r"(nthr) : "memory");
        issue();
      }
      chip_fold_warp(t, part, id);
    }
    chip_fold(part, tot);
  } else {
    asm volatile("bar.sync 1, %0;" ::"r"(nthr) : "memory");
    issue();
  }
  for (unsigned spins = 1;; ++spins) {
    if (__all_sync(0xffffffffu, check()) || over(spins)) break;
    issue();
  }
}

// les_cg_brick.cu: a brick's columns and planes at most; the kernel for bricks of at
// most zp planes (a multiple of 8), its shared memory and the elements of its arrays
constexpr int kBrickX = 32, kBrickY = 16, kBrickPlanes = 64;
size_t brick_smem(int zp, int* np, int* ng);
const void* brick_kernel(int zp);

}  // namespace les
