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
  double* partials;    // two slots of kSumSlot words per block (the set-up and gauge sums)
  unsigned* counters;  // kChipSpread arrival counters of the iterations' sums, kChipLine apart, zeroed
  void* spread;        // [2 slots][kChipSpread copies][4 values][gridDim.x] partials of those sums
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

// The grid-wide sum of p.q, r.r, r.q and q.q at iteration `iter`: each warp's four
// values by a transposing butterfly; warp 0 combines the warps' (FP32 ones as
// compensated pairs), writes them into kChipSpread copies, arrives on one of
// kChipSpread counters and waits for all of them; warps 0 .. 3 fold one value each
// from the block's copy, in block order, so every block obtains the same totals in
// tot.  meanwhile() runs in the other warps while warp 0 waits and must not depend
// on the sum; load() runs in every thread once all blocks have arrived and may read
// what they published before; in warps 0 .. 3 its loads follow the fold's own, or with
// LoadFirst precede them, which takes fewer registers.  At the return tot and fail are valid in warps 0 .. 3.
struct ChipNothing {
  __device__ __forceinline__ void operator()() const {}
};
template <bool LoadFirst, typename T, typename Acc, typename Meanwhile, typename Load>
__device__ __forceinline__ void chip_sum(const ChipArgs<T>& f, int iter, T d0, T d1, T d2, T d3, T (&shv)[4][kChipWarps],
                                         Acc (&tot)[4], int& fail, Meanwhile&& meanwhile, Load&& load) {
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarp = nthr >> 5;
  const unsigned G = gridDim.x;
  // after the butterfly lanes 8k .. 8k + 7 hold the warp's value k
  {
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
    acc_store(slot + ((size_t)(lane >> 2) * 4 + (lane & 3)) * G + blockIdx.x, mine);
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
  if (LoadFirst || warp >= 4) load();
  if (warp < 4) {
    for (int k = warp; k < 4; k += nwarp) {
      Acc t = acc_of(T(0));
      for (unsigned b0 = lane; b0 < G; b0 += 32 * 5) {
        Acc w[5];
#pragma unroll
        for (int u = 0; u < 5; ++u)
          w[u] = b0 + 32 * u < G ? acc_load(mycopy + (size_t)k * G + b0 + 32 * u) : acc_of(T(0));
        if (!LoadFirst && k == warp && b0 == (unsigned)lane) load();
#pragma unroll
        for (int u = 0; u < 5; ++u) t = acc_add(t, w[u]);
      }
      if (!LoadFirst && k == warp && (unsigned)lane >= G) load();
      t = acc_warp(t);
      if (lane == 0) tot[k] = t;
    }
    asm volatile("bar.sync 3, %0;" ::"r"(32 * min(nwarp, 4)) : "memory");
  }
}

// les_cg_brick.cu: a brick's columns and planes at most; the kernel for bricks of at
// most zp planes (a multiple of 8), its shared memory and the elements of its arrays
constexpr int kBrickX = 32, kBrickY = 16, kBrickPlanes = 64;
size_t brick_smem(int zp, int* np, int* ng);
const void* brick_kernel(int zp);

}  // namespace les
