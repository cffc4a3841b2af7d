// les_cg_chip.cu -- the on-chip conjugate-gradient Poisson solve (Sec. 2.4:
// L_c psi = b, compact 7-point Laplacian, periodic in x and y, mirror or
// periodic in z; mean of b removed, psi returned with zero mean) for any
// grid whose vectors fit in the registers of one block per SM, FP32 or FP64.
//
// Each block of one persistent cooperative launch owns a brick of the grid
// for the whole solve.  The brick extents along x, y and z differ by at most
// one node between blocks, so no extent has to divide the grid.  A thread
// owns one (x, y) column of the brick and a run of at most ZP planes of it,
// and keeps p, r, q = L_c p and x of those nodes in registers.  Its z
// neighbours are its own registers; the x and y neighbours, and the z
// neighbours past either end of the run, come from a copy of p in shared
// memory with a one-node ghost layer.  A brick that spans a periodic extent
// reads its own far side, and a wall mirrors the node itself, so such sides
// have no ghosts.  The ghost nodes are dealt to the threads: an iteration
// loads the neighbours' published q faces and forms the ghost r and p from
// them, so one exchange per iteration is enough.  Where a thread has few
// planes and at most four ghosts (XS = false), x and the ghosts' r and p are
// registers too; else x, the ghosts' r and their offsets lie in shared memory
// (XS = true), which leaves room for 24 FP32 or 12 FP64 planes of p, r and q.
//
// The iteration is that of les_cg_resident.cu: one grid-wide sum of p.q,
// r.r, r.q and q.q per iteration (alpha, and beta from |r - alpha q|^2
// expanded in the four; les_chip.cuh).  With XS = false the faces' q are tagged words;
// with more faces these cost more than they save (150 x 140 x 70 FP32: 13 us per
// iteration instead of 9.3 at the time), and counters order them.
//
// What bounds it: the latency of the grid sum (2.1 us of an iteration on the
// smallest grids) and, in FP64, the
// arithmetic: a scheduler issues an FP64 warp instruction every 64 cycles, so
// a five-step butterfly of four values in 16 warps alone costs 5000 cycles.
// The four values are therefore reduced by a transposing butterfly (six
// additions per warp instead of twenty), the plan weighs warps against planes
// per thread, the FP64 stencil takes six operations, and x += alpha p is left
// to the next sum's wait.
//
// Measured (GB300, us per iteration; before: the
// shared-memory kernel, or the one-pass streaming kernel where no whole
// bricks fit):
//   FP64  32^3 9.9 -> 4.7, 256 x 4 x 32 10.1 -> 4.7, 64 x 64 x 48 16.9 -> 9.3,
//         50 x 47 x 33 28.3 -> 6.9, 77 x 130 x 50 66.8 -> 16.5, 96^3 77 -> 27
//   FP32  32^3 4.2 -> 2.1, 64^3 5.0 -> 2.8, 96^3 7.3 -> 4.8, 160 x 160 x 48
//         8.4 -> 5.8, 100 x 76 x 61 23.6 -> 3.8, 150 x 140 x 70 36.7 -> 8.7
// (in FP32 3 to 6 % of it for sums that are compensated from the threads on, and
// scalars from the whole totals).
// FP32 grids 128 nodes wide keep les_cg_regs.cu, whose four-node lanes read
// x neighbours by shuffles: 128 x 64 x 64 2.7 there, 64 x 128 x 64 3.4 here; 128 x
// 128 x 96 4.5, 96 x 128 x 128 7.5.
#include <algorithm>
#include <cmath>
#include <string>

#include "les_chip.cuh"

namespace les {
namespace {

template <typename T, int ZP, bool XS>
__global__ void __launch_bounds__(kChipThreads, 1) k_cg_chip(ChipArgs<T> f) {
  using Acc = decltype(Dot<T>().acc());  // FP32 pair (FP32 solve) or FP64
  extern __shared__ __align__(16) unsigned char smraw[];
  constexpr int NG = XS ? 1 : kChipGhosts;  // ghosts per thread held in registers
  T* P = reinterpret_cast<T*>(smraw);  // p with its ghost layer
  const int tid = threadIdx.x, nthr = blockDim.x;
  const int warp = tid >> 5;
  int i0, j0, k0, bx, by, bz;
  chip_part(f.nx, f.px, blockIdx.x % f.px, i0, bx);
  chip_part(f.ny, f.py, (blockIdx.x / f.px) % f.py, j0, by);
  chip_part(f.nz, f.pz, blockIdx.x / (f.px * f.py), k0, bz);
  const int SY = bx + 2, SZ = SY * (by + 2);
  const int gpl = f.nx * f.ny;
  const bool low = f.walls && k0 == 0, high = f.walls && k0 + bz == f.nz;  // the brick touches a wall
  const T cx = f.cx, cy = f.cy, cz = f.cz;

  // this thread's column and run of planes
  const int ncol = bx * by;
  const int run = tid / ncol;
  const int col = tid - run * ncol;
  const bool active = run < f.zs;
  const int ly = col / bx, lx = col - ly * bx;
  const int zq = bz / f.zs, zr = bz - zq * f.zs;
  const int z0 = run * zq + min(run, zr);
  const int nzp = active ? zq + (run < zr ? 1 : 0) : 0;
  int pown = (z0 + 1) * SZ + (ly + 1) * SY + lx + 1;
  int gown = (k0 + z0) * gpl + (j0 + ly) * f.nx + i0 + lx;
  // offsets of the neighbours in P: a brick that spans a periodic extent
  // wraps onto itself, a wall mirrors the node
  const int oxm = f.px == 1 && lx == 0 ? bx - 1 : -1, oxp = f.px == 1 && lx == bx - 1 ? 1 - bx : 1;
  const int oym = f.py == 1 && ly == 0 ? (by - 1) * SY : -SY, oyp = f.py == 1 && ly == by - 1 ? (1 - by) * SY : SY;
  int ozm = -SZ, ozp = SZ;  // below the run's first plane, above its last
  if (z0 == 0) {
    if (low) ozm = 0;
    else if (!f.walls && f.pz == 1) ozm = (bz - 1) * SZ;
  }
  if (z0 + nzp == bz) {
    if (high) ozp = 0;
    else if (!f.walls && f.pz == 1) ozp = (1 - bz) * SZ;
  }
  // nodes that a neighbouring brick reads
  const bool fcol = (f.px > 1 && (lx == 0 || lx == bx - 1)) || (f.py > 1 && (ly == 0 || ly == by - 1));
  const bool flow = f.pz > 1 && !low && z0 == 0, fhigh = f.pz > 1 && !high && z0 + nzp == bz;
  auto is_face = [&](int j) { return fcol || (flow && j == 0) || (fhigh && j == nzp - 1); };

  // the brick's ghost nodes: the z faces, then the y faces, then the x faces
  const int nlo = f.pz > 1 && !low ? ncol : 0, nhi = f.pz > 1 && !high ? ncol : 0;
  const int nyf = f.py > 1 ? bx * bz : 0, nxf = f.px > 1 ? by * bz : 0;  // nodes per y and x face
  const int ngh = nlo + nhi + 2 * (nyf + nxf);
  // offsets of ghost node id in P and in global memory.  A ghost beyond a
  // wall does not occur: the sides that touch one have none.
  auto ghost_at = [&](int id) -> int2 {
    int gx = 0, gy = 0, gz = 0;
    if (id < nlo + nhi) {
      gz = id < nlo ? -1 : bz;
      id -= id < nlo ? 0 : nlo;
      gy = id / bx, gx = id - gy * bx;
    } else if ((id -= nlo + nhi) < 2 * nyf) {
      gy = id < nyf ? -1 : by;
      id -= id < nyf ? 0 : nyf;
      gz = id / bx, gx = id - gz * bx;
    } else {
      id -= 2 * nyf;
      gx = id < nxf ? -1 : bx;
      id -= id < nxf ? 0 : nxf;
      gz = id / by, gy = id - gz * by;
    }
    return make_int2((gz + 1) * SZ + (gy + 1) * SY + gx + 1,
                     chip_wrap(k0 + gz, f.nz) * gpl + chip_wrap(j0 + gy, f.ny) * f.nx + chip_wrap(i0 + gx, f.nx));
  };
  // XS: x by plane and thread, then r, q and the offsets of the ghost nodes
  T* XM = P + f.smem_p;
  T* GR = XM + ZP * nthr;
  T* GQ = GR + f.smem_g;
  int2* GT = reinterpret_cast<int2*>(GQ + f.smem_g);
  int gsm[NG], ggl[NG];  // else: this thread's ghosts (-1: none)
  if constexpr (XS) {
    for (int id = tid; id < ngh; id += nthr) GT[id] = ghost_at(id);
    gsm[0] = ggl[0] = 0;
  } else {
#pragma unroll
    for (int g = 0; g < NG; ++g) {
      const int id = tid + g * nthr;
      gsm[g] = -1;
      ggl[g] = 0;
      if (id < ngh) {
        const int2 o = ghost_at(id);
        gsm[g] = o.x;
        ggl[g] = o.y;
      }
    }
  }

  T p[ZP] = {}, r[ZP] = {}, q[ZP] = {};
  T xr[XS ? 1 : ZP] = {};
  auto get_x = [&](int j) -> T { return XS ? XM[j * nthr + tid] : xr[XS ? 0 : j]; };
  auto set_x = [&](int j, T v) {
    if constexpr (XS) XM[j * nthr + tid] = v;
    else xr[j] = v;
  };
  // x += alpha p of an iteration is added during the next sum's wait, where
  // registers for the old p are left (warp 0, which waits, adds it at once)
  constexpr bool kDefer = !XS && ZP * sizeof(T) <= 32;
  T po[kDefer ? ZP : 1] = {};
  T rgh[NG] = {}, pgh[NG] = {};  // r and p at the ghost nodes
  // L_c p at plane j of the run.  FP32: second differences formed before
  // scaling, as in the other CG kernels.  FP64, where each operation counts:
  // q' with L_c p = -c0 q', c0 the centre coefficient -- six operations instead
  // of nine.  The recurrences of r and p do not see the factor; the update of x
  // takes it up (its alpha is -1 / c0 times theirs).
  constexpr bool kScaled = sizeof(T) == 8;
  const T c0 = T(2) * (cx + cy + cz);
  const T ax = cx / c0, ay = cy / c0, az = cz / c0, mc0 = T(-1) / c0;
  auto stencil = [&](int j, bool inner) -> T {  // inner: plane j + 1 is surely of the run
    const T* pj = P + pown + j * SZ;
    const T d = j > 0 ? p[j > 0 ? j - 1 : 0] : pj[ozm];
    const T u = (j + 1 < ZP && (inner || j + 1 < nzp)) ? p[j + 1 < ZP ? j + 1 : ZP - 1] : pj[ozp];
    if constexpr (kScaled) {
      return fma(-az, d + u, fma(-ay, pj[oym] + pj[oyp], fma(-ax, pj[oxm] + pj[oxp], p[j])));
    } else {
      const T c2 = T(2) * p[j];
      return (pj[oxm] + pj[oxp] - c2) * cx + (pj[oym] + pj[oyp] - c2) * cy + (d + u - c2) * cz;
    }
  };

  // body(plane, its upper neighbour is surely of the run) up this thread's run.  The
  // plane counts are instantiated in steps of KT, so a run lacks KT planes at most; a
  // warp whose runs all have the others has no test between those, and their chains
  // overlap (FP32: 96^3 5.0 -> 4.7 us per iteration, 150 x 140 x 70 9.4 -> 8.2 as the
  // sums were then; FP64 waits for its arithmetic, not for chains, and loses 2 % by the
  // longer code).
  constexpr int KT = XS ? 4 : 2, ZF = sizeof(T) == 4 && ZP > KT ? ZP - KT : 0;
  const bool full = __all_sync(0xffffffffu, nzp >= ZF);
  auto each_plane = [&](auto&& body) {
    if (ZF > 0 && full) {
#pragma unroll
      for (int j = 0; j < ZF; ++j) body(j, j + 1 < ZF);
#pragma unroll
      for (int j = ZF; j < ZP; ++j)
        if (j < nzp) body(j, false);
    } else {
#pragma unroll
      for (int j = 0; j < ZP; ++j)
        if (j < nzp) body(j, false);
    }
  };

  // A at the ghost nodes into P (keep: as r and p there), outside the iterations
  auto fill_ghosts = [&](const T* A, bool keep) {
    if constexpr (XS) {
      for (int id = tid; id < ngh; id += nthr) {
        const int2 o = GT[id];
        const T v = __ldcg(A + o.y);
        P[o.x] = v;
        if (keep) GR[id] = v;
      }
    } else {
#pragma unroll
      for (int g = 0; g < NG; ++g)
        if (gsm[g] >= 0) {
          const T v = __ldcg(A + ggl[g]);
          P[gsm[g]] = v;
          if (keep) rgh[g] = pgh[g] = v;
        }
    }
  };

  GridSync gs{f.bar, f.partials, f.spin_cycles, f.expected, 0u};
  __shared__ struct {
    T mean, ta, tb, tx;  // alpha and beta of r and p, alpha of x
    T scale, xs;         // of r, p and q (FP64: 1); alpha of x over that of r
    int status, restart;
    double bb, rel;  // |b - mean|^2 and the relative residual of x0
  } sc;
  __shared__ Acc shv[4][kChipWarps];
  __shared__ Acc part[32];
  __shared__ int s_fail;
  double rr = 0.0, bb = 0.0, rel = 0.0;  // meaningful in thread 0
  int status = 0;  // 0 running, 1 converged, 2 maxit, 3 breakdown, 4 zero rhs, 5 timeout
  Acc rr_own{};  // this thread's share of r.r for the next sum

  // XS = false: a node's tagged word among the published faces of q (with an odd number
  // of nodes the last one ends in the padding of its array, whose size is a multiple of
  // 256 bytes)
  constexpr int W = Tagged<T>::BYTES;
  const int half = (int)(f.n / 2);
  auto word = [&](int s, int g) { return (g < half ? f.qt[0][s] : f.qt[1][s] - (size_t)half * W) + (size_t)g * W; };
  chip_sum_clear<Acc>(f.spread);  // no tag of an earlier solve: cleared here, for everyone after the first sum
  if constexpr (!XS) {
#pragma unroll
    for (int j = 0; j < ZP; ++j)
      if (j < nzp && is_face(j)) {
        tagged_clear<T>(word(0, gown + j * gpl));
        tagged_clear<T>(word(1, gown + j * gpl));
      }
  }
  if (tid == 0) s_fail = 0;

  // mean of b (b held in r, x0 in p), FP32: |b|_1 and |x0|_1
  {
    constexpr int NV = kScaled ? 1 : 3;
    ChipRun<T, ZP> a[NV];
#pragma unroll
    for (int j = 0; j < ZP; ++j)
      if (j < nzp) {
        r[j] = __ldcg(f.b + gown + j * gpl);
        p[j] = __ldcg(f.x + gown + j * gpl);
        a[0].add(j, r[j]);
        if constexpr (!kScaled) {
          a[1].add(j, fabsf(r[j]));
          a[2].add(j, fabsf(p[j]));
        }
      }
    Acc v[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) v[k] = a[k].total();
    double t[NV];
    const bool ok = grid_sum_t0<NV>(v, gs, t);
    if (tid == 0) {
      sc.status = ok ? 0 : 5;
      sc.mean = (T)(t[0] / (double)f.n);
      if constexpr (kScaled) sc.scale = T(1);
      else sc.scale = chip_scale(t[1], t[2], c0 * f.sc, (double)f.n);
      sc.xs = kScaled ? mc0 : f.isc / sc.scale;
    }
    __syncthreads();
    status = sc.status;
  }
  const T mean = sc.mean;
  // x0 with its ghosts in p and the copy; r = (b - mean) - L_c x0, scaled, published
  if (!status) {
#pragma unroll
    for (int j = 0; j < ZP; ++j)
      if (j < nzp) {
        set_x(j, p[j]);
        P[pown + j * SZ] = p[j];
      }
    fill_ghosts(f.x, false);
    __syncthreads();
    ChipRun<T, ZP> a2[2];
#pragma unroll
    for (int j = 0; j < ZP; ++j)
      if (j < nzp) {
        T bm = r[j] - mean;
        r[j] = kScaled ? fma(c0, stencil(j, false), bm) : (bm - f.sc * stencil(j, false)) * sc.scale;
        if constexpr (!kScaled) bm *= sc.scale;
        if (is_face(j)) __stcg(f.rg + gown + j * gpl, r[j]);
        a2[0].add(j, r[j] * r[j]);
        a2[1].add(j, bm * bm);
      }
    rr_own = a2[0].total();
    Acc v[2] = {rr_own, a2[1].total()};
    double s2[2];
    const bool ok = grid_sum_t0<2>(v, gs, s2);
    if (tid == 0) {
      // the plain solver judges a learned first guess: if it leaves a larger
      // residual than x0 = 0, restart from zero (r = b - mean b, r.r = |b|^2)
      sc.status = ok ? 0 : 5;
      sc.restart = ok && f.guard && s2[0] > s2[1];
      rr = sc.restart ? s2[1] : s2[0];
      bb = s2[1];
    }
    __syncthreads();
    status = sc.status;
    if (!status && sc.restart) {
      ChipRun<T, ZP> s;
#pragma unroll
      for (int j = 0; j < ZP; ++j)
        if (j < nzp) {
          set_x(j, T(0));
          r[j] = (__ldcg(f.b + gown + j * gpl) - mean) * sc.scale;
          s.add(j, r[j] * r[j]);
          if (is_face(j)) __stcg(f.rg + gown + j * gpl, r[j]);
        }
      rr_own = s.total();
      Dot<T> none[1];
      double t[1];
      const bool ok2 = grid_dot_t0<1>(none, gs, t);  // a grid barrier: the new faces are visible
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
        else if (!isfinite(bb)) status = 3;  // (r.r <= tol^2 |b|^2 would hold)
      }
    }
    sc.status = status;
    sc.bb = bb;
    sc.rel = rel;
  }
  __syncthreads();
  status = sc.status;
  Acc rr_stop, rr_last;  // rr_last meaningful in thread 0
  acc_from(f.tol * f.tol * sc.bb, rr_stop);
  acc_from(rr, rr_last);
  int iter = 0;
  T ta = T(0), tb = T(0), tx = T(0);
  if (!status) {
    // p_0 = r_0, with r_0 at the ghost nodes from the published faces
#pragma unroll
    for (int j = 0; j < ZP; ++j)
      if (j < nzp) {
        p[j] = r[j];
        P[pown + j * SZ] = p[j];
      }
    fill_ghosts(f.rg, true);
    __syncthreads();
    for (;;) {
      // the offsets of the planes are formed anew in each iteration: hoisted out
      // of the loop they would take the registers of the vectors
      asm volatile("" : "+r"(pown), "+r"(gown));
      T* qw = (iter & 1) ? f.qg1 : f.qg0;  // this iteration's q faces
      ChipRun<T, ZP> d0, d2, d3;           // p.q, r.q, q.q
      each_plane([&](int j, bool inner) {
        q[j] = stencil(j, inner);
        if (is_face(j)) {
          if constexpr (XS) __stcg(qw + gown + j * gpl, q[j]);
          else tagged_store(word(iter & 1, gown + j * gpl), q[j], iter);
        }
        d0.add(j, p[j] * q[j]);
        d2.add(j, r[j] * q[j]);
        d3.add(j, q[j] * q[j]);
      });
      Tagged<T> gq[NG];  // the q of the ghosts
      Acc tot[4];        // the totals, in warp 0
      constexpr int WORDS = sizeof(T) == 8 && ZP < 10 ? 5 : 3;
      auto deferred = [&] {
        if constexpr (kDefer) {
          if (iter > 0) {
#pragma unroll
            for (int j = 0; j < ZP; ++j) xr[XS ? 0 : j] += tx * po[kDefer ? j : 0];
          }
        }
      };
      if constexpr (XS) {
        chip_sum<1, WORDS>(
            f, iter, d0.total(), rr_own, d2.total(), d3.total(), shv, part, tot, s_fail, deferred,
            [&] {
              const int t0 = 32 * chip_ghost_warp<1>();
              for (int id = tid - t0; id < ngh; id += nthr - t0) cp_async(GQ + id, qw + GT[id].y);
              cp_commit();
            },
            ChipNothing{});
      } else {
        unsigned miss = 0;
#pragma unroll
        for (int g = 0; g < NG; ++g) miss |= gsm[g] >= 0 ? 1u << g : 0u;
        chip_sum<-1, WORDS>(
            f, iter, d0.total(), rr_own, d2.total(), d3.total(), shv, part, tot, s_fail, deferred,
            [&] {
#pragma unroll
              for (int g = 0; g < NG; ++g)
                if (miss >> g & 1u) tagged_load(gq[g], word(iter & 1, ggl[g]));
            },
            [&] {
#pragma unroll
              for (int g = 0; g < NG; ++g)
                if ((miss >> g & 1u) && tagged_ok(gq[g], iter)) miss &= ~(1u << g);
              return miss == 0u;
            });
      }
      if (warp == 0) {  // the status, alpha and beta
        T al = T(0), be = T(0);
        const bool good = chip_scalars(tot, al, be);
        if (tid == 0) {
          int st = 0;
          if (s_fail) {
            st = 5;
          } else {
            rr_last = tot[1];
            if (acc_le(tot[1], rr_stop)) st = 1;
            else if (iter >= f.maxit) st = 2;
            else if (!good) st = 3;
            sc.ta = al;
            sc.tb = be;
            sc.tx = al * sc.xs;
          }
          sc.status = st;
        }
      }
      if constexpr (XS) cp_wait<0>();
      __syncthreads();
      status = sc.status;
      if (status) break;
      ta = sc.ta;
      tb = sc.tb;
      tx = sc.tx;
      ChipRun<T, ZP> s;
      each_plane([&](int j, bool) {
        if (!kDefer || warp == 0) set_x(j, get_x(j) + tx * p[j]);
        else po[kDefer ? j : 0] = p[j];
        r[j] -= ta * q[j];
        s.add(j, r[j] * r[j]);
        p[j] = r[j] + tb * p[j];
        P[pown + j * SZ] = p[j];
      });
      rr_own = s.total();
      if constexpr (XS) {
        for (int id = tid; id < ngh; id += nthr) {
          const int at = GT[id].x;
          const T rv = GR[id] - ta * GQ[id];
          GR[id] = rv;
          P[at] = rv + tb * P[at];
        }
      } else {
#pragma unroll
        for (int g = 0; g < NG; ++g)
          if (gsm[g] >= 0) {
            rgh[g] -= ta * tagged_value(gq[g]);
            pgh[g] = rgh[g] + tb * pgh[g];
            P[gsm[g]] = pgh[g];
          }
      }
      iter += 1;
      __syncthreads();
    }
  }
  if (tid == 0) rel = (iter > 0 && sc.bb > 0.0) ? sqrt(acc_value(rr_last) / sc.bb) : sc.rel;

  // zero-mean gauge (or zero for a zero right side), written back to x
  if (status != 5) {
    ChipRun<T, ZP> s;
#pragma unroll
    for (int j = 0; j < ZP; ++j)
      if (j < nzp) s.add(j, get_x(j));
    Acc v[1] = {s.total()};
    double t[1];
    const bool ok = grid_sum_t0<1>(v, gs, t);
    if (tid == 0) {
      if (!ok) status = 5;
      else if (status < 3 && !isfinite(t[0])) status = 3;  // x has left the range
      sc.mean = (T)(t[0] / (double)f.n);
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
    if (status != 5) {
      const T mx = sc.mean;
#pragma unroll
      for (int j = 0; j < ZP; ++j)
        if (j < nzp) __stcg(f.x + gown + j * gpl, status == 4 ? T(0) : get_x(j) - mx);
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    f.ctl->iter = iter;
    f.ctl->rel = rel;
    f.ctl->done = status;
  }
}

// planes per thread with x and the ghosts in registers, and at most
template <typename T>
constexpr int kChipRegPlanes = sizeof(T) == 4 ? 8 : 4;
template <typename T>
constexpr int kChipMaxPlanes = sizeof(T) == 4 ? 24 : 12;

// the instantiated plane counts that hold zp planes
inline int chip_planes(int zp, bool xs, size_t es) {
  static constexpr int r4[] = {1, 2, 4, 6, 8}, x4[] = {4, 8, 12, 16, 20, 24}, r8[] = {1, 2, 4}, x8[] = {4, 6, 8, 10, 12};
  const int* t = es == 4 ? (xs ? x4 : r4) : (xs ? x8 : r8);
  while (*t < zp) ++t;
  return *t;
}

// Bricks of bx x by x bz nodes (rounded up), at most one per SM; for each
// (px, py) as many bricks along z as the SMs hold, in runs that fit a block's
// threads and a thread's planes.  Taken is the plan with the least time of
// the busiest block in the model below (cycles; the latency of the grid sum
// is common to all).  The model is a fit to some hundred timed plans: on 64^3
// FP32 eight planes per thread in 16 warps take 4.1 us, four 3.3 us; on 32^3
// FP64 two warps of four planes take 7.8 us, four of two 5.5, eight of one
// 5.8; it picks within 0.1 us of the fastest timed plan on the grids above.
template <typename T>
bool make_chip_plan(const Grid<T>& g, int nsm, size_t smem_max, int max_blocks, ChipPlan& best) {
  const int gmax = std::min(nsm, max_blocks);
  double cost = 0;
  bool found = false;
  for (int px = 1; px <= std::min(g.nx, gmax); ++px) {
    const int bx = (g.nx + px - 1) / px;
    if (px > 1 && (g.nx + px - 2) / (px - 1) == bx) continue;  // as large, with more bricks
    for (int py = 1; px * py <= gmax && py <= g.ny; ++py) {
      const int by = (g.ny + py - 1) / py, ncol = bx * by;
      if (ncol > kChipThreads || (py > 1 && (g.ny + py - 2) / (py - 1) == by)) continue;
      int pz = std::min(g.nz, gmax / (px * py));
      const int bz = (g.nz + pz - 1) / pz;
      pz = (g.nz + bz - 1) / bz;
      const size_t np = ((size_t)(bx + 2) * (by + 2) * (bz + 2) + 1) / 2 * 2;
      const int yg = py > 1 ? 2 * bx * bz : 0, xg = px > 1 ? 2 * by * bz : 0, zg = pz > 1 ? 2 * ncol : 0;
      for (int zs = 1; zs <= g.nz / pz && ncol * zs <= kChipThreads; ++zs) {
        const int zp = (bz + zs - 1) / zs, nw = (ncol * zs + 31) / 32;
        if (zp > kChipMaxPlanes<T>) continue;
        const int gh = zg + yg + xg, ng = (gh + 1) / 2 * 2;
        const bool xs = zp > kChipRegPlanes<T> || gh > kChipGhosts * 32 * nw;
        const int zi = chip_planes(zp, xs, sizeof(T));
        const size_t smem =
            (np + (xs ? (size_t)zi * 32 * nw + 2 * (size_t)ng : 0)) * sizeof(T) + (xs ? ng * sizeof(int2) : 0);
        if (smem > smem_max) continue;
        // per scheduler: 60 cycles per warp and plane; per thread: the chain
        // of its planes and ghosts; an x face is a strided access
        const int wps = (nw + 3) / 4, gt = (gh + 32 * nw - 1) / (32 * nw);
        double c = (xs ? 75.0 : 60.0) * wps * zp;
        // FP64: a warp instruction every 64 cycles of a scheduler -- 13 per
        // node, six of the reduction, two per ghost
        if (sizeof(T) == 8) c = 86.0 * (wps * (13.0 * zp + 6.0) + 2.0 * gh / 128.0);
        c += 200.0 * zp + 150.0 * gt + 3.0 * xg;
        if (!found || c < cost) {
          found = true;
          cost = c;
          best.px = px, best.py = py, best.pz = pz;
          best.zs = zs, best.zp = zi, best.threads = 32 * nw;
          best.xs = xs;
          best.np = (int)np, best.ng = ng;
          best.smem = smem;
        }
      }
    }
  }
  if (found || sizeof(T) != 4) return found;
  // larger FP32 grids: p in shared memory, r in registers (les_cg_brick.cu)
  const int px = (g.nx + kBrickX - 1) / kBrickX, py = (g.ny + kBrickY - 1) / kBrickY;
  if (px < 2 || py < 2 || px * py > gmax) return false;
  int pz = std::min(g.nz, gmax / (px * py));
  const int bz = (g.nz + pz - 1) / pz;
  pz = (g.nz + bz - 1) / bz;
  const int zp = (bz + 7) / 8 * 8;
  int np = 0, ng = 0;
  if (zp > kBrickPlanes || zp < 24 || brick_smem(zp, &np, &ng) > smem_max) return false;
  best.px = px, best.py = py, best.pz = pz;
  best.zs = 1, best.zp = zp, best.threads = kBrickX * kBrickY;
  best.brick = true;
  best.np = np, best.ng = ng;
  best.smem = brick_smem(zp, &np, &ng);
  return true;
}

template <typename T, bool XS, int... Z>
const void* chip_kernel_of(int zp) {
  const void* k = nullptr;
  ((zp == Z ? (void)(k = (const void*)k_cg_chip<T, Z, XS>) : (void)0), ...);
  return k;
}
template <typename T>
const void* chip_kernel(int zp, bool xs) {
  if constexpr (sizeof(T) == 4)
    return xs ? chip_kernel_of<T, true, 4, 8, 12, 16, 20, 24>(zp) : chip_kernel_of<T, false, 1, 2, 4, 6, 8>(zp);
  else
    return xs ? chip_kernel_of<T, true, 4, 6, 8, 10, 12>(zp) : chip_kernel_of<T, false, 1, 2, 4>(zp);
}

}  // namespace

template <typename T>
int poisson_solve_chip(const SolverArgs<T>& a, const FusedCfg& fc, const T* b, T* x, double tol, int maxit,
                       int* iters, double* rel, std::string* err, bool* used) {
  *used = false;
  if (!(a.op == LES_OP_COMPACT && a.solver == LES_SOLVER_CG && a.g.nz >= 2 && a.bar && a.r && a.q && a.p0 && a.p1) ||
      (long long)a.g.nx * a.g.ny * a.g.nz > (long long)kChipThreads * (sizeof(T) == 4 ? kBrickPlanes : kChipMaxPlanes<T>) * a.nsm)
    return LES_OK;
  int dev = 0, nsm = 0, smem_optin = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) != cudaSuccess) {
    if (err) *err = std::string("register-brick CG: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  // the plan depends on the grid, the device and the block cap alone: kept
  // by the handle (a search takes tens of microseconds)
  ChipPlan local, &pl = a.chip ? *a.chip : local;
  if (pl.nsm != nsm || pl.max_blocks != fc.max_blocks) {
    pl = ChipPlan{};
    pl.nsm = nsm;
    pl.max_blocks = fc.max_blocks;
    // leave room for the reductions' static shared memory (about 2 KB)
    pl.fits = make_chip_plan(a.g, nsm, (size_t)std::max(0, smem_optin - 4096), fc.max_blocks, pl);
  }
  if (!pl.fits) return LES_OK;
  const void* kern = pl.brick ? brick_kernel(pl.zp) : chip_kernel<T>(pl.zp, pl.xs);
  const unsigned G = (unsigned)(pl.px * pl.py * pl.pz);
  int per_sm = 0;
  if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pl.smem)) != cudaSuccess ||
      (e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, pl.threads, pl.smem)) != cudaSuccess) {
    if (err) *err = std::string("register-brick CG occupancy: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  if (per_sm < 1 || (long long)G > (long long)per_sm * nsm) return LES_OK;  // not co-resident
  ChipArgs<T> f;
  f.nx = a.g.nx;
  f.ny = a.g.ny;
  f.nz = a.g.nz;
  f.walls = a.g.walls;
  // the largest eigenvalue is 2 c0, c0 = 2 (1/dx^2 + 1/dy^2 + 1/dz^2)
  const double c0 = 2.0 * ((double)a.g.idx * a.g.idx + (double)a.g.idy * a.g.idy + (double)a.g.idz * a.g.idz);
  f.sc = sizeof(T) == 4 ? (T)std::ldexp(1.0, std::ilogb(c0) + 2) : T(1);
  f.isc = T(1) / f.sc;
  f.cx = a.g.idx * a.g.idx * f.isc;
  f.cy = a.g.idy * a.g.idy * f.isc;
  f.cz = a.g.idz * a.g.idz * f.isc;
  f.px = pl.px;
  f.py = pl.py;
  f.pz = pl.pz;
  f.zs = pl.zs;
  f.smem_p = pl.np;
  f.smem_g = pl.ng;
  f.n = (long long)f.nx * f.ny * f.nz;
  f.b = b;
  f.x = x;
  f.rg = a.r;
  f.qg0 = a.p0;
  f.qg1 = a.p1;
  f.qt[0][0] = reinterpret_cast<char*>(a.p0);
  f.qt[1][0] = reinterpret_cast<char*>(a.p1);
  f.qt[0][1] = reinterpret_cast<char*>(a.q);
  f.qt[1][1] = reinterpret_cast<char*>(a.r);
  f.partials = a.partials;
  // past the set-up sums' two slots: the counters, then the iterations' partials
  f.counters = reinterpret_cast<unsigned*>(a.partials + 2 * (size_t)kSumSlot * G);
  f.spread = a.partials + 2 * (size_t)kSumSlot * G + kChipSpread * kChipLine / 2;
  f.missing = (unsigned)std::max(0, fc.missing);
  f.bar = a.bar;
  f.ctl = a.ctl;
  f.tol = tol;
  f.maxit = maxit;
  f.spin_cycles = fc.spin_cycles;
  // the test hook's missing arrivals apply to the iterations' sums (whose
  // wait is this kernel's own); the set-up sums wait for the launched blocks
  f.expected = G;
  f.guard = a.guard;
  *used = true;
  if ((e = cudaMemsetAsync(a.bar, 0, sizeof(FusedBar), a.st)) != cudaSuccess ||
      (e = cudaMemsetAsync(f.counters, 0, kChipSpread * kChipLine * sizeof(unsigned), a.st)) != cudaSuccess) {
    if (err) *err = std::string("register-brick CG barrier reset: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  void* args[] = {&f};
  {
    ProfScope ps(a.prof, KI_CG_RESIDENT, a.st);
    e = cudaLaunchCooperativeKernel(kern, dim3(G), dim3(pl.threads), args, pl.smem, a.st);
  }
  if (e != cudaSuccess) {
    if (err) *err = std::string("register-brick CG launch: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  if ((e = cudaMemcpyAsync(a.ctl_host, a.ctl, sizeof(SolverCtl), cudaMemcpyDeviceToHost, a.st)) != cudaSuccess ||
      (e = cudaStreamSynchronize(a.st)) != cudaSuccess) {
    if (err) *err = std::string("register-brick CG: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  const SolverCtl& c = *a.ctl_host;
  if (iters) *iters = c.iter;
  if (rel) *rel = c.rel;
  // algorithmic traffic of the solve, as for every CG kernel (its vectors
  // stay on chip)
  if (a.prof) a.prof->bytes[KI_CG_RESIDENT] += (kCgSetupFields + kCgIterFields * c.iter) * (double)f.n * sizeof(T);
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
      if (err) *err = "poisson: register-brick CG returned no status";
      return LES_ERR_CUDA;
  }
}

template int poisson_solve_chip<float>(const SolverArgs<float>&, const FusedCfg&, const float*, float*, double, int,
                                       int*, double*, std::string*, bool*);
template int poisson_solve_chip<double>(const SolverArgs<double>&, const FusedCfg&, const double*, double*, double,
                                        int, int*, double*, std::string*, bool*);

}  // namespace les
