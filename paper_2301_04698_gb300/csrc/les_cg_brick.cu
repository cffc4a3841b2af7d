// les_cg_brick.cu -- the on-chip conjugate-gradient Poisson solve (Sec. 2.4, as in
// les_cg_chip.cu) for FP32 grids too large to keep every vector on chip: 12 288
// to 32 768 nodes per SM, up to 4.9 million in all on 152 SMs.
//
// A brick of at most 32 x 16 columns keeps p with its ghost layer in shared memory
// and r in registers: a lane and a warp own a column, its planes at compile-time
// offsets.  q = L_c p is not kept: it is formed for the dot products and again, from
// the unchanged p, for r -= alpha q; only then is p overwritten.  x is the one vector
// that streams, 8 bytes per node and iteration.  The faces' q are exchanged and the
// ghosts' r kept as in les_cg_chip.cu.
//
// What bounds it: instruction issue (about 75 per node and iteration) and shared
// memory, 12 accesses per node and iteration (five neighbours twice, p read and
// written).  Measured (GB300, us per iteration; before: the streaming kernels,
// which take 27 to 36 bytes per node through L2): 192 x 192 x 128 38.2 -> 19.3,
// 160 x 160 x 128 30.6 -> 12.8, 256 x 256 x 64 39.0 -> 18.6, 150 x 130 x 110 23.3 ->
// 12.6 (18.3, 12.7, 17.5 and 12.1 with warps summed and scalars formed in plain FP32).  Bricks of any extents, with their strides and column offsets in registers,
// spilled r and took 53 us on the first of these.
#include <algorithm>
#include <string>
#include <type_traits>

#include "les_chip.cuh"

namespace les {
namespace {

constexpr int BX = kBrickX, BY = kBrickY;       // columns of a brick at most: a lane and a warp each
constexpr int SY = BX + 2, SZ = SY * (BY + 2);  // strides of p with its ghost layer, whatever the brick's extents

// a predicated store, not a branch: the planes' arithmetic can overlap
__device__ __forceinline__ void store_if(bool p, float* at, float v) {
  asm volatile("{\n .reg .pred p;\n setp.ne.s32 p, %2, 0;\n @p st.global.cg.f32 [%0], %1;\n}" ::"l"(at), "f"(v),
               "r"((int)p)
               : "memory");
}

// ZP: a multiple of 8, at most 8 planes more than any brick of the grid has
template <int ZP>
__global__ void __launch_bounds__(BX* BY, 1) k_cg_brick(ChipArgs<float> f) {
  extern __shared__ __align__(16) unsigned char smraw[];
  float* P = reinterpret_cast<float*>(smraw);  // p with its ghost layer
  float* GR = P + f.smem_p;                    // r at the ghost nodes
  float* GQ = GR + f.smem_g;                   // the neighbours' q there
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int i0, j0, k0, bx, by, bz;
  chip_part(f.nx, f.px, blockIdx.x % f.px, i0, bx);
  chip_part(f.ny, f.py, (blockIdx.x / f.px) % f.py, j0, by);
  chip_part(f.nz, f.pz, blockIdx.x / (f.px * f.py), k0, bz);
  const int gpl = f.nx * f.ny;
  const bool low = f.walls && k0 == 0, high = f.walls && k0 + bz == f.nz;  // the brick touches a wall
  const bool zself = !f.walls && f.pz == 1;                                // ... or is its own z neighbour
  const float cx = f.cx, cy = f.cy, cz = f.cz;

  // this thread's column (without one it reads its place in P and writes nothing)
  const bool own = lane < bx && warp < by;
  float* const C = P + SZ + (warp + 1) * SY + lane + 1;  // p at its plane 0
  const int g0 = k0 * gpl + (j0 + warp) * f.nx + i0 + lane;
  // nodes that a neighbouring brick reads (px, py > 1)
  const bool fcol = own && (lane == 0 || lane == bx - 1 || warp == 0 || warp == by - 1);
  const bool flow = own && f.pz > 1 && !low, fhigh = own && f.pz > 1 && !high;
  auto is_face = [&](int j) { return fcol || (flow && j == 0) || (fhigh && j == bz - 1); };

  // body(id, place in P, offset in global memory) for the brick's ghost nodes, by the
  // warps from W0 on: the z faces a warp per row, the y faces a warp per row, the x faces
  // a half warp per plane
  auto each_ghost = [&](auto first, auto&& body) {
    constexpr int W0 = decltype(first)::value, NW = BY - W0;
    if (warp < W0) return;
    if (f.pz > 1)
#pragma unroll
      for (int y = warp - W0; y < BY; y += NW) {
        float* at = P + (y + 1) * SY + lane + 1;
        const int g = (j0 + y) * f.nx + i0 + lane;
        if (lane < bx && y < by) {
          if (!low) body(y * BX + lane, at, chip_wrap(k0 - 1, f.nz) * gpl + g);
          if (!high) body((BY + y) * BX + lane, at + SZ * (bz + 1), chip_wrap(k0 + bz, f.nz) * gpl + g);
        }
      }
    int id0 = 2 * BX * BY;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int g = k0 * gpl + chip_wrap(side ? j0 + by : j0 - 1, f.ny) * f.nx + i0 + lane;
      float* at = P + SZ + (side ? (by + 1) * SY : 0) + lane + 1;
      if (lane < bx)
        for (int z = warp - W0; z < bz; z += NW) body(id0 + z * BX + lane, at + z * SZ, g + z * gpl);
      id0 += ZP * BX;
    }
    const int y = lane & 15;
#pragma unroll
    for (int side = 0; side < 2; ++side) {
      const int g = k0 * gpl + (j0 + y) * f.nx + chip_wrap(side ? i0 + bx : i0 - 1, f.nx);
      float* at = P + SZ + (y + 1) * SY + (side ? bx + 1 : 0);
      if (y < by)
        for (int z = 2 * (warp - W0) + (lane >> 4); z < bz; z += 2 * NW)
          body(id0 + z * BY + y, at + z * SZ, g + z * gpl);
      id0 += ZP * BY;
    }
  };
  using AllWarps = std::integral_constant<int, 0>;
  using GhostWarps = std::integral_constant<int, kFoldWarps<F2>>;
  static_assert(BX == 32 && BY == 16, "the ghost loops' mapping");

  float r[ZP] = {};
  // body(j, offset in global memory) for the planes of the brick; only the last
  // eight can be missing
  auto planes = [&](auto&& body) {
    int g = g0;
    asm volatile("" : "+r"(g));  // formed anew in each loop: no registers kept for the planes' offsets
#pragma unroll
    for (int j = 0; j < ZP; ++j) {
      if (j < ZP - 8 || j < bz) body(j, g);
      g += gpl;
      if (j % 2) asm volatile("" ::: "memory");  // loads at most two planes ahead: registers
    }
  };
  // body(j, g, p at plane j, L_c p at plane j) up the column; second differences
  // formed before scaling, as in the other CG kernels
  auto march = [&](auto&& body) {
    float here = C[0];
    float below = low ? here : (zself ? C[SZ * (bz - 1)] : C[-SZ]);
    planes([&](int j, int g) {
      const float* pj = C + SZ * j;
      float above = pj[SZ];
      if (j >= ZP - 9 && j == bz - 1) above = high ? here : (zself ? C[0] : above);
      const float c2 = 2.f * here;
      const float q = (pj[-1] + pj[1] - c2) * cx + (pj[-SY] + pj[SY] - c2) * cy + (below + above - c2) * cz;
      body(j, g, here, q);
      below = here;
      here = above;
    });
  };
  // A at the ghost nodes into P (keep: as r there too), outside the iterations
  auto fill_ghosts = [&](const float* A, bool keep) {
    each_ghost(AllWarps{}, [&](int id, float* at, int g) {
      const float v = __ldcg(A + g);
      *at = v;
      if (keep) GR[id] = v;
    });
  };
  // the sum of a thread's column, of those that are the brick's
  auto total = [&](const ChipRun<float, ZP>& s) { return own ? s.total() : F2{0.f, 0.f}; };

  GridSync gs{f.bar, f.partials, f.spin_cycles, f.expected, 0u};
  __shared__ struct {
    float mean, ta, tb;
    float scale, xs;  // of r, p and q; alpha of x over that of r
    int status, restart;
    double bb, rel;  // |b - mean|^2 and the relative residual of x0
  } sc;
  __shared__ F2 shv[4][kChipWarps];
  __shared__ F2 part[32];
  F2 tot[4];  // in warp 0
  __shared__ int s_fail;
  double rr = 0.0, bb = 0.0, rel = 0.0;  // meaningful in thread 0
  int status = 0;  // 0 running, 1 converged, 2 maxit, 3 breakdown, 4 zero rhs, 5 timeout
  F2 rr_own{0.f, 0.f};  // this thread's share of r.r for the next sum

  chip_sum_clear<F2>(f.spread);  // no tag of an earlier solve: cleared here, for everyone after the first sum
  if (tid == 0) s_fail = 0;

  // mean of b (b held in r, x0 in P); |b|_1 and |x0|_1
  {
    ChipRun<float, ZP> s, sb, sx;
    planes([&](int j, int g) {
      float xv = 0.f;
      if (own) {
        r[j] = __ldcg(f.b + g);
        xv = __ldcg(f.x + g);
        C[SZ * j] = xv;
      }
      s.add(j, r[j]);
      sb.add(j, fabsf(r[j]));
      sx.add(j, fabsf(xv));
    });
    F2 v[3] = {total(s), total(sb), total(sx)};
    double t[3];
    const bool ok = grid_sum_t0<3>(v, gs, t);
    if (tid == 0) {
      sc.status = ok ? 0 : 5;
      sc.mean = (float)(t[0] / (double)f.n);
      sc.scale = chip_scale(t[1], t[2], 2.f * (cx + cy + cz) * f.sc, (double)f.n);
      sc.xs = f.isc / sc.scale;
    }
    __syncthreads();
    status = sc.status;
  }
  const float mean = sc.mean;
  // x0 with its ghosts in P; r = (b - mean) - L_c x0, scaled, published
  if (!status) {
    fill_ghosts(f.x, false);
    __syncthreads();
    ChipRun<float, ZP> s0, s1;
    march([&](int j, int g, float, float q) {
      float bm = r[j] - mean;
      r[j] = (bm - f.sc * q) * sc.scale;
      bm *= sc.scale;
      if (is_face(j)) __stcg(f.rg + g, r[j]);
      s0.add(j, r[j] * r[j]);
      s1.add(j, bm * bm);
    });
    rr_own = total(s0);
    F2 v[2] = {rr_own, total(s1)};
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
      ChipRun<float, ZP> s;
      planes([&](int j, int g) {
        if (!own) return;
        __stcg(f.x + g, 0.f);
        r[j] = (__ldcg(f.b + g) - mean) * sc.scale;
        s.add(j, r[j] * r[j]);
        if (is_face(j)) __stcg(f.rg + g, r[j]);
      });
      rr_own = total(s);
      Dot<float> none[1];
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
  F2 rr_stop, rr_last;  // rr_last meaningful in thread 0
  acc_from(f.tol * f.tol * sc.bb, rr_stop);
  acc_from(rr, rr_last);
  int iter = 0;
  if (!status) {
    // p_0 = r_0, with r_0 at the ghost nodes from the published faces
    planes([&](int j, int) {
      if (own) C[SZ * j] = r[j];
    });
    fill_ghosts(f.rg, true);
    __syncthreads();
    for (;;) {
      float* qw = (iter & 1) ? f.qg1 : f.qg0;  // this iteration's q faces
      ChipRun<float, ZP> d0, d2, d3;           // p.q, r.q, q.q
      march([&](int j, int g, float pv, float q) {
        // three planes of four by a predicated store, whose arithmetic can overlap;
        // a branch at the fourth keeps the compiler from spreading all of them
        // (64 planes in one stretch spill)
        if (j % 4 < 3) store_if(is_face(j), qw + g, q);
        else if (is_face(j)) __stcg(qw + g, q);
        d0.add(j, pv * q);
        d2.add(j, r[j] * q);
        d3.add(j, q * q);
      });
      chip_sum<GhostWarps::value, 3>(
          f, iter, total(d0), rr_own, total(d2), total(d3), shv, part, tot, s_fail, ChipNothing{},
          [&] {
            each_ghost(GhostWarps{}, [&](int id, float*, int g) { cp_async(GQ + id, qw + g); });
            cp_commit();
          },
          ChipNothing{});
      if (tid == 0) {  // the status, alpha and beta
        int st = 0;
        if (s_fail) {
          st = 5;
        } else {
          rr_last = tot[1];
          float al = 0.f, be = 0.f;
          if (acc_le(tot[1], rr_stop)) st = 1;
          else if (iter >= f.maxit) st = 2;
          else if (!chip_scalars(tot, al, be)) st = 3;
          sc.ta = al;
          sc.tb = be;
        }
        sc.status = st;
      }
      __syncthreads();
      status = sc.status;
      if (status) {
        cp_wait<0>();
        break;
      }
      const float ta = sc.ta, tb = sc.tb;
      // r -= alpha q, with q from p as it was
      ChipRun<float, ZP> s;
      march([&](int j, int, float, float q) {
        r[j] -= ta * q;
        s.add(j, r[j] * r[j]);
      });
      rr_own = total(s);
      cp_wait<0>();
      __syncthreads();  // every reader of p is done, and the copies of the ghosts' q have landed
      each_ghost(AllWarps{}, [&](int id, float* at, int) {
        const float rv = GR[id] - ta * GQ[id];
        GR[id] = rv;
        *at = rv + tb * *at;
      });
      // x += alpha p, p = r + beta p; the loads of eight planes of x together
      if (own) {
        int g = g0;
        asm volatile("" : "+r"(g));
        const float tx = ta * sc.xs;  // alpha of x
#pragma unroll
        for (int b = 0; b < ZP; b += 8) {
          float xv[8];
#pragma unroll
          for (int c = 0; c < 8; ++c)
            if (b < ZP - 8 || b + c < bz) xv[c] = __ldcg(f.x + g + c * gpl);
#pragma unroll
          for (int c = 0; c < 8; ++c)
            if (b < ZP - 8 || b + c < bz) {
              const float pv = C[SZ * (b + c)];
              __stcg(f.x + g + c * gpl, xv[c] + tx * pv);
              C[SZ * (b + c)] = r[b + c] + tb * pv;
            }
          g += 8 * gpl;
        }
      }
      iter += 1;
      __syncthreads();
    }
  }
  if (tid == 0) rel = (iter > 0 && sc.bb > 0.0) ? sqrt(acc_value(rr_last) / sc.bb) : sc.rel;

  // zero-mean gauge (or zero for a zero right side); x held in r
  if (status != 5) {
    ChipRun<float, ZP> s;
    planes([&](int j, int g) {
      if (own) r[j] = __ldcg(f.x + g);
      s.add(j, r[j]);
    });
    F2 v[1] = {total(s)};
    double t[1];
    const bool ok = grid_sum_t0<1>(v, gs, t);
    if (tid == 0) {
      if (!ok) status = 5;
      else if (status < 3 && !isfinite(t[0])) status = 3;  // x has left the range
      sc.mean = (float)(t[0] / (double)f.n);
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
    if (status != 5) {
      const float mx = sc.mean;
      planes([&](int j, int g) {
        if (own) __stcg(f.x + g, status == 4 ? 0.f : r[j] - mx);
      });
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    f.ctl->iter = iter;
    f.ctl->rel = rel;
    f.ctl->done = status;
  }
}

}  // namespace

size_t brick_smem(int zp, int* np, int* ng) {
  *np = SZ * (zp + 2);
  *ng = 2 * BX * BY + 2 * zp * (BX + BY);
  return ((size_t)*np + 2 * (size_t)*ng) * sizeof(float);
}
const void* brick_kernel(int zp) {
  switch (zp) {
    case 24: return (const void*)k_cg_brick<24>;
    case 32: return (const void*)k_cg_brick<32>;
    case 40: return (const void*)k_cg_brick<40>;
    case 48: return (const void*)k_cg_brick<48>;
    case 56: return (const void*)k_cg_brick<56>;
    case 64: return (const void*)k_cg_brick<64>;
    default: return nullptr;
  }
}

}  // namespace les
