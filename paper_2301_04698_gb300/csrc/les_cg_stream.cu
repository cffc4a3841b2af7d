// les_cg_stream.cu -- two-phase streaming conjugate-gradient Poisson solve in
// one persistent cooperative launch, for grids of any extents that do not fit
// on chip (Sec. 2.4: L_c psi = b, compact 7-point Laplacian, periodic in x and
// y, mirror or periodic in z; mean of b removed, psi returned with zero mean).
//
// Per iteration, each phase followed by a grid-wide sum:
//   A  x += alpha_{i-1} p_{i-1},  p_i = r_i + beta p_{i-1},  q = L_c p_i,  p.q
//   B  r -= alpha_i q,  r.r
// A block marches a tile of WX x WY columns through a run of planes.  A thread
// holds its nodes' p of the plane below and of the current plane in registers;
// the plane passes through shared memory (double-buffered, one barrier per
// plane) for the x and y neighbours, with a ring of one node around the tile
// whose p is formed again.  The loads of the next plane are in flight during
// the arithmetic of this one.  The tiles of a grid differ by at most one node
// in either extent, so no extent has to be a multiple of anything.
//
// What bounds it: FP64 arithmetic.  An SM issues an FP64 warp instruction every
// 16 cycles (1.25 TFLOP/s), so an iteration costs at least 11 operations per
// node / 2 per SM and clock = 18 ps per node, above the 11 ps of its 9 streamed
// fields (72 bytes).  Hence: the operator is scaled by its centre coefficient,
// q' = p - ax (w + e) - ay (s + n) - az (d + u), six operations instead of
// nine (p.L_c p, r -= alpha q and beta do not see the factor, the update of x
// takes it up); x is updated in phase A, where p_{i-1}
// is at hand, which takes a field off phase B; the one-pass kernels' second
// stencil and two more sums, which save bytes, would cost nine operations.
// FP32 keeps the second differences formed before scaling.
// Measured (GB300, FP64, us per iteration): 256 x 256 x 128 187, 512 x 512 x 128 680;
// with runs dealt in turns, before the planes were shared out equally, 192 and 719.
#include <algorithm>
#include <string>

#include "les_internal.h"
#include "les_stream.cuh"

namespace les {
namespace {

template <typename T>
struct StreamArgs {
  int nx, ny, nz, walls;
  T cx, cy, cz;                   // 1/dx^2, 1/dy^2, 1/dz^2
  int ntx, nty, nchunk;           // tiles along x and y, runs of planes per tile (0: equal shares)
  int nunits;
  long long n;
  const T* b;
  T* x;
  T* r;
  T* p[2];                        // p_i in p[i & 1]
  T* q;
  double* partials;
  FusedBar* bar;
  SolverCtl* ctl;
  double tol;
  int maxit;
  long long spin_cycles;
  unsigned expected;
  int guard;
};

template <typename T, typename S, bool Shares>
__global__ void __launch_bounds__(kStreamThreads, 2) k_cg_stream(StreamArgs<T> f) {
  constexpr int NO = S::NO, NWX = S::NWX, SP = S::SP, SN = S::SN;
  __shared__ T sm[2][SN];
  __shared__ struct {
    T ta, tb, mean;
    int status, restart;
    int e;  // the size of the sums (binary exponent): that of |b - mean|^2
  } sc;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int plane = f.nx * f.ny;
  const T cx = f.cx, cy = f.cy, cz = f.cz;
  // FP64: L_c p = -c0 q' with q' = p - ax (w + e) - ay (s + n) - az (d + u);
  // alpha of r -= alpha' q' is -c0 times that of x += alpha p
  const T c0 = T(2) * (cx + cy + cz);
  const T ax = cx / c0, ay = cy / c0, az = cz / c0;
  constexpr bool kScaled = sizeof(T) == 8;
  GridSync gs{f.bar, f.partials, f.spin_cycles, f.expected, 0u};
  const long long gstride = (long long)gridDim.x * kStreamThreads;
  const long long gtid = (long long)blockIdx.x * kStreamThreads + tid;

  // set-up sweeps: the 7-point operator straight from global memory
  auto lap_global = [&](const T* v, long long m) -> T {
    const int k = (int)(m / plane), o = (int)(m - (long long)k * plane), j = o / f.nx, i = o - j * f.nx;
    const T* pl = v + (size_t)k * plane;
    const T c2 = T(2) * __ldcg(pl + o);
    const T xm = __ldcg(pl + (i == 0 ? o + f.nx - 1 : o - 1)), xp = __ldcg(pl + (i == f.nx - 1 ? o + 1 - f.nx : o + 1));
    const T ym = __ldcg(pl + (j == 0 ? o + plane - f.nx : o - f.nx));
    const T yp = __ldcg(pl + (j == f.ny - 1 ? o + f.nx - plane : o + f.nx));
    const T zm = __ldcg(v + (size_t)stream_z(k - 1, f.nz, f.walls) * plane + o);
    const T zp = __ldcg(v + (size_t)stream_z(k + 1, f.nz, f.walls) * plane + o);
    return (xm + xp - c2) * cx + (ym + yp - c2) * cy + (zm + zp - c2) * cz;
  };

  double rr = 0.0, bb = 0.0, rel = 0.0;  // meaningful in thread 0
  int status = 0;  // 0 running, 1 converged, 2 maxit, 3 breakdown, 4 zero rhs, 5 timeout
  {
    StreamSum<T> s[1];
    for (long long m = gtid; m < f.n; m += gstride) {
      s[0].add(__ldcg(f.b + m));
      s[0].tick();
    }
    double t[1];
    const bool ok = stream_sum<1>(s, gs, t);
    if (tid == 0) {
      sc.status = ok ? 0 : 5;
      sc.mean = (T)(t[0] / (double)f.n);
    }
    __syncthreads();
    status = sc.status;
  }
  const T mean = sc.mean;
  if (!status) {
    StreamSum<T> s[2];
    for (long long m = gtid; m < f.n; m += gstride) {
      const T bm = __ldcg(f.b + m) - mean;
      const T rv = bm - lap_global(f.x, m);
      __stcg(f.r + m, rv);
      s[0].add(rv * rv);
      s[1].add(bm * bm);
      s[0].tick();
      s[1].tick();
    }
    double t[2];
    const bool ok = stream_sum<2>(s, gs, t);
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
        __stcg(f.r + m, __ldcg(f.b + m) - mean);
      }
      StreamSum<T> none[1];
      double t1[1];
      const bool ok2 = stream_sum<1>(none, gs, t1);  // a grid barrier: r_0 complete everywhere
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
    sc.ta = sc.tb = T(0);
    sc.e = (__double2hiint(bb) >> 20 & 0x7ff) - 1023;
  }
  __syncthreads();
  status = sc.status;

  int iter = 0;  // updates of r so far; x lacks the last one's alpha p until the next phase A
  T ta = T(0);   // alpha of the last update, as x takes it
  bool pend = false;
  while (!status) {
    const bool first = iter == 0;
    const T tb = sc.tb;
    const T* po = f.p[(iter + 1) & 1];
    T* pw = f.p[iter & 1];
    StreamSum<T> s;
    StreamTurns<Shares> turns(f.nunits);
    int tile, k0, kn;
    while (turns.next(f.nchunk, f.nz, tile, k0, kn)) {
      int x0, y0, w, h;
      stream_part(f.nx, f.ntx, tile % f.ntx, x0, w);
      stream_part(f.ny, f.nty, tile / f.ntx, y0, h);
      // this thread's nodes (offset in a plane; -1: none) and its ring node
      int go[NO];
#pragma unroll
      for (int m = 0; m < NO; ++m) {
        const int ex = lane + 32 * (m % NWX), ey = warp + 8 * (m / NWX);
        go[m] = ex < w && ey < h ? (y0 + ey) * f.nx + x0 + ex : -1;
      }
      const int eo = (warp + 1) * SP + lane + 1;  // of node 0 in sm; node m: + 8 (m / NWX) SP + 32 (m mod NWX)
      int gr, er;
      stream_ring<S>(tid, x0, y0, w, h, f.nx, f.ny, gr, er);
      T rv[NO], ov[NO], xv[NO], rh = T(0), oh = T(0);  // r, p_{i-1}, x of the plane in flight; its ring
      auto load = [&](int kk, bool inside) {
        const size_t base = (size_t)stream_z(kk, f.nz, f.walls) * plane;
#pragma unroll
        for (int m = 0; m < NO; ++m) {
          rv[m] = ov[m] = xv[m] = T(0);
          if (go[m] >= 0) {
            rv[m] = __ldcg(f.r + base + go[m]);
            if (!first) {
              ov[m] = __ldcg(po + base + go[m]);
              if (inside) xv[m] = __ldcg(f.x + base + go[m]);
            }
          }
        }
        if (inside && gr >= 0) {
          rh = __ldcg(f.r + base + gr);
          if (!first) oh = __ldcg(po + base + gr);
        }
      };
      T pd[NO], pc[NO], part[NO];  // p of the plane below and of this one; q without the node above
      load(k0 - 1, false);
#pragma unroll
      for (int m = 0; m < NO; ++m) pc[m] = first ? rv[m] : rv[m] + tb * ov[m], part[m] = T(0);
      load(k0, true);
      __syncthreads();  // the previous unit's readers are done with sm
      for (int k = k0; k <= k0 + kn; ++k) {
        const bool inside = k < k0 + kn;
        T pv[NO];
        T* pl = sm[k & 1];
        const size_t base = (size_t)k * plane;
#pragma unroll
        for (int m = 0; m < NO; ++m) {
          pv[m] = first ? rv[m] : rv[m] + tb * ov[m];
          if (inside && go[m] >= 0) {
            pl[eo + 8 * (m / NWX) * SP + 32 * (m % NWX)] = pv[m];
            if (!first) __stcg(f.x + base + go[m], xv[m] + ta * ov[m]);
          }
        }
        if (inside && gr >= 0) pl[er] = first ? rh : rh + tb * oh;
        if (inside) load(k + 1, k + 1 < k0 + kn);
        // the plane below is complete with this plane's p
        if (k > k0) {
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            T qv;
            if constexpr (kScaled) qv = fma(-az, pv[m], part[m]);
            else qv = part[m] + (pd[m] + pv[m] - T(2) * pc[m]) * cz;
            if (go[m] >= 0) {
              __stcg(f.q + base - plane + go[m], qv);
              __stcg(pw + base - plane + go[m], pc[m]);
              s.add(pc[m] * qv);
            }
          }
          s.tick();
        }
        if (!inside) break;
        __syncthreads();  // plane k is in sm (the other buffer's readers passed the barrier before)
#pragma unroll
        for (int m = 0; m < NO; ++m) {
          const T* e = pl + eo + 8 * (m / NWX) * SP + 32 * (m % NWX);
          if constexpr (kScaled) {
            const T t = fma(-ax, e[-1] + e[1], pv[m]);
            part[m] = fma(-az, pc[m], fma(-ay, e[-SP] + e[SP], t));
          } else {
            const T c2 = T(2) * pv[m];
            part[m] = (e[-1] + e[1] - c2) * cx + (e[-SP] + e[SP] - c2) * cy;
          }
          pd[m] = pc[m];
          pc[m] = pv[m];
        }
      }
    }
    double pq, rr_new;
    bool ok = stream_sum_scaled(s, sc.e, gs, pq);
    if (tid == 0) {
      if (!ok) status = 5;
      else if (pq == 0.0 || !isfinite(pq)) status = 3;
      else sc.ta = (T)(rr / pq);
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
    pend = false;  // phase A has added the last alpha p
    if (status) break;
    const T tq = sc.ta;
    ta = kScaled ? -tq / c0 : tq;
    pend = true;
    // B: r -= alpha q, r.r
    StreamSum<T> sb;
    {
      constexpr int V = StreamVec<T>::N, U = 4;
      const long long nv = f.n / V;
      for (long long v0 = gtid; v0 < nv; v0 += U * gstride) {
        StreamVec<T> ra[U], qa[U];
#pragma unroll
        for (int j = 0; j < U; ++j)
          if (v0 + j * gstride < nv) {
            ra[j] = svld(f.r + (v0 + j * gstride) * V);
            qa[j] = svld(f.q + (v0 + j * gstride) * V);
          }
#pragma unroll
        for (int j = 0; j < U; ++j)
          if (v0 + j * gstride < nv) {
#pragma unroll
            for (int e = 0; e < V; ++e) {
              ra[j].v[e] -= tq * qa[j].v[e];
              sb.add(ra[j].v[e] * ra[j].v[e]);
            }
            sb.tick();
            svst(f.r + (v0 + j * gstride) * V, ra[j]);
          }
      }
      for (long long m = nv * V + gtid; m < f.n; m += gstride) {
        const T v = __ldcg(f.r + m) - tq * __ldcg(f.q + m);
        sb.add(v * v);
        sb.tick();
        __stcg(f.r + m, v);
      }
    }
    ok = stream_sum_scaled(sb, sc.e, gs, rr_new);
    iter += 1;
    if (tid == 0) {
      if (!ok) {
        status = 5;
      } else {
        rel = sqrt(rr_new / bb);
        sc.tb = (T)(rr_new / rr);
        rr = rr_new;
        if (rel <= f.tol) status = 1;
        else if (iter >= f.maxit) status = 2;
        else if (!isfinite(rr_new)) status = 3;
      }
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
  }

  // x with the last alpha p, then the zero-mean gauge (or zero for a zero right side)
  if (status != 5) {
    const T* po = f.p[(iter + 1) & 1];
    StreamSum<T> s[1];
    for (long long m = gtid; m < f.n; m += gstride) {
      T v = __ldcg(f.x + m);
      if (pend) {
        v += ta * __ldcg(po + m);
        __stcg(f.x + m, v);
      }
      s[0].add(v);
      s[0].tick();
    }
    double t[1];
    const bool ok = stream_sum<1>(s, gs, t);
    if (tid == 0) {
      if (!ok) status = 5;
      sc.mean = (T)(t[0] / (double)f.n);
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
    if (status != 5) {
      const T mx = sc.mean;
      for (long long m = gtid; m < f.n; m += gstride)
        __stcg(f.x + m, status == 4 ? T(0) : __ldcg(f.x + m) - mx);
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    f.ctl->iter = iter;
    f.ctl->rel = rel;
    f.ctl->done = status;
  }
}

template <typename T, bool Shares>
const void* stream_kernel(int shape) {
  if (shape == 0) return (const void*)k_cg_stream<T, Tile64, Shares>;
  if (shape == 1) return (const void*)k_cg_stream<T, Tile32, Shares>;
  return (const void*)k_cg_stream<T, Tile32s, Shares>;
}
template <typename T>
const void* stream_kernel(const StreamPlan& pl) {
  if constexpr (sizeof(T) == 8)  // the plans of FP32 have none
    if (pl.nchunk == 0) return stream_kernel<T, true>(pl.shape);
  return stream_kernel<T, false>(pl.shape);
}

}  // namespace

template <typename T>
int poisson_solve_stream(const SolverArgs<T>& a, const FusedCfg& fc, const T* b, T* x, double tol, int maxit,
                         int* iters, double* rel, std::string* err) {
  int dev = 0, nsm = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) {
    if (err) *err = std::string("streaming CG: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  int per_sm = 2;
  StreamPlan pl;
  const void* kern = nullptr;
  for (int pass = 0; pass < 2; ++pass) {  // the plan depends on the resident blocks, they on the shape
    pl = make_stream_plan(a.g.nx, a.g.ny, a.g.nz, std::min<long long>((long long)per_sm * nsm, fc.max_blocks),
                          sizeof(T) == 8);
    kern = stream_kernel<T>(pl);
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kStreamThreads, 0)) != cudaSuccess) {
      if (err) *err = std::string("streaming CG occupancy: ") + cudaGetErrorString(e);
      return LES_ERR_CUDA;
    }
    per_sm = std::min(per_sm, 8);  // the partials hold 2 x kSumSlot words of 8 blocks per SM
    if (per_sm < 1) {
      if (err) *err = "streaming CG: no block fits on an SM";
      return LES_ERR_CUDA;
    }
  }
  const long long G = std::max<long long>(1, std::min<long long>((long long)per_sm * nsm, fc.max_blocks));
  StreamArgs<T> f;
  f.nx = a.g.nx;
  f.ny = a.g.ny;
  f.nz = a.g.nz;
  f.walls = a.g.walls;
  f.cx = a.g.idx * a.g.idx;
  f.cy = a.g.idy * a.g.idy;
  f.cz = a.g.idz * a.g.idz;
  f.ntx = pl.ntx;
  f.nty = pl.nty;
  f.nchunk = pl.nchunk;
  f.nunits = (int)pl.units;
  f.n = (long long)f.nx * f.ny * f.nz;
  f.b = b;
  f.x = x;
  f.r = a.r;
  f.p[0] = a.p0;
  f.p[1] = a.p1;
  f.q = a.q;
  f.partials = a.partials;
  f.bar = a.bar;
  f.ctl = a.ctl;
  f.tol = tol;
  f.maxit = maxit;
  f.spin_cycles = fc.spin_cycles;
  f.expected = (unsigned)G + (unsigned)std::max(0, fc.missing);
  f.guard = a.guard;
  if ((e = cudaMemsetAsync(a.bar, 0, sizeof(FusedBar), a.st)) != cudaSuccess) {
    if (err) *err = std::string("streaming CG barrier reset: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  void* args[] = {&f};
  {
    ProfScope ps(a.prof, KI_CG_FUSED, a.st);
    e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)G), dim3(kStreamThreads), args, 0, a.st);
  }
  if (e != cudaSuccess) {
    if (err) *err = std::string("streaming CG launch: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  if ((e = cudaMemcpyAsync(a.ctl_host, a.ctl, sizeof(SolverCtl), cudaMemcpyDeviceToHost, a.st)) != cudaSuccess ||
      (e = cudaStreamSynchronize(a.st)) != cudaSuccess) {
    if (err) *err = std::string("streaming CG: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  const SolverCtl& c = *a.ctl_host;
  if (iters) *iters = c.iter;
  if (rel) *rel = c.rel;
  // algorithmic traffic of the solve (this kernel streams 9 fields per iteration: A r,
  // p, x in, p, q, x out; B r, q in, r out)
  if (a.prof) a.prof->bytes[KI_CG_FUSED] += (kCgSetupFields + kCgIterFields * c.iter) * (double)f.n * sizeof(T);
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
      if (err) *err = "poisson: streaming solver returned no status";
      return LES_ERR_CUDA;
  }
}

template int poisson_solve_stream<float>(const SolverArgs<float>&, const FusedCfg&, const float*, float*, double, int,
                                         int*, double*, std::string*);
template int poisson_solve_stream<double>(const SolverArgs<double>&, const FusedCfg&, const double*, double*, double,
                                          int, int*, double*, std::string*);

}  // namespace les
