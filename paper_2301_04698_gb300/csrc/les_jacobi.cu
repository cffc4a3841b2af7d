// les_jacobi.cu -- weighted Jacobi, the paper's Poisson solver (Sec. 2.4), in one
// persistent cooperative launch: x <- x + omega (b - L_c x) / diag(L_c), with the
// compact 7-point Laplacian, periodic in x and y, mirror or periodic in z; the
// mean of b is removed and x returned with zero mean.
//
// A sweep marches tiles of any extents as the streaming CG does (les_stream.cuh):
// a plane of x passes through shared memory for its x and y neighbours, the z
// neighbours are the march's registers, and the residual of the plane below is
// complete when the plane above arrives.  A grid-wide sum per sweep gives the
// residual norm of the x it read; x is double-buffered.
//
// The norm decides when the solver stops, for residuals of any size that FP32 holds, so
// no square is rounded to FP32 or leaves its range: the first sweep of an FP32 solve
// squares and adds in FP64, the later ones in FP32 with each square's and addition's
// rounding error kept, of residuals scaled by a power of two to the size of the last
// sweep's.
//
// What bounds it: per sweep three fields (x and b in, x out) and the grid sum
// (about 3 us).  Measured on 256 x 256 x 64 in FP32 (the fields lie in L2): a
// launch per sweep, with every neighbour through L1 and a division per node, 70
// us; here 15.  Of a solve's 108 us beside its sweeps 39 are FP64 arithmetic (the right
// side's norm, the first sweep).
#include <algorithm>
#include <cmath>
#include <string>
#include <type_traits>

#include "les_internal.h"
#include "les_stream.cuh"

namespace les {
namespace {

template <typename T>
struct JacobiArgs {
  int nx, ny, nz, walls;
  T cx, cy, cz;          // 1/dx^2, 1/dy^2, 1/dz^2
  T wd, wd_wall;         // omega / diag(L_c), inside and on a plane next to a wall
  int ntx, nty, nchunk;  // tiles along x and y, runs of planes per tile
  long long n, nunits;
  int en;                // binary exponent of n
  const T* b;
  T* x[2];               // x_s in x[s & 1]; x[0] the caller's
  double* partials;
  FusedBar* bar;
  SolverCtl* ctl;
  double tol;
  int maxit;
  long long spin_cycles;
  unsigned expected;
};

template <typename T, typename S>
__global__ void __launch_bounds__(kStreamThreads, 2) k_jacobi_stream(JacobiArgs<T> f) {
  constexpr int NO = S::NO, NWX = S::NWX, SP = S::SP, SN = S::SN;
  __shared__ T sm[2][SN];
  __shared__ struct {
    T mean;
    int e;  // FP32: the residuals' size (binary exponent) at the last sweep
    int status;
  } sc;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int plane = f.nx * f.ny;
  const T cx = f.cx, cy = f.cy, cz = f.cz;
  GridSync gs{f.bar, f.partials, f.spin_cycles, f.expected, 0u};
  const long long gstride = (long long)gridDim.x * kStreamThreads;
  const long long gtid = (long long)blockIdx.x * kStreamThreads + tid;
  double bb = 0.0, rel = 0.0;  // meaningful in thread 0
  int status = 0;  // 0 running, 1 converged, 2 maxit, 3 non-finite, 4 zero rhs, 5 timeout

  // sums over the nodes: of FP64 terms in FP64, of FP32 ones with the additions' rounding
  // errors kept
  auto sum_of = [&](auto&& term) {
    double v[1] = {0.0}, t[1];
    if constexpr (std::is_same<decltype(term(gtid)), float>::value) {
      F2 a{0.f, 0.f};
#pragma unroll 4
      for (long long m = gtid; m < f.n; m += gstride) f2_acc(a, term(m));
      v[0] = f2_value(a);
    } else {
#pragma unroll 4
      for (long long m = gtid; m < f.n; m += gstride) v[0] += term(m);
    }
    const bool ok = grid_sum_t0<1>(v, gs, t);
    if (tid == 0 && !ok) status = 5;
    return t[0];
  };
  {
    const double t = sum_of([&](long long m) { return __ldcg(f.b + m); });
    if (tid == 0) {
      sc.status = status;
      sc.mean = (T)(t / (double)f.n);
    }
    __syncthreads();
    status = sc.status;
  }
  const T mean = sc.mean;
  if (!status) {
    const double t = sum_of([&](long long m) {
      const double v = (double)(__ldcg(f.b + m) - mean);
      return v * v;
    });
    if (tid == 0) {
      bb = t;
      if (!status && bb == 0.0) status = 4;
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
  }

  int sweep = 0;
  // the sweep's sum of squares, FP64 or compensated, into t (thread 0)
  auto relax = [&](auto exact, double (&t)[1]) -> bool {
    constexpr bool EXACT = decltype(exact)::value;
    const T* xin = f.x[sweep & 1];
    T* xout = f.x[(sweep + 1) & 1];
    const float scale = EXACT ? 1.f : __int_as_float((127 - sc.e) << 23);
    double sd[1] = {0.0};
    F2 sf[1] = {F2{0.f, 0.f}};
    auto square = [&](T r) {
      if constexpr (EXACT) {
        sd[0] += (double)r * (double)r;
      } else {
        const float v = r * scale, p = v * v;
        f2_acc(sf[0], p);
        sf[0].lo += fmaf(v, v, -p);
      }
    };
    for (long long u = blockIdx.x; u < f.nunits; u += gridDim.x) {
      const int tile = (int)(u / f.nchunk), chunk = (int)(u - (long long)tile * f.nchunk);
      int x0, y0, w, h, k0, kn;
      stream_part(f.nx, f.ntx, tile % f.ntx, x0, w);
      stream_part(f.ny, f.nty, tile / f.ntx, y0, h);
      stream_part(f.nz, f.nchunk, chunk, k0, kn);
      int go[NO];
#pragma unroll
      for (int m = 0; m < NO; ++m) {
        const int ex = lane + 32 * (m % NWX), ey = warp + 8 * (m / NWX);
        go[m] = ex < w && ey < h ? (y0 + ey) * f.nx + x0 + ex : -1;
      }
      const int eo = (warp + 1) * SP + lane + 1;
      int gr, er;
      stream_ring<S>(tid, x0, y0, w, h, f.nx, f.ny, gr, er);
      // a whole tile's lanes all have nodes: without the tests the nodes' chains overlap
      // (256 x 256 x 64 FP32: 16.8 -> 15.0 us per sweep)
      auto march = [&](auto whole) {
        constexpr bool FULL = decltype(whole)::value;
        T xv[NO], bv[NO], rh = T(0);  // x and b of the plane in flight; the ring's x
        auto load = [&](int kk, bool inside) {
          const size_t base = (size_t)stream_z(kk, f.nz, f.walls) * plane;
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            xv[m] = bv[m] = T(0);
            if (FULL || go[m] >= 0) {
              xv[m] = __ldcg(xin + base + go[m]);
              if (inside) bv[m] = __ldcg(f.b + base + go[m]);
            }
          }
          if (inside && gr >= 0) rh = __ldcg(xin + base + gr);
        };
        T pd[NO], pc[NO], bc[NO], part[NO];  // x below, x and b - mean here, L_c x without z
        load(k0 - 1, false);
#pragma unroll
        for (int m = 0; m < NO; ++m) pc[m] = xv[m], bc[m] = part[m] = pd[m] = T(0);
        load(k0, true);
        __syncthreads();  // the previous unit's readers are done with sm
        for (int k = k0; k <= k0 + kn; ++k) {
          const bool inside = k < k0 + kn;
          T pv[NO], bn[NO];
          T* pl = sm[k & 1];
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            pv[m] = xv[m];
            bn[m] = bv[m] - mean;
            if (inside && (FULL || go[m] >= 0)) pl[eo + 8 * (m / NWX) * SP + 32 * (m % NWX)] = pv[m];
          }
          if (inside && gr >= 0) pl[er] = rh;
          if (inside) load(k + 1, k + 1 < k0 + kn);
          if (k > k0) {  // plane k - 1 is complete with this plane's x
            const size_t base = (size_t)(k - 1) * plane;
            const T wd = f.walls && (k - 1 == 0 || k == f.nz) ? f.wd_wall : f.wd;
#pragma unroll
            for (int m = 0; m < NO; ++m)
              if (FULL || go[m] >= 0) {
                const T r = bc[m] - (part[m] + (pd[m] + pv[m] - T(2) * pc[m]) * cz);
                __stcg(xout + base + go[m], pc[m] + wd * r);
                square(r);
              }
          }
          if (!inside) break;
          __syncthreads();  // plane k is in sm (the other buffer's readers passed the barrier before)
#pragma unroll
          for (int m = 0; m < NO; ++m) {
            const T* e = pl + eo + 8 * (m / NWX) * SP + 32 * (m % NWX);
            const T c2 = T(2) * pv[m];
            part[m] = (e[-1] + e[1] - c2) * cx + (e[-SP] + e[SP] - c2) * cy;
            pd[m] = pc[m];
            pc[m] = pv[m];
            bc[m] = bn[m];
          }
        }
      };
      if (w == S::WX && h == S::WY) march(std::true_type{});
      else march(std::false_type{});
    }
    if constexpr (EXACT) {
      return grid_sum_t0<1>(sd, gs, t);
    } else {
      const bool ok = grid_sum_t0<1>(sf, gs, t);
      if (tid == 0) t[0] *= pow2(2 * sc.e);
      return ok;
    }
  };
  while (!status) {
    double t[1];
    bool ok;
    if constexpr (sizeof(T) == 8) ok = relax(std::true_type{}, t);
    else ok = sweep == 0 ? relax(std::true_type{}, t) : relax(std::false_type{}, t);
    if (tid == 0) {
      if (!ok) {
        status = 5;
      } else {
        // the residual of x_s, which stays in its buffer
        rel = sqrt(t[0] / bb);
        if (!isfinite(t[0])) status = 3;
        else if (rel <= f.tol) status = 1;
        else if (sweep >= f.maxit) status = 2;
        else sc.e = max(-126, min(126, ((__double2hiint(t[0]) >> 20 & 0x7ff) - 1023 - f.en) >> 1));
      }
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
    if (!status) ++sweep;
  }

  // zero-mean gauge (or zero for a zero right side) into the caller's array
  if (status != 5) {
    const T* src = f.x[sweep & 1];
    const double t = sum_of([&](long long m) { return __ldcg(src + m); });
    if (tid == 0) {
      sc.mean = (T)(t / (double)f.n);
      sc.status = status;
    }
    __syncthreads();
    status = sc.status;
    if (status != 5) {
      const T mx = sc.mean;
      for (long long m = gtid; m < f.n; m += gstride)
        __stcg(f.x[0] + m, status == 4 ? T(0) : __ldcg(src + m) - mx);
    }
  }
  if (blockIdx.x == 0 && tid == 0) {
    f.ctl->iter = sweep;
    f.ctl->rel = rel;
    f.ctl->done = status;
  }
}

template <typename T>
const void* jacobi_kernel(int shape) {
  if (shape == 0) return (const void*)k_jacobi_stream<T, Tile64>;
  if (shape == 1) return (const void*)k_jacobi_stream<T, Tile32>;
  return (const void*)k_jacobi_stream<T, Tile32s>;
}

}  // namespace

template <typename T>
int poisson_solve_jacobi(const SolverArgs<T>& a, const FusedCfg& fc, const T* b, T* x, double tol, int maxit,
                         int* iters, double* rel, std::string* err) {
  int dev = 0, nsm = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
      (e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) {
    if (err) *err = std::string("weighted Jacobi: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  int per_sm = 2;
  StreamPlan pl;
  const void* kern = nullptr;
  for (int pass = 0; pass < 2; ++pass) {  // the plan depends on the resident blocks, they on the shape
    pl = make_stream_plan(a.g.nx, a.g.ny, a.g.nz, std::min<long long>((long long)per_sm * nsm, fc.max_blocks), false);
    kern = jacobi_kernel<T>(pl.shape);
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kStreamThreads, 0)) != cudaSuccess) {
      if (err) *err = std::string("weighted Jacobi occupancy: ") + cudaGetErrorString(e);
      return LES_ERR_CUDA;
    }
    per_sm = std::min(per_sm, 8);  // the partials hold 2 x kSumSlot words of 8 blocks per SM
    if (per_sm < 1) {
      if (err) *err = "weighted Jacobi: no block fits on an SM";
      return LES_ERR_CUDA;
    }
  }
  long long G = std::min<long long>((long long)per_sm * nsm, fc.max_blocks);
  G = std::max<long long>(1, std::min(G, pl.units));
  JacobiArgs<T> f;
  f.nx = a.g.nx;
  f.ny = a.g.ny;
  f.nz = a.g.nz;
  f.walls = a.g.walls;
  f.cx = a.g.idx * a.g.idx;
  f.cy = a.g.idy * a.g.idy;
  f.cz = a.g.idz * a.g.idz;
  f.wd = (T)(a.omega / (-2.0 * ((double)f.cx + (double)f.cy + (double)f.cz)));
  f.wd_wall = (T)(a.omega / (-2.0 * ((double)f.cx + (double)f.cy) - (double)f.cz));
  f.ntx = pl.ntx;
  f.nty = pl.nty;
  f.nchunk = pl.nchunk;
  f.nunits = pl.units;
  f.n = (long long)f.nx * f.ny * f.nz;
  f.en = std::ilogb((double)f.n);
  f.b = b;
  f.x[0] = x;
  f.x[1] = a.p0;
  f.partials = a.partials;
  f.bar = a.bar;
  f.ctl = a.ctl;
  f.tol = tol;
  f.maxit = maxit;
  f.spin_cycles = fc.spin_cycles;
  f.expected = (unsigned)G + (unsigned)std::max(0, fc.missing);
  if ((e = cudaMemsetAsync(a.bar, 0, sizeof(FusedBar), a.st)) != cudaSuccess) {
    if (err) *err = std::string("weighted Jacobi barrier reset: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  void* args[] = {&f};
  {
    ProfScope ps(a.prof, KI_JACOBI, a.st);
    e = cudaLaunchCooperativeKernel(kern, dim3((unsigned)G), dim3(kStreamThreads), args, 0, a.st);
  }
  if (e != cudaSuccess) {
    if (err) *err = std::string("weighted Jacobi launch: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  if ((e = cudaMemcpyAsync(a.ctl_host, a.ctl, sizeof(SolverCtl), cudaMemcpyDeviceToHost, a.st)) != cudaSuccess ||
      (e = cudaStreamSynchronize(a.st)) != cudaSuccess) {
    if (err) *err = std::string("weighted Jacobi: ") + cudaGetErrorString(e);
    return LES_ERR_CUDA;
  }
  const SolverCtl& c = *a.ctl_host;
  if (iters) *iters = c.iter;
  if (rel) *rel = c.rel;
  // the means of b and x and |b|^2: 3, the gauge: x in and out; per pass over the grid,
  // one more than the sweeps counted, x and b in, x out: 3
  if (a.prof) a.prof->bytes[KI_JACOBI] += (5.0 + 3.0 * (c.iter + 1)) * (double)f.n * sizeof(T);
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
      if (err) *err = "poisson: the Jacobi solver returned no status";
      return LES_ERR_CUDA;
  }
}

template int poisson_solve_jacobi<float>(const SolverArgs<float>&, const FusedCfg&, const float*, float*, double, int,
                                         int*, double*, std::string*);
template int poisson_solve_jacobi<double>(const SolverArgs<double>&, const FusedCfg&, const double*, double*, double,
                                          int, int*, double*, std::string*);

}  // namespace les
