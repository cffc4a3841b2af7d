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
// What bounds it: per sweep three fields (x and b in, x out) and the grid sum
// (about 3 us).  Measured on 256 x 256 x 64 in FP32 (the fields lie in L2): a
// launch per sweep, with every neighbour through L1 and a division per node, 70
// us; here 15.
#include <algorithm>
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

  // this thread's sums over the nodes of v
  auto sum_of = [&](auto&& term) {
    StreamSum<T> s[1];
    for (long long m = gtid; m < f.n; m += gstride) {
      s[0].add(term(m));
      s[0].tick();
    }
    double t[1];
    const bool ok = stream_sum<1>(s, gs, t);
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
      const T v = __ldcg(f.b + m) - mean;
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
  while (!status) {
    const T* xin = f.x[sweep & 1];
    T* xout = f.x[(sweep + 1) & 1];
    StreamSum<T> s[1];
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
                s[0].add(r * r);
              }
            s[0].tick();
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
    double t[1];
    const bool ok = stream_sum<1>(s, gs, t);
    if (tid == 0) {
      if (!ok) {
        status = 5;
      } else {
        // the residual of x_s, which stays in its buffer
        rel = sqrt(t[0] / bb);
        if (!isfinite(t[0])) status = 3;
        else if (rel <= f.tol) status = 1;
        else if (sweep >= f.maxit) status = 2;
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
