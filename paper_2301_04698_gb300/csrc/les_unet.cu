// les_unet.cu -- the learned Poisson warm start: a 3-level 3-D U-Net trained
// and evaluated with this library's own BF16 tensor-core kernels (FP32
// accumulation).  Not in the paper; it predicts the first guess psi_0 of the
// pressure-correction solve (Sec. 2.4) from its right-hand side b:
//
//   x0 = b / s, s = rms(b);  e1 = B(x0; 1->16);  e2 = B(pool e1; 16->32);
//   e3 = B(pool e2; 32->64);  g2 = B([up e3, e2]; 96->32);
//   g1 = B([up g2, e1]; 48->16);  y = conv1(g1; 16->1);  psi_0 = s (y - mean y)
//
// with B(.; a->c) two 3x3x3 periodic convolutions each followed by a leaky
// ReLU (slope 0.1), pool a 2x2x2 mean, up nearest-neighbour doubling and
// [.,.] channel concatenation.  Weights travel as one flat FP32 vector, layer
// by layer, W[cout][cin][kz][ky][kx] then bias[cout].
//
// Activations are channels-last BF16 ([batch][z][y][x][c], c padded to a
// multiple of 16); weights [cout / 16][tap][16][cin + 8].  A convolution (k_conv) is an
// implicit GEMM on the tensor cores, mma.sync m16n8k16 BF16 -> FP32: rows are
// voxels, K runs over (tap, 16 channels), N over output channels.  A block
// stages its tile's input with a halo of one voxel and the weights of its
// output channels in shared memory once, and feeds the 27 taps from there
// with ldmatrix; voxel and weight rows are an odd number of 16-byte units, so
// the eight rows of a matrix fall on different banks.  Nearest doubling is
// read through halved coordinates, concatenation from two arrays, and the
// epilogue adds bias and activation (or, going back, multiplies by the
// activation's slope), pools, and on the last layer applies the 1x1 head.
// The input gradient is the same kernel on flipped, transposed weights.  The
// weight gradient (k_wgrad) is a GEMM over voxels: a warp per (dz, dy) keeps
// its three taps of every output channel and 16 input channels in registers
// while the block walks its share of the tiles; the FP32 partials of the
// shares are summed in order (deterministic).  Adam keeps FP32 master weights.
//
// What bounds it: at 32^3 and batch 1 the 13 short kernels' launches and
// latencies (5 to 10 us each, the MMAs 1 to 3 of them; each loads its weights
// before it waits for its predecessor); at batch 16 the shared-memory reads, 3
// wavefronts per MMA with two output fragments and 2 with four (the LSU pipe is
// 55 % busy, the tensor pipe 36 %).  mma.sync, not tcgen05: N is 16 to 64, and
// every sum runs over taps and channels in one order, so the results do not
// depend on the tile.  Blocks that keep their weights and stage the next tile
// during the MMAs were no faster (two input buffers cost the second block).
// Measured (GB300, 32^3): forward at batch 1 437 us with an operand fetched
// from global memory per MMA, 82 now; training gradient at batch 16 8990, 1090.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "les_internal.h"

namespace les {
namespace {

using bf16 = __nv_bfloat16;
constexpr float kLeak = 0.1f;

struct LayerDef {
  const char* name;
  int cin, cout, k;
};
constexpr LayerDef kLayers[] = {{"enc1a", 1, 16, 3},  {"enc1b", 16, 16, 3}, {"enc2a", 16, 32, 3},
                                {"enc2b", 32, 32, 3}, {"enc3a", 32, 64, 3}, {"enc3b", 64, 64, 3},
                                {"dec2a", 96, 32, 3}, {"dec2b", 32, 32, 3}, {"dec1a", 48, 16, 3},
                                {"dec1b", 16, 16, 3}, {"head", 16, 1, 1}};
constexpr int kNL = 11;
enum { L_E1A, L_E1B, L_E2A, L_E2B, L_E3A, L_E3B, L_D2A, L_D2B, L_D1A, L_D1B, L_HEAD };

__host__ __device__ inline int pad16(int c) { return (c + 15) / 16 * 16; }
__host__ __device__ inline int pad8(int c) { return (c + 7) / 8 * 8; }

// ---- tensor-core primitives ---------------------------------------------------
__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void ldsm4t(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
// Programmatic dependent launch: a kernel starts while its predecessor in the
// stream drains, and waits here before it touches what that one writes (every
// kernel of a chain waits, so whatever ran before the predecessor is complete
// too).  Only weights, which the chain does not write, are read before.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

__device__ __forceinline__ unsigned ld32(const bf16* p) { return *reinterpret_cast<const unsigned*>(p); }
__device__ __forceinline__ unsigned pack2(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const unsigned*>(&v);
}
// eight BF16 values of a 16-byte chunk
struct Chunk {
  float v[8];
};
__device__ __forceinline__ Chunk unpack8(uint4 u) {
  Chunk c;
  const unsigned w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    c.v[2 * q] = __uint_as_float(w[q] << 16);
    c.v[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u);
  }
  return c;
}
__device__ __forceinline__ uint4 pack8(const Chunk& c) {
  return make_uint4(pack2(c.v[0], c.v[1]), pack2(c.v[2], c.v[3]), pack2(c.v[4], c.v[5]), pack2(c.v[6], c.v[7]));
}
// leaky ReLU backward from the post-activation (same sign as the
// pre-activation): g is BF16 already, the product is rounded to BF16
__device__ __forceinline__ uint4 act_back(uint4 post, uint4 g) {
  const Chunk p = unpack8(post);
  Chunk c = unpack8(g);
#pragma unroll
  for (int q = 0; q < 8; ++q) c.v[q] = p.v[q] > 0.f ? c.v[q] : kLeak * c.v[q];
  return pack8(c);
}
// periodic coordinate of a staged voxel: at most one before the grid, and any
// number past it (ragged tiles)
__device__ __forceinline__ int wrap_tile(int i, int n) { return i < 0 ? i + n : (i >= n ? i % n : i); }

// ---- convolution as an implicit GEMM --------------------------------------------
// Block tiles: 4 x 4 x 4 voxels by 4 warps, a z-plane each, where the grid is
// small, and 4 x 8 x 8 by 8 warps of two row groups each (half the weight
// loads per voxel, 1.5 times the MMAs per shared-memory read).
template <int CFG>
struct Tile;
template <>
struct Tile<0> {
  static constexpr int Z = 4, Y = 4, X = 4, W = 4, MT = 1;
};
template <>
struct Tile<1> {
  static constexpr int Z = 4, Y = 8, X = 8, W = 8, MT = 2;
};
// staged input of KC x 16 channels, in 16-byte units: S per voxel (odd), P per
// row (4 mod 8 where the rows of a matrix span two tile rows), PZ per plane
template <int CFG, int KC>
struct Staged {
  using T = Tile<CFG>;
  static constexpr int S = 2 * KC + 1;
  static constexpr int U = (T::X + 2) * S;
  static constexpr int P = T::X == 4 ? (U + 3) / 8 * 8 + 4 : U;
  static constexpr int PZ = (T::Y + 2) * P;
  static constexpr int IN = (T::Z + 2) * PZ;
};
template <int CFG, int KC, int NFB>
constexpr size_t conv_smem() {
  return 16 * ((size_t)Staged<CFG, KC>::IN + 27 * 8 * NFB * (2 * KC + 1));
}

struct ConvArgs {
  const bf16* in0;
  int c0, up0;  // channels of in0 (multiple of 16); 1: in0 lives on the halved grid
  const bf16* in1;
  int c1;          // channels of in1 (0 if absent)
  const bf16* w;   // [cout / 16][27][16][16 KC + 8]
  int cout;
  const float* bias;  // forward: bias and leaky ReLU; NULL: neither
  const bf16* post;   // backward: activations whose slope multiplies the result (oc0 channels)
  bf16* out0;
  int oc0;
  bf16* out1;
  int oc1;
  bf16* pool;         // 2 x 2 x 2 means of the output (oc0 channels)
  const bf16* hw;     // head: y = hw . output + hb, and the tile's FP64 sum of y
  const float* hb;
  float* y;
  double* ysum;
  int n, tx, ty, tz;  // grid, tiles along x, y, z
};

// Where the rows and columns of a halo tile lie: element offsets of its rows in
// both inputs and of its columns within a row (periodic, halved for an input on
// the coarser grid).  Made once per tile by one thread per row, so that a
// 16-byte copy costs a dozen instructions: formed per copy, the wraps and
// products took longer than the MMAs.
template <int CFG>
struct HaloTable {
  using T = Tile<CFG>;
  static constexpr int HX = T::X + 2, HY = T::Y + 2, ROWS = (T::Z + 2) * HY;
  long long r0[ROWS], r1[ROWS];
  int x0[HX], x1[HX];
  __device__ __forceinline__ void make(int c0, int up0, int c1, int n, long long b, int z0, int y0, int xs) {
    const int t = threadIdx.x, m = n >> 1;
    if (t < ROWS) {
      const int gz = wrap_tile(z0 - 1 + t / HY, n), gy = wrap_tile(y0 - 1 + t % HY, n);
      const long long r = (b * n + gz) * n + gy;
      r0[t] = (up0 ? ((b * m + (gz >> 1)) * m + (gy >> 1)) * m : r * n) * c0;
      r1[t] = r * n * c1;
    } else if (t < ROWS + HX) {
      const int gx = wrap_tile(xs - 1 + t - ROWS, n);
      x0[t - ROWS] = (up0 ? gx >> 1 : gx) * c0;
      x1[t - ROWS] = gx * c1;
    }
  }
};
// Channels [ch0, ch0 + 8 NC) of [in0, in1] of a halo tile into shared memory.
template <int CFG, int NC, int S, int P, int PZ, int NTHR>
__device__ __forceinline__ void stage_halo(unsigned sm, const HaloTable<CFG>& tab, const bf16* in0, int c0,
                                           const bf16* in1, int ch0) {
  using H = HaloTable<CFG>;
  constexpr int N = H::ROWS * H::HX * NC;
#pragma unroll 4
  for (int e = threadIdx.x; e < N; e += NTHR) {
    const int row = e / (H::HX * NC), k = e - row * (H::HX * NC), x = k / NC, c = k - x * NC;
    const int z = row / H::HY, y = row - z * H::HY, ch = ch0 + 8 * c;
    const bf16* src = ch < c0 ? in0 + (tab.r0[row] + tab.x0[x] + ch) : in1 + (tab.r1[row] + tab.x1[x] + (ch - c0));
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sm + 16u * (unsigned)(z * PZ + y * P + x * S + c)),
                 "l"(src)
                 : "memory");
  }
}

template <int CFG, int KC, int NFB>
__global__ void __launch_bounds__(32 * Tile<CFG>::W) k_conv(ConvArgs a) {
  using T = Tile<CFG>;
  using G = Staged<CFG, KC>;
  constexpr int NB = 8 * NFB, NTHR = 32 * T::W, WS = 2 * KC + 1, MT = T::MT;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ double shd[32];
  __shared__ HaloTable<CFG> tab;
  const unsigned sin = (unsigned)__cvta_generic_to_shared(smraw), sw = sin + 16u * G::IN;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gid = lane >> 2, tig = lane & 3;
  const int co0 = blockIdx.y * NB;
  // the weights first: they do not depend on the kernel before.  Their rows are
  // padded in global memory as they are here, so the copy is a plain one.
  {
    constexpr int NCH = 27 * NB * WS;
    const bf16* src = a.w + (size_t)blockIdx.y * NCH * 8;
#pragma unroll 4
    for (int e = threadIdx.x; e < NCH; e += NTHR)
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(sw + 16u * (unsigned)e), "l"(src + 8 * e)
                   : "memory");
  }
  const int tps = a.tx * a.ty * a.tz;
  const long long b = blockIdx.x / tps;
  const int tile = blockIdx.x - (int)b * tps;
  const int x0 = (tile % a.tx) * T::X, y0 = (tile / a.tx) % a.ty * T::Y, z0 = tile / (a.tx * a.ty) * T::Z;
  tab.make(a.c0, a.up0, a.c1, a.n, b, z0, y0, x0);
  __syncthreads();
  pdl_launch();
  pdl_wait();
  stage_halo<CFG, 2 * KC, G::S, G::P, G::PZ, NTHR>(sin, tab, a.in0, a.c0, a.in1, 0);
  cp_commit();
  cp_wait<0>();
  __syncthreads();

  // the lane's row of each A matrix (voxel lane mod 16, channel half lane / 16)
  // and of a B matrix pair
  auto voxel = [&](int mt, int row, int& z, int& y, int& x) {
    if (CFG == 0) {
      z = warp, y = row >> 2, x = row & 3;
    } else {
      const int q = warp * MT + mt;
      z = q >> 2, y = ((q & 3) << 1) + (row >> 3), x = row & 7;
    }
  };
  const unsigned pb = sw + 16u * (unsigned)(((lane & 7) + ((lane >> 4) & 1) * 8) * WS + ((lane >> 3) & 1));
  unsigned pa[MT];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    int z, y, x;
    voxel(mt, lane & 15, z, y, x);
    pa[mt] = sin + 16u * (unsigned)(z * G::PZ + y * G::P + x * G::S + (lane >> 4));
  }
  float acc[MT][NFB][4];
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int f = 0; f < NFB; ++f) acc[mt][f][0] = acc[mt][f][1] = acc[mt][f][2] = acc[mt][f][3] = 0.f;
  // the operands of a step are loaded while the MMAs of the one before run
  unsigned A[MT][4], B[NFB / 2][4];
  auto load = [&](unsigned (&fa)[MT][4], unsigned (&fb)[NFB / 2][4], int zy, int step) {
    const int tx = step / KC, kc = step % KC;
    const unsigned oa = 16u * (unsigned)((zy / 3) * G::PZ + (zy % 3) * G::P + tx * G::S + 2 * kc);
    const unsigned ob = 16u * (unsigned)((zy * 3 + tx) * 16 * WS + 2 * kc);
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) ldsm4(fa[mt], pa[mt] + oa);
#pragma unroll
    for (int h = 0; h < NFB / 2; ++h) ldsm4(fb[h], pb + ob + 16u * (unsigned)(27 * 16 * h * WS));
  };
  load(A, B, 0, 0);
#pragma unroll 1
  for (int zy = 0; zy < 9; ++zy) {
#pragma unroll
    for (int step = 0; step < 3 * KC; ++step) {
      unsigned An[MT][4], Bn[NFB / 2][4];
      // (after the very last step the first of the last group again, unused)
      if (step + 1 < 3 * KC) load(An, Bn, zy, step + 1);
      else load(An, Bn, zy < 8 ? zy + 1 : 8, 0);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt)
#pragma unroll
        for (int f = 0; f < NFB; ++f) mma_bf16(acc[mt][f], A[mt], B[f >> 1][2 * (f & 1)], B[f >> 1][2 * (f & 1) + 1]);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
#pragma unroll
        for (int mt = 0; mt < MT; ++mt) A[mt][q] = An[mt][q];
#pragma unroll
        for (int h = 0; h < NFB / 2; ++h) B[h][q] = Bn[h][q];
      }
    }
  }
  __syncthreads();  // the staged input is free: it takes the output tile

  // epilogue: bias and activation, rounded to BF16 into [voxel][NB + 8]
  bf16* so = reinterpret_cast<bf16*>(smraw);
  constexpr int OS = NB + 8;
  double ysum = 0.0;
#pragma unroll
  for (int mt = 0; mt < MT; ++mt) {
    unsigned packed[NFB][2];
#pragma unroll
    for (int f = 0; f < NFB; ++f) {
      const int co = co0 + f * 8 + tig * 2;
      float b0 = 0.f, b1 = 0.f;
      if (a.bias) {
        b0 = a.bias[co];
        b1 = a.bias[co + 1];
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        float u0 = acc[mt][f][2 * h], u1 = acc[mt][f][2 * h + 1];
        if (a.bias) {
          u0 += b0;
          u1 += b1;
          u0 = u0 > 0.f ? u0 : kLeak * u0;
          u1 = u1 > 0.f ? u1 : kLeak * u1;
        }
        packed[f][h] = pack2(u0, u1);
        const int row = (warp * MT + mt) * 16 + gid + 8 * h;
        *reinterpret_cast<unsigned*>(so + row * OS + f * 8 + tig * 2) = packed[f][h];
      }
    }
    if (NFB == 2 && a.hw) {
      // the output fragments are the A fragments of the 1x1 head
      const unsigned H[4] = {packed[0][0], packed[0][1], packed[1][0], packed[1][1]};
      float yv[4] = {0.f, 0.f, 0.f, 0.f};
      mma_bf16(yv, H, ld32(a.hw + gid * 16 + tig * 2), ld32(a.hw + gid * 16 + tig * 2 + 8));
      if (tig == 0) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          int z, y, x;
          voxel(mt, gid + 8 * h, z, y, x);
          if (z0 + z < a.n && y0 + y < a.n && x0 + x < a.n) {
            const float v = yv[2 * h] + a.hb[0];
            a.y[((b * a.n + z0 + z) * a.n + y0 + y) * a.n + x0 + x] = v;
            ysum += (double)v;
          }
        }
      }
    }
  }
  __syncthreads();
  // stored 16 bytes at a time; row q of the tile is voxel (q)
  for (int e = threadIdx.x; e < T::Z * T::Y * T::X * NFB; e += NTHR) {
    const int q = e / NFB, c = e - q * NFB;
    const int z = z0 + q / (T::Y * T::X), y = y0 + q / T::X % T::Y, x = x0 + q % T::X;
    if (z >= a.n || y >= a.n || x >= a.n) continue;
    const size_t v = (size_t)((b * a.n + z) * a.n + y) * a.n + x;
    uint4 o = *reinterpret_cast<const uint4*>(so + q * OS + 8 * c);
    const int co = co0 + 8 * c;
    if (a.post) o = act_back(__ldg(reinterpret_cast<const uint4*>(a.post + v * a.oc0 + co)), o);
    if (co < a.oc0) *reinterpret_cast<uint4*>(a.out0 + v * a.oc0 + co) = o;
    else *reinterpret_cast<uint4*>(a.out1 + v * a.oc1 + (co - a.oc0)) = o;
  }
  if (a.pool) {
    const int m = a.n >> 1;
    for (int e = threadIdx.x; e < T::Z * T::Y * T::X / 8 * NFB; e += NTHR) {
      const int q = e / NFB, c = e - q * NFB;
      const int x = q % (T::X / 2), y = q / (T::X / 2) % (T::Y / 2), z = q / (T::X / 2 * (T::Y / 2));
      if (z0 + 2 * z >= a.n || y0 + 2 * y >= a.n || x0 + 2 * x >= a.n) continue;
      Chunk s = {};
#pragma unroll
      for (int r8 = 0; r8 < 8; ++r8) {
        const int r = ((2 * z + (r8 >> 2)) * T::Y + 2 * y + ((r8 >> 1) & 1)) * T::X + 2 * x + (r8 & 1);
        const Chunk u = unpack8(*reinterpret_cast<const uint4*>(so + r * OS + 8 * c));
#pragma unroll
        for (int i = 0; i < 8; ++i) s.v[i] += u.v[i];
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) s.v[i] *= 0.125f;
      *reinterpret_cast<uint4*>(a.pool + (size_t)(((b * m + z0 / 2 + z) * m + y0 / 2 + y) * m + x0 / 2 + x) * a.oc0 +
                                co0 + 8 * c) = pack8(s);
    }
  }
  if (a.hw) {
    const double t = block_reduce<false>(ysum, shd);
    if (threadIdx.x == 0) a.ysum[blockIdx.x] = t;
  }
}

// ---- weight gradient: gW[t][co][ci] = sum_v g[v][co] in[nbr(v, t)][ci] ----------
struct WgradArgs {
  const bf16* g;  // [voxels][16 CO]
  const bf16* in0;
  int c0, up0;
  const bf16* in1;
  int c1;
  float* part;   // [shares][27][16 CO][cin]
  float* bpart;  // [shares][16 CO]
  int cin, n, tx, ty, tz;
  long long ntiles;
};
constexpr int kWgWarps = 9;  // one per (dz, dy)
// Tiles whose products the accumulators take before they are added to the share's
// partials: 16 x 256 voxels, 256 MMAs in a chain, whatever the grid and the batch.  The
// error of a chain grows with its length: the gradient of one sample at 64^3 repeated 16
// and 64 times is off by 1.5e-4 and 6.8e-4 of a layer's norm with chains as long as the
// shares (162 and 649 tiles), by 1e-5 at most with these.
constexpr int kWgFold = 16;

template <int CO>
constexpr size_t wgrad_smem() {
  return 2 * 16 * ((size_t)Staged<1, 1>::IN + 256 * (2 * CO + 1));
}

// Block (ci slice, share): 16 input channels, every (share)-th tile.  A row of
// voxel pairs is 16 K entries; both operands come transposed from rows of
// voxels by ldmatrix.  The bias gradient is one more column, of ones, in the
// blocks of the first slice.
template <int CO>
__global__ void __launch_bounds__(32 * kWgWarps) k_wgrad(WgradArgs a) {
  using T = Tile<1>;
  using G = Staged<1, 1>;
  constexpr int NTHR = 32 * kWgWarps, GS = 2 * CO + 1, STAGE = G::IN + 256 * GS;
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ HaloTable<1> tab[2];
  const unsigned sm = (unsigned)__cvta_generic_to_shared(smraw);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int gid = lane >> 2, tig = lane & 3;
  const int tps = a.tx * a.ty * a.tz;
  auto origin = [&](long long tile, long long& b, int& z0, int& y0, int& x0) {
    b = tile / tps;
    const int q0 = (int)(tile - b * tps);
    x0 = (q0 % a.tx) * T::X, y0 = (q0 / a.tx) % a.ty * T::Y, z0 = q0 / (a.tx * a.ty) * T::Z;
  };
  auto table = [&](long long tile, int buf) {
    long long b;
    int z0, y0, x0;
    origin(tile, b, z0, y0, x0);
    tab[buf].make(a.c0, a.up0, a.c1, a.n, b, z0, y0, x0);
  };
  auto stage = [&](long long tile, int buf) {
    const unsigned s0 = sm + 16u * (unsigned)(buf * STAGE);
    long long b;
    int z0, y0, x0;
    origin(tile, b, z0, y0, x0);
    stage_halo<1, 2, G::S, G::P, G::PZ, NTHR>(s0, tab[buf], a.in0, a.c0, a.in1, 16 * blockIdx.x);
    for (int e = threadIdx.x; e < 256 * 2 * CO; e += NTHR) {
      const int q = e / (2 * CO), c = e - q * (2 * CO);
      const int z = z0 + (q >> 6), y = y0 + ((q >> 3) & 7), x = x0 + (q & 7);
      // voxels beyond the grid contribute nothing: zero bytes are copied
      const bool in = z < a.n && y < a.n && x < a.n;
      const bf16* src = in ? a.g + (size_t)(((b * a.n + z) * a.n + y) * a.n + x) * (16 * CO) + 8 * c : a.g;
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(s0 + 16u * (unsigned)(G::IN + q * GS + c)),
                   "l"(src), "r"(in ? 16 : 0)
                   : "memory");
    }
  };
  float acc[3][CO][2][4], ab[CO][4];
#pragma unroll
  for (int o = 0; o < CO; ++o) {
#pragma unroll
    for (int k = 0; k < 4; ++k) ab[o][k] = 0.f;
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
      for (int f = 0; f < 2; ++f)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[t][o][f][k] = 0.f;
  }
  const int dz = warp / 3, dy = warp % 3;
  // lane addresses: A (voxel, channel half) of g, B of the input halo
  const unsigned oa = 16u * (unsigned)(G::IN + ((lane & 7) + ((lane >> 4) & 1) * 8) * GS + ((lane >> 3) & 1));
  const unsigned ob = 16u * (unsigned)(dz * G::PZ + (dy + ((lane >> 3) & 1)) * G::P + (lane & 7) * G::S + (lane >> 4));
  const bool bias = blockIdx.x == 0 && warp == 4;
  // the accumulators into the share's partials (added from the second time on)
  bool more = false;
  int held = 0;  // tiles in the accumulators
  auto fold = [&] {
    unsigned share = blockIdx.y;
    asm volatile("" : "+r"(share));  // addresses formed here, not held through the loop
    const int cout = 16 * CO;
    float* base = a.part + (size_t)share * 27 * cout * a.cin + 16 * blockIdx.x;
#pragma unroll
    for (int t = 0; t < 3; ++t)
#pragma unroll
      for (int o = 0; o < CO; ++o)
#pragma unroll
        for (int f = 0; f < 2; ++f)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float* q = base + ((size_t)(warp * 3 + t) * cout + o * 16 + gid + 8 * h) * a.cin + f * 8 + tig * 2;
            float2 v = make_float2(acc[t][o][f][2 * h], acc[t][o][f][2 * h + 1]);
            if (more) {
              const float2 u = *reinterpret_cast<const float2*>(q);
              v.x += u.x;
              v.y += u.y;
            }
            *reinterpret_cast<float2*>(q) = v;
            acc[t][o][f][2 * h] = acc[t][o][f][2 * h + 1] = 0.f;
          }
    if (bias && tig == 0)
#pragma unroll
      for (int o = 0; o < CO; ++o)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float* q = a.bpart + (size_t)share * cout + o * 16 + gid + 8 * h;
          *q = ab[o][2 * h] + (more ? *q : 0.f);
        }
#pragma unroll
    for (int o = 0; o < CO; ++o) ab[o][0] = ab[o][1] = ab[o][2] = ab[o][3] = 0.f;
    more = true;
    held = 0;
  };
  int buf = 0;
  long long tile = blockIdx.y;
  table(tile, 0);
  if (tile + gridDim.y < a.ntiles) table(tile + gridDim.y, 1);
  __syncthreads();
  pdl_launch();
  pdl_wait();
  stage(tile, 0);
  cp_commit();
  for (; tile < a.ntiles; tile += gridDim.y, buf ^= 1) {
    if (tile + gridDim.y < a.ntiles) stage(tile + gridDim.y, buf ^ 1);
    cp_commit();
    cp_wait<1>();
    __syncthreads();
    // the table of the tile after the next (this buffer's was read above)
    if (tile + 2 * (long long)gridDim.y < a.ntiles) table(tile + 2 * (long long)gridDim.y, buf);
    const unsigned s0 = sm + 16u * (unsigned)(buf * STAGE);
#pragma unroll 2
    for (int q = 0; q < 16; ++q) {  // two rows of eight voxels each
      const int z = q >> 2, y = (q & 3) * 2;
      unsigned A[CO][4];
#pragma unroll
      for (int o = 0; o < CO; ++o) ldsm4t(A[o], s0 + oa + 16u * (unsigned)(q * 16 * GS + 2 * o));
#pragma unroll
      for (int t = 0; t < 3; ++t) {
        unsigned B[4];
        ldsm4t(B, s0 + ob + 16u * (unsigned)(z * G::PZ + y * G::P + t * G::S));
#pragma unroll
        for (int o = 0; o < CO; ++o) {
          mma_bf16(acc[t][o][0], A[o], B[0], B[1]);
          mma_bf16(acc[t][o][1], A[o], B[2], B[3]);
        }
      }
      if (bias)
#pragma unroll
        for (int o = 0; o < CO; ++o) mma_bf16(ab[o], A[o], 0x3F803F80u, 0x3F803F80u);
    }
    if (++held == kWgFold || tile + gridDim.y >= a.ntiles) fold();
    __syncthreads();  // the buffer is free for the tile after the next
  }
}

// The partials of every layer, summed over their shares in order, into the
// flat FP32 gradient (W[co][ci][tap] of the real channels, then the biases).
// A warp owns 32 consecutive values of a layer's [tap][co][ci] partials.
struct ReduceLayer {
  const float* part;
  const float* bpart;
  int shares, ntap, cout, coutp, cin, cinp;
  long long off;  // of the layer in the flat gradient
  int block0;     // first block of the layer
};
struct ReduceArgs {
  ReduceLayer l[kNL];
  float* grad;
};
constexpr int kRedWarps = 8;
__global__ void __launch_bounds__(32 * kRedWarps) k_grad_reduce(ReduceArgs a) {
  pdl_launch();
  pdl_wait();
  int li = 0;
  while (li + 1 < kNL && (int)blockIdx.x >= a.l[li + 1].block0) ++li;
  const ReduceLayer& L = a.l[li];
  const int nw = L.ntap * L.coutp * L.cinp, total = nw + L.cout;
  const int i = ((int)blockIdx.x - L.block0) * 32 + (threadIdx.x & 31), warp = threadIdx.x >> 5;
  // each warp sums every kRedWarps-th share, then the warps in order
  __shared__ float sh[kRedWarps][32];
  float s = 0.f;
  if (i < total) {
    const float* p = i < nw ? L.part + i : L.bpart + (i - nw);
    const size_t step = i < nw ? (size_t)nw : (size_t)L.coutp;
#pragma unroll 8
    for (int q = warp; q < L.shares; q += kRedWarps) s += p[q * step];
  }
  sh[warp][threadIdx.x & 31] = s;
  __syncthreads();
  if (warp != 0 || i >= total) return;
  s = 0.f;
#pragma unroll
  for (int q = 0; q < kRedWarps; ++q) s += sh[q][threadIdx.x];
  const int nreal = L.cout * L.cin * L.ntap;
  if (i >= nw) {
    a.grad[L.off + nreal + (i - nw)] = s;
    return;
  }
  const int ci = i % L.cinp, co = i / L.cinp % L.coutp, t = i / (L.cinp * L.coutp);
  if (ci < L.cin && co < L.cout) a.grad[L.off + ((size_t)co * L.cin + ci) * L.ntap + t] = s;
}

// ---- elementwise and resampling ---------------------------------------------------
// Back through the 1x1 head: s = slope(post) * (gy w), gy the BF16 gradient of
// y, and the head's own gradients sum gy post, sum gy (FP32 partials per block).
// Thread pairs own the two 8-channel chunks of a voxel.
__global__ void __launch_bounds__(256) k_head_back(const bf16* gy, const bf16* hw /* [8][16], row 0 */, const bf16* post,
                                                   long long nvox, bf16* s, float* part, float* bpart) {
  pdl_launch();
  pdl_wait();
  __shared__ float sh[8][2][9];
  const int half = threadIdx.x & 1;
  const Chunk w = unpack8(__ldg(reinterpret_cast<const uint4*>(hw + 8 * half)));
  float acc[9] = {};
  for (long long i = (blockIdx.x * 256LL + threadIdx.x) >> 1; i < nvox;) {
    float run[9] = {};  // sums of 256 voxels, so that no chain of additions grows with the grid
    for (int n = 0; n < 256 && i < nvox; ++n, i += gridDim.x * 128LL) {
      const float g = __bfloat162float(gy[i]);
      const uint4 pu = __ldg(reinterpret_cast<const uint4*>(post + i * 16 + 8 * half));
      const Chunk p = unpack8(pu);
      Chunk c;
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        c.v[q] = g * w.v[q];
        run[q] += g * p.v[q];
      }
      run[8] += g;
      *reinterpret_cast<uint4*>(s + i * 16 + 8 * half) = act_back(pu, pack8(c));
    }
#pragma unroll
    for (int q = 0; q < 9; ++q) acc[q] += run[q];
  }
#pragma unroll
  for (int q = 0; q < 9; ++q)
#pragma unroll
    for (int o = 16; o > 1; o >>= 1) acc[q] += __shfl_xor_sync(0xffffffffu, acc[q], o);
  if ((threadIdx.x & 31) < 2)
#pragma unroll
    for (int q = 0; q < 9; ++q) sh[threadIdx.x >> 5][half][q] = acc[q];
  __syncthreads();
  if (threadIdx.x < 18) {
    const int h = threadIdx.x / 9, q = threadIdx.x - 9 * h;
    float t = 0.f;
#pragma unroll
    for (int k = 0; k < 8; ++k) t += sh[k][h][q];
    if (q < 8) part[(size_t)blockIdx.x * 16 + 8 * h + q] = t;
    else if (h == 0) bpart[blockIdx.x] = t;
  }
}
// Back through nearest doubling and the activation below it: the sum of the 8
// fine children, rounded to BF16, times the slope at post.  c channels, coarse
// grid m.
__global__ void __launch_bounds__(256) k_up_back(const bf16* gout, int c, int m, long long total /* chunks */,
                                                 const bf16* post, bf16* s) {
  pdl_launch();
  pdl_wait();
  const int n = 2 * m, nc = c / 8;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < total; i += gridDim.x * 256LL) {
    const int ch = (int)(i % nc);
    const long long v = i / nc;
    const int x = (int)(v % m), y = (int)(v / m % m), z = (int)(v / ((long long)m * m) % m);
    const long long b = v / ((long long)m * m * m);
    Chunk t = {};
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const long long f = ((b * n + 2 * z + (q >> 2)) * n + 2 * y + ((q >> 1) & 1)) * n + 2 * x + (q & 1);
      const Chunk u = unpack8(__ldg(reinterpret_cast<const uint4*>(gout + f * c + 8 * ch)));
#pragma unroll
      for (int k = 0; k < 8; ++k) t.v[k] += u.v[k];
    }
    *reinterpret_cast<uint4*>(s + i * 8) = act_back(__ldg(reinterpret_cast<const uint4*>(post + i * 8)), pack8(t));
  }
}
// Back through the 2 x 2 x 2 mean, added to the gradient that reached the same
// activations over the skip connection, times the slope at post.  Fine grid n.
__global__ void __launch_bounds__(256) k_pool_back(const bf16* gout, int c, int n, long long total /* chunks */,
                                                   const bf16* gskip, const bf16* post, bf16* s) {
  pdl_launch();
  pdl_wait();
  const int m = n / 2, nc = c / 8;
  for (long long i = blockIdx.x * 256LL + threadIdx.x; i < total; i += gridDim.x * 256LL) {
    const int ch = (int)(i % nc);
    const long long v = i / nc;
    const int x = (int)(v % n), y = (int)(v / n % n), z = (int)(v / ((long long)n * n) % n);
    const long long b = v / ((long long)n * n * n);
    const long long q = ((b * m + z / 2) * m + y / 2) * m + x / 2;
    const Chunk g = unpack8(__ldg(reinterpret_cast<const uint4*>(gout + q * c + 8 * ch)));
    Chunk t = unpack8(__ldg(reinterpret_cast<const uint4*>(gskip + i * 8)));
#pragma unroll
    for (int k = 0; k < 8; ++k) t.v[k] = g.v[k] * 0.125f + t.v[k];
    *reinterpret_cast<uint4*>(s + i * 8) = act_back(__ldg(reinterpret_cast<const uint4*>(post + i * 8)), pack8(t));
  }
}

// per-sample FP64 sum of squares of b (n3 values per sample)
template <typename T>
__global__ void k_sumsq(const T* b, long long n3, double* out) {
  __shared__ double sh[32];
  const int s = blockIdx.y;
  double acc = 0.0;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n3; i += (long long)gridDim.x * blockDim.x) {
    const double x = (double)b[(size_t)s * n3 + i];
    acc += x * x;
  }
  const double r = block_reduce<false>(acc, sh);
  if (threadIdx.x == 0) out[(size_t)s * gridDim.x + blockIdx.x] = r;
}
constexpr int kSumBlocks = 64;  // partials of sum b^2 per sample
// The scale s = sqrt(mean b^2) of sample `q` from its partials (one warp, the
// result in every lane)
__device__ __forceinline__ double sample_scale(const double* part, long long q, long long n3) {
  const int lane = threadIdx.x & 31;
  const double* p = part + q * kSumBlocks;
  return sqrt(warp_sum(p[lane] + p[lane + 32]) / (double)n3);
}
// x0[v][0] = b / s, other 15 channels 0; optional normalised target t = psi / s.
// A grid row of blocks per sample; its first block keeps s.
template <typename T>
__global__ void __launch_bounds__(256) k_pack(const T* b, const T* psi, long long n3, const double* part, double* scale,
                                              double out_scale, bf16* x0, float* tgt) {
  __shared__ double sh[2];  // 1 / s, 1 / (s out_scale): one thread's divisions
  pdl_launch();
  pdl_wait();
  const long long s = blockIdx.y;
  if (threadIdx.x < 32) {
    const double sc = sample_scale(part, s, n3);
    if (threadIdx.x == 0) {
      sh[0] = sc > 0.0 ? 1.0 / sc : 0.0;
      sh[1] = sh[0] / out_scale;
      if (blockIdx.x == 0) scale[s] = sc;
    }
  }
  __syncthreads();
  const double inv = sh[0], invt = sh[1];
  for (long long v = blockIdx.x * 256LL + threadIdx.x; v < n3; v += gridDim.x * 256LL) {
    const long long i = s * n3 + v;
    uint4* o = reinterpret_cast<uint4*>(x0 + i * 16);
    o[0] = make_uint4(pack2((float)((double)b[i] * inv), 0.f), 0u, 0u, 0u);
    o[1] = make_uint4(0u, 0u, 0u, 0u);
    if (tgt) tgt[i] = (float)((double)psi[i] * invt);
  }
}
// MSE over batch x n3 of y vs t; gy = 2 (y - t) / count in BF16
__global__ void k_loss(const float* y, const float* t, long long total, bf16* gy, double* part) {
  __shared__ double sh[32];
  pdl_launch();
  pdl_wait();
  double acc = 0.0;
  const float inv = 2.f / (float)total;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    acc += (double)d * d;
    gy[i] = __float2bfloat16(d * inv);
  }
  const double r = block_reduce<false>(acc, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = r;
}
// Energy norm of the error on the periodic n^3 grid (unit spacing) over
// batch samples: loss = sum d (6 d - sum of the six neighbours) / count,
// d = y - t; gy = 2 (6 d - sum of the six neighbours) / count.
__global__ void k_loss_energy(const float* y, const float* t, int n, long long total, bf16* gy, double* part) {
  __shared__ double sh[32];
  pdl_launch();
  pdl_wait();
  double acc = 0.0;
  const float inv = 2.f / (float)total;
  const long long n3 = (long long)n * n * n;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const long long s0 = (i / n3) * n3;
    const int v = (int)(i - s0);
    const int x = v % n, yy = (v / n) % n, z = v / (n * n);
    auto d = [&](int xx, int yv, int zz) {
      const long long q = s0 + ((long long)zz * n + yv) * n + xx;
      return y[q] - t[q];
    };
    const float d0 = d(x, yy, z);
    const int xm = x == 0 ? n - 1 : x - 1, xp = x == n - 1 ? 0 : x + 1;
    const int ym = yy == 0 ? n - 1 : yy - 1, yp = yy == n - 1 ? 0 : yy + 1;
    const int zm = z == 0 ? n - 1 : z - 1, zp = z == n - 1 ? 0 : z + 1;
    const float ld = 6.f * d0 - (d(xm, yy, z) + d(xp, yy, z)) - (d(x, ym, z) + d(x, yp, z)) -
                     (d(x, yy, zm) + d(x, yy, zp));
    acc += (double)d0 * ld;
    gy[i] = __float2bfloat16(ld * inv);
  }
  const double r = block_reduce<false>(acc, sh);
  if (threadIdx.x == 0) part[blockIdx.x] = r;
}
__global__ void k_sum_part(const double* part, int n, double* out) {
  __shared__ double sh[32];
  pdl_launch();
  pdl_wait();
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += part[i];
  const double r = block_reduce<false>(acc, sh);
  if (threadIdx.x == 0) *out = r;
}
// psi_0 = s (y - mean y), the mean from the head's tile sums.  A grid row of
// blocks per sample.
template <typename T>
__global__ void __launch_bounds__(256) k_unpack(const float* y, long long n3, const double* scale, double out_scale,
                                                const double* ysum, int tiles, T* psi) {
  __shared__ double sh[32];
  __shared__ double mean;
  pdl_launch();
  pdl_wait();
  const long long s = blockIdx.y;
  double t = 0.0;
  for (int q = threadIdx.x; q < tiles; q += 256) t += ysum[s * tiles + q];
  t = block_reduce<false>(t, sh);
  if (threadIdx.x == 0) mean = t / (double)n3;
  __syncthreads();
  const double m = mean, sc = scale[s] * out_scale;
  for (long long v = blockIdx.x * 256LL + threadIdx.x; v < n3; v += gridDim.x * 256LL)
    psi[s * n3 + v] = (T)(sc * ((double)y[s * n3 + v] - m));
}

// master FP32 (flat) -> forward BF16 [co / 16][tap][16][ci_pad16 + 8] and
// backward BF16 [ci / 16][flipped tap][16][co_pad16 + 8] weights (the padding
// stays zero), FP32 bias; the 1x1 head forward only, as [co_pad8][ci_pad16].
// A grid row of blocks per layer.
struct WeightLayer {
  bf16 *wf, *wb;
  float* bias;
  long long off;
  int cin, cout, ntap;
};
struct WeightArgs {
  WeightLayer l[kNL];
  const float* flat;
};
__global__ void k_weights(WeightArgs a) {
  const WeightLayer& L = a.l[blockIdx.y];
  const float* flat = a.flat + L.off;
  const int cinp = pad16(L.cin), coutp = pad8(L.cout), coutp16 = pad16(L.cout), ntap = L.ntap;
  const int total = ntap * coutp16 * cinp;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    const int ci = i % cinp, co = (i / cinp) % coutp16, t = i / (cinp * coutp16);
    const float w = (co < L.cout && ci < L.cin) ? flat[((size_t)co * L.cin + ci) * ntap + t] : 0.f;
    if (ntap == 1) {
      if (co < coutp) L.wf[(size_t)co * cinp + ci] = __float2bfloat16(w);
      continue;
    }
    L.wf[(((size_t)(co >> 4) * ntap + t) * 16 + (co & 15)) * (cinp + 8) + ci] = __float2bfloat16(w);
    // backward data: out channel = ci, in channel = co, tap flipped
    L.wb[(((size_t)(ci >> 4) * ntap + ntap - 1 - t) * 16 + (ci & 15)) * (coutp16 + 8) + co] = __float2bfloat16(w);
  }
  if (blockIdx.x == 0)
    for (int co = threadIdx.x; co < coutp; co += blockDim.x)
      L.bias[co] = co < L.cout ? flat[(size_t)L.cout * L.cin * ntap + co] : 0.f;
}

__global__ void k_adam(float* w, const float* g, float* m, float* v, long long n, float lr, float b1, float b2,
                       float eps, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    w[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

}  // namespace
}  // namespace les

// ============================================================================
// host side
// ============================================================================
using namespace les;

struct les_unet {
  int n = 0, batch = 0;
  cudaStream_t st = nullptr;
  char* ws = nullptr;
  size_t ws_bytes = 0;
  int nsm = 152;
  size_t nparams = 0;
  size_t woff[kNL] = {};  // flat offsets of each layer's W (bias follows)
  // device buffers
  float *master = nullptr, *grad = nullptr, *m1 = nullptr, *m2 = nullptr;
  bf16* wf[kNL] = {};
  bf16* wb[kNL] = {};
  float* bias[kNL] = {};
  bf16 *x0, *a1a, *e1, *p1, *a2a, *e2, *p2, *a3a, *e3, *a4a, *g2, *a5a, *g1, *gy;
  float *y, *tgt;
  bf16 *G0, *G1, *G2, *G3, *G4;  // gradient scratch
  float *wpart[kNL] = {}, *bpart[kNL] = {};  // weight and bias gradient partials of the layers' shares
  double *scale, *ysum, *dpart, *loss;
  int step = 0;
  int loss_kind = 0;       // 0 mean squared error, 1 energy norm of the error
  double out_scale = 1.0;  // psi_0 = s * out_scale * (y - mean y)
  std::string err;
  Profiler* prof = nullptr;
};

namespace {

struct Carve {
  char* base;
  size_t off = 0;
  bool dry;
  template <typename P>
  P* take(size_t bytes) {
    off = (off + 255) / 256 * 256;
    P* p = dry ? nullptr : reinterpret_cast<P*>(base + off);
    off += bytes;
    return p;
  }
};

int level_of(int l) { return (l <= L_E1B || l >= L_D1A) ? 0 : ((l <= L_E2B || l >= L_D2A) ? 1 : 2); }
long long tiles_of(int cfg, int n, long long batch) {
  const int zy = cfg ? 8 : 4;
  const long long t = (n + zy - 1) / zy;
  return batch * ((n + 3) / 4) * t * t;
}
// Shares of the voxel tiles in a weight gradient: a wave of blocks per slice of
// 16 input channels, but no more partials than 2 M floats (8 MB).
int wgrad_shares(const les_unet* u, int l, long long batch) {
  const LayerDef& L = kLayers[l];
  if (l == L_HEAD) return 2 * u->nsm;
  const int cinp = pad16(L.cin);
  const long long tiles = tiles_of(1, u->n >> level_of(l), batch);
  const long long cap = std::max<long long>(1, (2LL << 20) / (27LL * L.cout * cinp));
  const long long wave = std::max<long long>(1, 2LL * u->nsm / (cinp / 16));
  return (int)std::max<long long>(1, std::min(tiles, std::min(cap, wave)));
}

size_t layout(les_unet* u, char* base, bool dry) {
  Carve c{base, 0, dry};
  const size_t n3 = (size_t)u->n * u->n * u->n, B = (size_t)u->batch;
  const size_t v1 = B * n3, v2 = v1 / 8, v3 = v2 / 8;
  size_t np = 0;
  for (int l = 0; l < kNL; ++l) {
    u->woff[l] = np;
    np += (size_t)kLayers[l].cout * kLayers[l].cin * kLayers[l].k * kLayers[l].k * kLayers[l].k + kLayers[l].cout;
  }
  u->nparams = np;
  u->master = c.take<float>(np * 4);
  u->grad = c.take<float>(np * 4);
  u->m1 = c.take<float>(np * 4);
  u->m2 = c.take<float>(np * 4);
  for (int l = 0; l < kNL; ++l) {
    const LayerDef& L = kLayers[l];
    const int nt = L.k * L.k * L.k, cinp = pad16(L.cin), cop = pad8(L.cout), cop16 = pad16(L.cout);
    u->wf[l] = c.take<bf16>((size_t)nt * cop16 * (cinp + 8) * 2);
    u->wb[l] = c.take<bf16>((size_t)nt * cinp * (cop16 + 8) * 2);
    u->bias[l] = c.take<float>((size_t)cop * 4);
    const size_t sh = (size_t)wgrad_shares(u, l, u->batch);
    u->wpart[l] = c.take<float>(sh * (l == L_HEAD ? 16 : (size_t)nt * L.cout * cinp) * 4);
    u->bpart[l] = c.take<float>(sh * (size_t)L.cout * 4);
  }
  u->x0 = c.take<bf16>(v1 * 16 * 2);
  u->a1a = c.take<bf16>(v1 * 16 * 2);
  u->e1 = c.take<bf16>(v1 * 16 * 2);
  u->p1 = c.take<bf16>(v2 * 16 * 2);
  u->a2a = c.take<bf16>(v2 * 32 * 2);
  u->e2 = c.take<bf16>(v2 * 32 * 2);
  u->p2 = c.take<bf16>(v3 * 32 * 2);
  u->a3a = c.take<bf16>(v3 * 64 * 2);
  u->e3 = c.take<bf16>(v3 * 64 * 2);
  u->a4a = c.take<bf16>(v2 * 32 * 2);
  u->g2 = c.take<bf16>(v2 * 32 * 2);
  u->a5a = c.take<bf16>(v1 * 16 * 2);
  u->g1 = c.take<bf16>(v1 * 16 * 2);
  u->gy = c.take<bf16>(v1 * 2);
  u->y = c.take<float>(v1 * 4);
  u->tgt = c.take<float>(v1 * 4);
  u->G0 = c.take<bf16>(v1 * 16 * 2);  // gradient at e1 over the skip connection
  u->G1 = c.take<bf16>(v2 * 32 * 2);  // ... at e2
  u->G2 = c.take<bf16>(v1 * 32 * 2);  // gradient on its way between levels
  u->G3 = c.take<bf16>(v1 * 16 * 2);  // gradients before the activations of a block's second
  u->G4 = c.take<bf16>(v1 * 16 * 2);  // ... and first convolution
  u->scale = c.take<double>(B * 8);
  u->ysum = c.take<double>((size_t)tiles_of(0, u->n, u->batch) * 8);
  u->dpart = c.take<double>((4096 + B * kSumBlocks) * 8);
  u->loss = c.take<double>(8);
  return c.off + 256;
}

int unet_fail(les_unet* u, cudaError_t e, const char* where) {
  u->err = std::string(where) + ": " + cudaGetErrorString(e);
  return LES_ERR_CUDA;
}

unsigned eblocks(long long total) { return (unsigned)std::min<long long>((total + 255) / 256, 8192); }

// launch that may start while the kernel before it in the stream drains (the
// kernel waits with pdl_wait)
template <typename... K, typename... A>
cudaError_t launch_pdl(void (*k)(K...), dim3 grid, int threads, size_t smem, cudaStream_t st, A... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3((unsigned)threads);
  c.dynamicSmemBytes = smem;
  c.stream = st;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  c.attrs = &at;
  c.numAttrs = 1;
  return cudaLaunchKernelEx(&c, k, K(args)...);
}

using ConvKernel = void (*)(ConvArgs);
struct ConvChoice {
  ConvKernel k = nullptr;
  size_t smem = 0;
};
template <int CFG, int KC, int NFB>
ConvChoice choice() {
  return {k_conv<CFG, KC, NFB>, conv_smem<CFG, KC, NFB>()};
}
template <int KC>
ConvChoice choice_kc(int cfg, int nfb) {
  if (cfg) return nfb == 4 ? choice<1, KC, 4>() : choice<1, KC, 2>();
  return nfb == 4 ? choice<0, KC, 4>() : choice<0, KC, 2>();
}
ConvChoice conv_kernel(int kc, int cfg, int nfb) {
  switch (kc) {
    case 1: return choice_kc<1>(cfg, nfb);
    case 2: return choice_kc<2>(cfg, nfb);
    case 3: return choice_kc<3>(cfg, nfb);
    case 4: return choice_kc<4>(cfg, nfb);
    case 6: return choice_kc<6>(cfg, nfb);
    default: return {};
  }
}
constexpr size_t kConvSmemMax = 227 * 1024 - 4096;  // beside the tables

// shared-memory limits of the kernels, once per network
cudaError_t kernel_limits() {
  for (int kc : {1, 2, 3, 4, 6})
    for (int cfg : {0, 1})
      for (int nfb : {2, 4}) {
        const ConvChoice c = conv_kernel(kc, cfg, nfb);
        if (c.smem > kConvSmemMax) continue;
        const cudaError_t e = cudaFuncSetAttribute(c.k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)c.smem);
        if (e != cudaSuccess) return e;
      }
  cudaError_t e = cudaFuncSetAttribute(k_wgrad<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wgrad_smem<1>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_wgrad<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wgrad_smem<2>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_wgrad<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)wgrad_smem<4>());
  return e;
}

// The widest tile and output slice that still give every SM a block: large
// tiles halve the weight and halo loads per voxel, small ones fill the chip on
// the coarse levels.
cudaError_t conv(les_unet* u, int n, int batch, ConvArgs a) {
  const int kc = (a.c0 + a.c1) / 16, cout = a.oc0 + a.oc1;
  a.n = n;
  static constexpr int order[4][2] = {{1, 4}, {1, 2}, {0, 4}, {0, 2}};
  int cfg = 0, nfb = 2;
  for (const auto& o : order) {
    if (cout % (8 * o[1]) || conv_kernel(kc, o[0], o[1]).smem > kConvSmemMax) continue;
    if (tiles_of(o[0], n, batch) * (cout / (8 * o[1])) < u->nsm - u->nsm / 4) continue;
    cfg = o[0], nfb = o[1];
    break;
  }
  const ConvChoice c = conv_kernel(kc, cfg, nfb);
  if (!c.k) return cudaErrorInvalidValue;
  a.tz = (n + 3) / 4;
  a.ty = a.tx = cfg ? (n + 7) / 8 : (n + 3) / 4;
  ProfScope ps(u->prof, KI_UNET_CONV, u->st);
  return launch_pdl(c.k, dim3((unsigned)tiles_of(cfg, n, batch), (unsigned)(cout / (8 * nfb))), cfg ? 256 : 128, c.smem,
                    u->st, a);
}
// tiles per sample of the last convolution (whose tiles sum y)
int head_tiles(const les_unet* u, int batch) {
  const long long t1 = tiles_of(1, u->n, batch);
  const bool big = t1 >= u->nsm - u->nsm / 4;
  return (int)(tiles_of(big ? 1 : 0, u->n, 1));
}

// forward convolution of layer l
cudaError_t conv_fwd(les_unet* u, int l, int n, int batch, const bf16* in0, int c0, int up0, const bf16* in1, int c1,
                     bf16* out, bf16* pool) {
  ConvArgs a{};
  a.in0 = in0, a.c0 = c0, a.up0 = up0, a.in1 = in1, a.c1 = c1;
  a.w = u->wf[l];
  a.bias = u->bias[l];
  a.out0 = out, a.oc0 = kLayers[l].cout;
  a.pool = pool;
  if (l == L_D1B) a.hw = u->wf[L_HEAD], a.hb = u->bias[L_HEAD], a.y = u->y, a.ysum = u->ysum;
  return conv(u, n, batch, a);
}
// input gradient of layer l from g (its pre-activation gradient), times the
// slope of the activations post where given
cudaError_t conv_back(les_unet* u, int l, int n, int batch, const bf16* g, const bf16* post, bf16* out0, int oc0,
                      bf16* out1, int oc1) {
  ConvArgs a{};
  a.in0 = g, a.c0 = kLayers[l].cout;
  a.w = u->wb[l];
  a.post = post;
  a.out0 = out0, a.oc0 = oc0, a.out1 = out1, a.oc1 = oc1;
  return conv(u, n, batch, a);
}

// weight and bias gradient partials of layer l given g (gradient at its pre-activation)
cudaError_t wgrad(les_unet* u, int l, int n, int batch, const bf16* g, const bf16* in0, int c0, int up0, const bf16* in1,
                  int c1) {
  const LayerDef& L = kLayers[l];
  WgradArgs a{g, in0, c0, up0, in1, c1, u->wpart[l], u->bpart[l], c0 + c1, n, (n + 7) / 8, (n + 7) / 8, (n + 3) / 4, 0};
  a.ntiles = tiles_of(1, n, batch);
  const dim3 grid((unsigned)((c0 + c1) / 16), (unsigned)wgrad_shares(u, l, batch));
  ProfScope ps(u->prof, KI_UNET_WGRAD, u->st);
  switch (L.cout / 16) {
    case 1: return launch_pdl(k_wgrad<1>, grid, 32 * kWgWarps, wgrad_smem<1>(), u->st, a);
    case 2: return launch_pdl(k_wgrad<2>, grid, 32 * kWgWarps, wgrad_smem<2>(), u->st, a);
    case 4: return launch_pdl(k_wgrad<4>, grid, 32 * kWgWarps, wgrad_smem<4>(), u->st, a);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t refresh_weights(les_unet* u) {
  WeightArgs a;
  a.flat = u->master;
  int most = 0;
  for (int l = 0; l < kNL; ++l) {
    const LayerDef& L = kLayers[l];
    a.l[l] = {u->wf[l], u->wb[l], u->bias[l], (long long)u->woff[l], L.cin, L.cout, L.k * L.k * L.k};
    most = std::max(most, L.k * L.k * L.k * pad16(L.cout) * pad16(L.cin));
  }
  k_weights<<<dim3((unsigned)((most + 1023) / 1024), kNL), 256, 0, u->st>>>(a);
  return cudaGetLastError();
}

#define CK(x)                             \
  if ((e = (x)) != cudaSuccess) return e;
// forward pass on the packed input x0 (batch b); y receives the head output
cudaError_t forward(les_unet* u, int b) {
  const int n1 = u->n, n2 = n1 / 2, n3 = n2 / 2;
  cudaError_t e;
  CK(conv_fwd(u, L_E1A, n1, b, u->x0, 16, 0, nullptr, 0, u->a1a, nullptr));
  CK(conv_fwd(u, L_E1B, n1, b, u->a1a, 16, 0, nullptr, 0, u->e1, u->p1));
  CK(conv_fwd(u, L_E2A, n2, b, u->p1, 16, 0, nullptr, 0, u->a2a, nullptr));
  CK(conv_fwd(u, L_E2B, n2, b, u->a2a, 32, 0, nullptr, 0, u->e2, u->p2));
  CK(conv_fwd(u, L_E3A, n3, b, u->p2, 32, 0, nullptr, 0, u->a3a, nullptr));
  CK(conv_fwd(u, L_E3B, n3, b, u->a3a, 64, 0, nullptr, 0, u->e3, nullptr));
  CK(conv_fwd(u, L_D2A, n2, b, u->e3, 64, 1, u->e2, 32, u->a4a, nullptr));
  CK(conv_fwd(u, L_D2B, n2, b, u->a4a, 32, 0, nullptr, 0, u->g2, nullptr));
  CK(conv_fwd(u, L_D1A, n1, b, u->g2, 32, 1, u->e1, 16, u->a5a, nullptr));
  CK(conv_fwd(u, L_D1B, n1, b, u->a5a, 16, 0, nullptr, 0, u->g1, nullptr));
  return cudaSuccess;
}

// full backward from gy; fills u->grad.  Per block B(.; a -> c): G3 holds the
// gradient before the second activation, G4 before the first.
cudaError_t backward(les_unet* u, int b) {
  const int n1 = u->n, n2 = n1 / 2, n3 = n2 / 2;
  const long long v1 = (long long)b * n1 * n1 * n1, v2 = v1 / 8, v3 = v2 / 8;
  cudaError_t e;
  auto blocks = [&](long long total) { return dim3((unsigned)std::min<long long>((total + 255) / 256, 16LL * u->nsm)); };
  const int hsh = wgrad_shares(u, L_HEAD, b);
  CK(launch_pdl(k_head_back, dim3((unsigned)hsh), 256, 0, u->st, u->gy, u->wf[L_HEAD], u->g1, v1, u->G3, u->wpart[L_HEAD],
                u->bpart[L_HEAD]));
  CK(wgrad(u, L_D1B, n1, b, u->G3, u->a5a, 16, 0, nullptr, 0));
  CK(conv_back(u, L_D1B, n1, b, u->G3, u->a5a, u->G4, 16, nullptr, 0));
  CK(wgrad(u, L_D1A, n1, b, u->G4, u->g2, 32, 1, u->e1, 16));
  CK(conv_back(u, L_D1A, n1, b, u->G4, nullptr, u->G2, 32, u->G0, 16));
  CK(launch_pdl(k_up_back, blocks(v2 * 4), 256, 0, u->st, u->G2, 32, n2, v2 * 4, u->g2, u->G3));
  CK(wgrad(u, L_D2B, n2, b, u->G3, u->a4a, 32, 0, nullptr, 0));
  CK(conv_back(u, L_D2B, n2, b, u->G3, u->a4a, u->G4, 32, nullptr, 0));
  CK(wgrad(u, L_D2A, n2, b, u->G4, u->e3, 64, 1, u->e2, 32));
  CK(conv_back(u, L_D2A, n2, b, u->G4, nullptr, u->G2, 64, u->G1, 32));
  CK(launch_pdl(k_up_back, blocks(v3 * 8), 256, 0, u->st, u->G2, 64, n3, v3 * 8, u->e3, u->G3));
  CK(wgrad(u, L_E3B, n3, b, u->G3, u->a3a, 64, 0, nullptr, 0));
  CK(conv_back(u, L_E3B, n3, b, u->G3, u->a3a, u->G4, 64, nullptr, 0));
  CK(wgrad(u, L_E3A, n3, b, u->G4, u->p2, 32, 0, nullptr, 0));
  CK(conv_back(u, L_E3A, n3, b, u->G4, nullptr, u->G2, 32, nullptr, 0));
  CK(launch_pdl(k_pool_back, blocks(v2 * 4), 256, 0, u->st, u->G2, 32, n2, v2 * 4, u->G1, u->e2, u->G3));
  CK(wgrad(u, L_E2B, n2, b, u->G3, u->a2a, 32, 0, nullptr, 0));
  CK(conv_back(u, L_E2B, n2, b, u->G3, u->a2a, u->G4, 32, nullptr, 0));
  CK(wgrad(u, L_E2A, n2, b, u->G4, u->p1, 16, 0, nullptr, 0));
  CK(conv_back(u, L_E2A, n2, b, u->G4, nullptr, u->G2, 16, nullptr, 0));
  CK(launch_pdl(k_pool_back, blocks(v1 * 2), 256, 0, u->st, u->G2, 16, n1, v1 * 2, u->G0, u->e1, u->G3));
  CK(wgrad(u, L_E1B, n1, b, u->G3, u->a1a, 16, 0, nullptr, 0));
  CK(conv_back(u, L_E1B, n1, b, u->G3, u->a1a, u->G4, 16, nullptr, 0));
  CK(wgrad(u, L_E1A, n1, b, u->G4, u->x0, 16, 0, nullptr, 0));
  ReduceArgs r;
  r.grad = u->grad;
  int blk = 0;
  for (int l = 0; l < kNL; ++l) {
    const LayerDef& L = kLayers[l];
    const int nt = L.k * L.k * L.k, cinp = pad16(L.cin);
    r.l[l] = {u->wpart[l], u->bpart[l], wgrad_shares(u, l, b), nt, L.cout, L.cout, L.cin, cinp, (long long)u->woff[l], blk};
    blk += (nt * L.cout * cinp + L.cout + 31) / 32;
  }
  return launch_pdl(k_grad_reduce, dim3((unsigned)blk), 32 * kRedWarps, 0, u->st, r);
}
#undef CK

template <typename T>
cudaError_t pack_inputs(les_unet* u, const T* b, const T* psi, int batch) {
  const long long n3 = (long long)u->n * u->n * u->n;
  // an ordinary launch: whatever wrote the weights is complete before the
  // chain of overlapping launches begins
  k_sumsq<T><<<dim3(kSumBlocks, batch), 256, 0, u->st>>>(b, n3, u->dpart + 4096);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const unsigned bx = (unsigned)std::min<long long>((n3 + 255) / 256, std::max(1, 16 * u->nsm / batch));
  return launch_pdl(k_pack<T>, dim3(bx, (unsigned)batch), 256, 0, u->st, b, psi, n3, u->dpart + 4096, u->scale,
                    u->out_scale, u->x0, psi ? u->tgt : (float*)nullptr);
}

template <typename T>
int run_forward(les_unet* u, const T* b, int batch, T* psi0) {
  cudaError_t e;
  if ((e = pack_inputs<T>(u, b, (const T*)nullptr, batch)) != cudaSuccess) return unet_fail(u, e, "pack");
  if ((e = forward(u, batch)) != cudaSuccess) return unet_fail(u, e, "forward");
  const long long n3 = (long long)u->n * u->n * u->n;
  const unsigned bx = (unsigned)std::min<long long>((n3 + 255) / 256, std::max(1, 16 * u->nsm / batch));
  e = launch_pdl(k_unpack<T>, dim3(bx, (unsigned)batch), 256, 0, u->st, u->y, n3, u->scale, u->out_scale, u->ysum,
                 head_tiles(u, batch), psi0);
  return e == cudaSuccess ? LES_OK : unet_fail(u, e, "unpack");
}

template <typename T>
int run_loss_grad(les_unet* u, const T* b, const T* psi, int batch, double* loss) {
  cudaError_t e;
  if ((e = pack_inputs<T>(u, b, psi, batch)) != cudaSuccess) return unet_fail(u, e, "pack");
  if ((e = forward(u, batch)) != cudaSuccess) return unet_fail(u, e, "forward");
  const long long total = (long long)batch * u->n * u->n * u->n;
  const int nb = (int)std::min<long long>((total + 255) / 256, 4096);
  if (u->loss_kind == 1)
    e = launch_pdl(k_loss_energy, dim3((unsigned)nb), 256, 0, u->st, u->y, u->tgt, u->n, total, u->gy, u->dpart);
  else e = launch_pdl(k_loss, dim3((unsigned)nb), 256, 0, u->st, u->y, u->tgt, total, u->gy, u->dpart);
  if (e == cudaSuccess) e = launch_pdl(k_sum_part, dim3(1), 256, 0, u->st, u->dpart, nb, u->loss);
  if (e == cudaSuccess) e = backward(u, batch);
  if (e != cudaSuccess) return unet_fail(u, e, "backward");
  if (loss) {
    double h = 0;
    if ((e = cudaMemcpyAsync(&h, u->loss, 8, cudaMemcpyDeviceToHost, u->st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(u->st)) != cudaSuccess)
      return unet_fail(u, e, "loss readback");
    *loss = h / (double)total;
  }
  return LES_OK;
}

int check_n(int n) { return n >= 8 && n % 4 == 0 && n <= 512; }

}  // namespace

namespace les {
// used by the solver handle for LES_WARM_LEARNED
int unet_predict(les_unet* u, int precision, const void* b, void* psi0, cudaStream_t st, std::string* err) {
  u->st = st;
  const int rc = precision == 64 ? run_forward<double>(u, (const double*)b, 1, (double*)psi0)
                                 : run_forward<float>(u, (const float*)b, 1, (float*)psi0);
  if (rc != LES_OK && err) *err = u->err;
  return rc;
}
int unet_grid(const les_unet* u) { return u ? u->n : 0; }
}  // namespace les

extern "C" {

int64_t les_unet_param_count(void) {
  int64_t np = 0;
  for (int l = 0; l < kNL; ++l)
    np += (int64_t)kLayers[l].cout * kLayers[l].cin * kLayers[l].k * kLayers[l].k * kLayers[l].k + kLayers[l].cout;
  return np;
}

int les_unet_workspace_bytes(int32_t n, int32_t batch, size_t* bytes) {
  if (!bytes || !check_n(n) || batch < 1 || batch > 4096) return LES_ERR_INVALID_ARG;
  les_unet tmp;
  tmp.n = n;
  tmp.batch = batch;
  *bytes = layout(&tmp, nullptr, true);
  return LES_OK;
}

int les_unet_create(int32_t n, int32_t batch, void* workspace, size_t bytes, void* stream, les_unet** out) {
  if (!out) return LES_ERR_INVALID_ARG;
  *out = nullptr;
  size_t need = 0;
  if (les_unet_workspace_bytes(n, batch, &need) != LES_OK || !workspace || bytes < need ||
      ((uintptr_t)workspace % 256) != 0)
    return LES_ERR_INVALID_ARG;
  les_unet* u = new (std::nothrow) les_unet();
  if (!u) return LES_ERR_INVALID_ARG;
  u->n = n;
  u->batch = batch;
  u->st = (cudaStream_t)stream;
  u->ws = (char*)workspace;
  u->ws_bytes = bytes;
  layout(u, u->ws, false);
  cudaError_t e = kernel_limits();
  if (e == cudaSuccess) e = cudaMemsetAsync(u->ws, 0, need, u->st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(u->st);
  if (e != cudaSuccess) {
    delete u;
    return LES_ERR_CUDA;
  }
  *out = u;
  return LES_OK;
}

void les_unet_destroy(les_unet* u) { delete u; }

int les_unet_set_stream(les_unet* u, void* stream) {
  if (!u) return LES_ERR_INVALID_ARG;
  u->st = (cudaStream_t)stream;
  return LES_OK;
}

int les_unet_set_weights(les_unet* u, const float* w, int32_t on_device) {
  if (!u || !w) return LES_ERR_INVALID_ARG;
  cudaError_t e = cudaMemcpyAsync(u->master, w, u->nparams * 4,
                                  on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, u->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(u->m1, 0, u->nparams * 4, u->st);
  if (e == cudaSuccess) e = cudaMemsetAsync(u->m2, 0, u->nparams * 4, u->st);
  if (e == cudaSuccess) e = refresh_weights(u);
  if (e == cudaSuccess && !on_device) e = cudaStreamSynchronize(u->st);
  u->step = 0;
  return e == cudaSuccess ? LES_OK : unet_fail(u, e, "set_weights");
}

int les_unet_get_weights(les_unet* u, float* w, int32_t on_device) {
  if (!u || !w) return LES_ERR_INVALID_ARG;
  cudaError_t e = cudaMemcpyAsync(w, u->master, u->nparams * 4,
                                  on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, u->st);
  if (e == cudaSuccess && !on_device) e = cudaStreamSynchronize(u->st);
  return e == cudaSuccess ? LES_OK : unet_fail(u, e, "get_weights");
}

int les_unet_forward(les_unet* u, int32_t precision, const void* d_b, int32_t batch, void* d_psi0) {
  if (!u || !d_b || !d_psi0 || batch < 1 || batch > u->batch || (precision != 32 && precision != 64))
    return LES_ERR_INVALID_ARG;
  return precision == 64 ? run_forward<double>(u, (const double*)d_b, batch, (double*)d_psi0)
                         : run_forward<float>(u, (const float*)d_b, batch, (float*)d_psi0);
}

int les_unet_loss_grad(les_unet* u, int32_t precision, const void* d_b, const void* d_psi, int32_t batch,
                       double* loss, float* d_grad) {
  if (!u || !d_b || !d_psi || batch < 1 || batch > u->batch || (precision != 32 && precision != 64))
    return LES_ERR_INVALID_ARG;
  int rc = precision == 64 ? run_loss_grad<double>(u, (const double*)d_b, (const double*)d_psi, batch, loss)
                           : run_loss_grad<float>(u, (const float*)d_b, (const float*)d_psi, batch, loss);
  if (rc == LES_OK && d_grad) {
    cudaError_t e = cudaMemcpyAsync(d_grad, u->grad, u->nparams * 4, cudaMemcpyDeviceToDevice, u->st);
    if (e != cudaSuccess) return unet_fail(u, e, "grad copy");
  }
  return rc;
}

int les_unet_train_step(les_unet* u, int32_t precision, const void* d_b, const void* d_psi, int32_t batch, float lr,
                        double* loss) {
  int rc = les_unet_loss_grad(u, precision, d_b, d_psi, batch, loss, nullptr);
  if (rc != LES_OK) return rc;
  u->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)u->step), c2 = 1.f - std::pow(b2, (float)u->step);
  {
    ProfScope ps(u->prof, KI_UNET_ADAM, u->st);
    k_adam<<<eblocks((long long)u->nparams), 256, 0, u->st>>>(u->master, u->grad, u->m1, u->m2,
                                                              (long long)u->nparams, lr, b1, b2, 1e-8f, c1, c2);
  }
  cudaError_t e = refresh_weights(u);
  return e == cudaSuccess ? LES_OK : unet_fail(u, e, "adam");
}

int les_unet_set_loss(les_unet* u, int32_t kind) {
  if (!u || (kind != LES_UNET_LOSS_MSE && kind != LES_UNET_LOSS_ENERGY)) return LES_ERR_INVALID_ARG;
  u->loss_kind = kind;
  return LES_OK;
}

int les_unet_set_output_scale(les_unet* u, double scale) {
  if (!u || !(scale > 0) || !std::isfinite(scale)) return LES_ERR_INVALID_ARG;
  u->out_scale = scale;
  return LES_OK;
}

double les_unet_get_output_scale(const les_unet* u) { return u ? u->out_scale : 0.0; }

const char* les_unet_last_error(const les_unet* u) { return u ? u->err.c_str() : "no model"; }

}  // extern "C"
