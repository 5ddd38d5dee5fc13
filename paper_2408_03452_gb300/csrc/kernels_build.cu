// Coefficient and right-hand-side construction (once per solve).
//
// Transmissibility (arXiv 2408.03452, Section II.A, Eq. 4): the flux across
// the face between cells K and L is T_KL (p_L - p_K) with T_KL = Y_KL *
// lambda_KL.  The geometric factor Y is the two-point (half-transmissibility)
// form A_f / (h/(2 k_K) + h/(2 k_L)), which is the harmonic mean of the two
// permeabilities for unit cells; lambda_KL = 1/mu, the arithmetic mean of the
// two (equal) mobilities.  Faces on the outer boundary carry no flow.
// Dirichlet cells (Eq. 3) keep the identity row; their couplings to interior
// cells move to the right-hand side.
#include <cuda_bf16.h>

#include "fp64_div.cuh"
#include "tpfa_internal.cuh"

namespace tpfa {

namespace {

struct Geo {
  Num ax, ay, az;  // face area / mu for x, y, z faces
  Num hx, hy, hz;  // half the cell size along each axis
};

__device__ __forceinline__ double face_trans(double kK, double kL, const Num& a, const Num& half) {
  return div_rn(a, div_rn(half, kK) + div_rn(half, kL));
}

__device__ __forceinline__ bool is_dir(const uint8_t* m, int64_t c) { return m != nullptr && m[c] != 0; }

// Records of one run of z-planes of a 32 x 8 column, FP32 + FP64 (B16 = false)
// or BF16.
//
// The FP64 pipe (1/64 of the FP32 rate on GB300) bounds this kernel, so it is left
// the sums alone: divisions run in integer arithmetic (div_rn) and none is done
// twice.  The half-transmissibility h/(2k) of a cell is formed once (ISO: the three
// axes share it when the spacings are equal, else one per axis) and a face once, by
// the cell on its low side; neighbours read both from shared memory, along z from
// registers: 4.6 divisions per cell (ISO) instead of 18.  Values and their order of
// summation are those of the definition.  256^3, both record types: 4,736 us with 18
// divisions, 1,577 with 4.3 by the operator (16-row tiles), 708 with div_rn, 517 with
// 8-row tiles (four blocks per SM, whose barriers do not coincide; the same rows with
// three to six: 560, 517, 537, 524) and K loaded a plane ahead.  The nine sums per
// cell are busy for two thirds of that, issue and the integer pipe for 60 % each.
//
// BF16 record for the mixed-precision inner solve: (Tx', Ty', Tz', E), each
// rounded to nearest-even from FP64, with E = d_K + sum of the T_KL to
// Dirichlet neighbours (faces -x..+z in order; E = 1 and T' = 0 on Dirichlet
// cells).  The sweep forms D = sum of the six T' + E in FP32, so the BF16
// operator is the TPFA operator of the rounded face values: symmetric
// positive definite whenever the FP64 one is, with x'Ax within a factor
// (1 +- 2^-9) of the FP64 operator's.
constexpr int kBY = 8;                 // rows of a tile
constexpr int kBMin = 4;               // blocks per SM the registers are held to
constexpr int kBThreads = 32 * kBY;

template <bool ISO, bool B16>
__global__ void __launch_bounds__(kBThreads, kBMin)
build_trans_kernel(Grid g, Geo geo, const double* __restrict__ K, const uint8_t* __restrict__ mask,
                   const double* __restrict__ d, double d0, float4* __restrict__ coef,
                   double2* __restrict__ coef64, ushort4* __restrict__ coef16, int64_t nbx,
                   int64_t nby, int zc) {
  __shared__ double sX[kBY][34];             // h/(2k) along x, columns -1 .. 32
  __shared__ double sY[kBY + 2][32];         // h/(2k) along y, rows -1 .. 8
  __shared__ double fX[kBY][33];             // T of the faces x-1|x, x = 0 .. 32
  __shared__ double fY[kBY + 1][32];         // T of the faces y-1|y, y = 0 .. 8
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t bx = blockIdx.x % nbx, t_ = blockIdx.x / nbx;
  const int64_t X0 = 32 * bx, Y0 = kBY * (t_ % nby), z0 = (t_ / nby) * zc;
  const int64_t z1 = min(z0 + (int64_t)zc, g.nz);
  const int64_t x = X0 + tx, y = Y0 + ty;
  const bool in = x < g.nx && y < g.ny;
  const bool xp_in = in && x + 1 < g.nx, yp_in = in && y + 1 < g.ny;

  // this thread's halo work: warps 0 and 1 the rows below and above the tile,
  // warp 2 the columns left (lanes 0 ..) and right (lanes 16 ..) of it
  int64_t hc = -1;  // in-plane cell
  double* hs = nullptr;
  if (ty < 2) {
    const int64_t yy = ty == 0 ? Y0 - 1 : Y0 + kBY;
    hs = &sY[ty == 0 ? 0 : kBY + 1][tx];
    if (x < g.nx && yy >= 0 && yy < g.ny) hc = x + g.nx * yy;
  } else if (ty == 2 && (tx & 15) < kBY) {
    const int64_t xx = tx < 16 ? X0 - 1 : X0 + 32, yy = Y0 + (tx & 15);
    hs = &sX[tx & 15][tx < 16 ? 0 : 33];
    if (xx >= 0 && xx < g.nx && yy < g.ny) hc = xx + g.nx * yy;
  }

  // K of the next plane and of the halo cell are loaded one plane ahead; a cell's
  // Dirichlet flag comes from the plane below it
  int64_t c = x + g.nx * y + g.plane * z0;
  const double* hk = K + (hc >= 0 ? hc + g.plane * z0 : 0);
  double kc = 0.0, zlo = 0.0;   // own K; T of the face below the plane
  double sz = 0.0;              // own h/(2k) along z
  double kn = 0.0, kh = 0.0;
  bool own_dir = false;
  if (hc >= 0) kh = __ldg(hk);
  if (in) {
    kc = __ldg(K + c);
    if (z0 + 1 < g.nz) kn = __ldg(K + c + g.plane);
    own_dir = is_dir(mask, c);
    sz = div_rn(geo.hz, kc);
    if (z0 > 0) zlo = div_rn(geo.az, div_rn(geo.hz, __ldg(K + c - g.plane)) + sz);
  }
  for (int64_t z = z0; z < z1; ++z, c += g.plane) {
    const bool zp_in = in && z + 1 < g.nz;
    const double s_x = ISO ? sz : (in ? div_rn(geo.hx, kc) : 0.0);
    const double s_y = ISO ? sz : (in ? div_rn(geo.hy, kc) : 0.0);
    sX[ty][tx + 1] = s_x;
    sY[ty + 1][tx] = s_y;
    if (hs != nullptr) *hs = hc >= 0 ? div_rn(ISO || ty < 2 ? geo.hy : geo.hx, kh) : 0.0;
    bool dxp = false, dyp = false, dzp = false;
    if (mask != nullptr) {
      if (xp_in) dxp = mask[c + 1] != 0;
      if (yp_in) dyp = mask[c + g.nx] != 0;
      if (zp_in) dzp = mask[c + g.plane] != 0;
    }
    const double dc = d != nullptr && in ? d[c] : d0;
    double kn2 = 0.0, szn = 0.0, zhi = 0.0;
    if (z + 1 < z1) {
      hk += g.plane;
      if (hc >= 0) kh = __ldg(hk);
      if (in && z + 2 < g.nz) kn2 = __ldg(K + c + 2 * g.plane);
    }
    if (zp_in) {
      szn = div_rn(geo.hz, kn);
      zhi = div_rn(geo.az, sz + szn);
    }
    __syncthreads();
    // faces on the high side of the own cell, and those on the low side of the
    // tile (warps 3: x, 4: y)
    const double xp = xp_in ? div_rn(geo.ax, s_x + sX[ty][tx + 2]) : 0.0;
    const double yp = yp_in ? div_rn(geo.ay, s_y + sY[ty + 2][tx]) : 0.0;
    fX[ty][tx + 1] = xp;
    fY[ty + 1][tx] = yp;
    if (ty == 3 && tx < kBY)
      fX[tx][0] = (X0 > 0 && Y0 + tx < g.ny) ? div_rn(geo.ax, sX[tx][0] + sX[tx][1]) : 0.0;
    if (ty == 4) fY[0][tx] = (Y0 > 0 && x < g.nx) ? div_rn(geo.ay, sY[0][tx] + sY[1][tx]) : 0.0;
    __syncthreads();
    if (in) {
      const double xm = fX[ty][tx], ym = fY[ty][tx];
      double t0 = xp, t1 = yp, t2 = zhi, w;
      if (own_dir) {
        t0 = t1 = t2 = 0.0;
        w = 1.0;
      } else {
        // faces beyond the grid are zero, and so are the terms they add
        if (B16) {
          w = dc;
          if (x > 0 && is_dir(mask, c - 1)) w += xm;
          if (dxp) w += xp;
          if (y > 0 && is_dir(mask, c - g.nx)) w += ym;
          if (dyp) w += yp;
          if (z > 0 && is_dir(mask, c - g.plane)) w += zlo;
          if (dzp) w += zhi;
        } else {
          w = (((((xm + xp) + ym) + yp) + zlo) + zhi) + dc;
        }
        if (dxp) t0 = 0.0;
        if (dyp) t1 = 0.0;
        if (dzp) t2 = 0.0;
      }
      if (B16) {
        coef16[c] = make_ushort4(__bfloat16_as_ushort(__double2bfloat16(t0)),
                                 __bfloat16_as_ushort(__double2bfloat16(t1)),
                                 __bfloat16_as_ushort(__double2bfloat16(t2)),
                                 __bfloat16_as_ushort(__double2bfloat16(w)));
      } else {
        coef[c] = make_float4(__double2float_rn(t0), __double2float_rn(t1), __double2float_rn(t2),
                              __double2float_rn(w));
        if (coef64 != nullptr) {
          coef64[2 * c] = make_double2(t0, t1);
          coef64[2 * c + 1] = make_double2(t2, w);
        }
      }
    }
    own_dir = dzp;
    zlo = zhi;
    kc = kn;
    kn = kn2;
    sz = szn;
  }
}

// The same records, one thread per cell, every face formed by both its cells: for
// thin grids, which leave most threads of the 32 x 8 tiles idle.
template <bool B16>
__global__ void __launch_bounds__(kElemThreads)
build_trans_cell_kernel(Grid g, Geo geo, const double* __restrict__ K,
                        const uint8_t* __restrict__ mask, const double* __restrict__ d, double d0,
                        float4* __restrict__ coef, double2* __restrict__ coef64,
                        ushort4* __restrict__ coef16) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < g.n; c += stride) {
    const int64_t pos[3] = {c % g.nx, (c / g.nx) % g.ny, c / g.plane};
    const int64_t ext[3] = {g.nx, g.ny, g.nz}, step[3] = {1, g.nx, g.plane};
    const Num ar[3] = {geo.ax, geo.ay, geo.az}, hh[3] = {geo.hx, geo.hy, geo.hz};
    double t[3] = {0.0, 0.0, 0.0}, w = 1.0;
    if (!is_dir(mask, c)) {
      const double kc = K[c], dc = d != nullptr ? d[c] : d0;
      w = B16 ? dc : 0.0;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const int64_t lo = c - step[a], hi = c + step[a];
        if (pos[a] > 0 && (!B16 || is_dir(mask, lo))) w += face_trans(K[lo], kc, ar[a], hh[a]);
        if (pos[a] + 1 < ext[a]) {
          const double T = face_trans(kc, K[hi], ar[a], hh[a]);
          const bool dir = is_dir(mask, hi);
          if (!B16 || dir) w += T;
          if (!dir) t[a] = T;
        }
      }
      if (!B16) w += dc;
    }
    if (B16) {
      coef16[c] = make_ushort4(__bfloat16_as_ushort(__double2bfloat16(t[0])),
                               __bfloat16_as_ushort(__double2bfloat16(t[1])),
                               __bfloat16_as_ushort(__double2bfloat16(t[2])),
                               __bfloat16_as_ushort(__double2bfloat16(w)));
    } else {
      coef[c] = make_float4(__double2float_rn(t[0]), __double2float_rn(t[1]),
                            __double2float_rn(t[2]), __double2float_rn(w));
      if (coef64 != nullptr) {
        coef64[2 * c] = make_double2(t[0], t[1]);
        coef64[2 * c + 1] = make_double2(t[2], w);
      }
    }
  }
}

// The lifted couplings of a cell to its Dirichlet neighbours, added to s in the
// order of the faces -x, +x, -y, +y, -z, +z (bits 0 .. 5 of dir).
template <typename I>
__device__ __forceinline__ double lift_faces(double s, unsigned dir, I c, I nx, I plane,
                                             const Geo& geo, const double* __restrict__ K,
                                             const double* __restrict__ pD) {
  const I nb[6] = {c - 1, c + 1, c - nx, c + nx, c - plane, c + plane};
  const Num ar[3] = {geo.ax, geo.ay, geo.az}, hh[3] = {geo.hx, geo.hy, geo.hz};
  const double kc = K[c];
#pragma unroll
  for (int f = 0; f < 6; ++f) {
    if (!((dir >> f) & 1u)) continue;
    const double T = (f & 1) ? face_trans(kc, K[nb[f]], ar[f >> 1], hh[f >> 1])
                             : face_trans(K[nb[f]], kc, ar[f >> 1], hh[f >> 1]);
    s += T * (pD != nullptr ? pD[nb[f]] : 0.0);
  }
  return s;
}

// Right-hand side of a run of z-planes of a 32 x 8 column.  K is read only where a
// neighbour is a Dirichlet cell.  Latency bounds this kernel: the flags and q of a
// plane are loaded together and one plane ahead, those of x +- 1 come by shuffles
// and those of z -+ 1 from the planes around.  256^3 with Dirichlet x-ends: 370 us
// with K read everywhere and 64-bit divisions, 308 with one thread per cell, 254 with
// div_rn, 149 so; the warps at the two ends divide for one lane each.
template <typename I>
__global__ void __launch_bounds__(kBThreads)
build_rhs_kernel(Grid g, Geo geo, const double* __restrict__ K, const uint8_t* __restrict__ mask,
                 const double* __restrict__ q, const double* __restrict__ pD,
                 double* __restrict__ b, int64_t nbx, int64_t nby, int zc) {
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t bx = blockIdx.x % nbx, t_ = blockIdx.x / nbx;
  const int64_t x = 32 * bx + tx, y = kBY * (t_ % nby) + ty, z0 = (t_ / nby) * zc;
  const int64_t z1 = min(z0 + (int64_t)zc, g.nz);
  const bool in = x < g.nx && y < g.ny;
  const I nx = (I)g.nx, plane = (I)g.plane;
  I c = in ? (I)(x + g.nx * y + g.plane * z0) : 0;
  const bool ym = in && y > 0, yp = in && y + 1 < g.ny;
  // the lanes whose neighbour along x is another warp's load it
  const bool xl = in && tx == 0 && x > 0, xr = in && tx == 31 && x + 1 < g.nx;
  struct Plane {
    unsigned own, side, lo, hi;
    double q;
  };
  auto load = [&](I cc, int64_t z) {
    Plane p{0, 0, 0, 0, 0.0};
    if (in && z < g.nz) p.own = mask[cc];
    if (z < z1) {
      if (xl) p.side = mask[cc - 1];
      if (xr) p.side = mask[cc + 1];
      if (ym) p.lo = mask[cc - nx];
      if (yp) p.hi = mask[cc + nx];
      if (in && q != nullptr) p.q = q[cc];
    }
    return p;
  };
  Plane p = load(c, z0);
  unsigned below = in && z0 > 0 ? mask[c - plane] : 0u;
  for (int64_t z = z0; z < z1; ++z, c += plane) {
    const Plane n = load(c + plane, z + 1);
    unsigned left = __shfl_up_sync(0xffffffffu, p.own, 1);
    unsigned right = __shfl_down_sync(0xffffffffu, p.own, 1);
    if (tx == 0) left = p.side;
    if (tx == 31) right = p.side;
    if (in) {
      double s = p.q;
      const unsigned dir = (left != 0 ? 1u : 0u) | (right != 0 ? 2u : 0u) | (p.lo != 0 ? 4u : 0u) |
                           (p.hi != 0 ? 8u : 0u) | (below != 0 ? 16u : 0u) | (n.own != 0 ? 32u : 0u);
      if (p.own != 0)
        s = pD != nullptr ? pD[c] : 0.0;
      else if (dir != 0)
        s = lift_faces(s, dir, c, nx, plane, geo, K, pD);
      b[c] = s;
    }
    below = p.own;
    p = n;
  }
}

// The same, one thread per cell, for thin grids and for systems without Dirichlet
// cells; a cell's position takes two 32-bit divisions where the grid allows it (I).
template <typename I>
__global__ void __launch_bounds__(kElemThreads)
build_rhs_cell_kernel(Grid g, Geo geo, const double* __restrict__ K,
                      const uint8_t* __restrict__ mask, const double* __restrict__ q,
                      const double* __restrict__ pD, double* __restrict__ b) {
  const I nx = (I)g.nx, ny = (I)g.ny, nz = (I)g.nz, plane = (I)g.plane, n = (I)g.n;
  const I stride = (I)gridDim.x * blockDim.x;
  for (I c = (I)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += stride) {
    if (is_dir(mask, c)) {
      b[c] = pD != nullptr ? pD[c] : 0.0;
      continue;
    }
    double s = q != nullptr ? q[c] : 0.0;
    if (mask != nullptr) {
      const I row = c / nx, i = c - row * nx, k = c / plane, j = row - k * ny;
      const I nb[6] = {c - 1, c + 1, c - nx, c + nx, c - plane, c + plane};
      const bool ex[6] = {i > 0, i + 1 < nx, j > 0, j + 1 < ny, k > 0, k + 1 < nz};
      unsigned dir = 0u;
#pragma unroll
      for (int f = 0; f < 6; ++f)
        if (ex[f] && mask[nb[f]] != 0) dir |= 1u << f;
      if (dir != 0u) s = lift_faces(s, dir, c, nx, plane, geo, K, pD);
    }
    b[c] = s;
  }
}

// Point sources, added one after another by a single thread so that
// duplicates accumulate in a fixed order.  Sources on Dirichlet cells and
// indices outside the grid are ignored.
__global__ void add_sources_kernel(Grid g, const uint8_t* __restrict__ mask,
                                   const int64_t* __restrict__ idx, const double* __restrict__ val,
                                   int64_t n, double* __restrict__ b) {
  if (blockIdx.x != 0 || threadIdx.x != 0) return;
  for (int64_t t = 0; t < n; ++t) {
    const int64_t c = idx[t];
    if (c < 0 || c >= g.n || is_dir(mask, c)) continue;
    b[c] += val[t];
  }
}

// Known part of the accumulation term of one backward-Euler step:
// b_K += d_K p_K^n on interior cells.
__global__ void __launch_bounds__(kElemThreads)
accumulation_kernel(Grid g, const uint8_t* __restrict__ mask, const double* __restrict__ d,
                    double d0, const double* __restrict__ p_prev, double* __restrict__ b) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < g.n; c += stride)
    if (!is_dir(mask, c)) b[c] += (d != nullptr ? d[c] : d0) * p_prev[c];
}

Geo make_geo(const tpfa_grid& geo) {
  Geo o;
  o.ax = make_num((geo.dy * geo.dz) / geo.mu);
  o.ay = make_num((geo.dx * geo.dz) / geo.mu);
  o.az = make_num((geo.dx * geo.dy) / geo.mu);
  o.hx = make_num(0.5 * geo.dx);
  o.hy = make_num(0.5 * geo.dy);
  o.hz = make_num(0.5 * geo.dz);
  return o;
}

int grid_for(const Grid& g) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return elem_blocks(g, sms);
}

}  // namespace

// Tiles of 32 x kBY cells and z-runs of 16 planes, shorter until there are about
// four blocks per SM (a run repeats two divisions per column; 256^3: 600 us at 32
// planes, where the last of 3.4 waves is nearly empty, 577 at 16, 583 at 8).
struct Tiles {
  int64_t nbx, nby, zc, blocks;
};

static Tiles tile_grid(const Grid& g) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  Tiles t{(g.nx + 31) / 32, (g.ny + kBY - 1) / kBY, 16, 0};
  while (t.zc > 2 && t.nbx * t.nby * ((g.nz + t.zc - 1) / t.zc) < 4 * (int64_t)sms) t.zc /= 2;
  t.blocks = t.nbx * t.nby * ((g.nz + t.zc - 1) / t.zc);
  while (t.blocks > 0x7fffffff) {
    t.zc *= 2;
    t.blocks = t.nbx * t.nby * ((g.nz + t.zc - 1) / t.zc);
  }
  return t;
}

// a tile's cell costs 4.6 divisions against 18: tiles win down to a quarter full
static bool thin(const Grid& g, const Tiles& t) {
  return g.nx * g.ny * 4 < t.nbx * t.nby * 32 * kBY;
}

template <bool B16>
static cudaError_t launch_records(const Grid& g, const tpfa_grid& geo, const double* K,
                                  const uint8_t* mask, const double* d, double d0, float4* coef,
                                  double2* coef64, ushort4* coef16, cudaStream_t s) {
  const Geo o = make_geo(geo);
  const Tiles t = tile_grid(g);
  if (thin(g, t))
    build_trans_cell_kernel<B16><<<grid_for(g), kElemThreads, 0, s>>>(g, o, K, mask, d, d0, coef,
                                                                      coef64, coef16);
  else if (o.hx.v == o.hy.v && o.hy.v == o.hz.v)
    build_trans_kernel<true, B16><<<(unsigned)t.blocks, kBThreads, 0, s>>>(
        g, o, K, mask, d, d0, coef, coef64, coef16, t.nbx, t.nby, (int)t.zc);
  else
    build_trans_kernel<false, B16><<<(unsigned)t.blocks, kBThreads, 0, s>>>(
        g, o, K, mask, d, d0, coef, coef64, coef16, t.nbx, t.nby, (int)t.zc);
  return cudaGetLastError();
}

cudaError_t launch_build_trans(const Grid& g, const tpfa_grid& geo, const double* K,
                               const uint8_t* mask, const double* d, double d0, float4* coef,
                               double* coef64, cudaStream_t s) {
  return launch_records<false>(g, geo, K, mask, d, d0, coef, reinterpret_cast<double2*>(coef64),
                               nullptr, s);
}

cudaError_t launch_accumulation(const Grid& g, const uint8_t* mask, const double* d, double d0,
                                const double* p_prev, double* b, cudaStream_t s) {
  accumulation_kernel<<<grid_for(g), kElemThreads, 0, s>>>(g, mask, d, d0, p_prev, b);
  return cudaGetLastError();
}

cudaError_t launch_build_trans_bf16(const Grid& g, const tpfa_grid& geo, const double* K,
                                    const uint8_t* mask, const double* d, double d0,
                                    uint2* coef16, cudaStream_t s) {
  return launch_records<true>(g, geo, K, mask, d, d0, nullptr, nullptr,
                              reinterpret_cast<ushort4*>(coef16), s);
}

cudaError_t launch_build_rhs(const Grid& g, const tpfa_grid& geo, const double* K,
                             const uint8_t* mask, const double* q, const double* pD,
                             const int64_t* src_idx, const double* src_val, int64_t n_src,
                             double* b, cudaStream_t s) {
  const int blocks = grid_for(g);
  const Tiles t = tile_grid(g);
  const Geo o = make_geo(geo);
  // below 2^31 cells minus one grid stride, 32-bit indices cannot overflow
  const bool small = g.n < (int64_t)0x7fffffff - (int64_t)blocks * kElemThreads;
  if (mask == nullptr || thin(g, t)) {
    if (small)
      build_rhs_cell_kernel<uint32_t><<<blocks, kElemThreads, 0, s>>>(g, o, K, mask, q, pD, b);
    else
      build_rhs_cell_kernel<int64_t><<<blocks, kElemThreads, 0, s>>>(g, o, K, mask, q, pD, b);
  } else if (small) {
    build_rhs_kernel<uint32_t><<<(unsigned)t.blocks, kBThreads, 0, s>>>(g, o, K, mask, q, pD, b, t.nbx,
                                                                        t.nby, (int)t.zc);
  } else {
    build_rhs_kernel<int64_t><<<(unsigned)t.blocks, kBThreads, 0, s>>>(g, o, K, mask, q, pD, b, t.nbx,
                                                                       t.nby, (int)t.zc);
  }
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || n_src <= 0) return e;
  add_sources_kernel<<<1, 32, 0, s>>>(g, mask, src_idx, src_val, n_src, b);
  return cudaGetLastError();
}

}  // namespace tpfa
