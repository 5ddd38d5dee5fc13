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

#include "tpfa_internal.cuh"

namespace tpfa {

namespace {

struct Geo {
  double ax, ay, az;  // face area / mu for x, y, z faces
  double hx, hy, hz;  // cell size along each axis
};

__device__ __forceinline__ double face_trans(double kK, double kL, double a, double h) {
  const double half = 0.5 * h;
  return a / (half / kK + half / kL);
}

__device__ __forceinline__ bool is_dir(const uint8_t* m, int64_t c) { return m != nullptr && m[c] != 0; }

// Records of one run of z-planes of a 32 x 16 column, FP32 + FP64 (B16 = false)
// or BF16.
//
// FP64 arithmetic bounds this kernel (1/64 of the FP32 rate on GB300; a division
// is about eight operations), so no division is done twice: the
// half-transmissibility h/(2k) of a cell is formed once (ISO: the three axes
// share it when the spacings are equal, else one per axis) and a face once, by
// the cell on its low side; neighbours read both from shared memory, along z
// from registers.  4.3 divisions per cell (ISO) instead of 18; values and
// their order of summation are those of the definition.  256^3, both record
// types: 4,736 -> 1,4xx us.
//
// BF16 record for the mixed-precision inner solve: (Tx', Ty', Tz', E), each
// rounded to nearest-even from FP64, with E = d_K + sum of the T_KL to
// Dirichlet neighbours (faces -x..+z in order; E = 1 and T' = 0 on Dirichlet
// cells).  The sweep forms D = sum of the six T' + E in FP32, so the BF16
// operator is the TPFA operator of the rounded face values: symmetric
// positive definite whenever the FP64 one is, with x'Ax within a factor
// (1 +- 2^-9) of the FP64 operator's.
constexpr int kBY = 16;                // rows of a tile
constexpr int kBThreads = 32 * kBY;

template <bool ISO, bool B16>
__global__ void __launch_bounds__(kBThreads)
build_trans_kernel(Grid g, Geo geo, const double* __restrict__ K, const uint8_t* __restrict__ mask,
                   const double* __restrict__ d, double d0, float4* __restrict__ coef,
                   double2* __restrict__ coef64, ushort4* __restrict__ coef16, int64_t nbx,
                   int64_t nby, int zc) {
  __shared__ double sX[kBY][34];             // h/(2k) along x, columns -1 .. 32
  __shared__ double sY[kBY + 2][32];         // h/(2k) along y, rows -1 .. 16
  __shared__ double fX[kBY][33];             // T of the faces x-1|x, x = 0 .. 32
  __shared__ double fY[kBY + 1][32];         // T of the faces y-1|y, y = 0 .. 16
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  const int64_t bx = blockIdx.x % nbx, t_ = blockIdx.x / nbx;
  const int64_t X0 = 32 * bx, Y0 = kBY * (t_ % nby), z0 = (t_ / nby) * zc;
  const int64_t z1 = min(z0 + (int64_t)zc, g.nz);
  const int64_t x = X0 + tx, y = Y0 + ty;
  const bool in = x < g.nx && y < g.ny;
  const double hx = 0.5 * geo.hx, hy = 0.5 * geo.hy, hz = 0.5 * geo.hz;

  // this thread's halo work: warps 0 and 1 the rows below and above the tile,
  // warp 2 the columns left (lanes 0..15) and right of it
  int64_t hc = -1;  // in-plane cell
  double* hs = nullptr;
  double hh = 0.0;
  if (ty < 2) {
    const int64_t yy = ty == 0 ? Y0 - 1 : Y0 + kBY;
    hs = &sY[ty == 0 ? 0 : kBY + 1][tx];
    hh = hy;
    if (x < g.nx && yy >= 0 && yy < g.ny) hc = x + g.nx * yy;
  } else if (ty == 2) {
    const int64_t xx = tx < 16 ? X0 - 1 : X0 + 32, yy = Y0 + (tx & 15);
    hs = &sX[tx & 15][tx < 16 ? 0 : 33];
    hh = hx;
    if (xx >= 0 && xx < g.nx && yy < g.ny) hc = xx + g.nx * yy;
  }

  const int64_t c0 = x + g.nx * y;
  double kc = 0.0, zlo = 0.0;   // own K; T of the face below the plane
  double sz = 0.0;              // own h/(2k) along z
  if (in) {
    kc = __ldg(K + c0 + g.plane * z0);
    sz = hz / kc;
    if (z0 > 0) zlo = geo.az / (hz / __ldg(K + c0 + g.plane * (z0 - 1)) + sz);
  }
  for (int64_t z = z0; z < z1; ++z) {
    const int64_t c = c0 + g.plane * z;
    const double s_x = ISO ? sz : (in ? hx / kc : 0.0), s_y = ISO ? sz : (in ? hy / kc : 0.0);
    sX[ty][tx + 1] = s_x;
    sY[ty + 1][tx] = s_y;
    if (hs != nullptr) *hs = hc >= 0 ? hh / __ldg(K + hc + g.plane * z) : 0.0;
    double kn = 0.0, szn = 0.0, zhi = 0.0;
    if (in && z + 1 < g.nz) {
      kn = __ldg(K + c + g.plane);
      szn = hz / kn;
      zhi = geo.az / (sz + szn);
    }
    __syncthreads();
    // faces on the high side of the own cell, and those on the low side of the
    // tile (warps 3: x, 4: y)
    fX[ty][tx + 1] = (in && x + 1 < g.nx) ? geo.ax / (s_x + sX[ty][tx + 2]) : 0.0;
    fY[ty + 1][tx] = (in && y + 1 < g.ny) ? geo.ay / (s_y + sY[ty + 2][tx]) : 0.0;
    if (ty == 3 && tx < 16)
      fX[tx][0] = (X0 > 0 && Y0 + tx < g.ny) ? geo.ax / (sX[tx][0] + sX[tx][1]) : 0.0;
    if (ty == 4) fY[0][tx] = (Y0 > 0 && x < g.nx) ? geo.ay / (sY[0][tx] + sY[1][tx]) : 0.0;
    __syncthreads();
    if (in) {
      const double xm = fX[ty][tx], xp = fX[ty][tx + 1], ym = fY[ty][tx], yp = fY[ty + 1][tx];
      double t0 = xp, t1 = yp, t2 = zhi, w;
      const double dc = d != nullptr ? d[c] : d0;
      if (is_dir(mask, c)) {
        t0 = t1 = t2 = 0.0;
        w = 1.0;
      } else {
        // faces beyond the grid are zero, and so are the terms they add
        const bool dxp = x + 1 < g.nx && is_dir(mask, c + 1);
        const bool dyp = y + 1 < g.ny && is_dir(mask, c + g.nx);
        const bool dzp = z + 1 < g.nz && is_dir(mask, c + g.plane);
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
    zlo = zhi;
    kc = kn;
    sz = szn;
  }
}

// The same records, one thread per cell, every face formed by both its cells: for
// thin grids, which leave most threads of the 32 x 16 tiles idle.
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
    const double ar[3] = {geo.ax, geo.ay, geo.az}, hh[3] = {geo.hx, geo.hy, geo.hz};
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

// One thread per cell, grid-stride.  K is read only where a neighbour is a
// Dirichlet cell, and a cell's position takes two 32-bit divisions where the
// grid allows it (I; 256^3 with Dirichlet ends: 370 -> xx us).
template <typename I>
__global__ void __launch_bounds__(kElemThreads)
build_rhs_kernel(Grid g, Geo geo, const double* __restrict__ K, const uint8_t* __restrict__ mask,
                 const double* __restrict__ q, const double* __restrict__ pD,
                 double* __restrict__ b) {
  const I nx = (I)g.nx, ny = (I)g.ny, nz = (I)g.nz, plane = (I)g.plane, n = (I)g.n;
  const I stride = (I)gridDim.x * blockDim.x;
  for (I c = (I)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += stride) {
    if (is_dir(mask, c)) {
      b[c] = pD != nullptr ? pD[c] : 0.0;
      continue;
    }
    double s = q != nullptr ? q[c] : 0.0;
    if (mask != nullptr) {
      // lifted couplings to Dirichlet neighbours, faces -x, +x, -y, +y, -z, +z
      const I row = c / nx, i = c - row * nx, k = c / plane, j = row - k * ny;
      const I nb[6] = {c - 1, c + 1, c - nx, c + nx, c - plane, c + plane};
      const bool ex[6] = {i > 0, i + 1 < nx, j > 0, j + 1 < ny, k > 0, k + 1 < nz};
      const double ar[3] = {geo.ax, geo.ay, geo.az}, hh[3] = {geo.hx, geo.hy, geo.hz};
      unsigned dir = 0u;
#pragma unroll
      for (int f = 0; f < 6; ++f)
        if (ex[f] && mask[nb[f]] != 0) dir |= 1u << f;
      if (dir != 0u) {
        const double kc = K[c];
#pragma unroll
        for (int f = 0; f < 6; ++f) {
          if (!((dir >> f) & 1u)) continue;
          const double T = (f & 1) ? face_trans(kc, K[nb[f]], ar[f >> 1], hh[f >> 1])
                                   : face_trans(K[nb[f]], kc, ar[f >> 1], hh[f >> 1]);
          s += T * (pD != nullptr ? pD[nb[f]] : 0.0);
        }
      }
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
  o.ax = (geo.dy * geo.dz) / geo.mu;
  o.ay = (geo.dx * geo.dz) / geo.mu;
  o.az = (geo.dx * geo.dy) / geo.mu;
  o.hx = geo.dx; o.hy = geo.dy; o.hz = geo.dz;
  return o;
}

int grid_for(const Grid& g) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return elem_blocks(g, sms);
}

}  // namespace

// z-runs of the record kernel: 32 planes, shorter until there are about four
// blocks per SM (each run repeats two divisions per column)
template <bool B16>
static cudaError_t launch_records(const Grid& g, const tpfa_grid& geo, const double* K,
                                  const uint8_t* mask, const double* d, double d0, float4* coef,
                                  double2* coef64, ushort4* coef16, cudaStream_t s) {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t nbx = (g.nx + 31) / 32, nby = (g.ny + kBY - 1) / kBY;
  const Geo o = make_geo(geo);
  // a tile's cell costs 4.3 divisions against 18: tiles win down to a quarter full
  if (g.nx * g.ny * 4 < nbx * nby * 32 * kBY) {
    build_trans_cell_kernel<B16><<<grid_for(g), kElemThreads, 0, s>>>(g, o, K, mask, d, d0, coef,
                                                                      coef64, coef16);
    return cudaGetLastError();
  }
  int64_t zc = 32;
  while (zc > 2 && nbx * nby * ((g.nz + zc - 1) / zc) < 4 * (int64_t)sms) zc /= 2;
  int64_t blocks = nbx * nby * ((g.nz + zc - 1) / zc);
  while (blocks > 0x7fffffff) {
    zc *= 2;
    blocks = nbx * nby * ((g.nz + zc - 1) / zc);
  }
  if (o.hx == o.hy && o.hy == o.hz)
    build_trans_kernel<true, B16><<<(unsigned)blocks, kBThreads, 0, s>>>(
        g, o, K, mask, d, d0, coef, coef64, coef16, nbx, nby, (int)zc);
  else
    build_trans_kernel<false, B16><<<(unsigned)blocks, kBThreads, 0, s>>>(
        g, o, K, mask, d, d0, coef, coef64, coef16, nbx, nby, (int)zc);
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
  // below 2^31 cells minus one grid stride, 32-bit indices cannot overflow
  if (g.n < (int64_t)0x7fffffff - (int64_t)blocks * kElemThreads)
    build_rhs_kernel<uint32_t><<<blocks, kElemThreads, 0, s>>>(g, make_geo(geo), K, mask, q, pD, b);
  else
    build_rhs_kernel<int64_t><<<blocks, kElemThreads, 0, s>>>(g, make_geo(geo), K, mask, q, pD, b);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || n_src <= 0) return e;
  add_sources_kernel<<<1, 32, 0, s>>>(g, mask, src_idx, src_val, n_src, b);
  return cudaGetLastError();
}

}  // namespace tpfa
