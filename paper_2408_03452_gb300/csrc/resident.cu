// Resident conjugate gradient: the whole inner solve of a grid that fits on
// the chip, in one cooperative launch.
//
// A sweep of a small grid is bound by latency, not by memory: on 32^3 and 64^3
// grids the sweep loop (one graph-node launch and a march through ten planes
// per iteration) takes 20 us per iteration while the data of an iteration
// would move in well under 1 us.  Here every block owns a brick of 32 x 16 x
// CZ cells for the whole solve: the face transmissibilities, the diagonal and
// the search direction live in shared memory, r, q = A p and x in registers,
// and nothing but the brick faces and four partial sums crosses the chip per
// iteration.  Capacity: num_sms bricks of 8,192 cells (1.2 M cells on GB300).
//
// One grid-wide exchange per iteration.  With the q of a neighbour's face cell
// a block can form r and p of its halo cells itself (r_h -= alpha q_h, p_h =
// z_h + beta p_h), so the neighbours' q and the four dot products are the only
// things an iteration needs from other blocks, and both are complete at the
// same point.  They travel as words that carry their own sequence number
// ({value, epoch}, 8 bytes, single-copy atomic): a reader polls the data
// itself, so an iteration costs one store-to-load round trip through L2 and
// no fence, no counter and no second read.  Two buffers alternate: a block
// overwrites a buffer only after it has seen every block's sums of the
// iteration in between, which each block sends after it has read that buffer.
//
// Scalars.  FP64 runs at 1/64 of the FP32 rate on this chip, so beyond the
// thread sums (compensated FP32, as in the sweeps) the dot products are added
// as unevaluated pairs of floats (48 bits, fp32_pair.cuh) in a fixed order, and every
// block forms the same alpha and beta from them: pair quotients rounded once, which
// is what the sweeps' FP64 quotients round to.  Against the exact sums the totals are
// off by 1e-10 to 3e-10 (the thread sums' share), the same to four digits as with FP64
// trees, whose own share is 2e-16 against 9e-15; with the scalars in FP64 an iteration
// takes 1.0 us longer (32^3 3.06 against 2.04).  The operator is scaled by a power of
// two at load time (largest D in [1, 2)), which changes no mantissa and keeps the
// pairs inside the FP32 range; the solution is scaled back at the end.
//
// us per iteration (GB300, plain CG), the sweeps in their graph loop and here:
//   32^3 20.1 / 2.1    64^3 20.0 / 2.6    96x96x48 20.3 / 3.2
//   128x128x64 23.3 / 5.0    128^3 28.4 / 10.6 (the kernel for taller bricks below)
// The sweeps pay a graph-node launch and a march of a few planes on a few blocks;
// here an iteration costs one trip of words through L2 (1.5 us) and the brick's
// stencil, 0.2 us per plane.
#include <math.h>

#include "fp32_pair.cuh"
#include "sweep_common.cuh"

namespace tpfa {
namespace {

constexpr int kRW = 16;                 // warps per block = brick rows
constexpr int kRT = kRW * 32;           // threads
constexpr uint32_t kBeat = 64;          // iterations between signs of progress (batches)

__device__ __forceinline__ Dfl df_xor(Dfl a, int m) {
  return {__shfl_xor_sync(kFull, a.h, m), __shfl_xor_sync(kFull, a.l, m)};
}

// ---- sequence-numbered words -------------------------------------------------
__device__ __forceinline__ uint2 ll_load(const uint2* p) {
  unsigned long long w;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(w) : "l"(p) : "memory");
  return make_uint2((uint32_t)w, (uint32_t)(w >> 32));
}
__device__ __forceinline__ void ll_store(uint2* p, float v, uint32_t epoch) {
  const unsigned long long w = (unsigned long long)__float_as_uint(v) | ((unsigned long long)epoch << 32);
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"(w) : "memory");
}

// ---- layout ------------------------------------------------------------------
template <int CZ>
struct ResLayout {
  static constexpr int kTx = 0;                                   // [CZ][W][33], column 0: x - 1
  static constexpr int kTy = kTx + CZ * kRW * 33;                 // [CZ][W + 1][32], row 0: y - 1
  static constexpr int kTz = kTy + CZ * (kRW + 1) * 32;           // [CZ][W][32]
  static constexpr int kD = kTz + CZ * kRW * 32;
  static constexpr int kP = kD + CZ * kRW * 32;                   // [CZ][W + 2][34]
  static constexpr int kM = kP + CZ * (kRW + 2) * 34;             // Jacobi: M^-1 [CZ][W][32]
  static constexpr int floats(bool jac) { return kM + (jac ? CZ * kRW * 32 : 0); }
  // face words of a block: x lo, x hi [W][CZ], y lo, y hi [CZ][32], z lo, z hi [W][32]
  static constexpr int kFx = CZ * kRW, kFy = CZ * 32, kFz = kRW * 32;
  static constexpr int kFaces = 2 * (kFx + kFy + kFz);
};

// what every thread needs from the scalars of an iteration
struct ResNext {
  float alpha, beta;
  int done;
};

// Scalars of an iteration, formed by warp 0 (tall bricks: kept in shared memory, a
// dozen registers of every thread otherwise): alpha, beta and the stop test (as
// cg_finish).
struct ResScalars {
  Dfl rho, rho0, thresh;
  long long iter, sweeps;
  float alpha, beta;
  int done;

  __device__ __forceinline__ void init() {
    rho = rho0 = thresh = {0.f, 0.f};
    iter = sweeps = 0;
    alpha = beta = 0.f;
    done = kRunning;
  }
  __device__ __forceinline__ void update(const Dfl (&tot)[4], double rtol2, long long maxit) {
    rho = tot[0];
    if (iter == 0) {
      const float h = (float)rtol2, l = (float)(rtol2 - (double)h);
      rho0 = rho;
      thresh = df_add(df_mulf(rho0, h), df_mulf(rho0, l));
    }
    // alpha is the FP32 step the vectors take, so that rho - 2 alpha r'q +
    // alpha^2 q'q is the norm of the residual it leaves
    const float al = df_quot(rho, tot[1]);
    const Dfl u = df_mulf(tot[3], al);
    const Dfl v = df_mulf(df_add({2.f * tot[2].h, 2.f * tot[2].l}, {-u.h, -u.l}), al);
    Dfl rn = df_add(rho, {-v.h, -v.l});
    if (rn.h < 0.f) rn = {0.f, 0.f};
    alpha = al;
    beta = df_quot(rn, rho);
    // 0 unless one of the sums is infinite or NaN
    const float bad = fmaf(tot[0].h, 0.f, fmaf(tot[1].h, 0.f, fmaf(tot[2].h, 0.f, tot[3].h * 0.f)));
    const bool stay = bad == 0.f && tot[1].h > 0.f && !df_le(rho, thresh);
    ++iter;
    if (!stay || df_le(rn, thresh) || iter >= maxit || ++sweeps > 2 * maxit + 64) {
      done = stay ? (df_le(rn, thresh) ? kConvEst : iter >= maxit ? kMaxit : kGuard)
                  : (bad != 0.f ? kNonFinite : df_le(rho, thresh) ? kConvTrue : kBreakdown);
      if (!stay) {
        alpha = 0.f;
        --iter;
      }
    }
  }
  // after the last step: the true r'r of the residual it leaves; if the estimate
  // that stopped the loop was too optimistic, go on with the exact continuation
  __device__ __forceinline__ void finish(const Dfl (&tot)[4], long long maxit) {
    const Dfl prev = rho;
    rho = tot[0];
    if (done == kConvEst && !df_le(rho, thresh) && iter < maxit && isfinite(rho.h) && prev.h > 0.f) {
      beta = df_quot(rho, prev);
      done = kRunning;
    }
    alpha = 0.f;
  }
  __device__ __forceinline__ void report(CgState* st, double scale, bool fault) const {
    st->rho = (double)rho.h + (double)rho.l;
    st->rho0 = (double)rho0.h + (double)rho0.l;
    st->scale = scale;
    st->iter = iter;
    st->launches = 1;
    st->done = fault ? (int)kGuard : done;
  }
};

struct ResShared {
  float2 a[kRW][4], b[kRW][4];  // sums per warp: of the block, of all blocks
  float mx[kRW];
  ResScalars sc;
  ResNext next;
};

// the face words a thread waits for, where their offsets are not held: has(j), off(j)
template <class Has, class Off>
struct FaceWords {
  Has has;
  Off off;
};

// the block's sums of four values, sent to every block and added up in a fixed
// order; the neighbours' face words arrive in the same wait
// (NH: words a thread waits for; EARLY: first look before the sums are sent; BW: words
// of one look.  With 8 words their offsets and both halves take 24 registers, which the
// tall bricks do not have: there they are looked at four at a time and the offsets
// formed on the way, 128^3 10.6 against 12.6 us per iteration.)
template <int NH, bool EARLY, int BW = NH>
struct ResComm {
  uint2* part;
  const uint2* face;
  int nblk, blk;
  int hoff[BW == NH ? NH : 1];  // face words this thread reads (index in one buffer), -1: none
  size_t face_buf;

  __device__ __forceinline__ bool has(int j) const { return hoff[j] >= 0; }
  __device__ __forceinline__ int off(int j) const { return hoff[j]; }

  // warp-wide transposing sum of four pairs: lane l ends with value (l >> 3)
  __device__ __forceinline__ static Dfl warp4(const Dfl (&v)[4]) {
    const int lane = threadIdx.x & 31;
    const bool u = lane & 16;
    Dfl a = u ? v[2] : v[0], b = u ? v[3] : v[1];
    const Dfl sa = df_xor(u ? v[0] : v[2], 16), sb = df_xor(u ? v[1] : v[3], 16);
    a = df_acc(a, sa);
    b = df_acc(b, sb);
    const bool w = lane & 8;
    Dfl c = w ? b : a;
    c = df_acc(c, df_xor(w ? a : b, 8));
    c = df_acc(c, df_xor(c, 4));
    c = df_acc(c, df_xor(c, 2));
    return df_acc(c, df_xor(c, 1));
  }
  // sum over the block's warps: s[warp][value]; every lane gets value (lane & 3)
  __device__ __forceinline__ static Dfl warps16(const float2 (*s)[4]) {
    const int lane = threadIdx.x & 31, v = lane & 3, w = lane >> 2;
    const float2 a = s[w][v], b = s[w + 8][v];
    Dfl t = df_acc({a.x, a.y}, {b.x, b.y});
    t = df_acc(t, df_xor(t, 4));
    t = df_acc(t, df_xor(t, 8));
    t = df_acc(t, df_xor(t, 16));
    return df_fast(t.h, t.l);
  }

  // Sends this block's sums and waits for every block's and for the
  // neighbours' face words (FACES; wd.has(j): there is one, wd.off(j): its index in one
  // buffer).  The totals are there in warp 0 only.  Returns false when the wait ran out (or another block gave up).
  template <bool FACES, class Words>
  __device__ __forceinline__ bool exchange(const ResProb& a, const Dfl (&mine)[4], uint32_t epoch,
                                           const Words& wd, Dfl (&tot)[4], float (&qh)[NH],
                                           ResShared& sh) {
    auto& sA = sh.a;
    auto& sB = sh.b;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Dfl w = warp4(mine);
    if ((lane & 7) == 0) sA[warp][lane >> 3] = make_float2(w.h, w.l);
    __syncthreads();
    const uint32_t par = epoch & 1u;
    uint2* pb = part + (size_t)par * nblk * 8;
    const uint2* fb = face + par * face_buf;
    // a first look at the neighbours' words: they were sent before the
    // reduction, so they are there as a rule.  With short bricks it is in flight
    // while warp 0 sends the sums (64^3: 2.89 -> 2.66 us per iteration); with
    // tall ones the loads would only hold up those (128x128x64: 5.3 against 5.9)
    unsigned need = 0u;
    uint2 f[BW];
    auto look = [&](int j0) {
      if (!FACES) return;
#pragma unroll
      for (int j = 0; j < BW; ++j)
        if (j0 + j < NH && wd.has(j0 + j)) {
          need |= 1u << j;
          f[j] = ll_load(fb + wd.off(j0 + j));
        }
    };
    if (EARLY) look(0);
    if (warp == 0) {
      const Dfl t = warps16(sA);
      if (lane < 4) {
        ll_store(pb + ((size_t)blk * 4 + lane) * 2, t.h, epoch);
        ll_store(pb + ((size_t)blk * 4 + lane) * 2 + 1, t.l, epoch);
      }
    }
    if (!EARLY) look(0);
    bool ok = true;
    uint32_t polls = 0;
    auto give_up = [&]() -> bool {
      if (++polls >= a.poll_limit) return true;
      return (polls & 1023u) == 0u && *(volatile uint32_t*)a.abort != 0u;
    };
    auto await = [&](int j0) {
      while (need != 0u) {
#pragma unroll
        for (int j = 0; j < BW; ++j)
          if (j0 + j < NH && ((need >> j) & 1u) && f[j].y == epoch) {
            qh[j0 + j] = __uint_as_float(f[j].x);
            need &= ~(1u << j);
          }
        if (need != 0u && give_up()) {
          ok = false;
          break;
        }
#pragma unroll
        for (int j = 0; j < BW; ++j)
          if (j0 + j < NH && ((need >> j) & 1u)) f[j] = ll_load(fb + wd.off(j0 + j));
      }
    };
    await(0);
#pragma unroll
    for (int j0 = BW; j0 < NH; j0 += BW) {
      if (!ok) break;
      look(j0);
      await(j0);
    }
    // the sums of every block: item = 4 block + value, in order
    Dfl sum = {0.f, 0.f};
    for (int item = tid; ok && item < 4 * nblk;) {
      const uint2 h = ll_load(pb + (size_t)item * 2), l = ll_load(pb + (size_t)item * 2 + 1);
      if (h.y == epoch && l.y == epoch) {
        sum = df_acc(sum, {__uint_as_float(h.x), __uint_as_float(l.x)});
        item += kRT;
      } else if (give_up()) {
        ok = false;
      }
    }
    sum = df_acc(sum, df_xor(sum, 4));
    sum = df_acc(sum, df_xor(sum, 8));
    sum = df_acc(sum, df_xor(sum, 16));
    if (lane < 4) sB[warp][lane] = make_float2(sum.h, sum.l);
    if (__syncthreads_or(!ok)) {
      if (tid == 0) *(volatile uint32_t*)a.abort = 1u;
      return false;
    }
    if (warp == 0) {
      const Dfl t = warps16(sB);
#pragma unroll
      for (int v = 0; v < 4; ++v)
        tot[v] = {__shfl_sync(kFull, t.h, v), __shfl_sync(kFull, t.l, v)};
    }
    return true;
  }
};

// Power-of-two scale of the operator: the largest D of the grid, from every
// block's, scaled into [1, 2).
__device__ __forceinline__ float operator_scale(const ResProb& a, int blk, float dmax,
                                                uint32_t epoch, ResShared& sh, bool& fault) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  auto& sMax = sh.mx;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(kFull, dmax, o));
  if (lane == 0) sMax[warp] = dmax;
  __syncthreads();
  for (int w = 0; w < kRW; ++w) dmax = fmaxf(dmax, sMax[w]);
  uint2* pb = a.part + (size_t)(epoch & 1u) * a.nblk * 8;
  if (tid == 0) ll_store(pb + (size_t)blk * 8, dmax, epoch);
  uint32_t polls = 0;
  for (int i = tid; i < a.nblk && !fault; i += kRT) {
    for (;;) {
      const uint2 v = ll_load(pb + (size_t)i * 8);
      if (v.y == epoch) {
        dmax = fmaxf(dmax, __uint_as_float(v.x));
        break;
      }
      if (++polls >= a.poll_limit ||
          ((polls & 1023u) == 0u && *(volatile uint32_t*)a.abort != 0u)) {
        fault = true;
        break;
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) dmax = fmaxf(dmax, __shfl_xor_sync(kFull, dmax, o));
  if (lane == 0) sMax[warp] = dmax;
  fault = __syncthreads_or(fault);
  for (int w = 0; w < kRW; ++w) dmax = fmaxf(dmax, sMax[w]);
  if (!(dmax > 0.f && isfinite(dmax))) return 1.f;
  int e = ilogbf(dmax);
  e = e > 120 ? 120 : (e < -120 ? -120 : e);
  return exp2f((float)-e);
}

// One inner solve, run by the blocks blk = 0 .. a.nblk - 1 of its brick grid
// (BATCH: with signs of progress for the scheduler).
template <int CZ, bool JAC, bool BATCH>
__device__ __forceinline__ void resident_solve(const ResProb& a, int blk, float* sm,
                                               ResShared& sh) {
  using LY = ResLayout<CZ>;
  float* sTx = sm + LY::kTx;
  float* sTy = sm + LY::kTy;
  float* sTz = sm + LY::kTz;
  float* sD = sm + LY::kD;
  float* sP = sm + LY::kP;
  float* sM = sm + LY::kM;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int bx = blk % a.nbx, by = (blk / a.nbx) % a.nby, bz = blk / (a.nbx * a.nby);
  const Grid g = a.g;
  const int64_t gx = 32 * bx + lane, gy = kRW * by + warp, Z0 = (int64_t)CZ * bz;
  const bool inxy = gx < g.nx && gy < g.ny;
  const int64_t c0 = gx + g.nx * gy;  // in-plane cell
  CgState* st = a.st;
  const double scale = st->rr64 > 0.0 ? 1.0 / sqrt(st->rr64) : 1.0;

  // record of cell (x, y, z) as (Tx, Ty, Tz, D); zeros outside the grid
  const float4* c32 = static_cast<const float4*>(a.coef);
  const uint2* c16 = static_cast<const uint2*>(a.coef);
  auto rec = [&](int64_t x, int64_t y, int64_t z) -> float4 {
    if (x < 0 || y < 0 || z < 0 || x >= g.nx || y >= g.ny || z >= g.nz)
      return make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t c = x + g.nx * y + g.plane * z;
    if (!a.b16) return __ldg(c32 + c);
    const uint2 u = __ldg(c16 + c);
    return make_float4(bf16_lo(u.x), bf16_hi(u.x), bf16_lo(u.y), bf16_hi(u.y));
  };

  // ---- load the brick -------------------------------------------------------
  float dmax = 0.f;
  float tzlo = 0.f;  // Tz of the plane below the brick
  if (inxy) tzlo = rec(gx, gy, Z0 - 1).z;
  float tzm = tzlo;
#pragma unroll
  for (int k = 0; k < CZ; ++k) {
    const int64_t z = Z0 + k;
    float4 cf = rec(gx, gy, z);
    const float txl = lane == 0 ? rec(gx - 1, gy, z).x : 0.f;
    const float tyl = warp == 0 ? rec(gx, gy - 1, z).y : 0.f;
    if (a.b16) {
      const float txm = rec(gx - 1, gy, z).x, tym = rec(gx, gy - 1, z).y;
      if (inxy && z < g.nz) cf.w = (((((txm + cf.x) + tym) + cf.y) + tzm) + cf.z) + cf.w;
    }
    tzm = cf.z;
    sTx[(k * kRW + warp) * 33 + lane + 1] = cf.x;
    if (lane == 0) sTx[(k * kRW + warp) * 33] = txl;
    sTy[(k * (kRW + 1) + warp + 1) * 32 + lane] = cf.y;
    if (warp == 0) sTy[k * (kRW + 1) * 32 + lane] = tyl;
    sTz[(k * kRW + warp) * 32 + lane] = cf.z;
    sD[(k * kRW + warp) * 32 + lane] = cf.w;
    if (JAC)
      sM[(k * kRW + warp) * 32 + lane] =
          (inxy && z < g.nz) ? (a.b16 ? a.dinv[c0 + g.plane * z] : jac_inv(cf.w)) : 0.f;
    dmax = fmaxf(dmax, cf.w);
  }
  for (int i = tid; i < CZ * (kRW + 2) * 34; i += kRT) sP[i] = 0.f;

  ResComm<5, (CZ <= 8)> cm;
  cm.part = a.part;
  cm.face = a.face;
  cm.nblk = a.nblk;
  cm.blk = blk;
  cm.face_buf = (size_t)a.nblk * LY::kFaces;
  // halo cells of this thread: below, above, y - 1 and y + 16 of plane `warp`,
  // and one x-halo cell; their r, M^-1 and (z) p
  float rh[5], mh[5], pz[2] = {0.f, 0.f}, qh[5];
  const int xs = tid / LY::kFx, xi = tid % LY::kFx;  // x-halo: side, index w CZ + k
  int pslot[3];                                      // sP index of halo cells 2, 3, 4
  const unsigned halo =
      (bz > 0 ? 1u : 0u) | (bz + 1 < a.nbz ? 2u : 0u) | (warp < CZ && by > 0 ? 4u : 0u) |
      (warp < CZ && by + 1 < a.nby ? 8u : 0u) |
      ((xs == 0 && bx > 0) || (xs == 1 && bx + 1 < a.nbx) ? 16u : 0u);
  auto hindex = [&](int j) {
    constexpr int fy = 2 * LY::kFx, fz = 2 * (LY::kFx + LY::kFy);
    return j == 0   ? (blk - a.nbx * a.nby) * LY::kFaces + fz + LY::kFz + tid
           : j == 1 ? (blk + a.nbx * a.nby) * LY::kFaces + fz + tid
           : j == 2 ? (blk - a.nbx) * LY::kFaces + fy + LY::kFy + tid
           : j == 3 ? (blk + a.nbx) * LY::kFaces + fy + tid
           : xs == 0 ? (blk - 1) * LY::kFaces + LY::kFx + xi
                     : (blk + 1) * LY::kFaces + xi;
  };
#pragma unroll
  for (int j = 0; j < 5; ++j) cm.hoff[j] = ((halo >> j) & 1u) ? hindex(j) : -1;
  {
    const int xk = xi % CZ, xw = xi / CZ;
    pslot[0] = warp * (kRW + 2) * 34 + lane + 1;
    pslot[1] = (warp * (kRW + 2) + kRW + 1) * 34 + lane + 1;
    pslot[2] = (xk * (kRW + 2) + xw + 1) * 34 + (xs == 0 ? 0 : 33);
    const int64_t hx[5] = {gx, gx, gx, gx, 32 * (int64_t)bx + (xs == 0 ? -1 : 32)};
    const int64_t hy[5] = {gy, gy, kRW * (int64_t)by - 1, kRW * (int64_t)by + kRW,
                           kRW * (int64_t)by + xw};
    const int64_t hz[5] = {Z0 - 1, Z0 + CZ, Z0 + warp, Z0 + warp, Z0 + xk};
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      rh[j] = 0.f;
      mh[j] = 0.f;
      qh[j] = 0.f;
      if (((halo >> j) & 1u) && hx[j] < g.nx && hy[j] < g.ny && hz[j] < g.nz) {
        const int64_t c = hx[j] + g.nx * hy[j] + g.plane * hz[j];
        rh[j] = (float)(scale * a.r64[c]);
        if (JAC) mh[j] = a.b16 ? a.dinv[c] : jac_inv(__ldg(c32 + c).w);
      }
    }
  }

  float r[CZ], q[CZ], x[CZ];
#pragma unroll
  for (int k = 0; k < CZ; ++k) {
    r[k] = (inxy && Z0 + k < g.nz) ? (float)(scale * a.r64[c0 + g.plane * (Z0 + k)]) : 0.f;
    q[k] = 0.f;
    x[k] = 0.f;
  }

  uint32_t epoch = *(volatile uint32_t*)a.ctl;
  bool fault = false;
  const float tscale = operator_scale(a, blk, dmax, ++epoch, sh, fault);
  const float mscale = 1.f / tscale;  // exact: a power of two
  tzlo *= tscale;
#pragma unroll
  for (int k = 0; k < CZ; ++k) {
    sTx[(k * kRW + warp) * 33 + lane + 1] *= tscale;
    if (lane == 0) sTx[(k * kRW + warp) * 33] *= tscale;
    sTy[(k * (kRW + 1) + warp + 1) * 32 + lane] *= tscale;
    if (warp == 0) sTy[k * (kRW + 1) * 32 + lane] *= tscale;
    sTz[(k * kRW + warp) * 32 + lane] *= tscale;
    sD[(k * kRW + warp) * 32 + lane] *= tscale;
    if (JAC) sM[(k * kRW + warp) * 32 + lane] *= mscale;
  }
  if (JAC)
#pragma unroll
    for (int j = 0; j < 5; ++j) mh[j] *= mscale;

  // ---- iterations -------------------------------------------------------------
  float alpha = 0.f, beta = 0.f;
  int done = kRunning;
  ResScalars sc;  // (warp 0)
  sc.init();
  ResNext& sNext = sh.next;
  uint2* fmine = a.face + (size_t)blk * LY::kFaces;
  const bool fy0 = warp == 0 && by > 0, fy1 = warp == kRW - 1 && by + 1 < a.nby;

  // r -= alpha q, x += alpha p, p = z + beta p (with `dir`), on the own and the
  // halo cells; returns the sums of r'z
  auto step = [&](bool dir, Acc& s0) {
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      if (cm.hoff[j] < 0) continue;
      rh[j] = fmaf(-alpha, qh[j], rh[j]);
      if (!dir) continue;
      const float z = JAC ? rh[j] * mh[j] : rh[j];
      if (j < 2) {
        pz[j] = fmaf(beta, pz[j], z);
      } else {
        float* ps = sP + pslot[j - 2];
        *ps = fmaf(beta, *ps, z);
      }
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < CZ; ++k) {
      float* ps = sP + (k * (kRW + 2) + warp + 1) * 34 + lane + 1;
      const float p0 = *ps;
      x[k] = fmaf(alpha, p0, x[k]);
      r[k] = fmaf(-alpha, q[k], r[k]);
      const float z = JAC ? r[k] * sM[(k * kRW + warp) * 32 + lane] : r[k];
      if (dir) *ps = fmaf(beta, p0, z);
      s = fmaf(r[k], z, s);
      if ((k & 3) == 3 || k == CZ - 1) {
        kadd(s0, s);
        s = 0.f;
      }
    }
  };

  while (!fault) {
    Acc acc[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    step(true, acc[0]);
    __syncthreads();
    ++epoch;
    uint2* fo = fmine + (epoch & 1u) * cm.face_buf;
    float s1 = 0.f, s2 = 0.f, s3 = 0.f;
    float tz0 = tzlo, pm = pz[0];
    float pc = sP[(warp + 1) * 34 + lane + 1];
#pragma unroll
    for (int k = 0; k < CZ; ++k) {
      const float* ps = sP + (k * (kRW + 2) + warp + 1) * 34 + lane + 1;
      const float pp = k + 1 < CZ ? ps[(kRW + 2) * 34] : pz[1];
      const float* tx = sTx + (k * kRW + warp) * 33 + lane;
      const float* ty = sTy + (k * (kRW + 1) + warp) * 32 + lane;
      const int i = (k * kRW + warp) * 32 + lane;
      const float4 cf = make_float4(tx[1], ty[32], sTz[i], sD[i]);
      const float v = stencil7(cf, tx[0], ty[0], tz0, pc, ps[1], ps[-1], ps[34], ps[-34], pp, pm);
      q[k] = v;
      float z = r[k], mq = v;
      if (JAC) {
        const float m = sM[i];
        z *= m;
        mq *= m;
      }
      s1 = fmaf(pc, v, s1);
      s2 = fmaf(z, v, s2);
      s3 = fmaf(v, mq, s3);
      if ((k & 3) == 3 || k == CZ - 1) {
        kadd(acc[1], s1);
        kadd(acc[2], s2);
        kadd(acc[3], s3);
        s1 = s2 = s3 = 0.f;
      }
      tz0 = cf.z;
      pm = pc;
      pc = pp;
    }
    // the neighbours' words, once all of q is there: a store between the planes
    // would keep the loads of the next plane behind it (320 instead of 100
    // cycles per plane)
    if (bz > 0) ll_store(fo + 2 * (LY::kFx + LY::kFy) + tid, q[0], epoch);
    if (bz + 1 < a.nbz) ll_store(fo + 2 * (LY::kFx + LY::kFy) + LY::kFz + tid, q[CZ - 1], epoch);
    if (fy0 || fy1) {
      uint2* f = fo + 2 * LY::kFx + (fy0 ? 0 : LY::kFy) + lane;
#pragma unroll
      for (int k = 0; k < CZ; ++k) ll_store(f + k * 32, q[k], epoch);
    }
    if (bx > 0 || bx + 1 < a.nbx) {
      // lanes 0..15 take q[lane] of lane 0, lanes 16..31 q[lane - 16] of lane
      // 31: one store per warp instead of one per plane
      float v = 0.f;
#pragma unroll
      for (int k = 0; k < CZ; ++k) {
        const float t = __shfl_sync(kFull, q[k], lane < 16 ? 0 : 31);
        if ((lane & 15) == k) v = t;
      }
      if ((lane & 15) < CZ && (lane < 16 ? bx > 0 : bx + 1 < a.nbx))
        ll_store(fo + (lane < 16 ? 0 : LY::kFx) + warp * CZ + (lane & 15), v, epoch);
    }
    Dfl mine[4], tot[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) mine[v] = df_fast(acc[v].s, -acc[v].c);
    if (!cm.template exchange<true>(a, mine, epoch, cm, tot, qh, sh)) {
      fault = true;
      break;
    }
    if (BATCH && (epoch & (kBeat - 1u)) == 0u && blk == 0 && tid == 0)
      atomicAdd(a.beat, 1u);
    // the scalars are formed by warp 0 alone: in all 16 warps the same chain takes
    // twice as long
    if (warp == 0) {
      sc.update(tot, a.rtol2, a.maxit);
      if (lane == 0) sNext = {sc.alpha, sc.beta, sc.done};
    }
    __syncthreads();
    alpha = sNext.alpha;
    beta = sNext.beta;
    done = sNext.done;
    if (done == kRunning) continue;
    if (done != kConvEst && done != kMaxit) break;
    // the last step, and the true r'r (r' M^-1 r) of the residual it leaves
    Acc s0 = {0.f, 0.f};
    step(false, s0);
    ++epoch;
    // the face words of this exchange are not sent: nothing reads them
    mine[0] = df_fast(s0.s, -s0.c);
    mine[1] = mine[2] = mine[3] = {0.f, 0.f};
    const bool ok = cm.template exchange<false>(a, mine, epoch, cm, tot, qh, sh);
    if (!ok) {
      fault = true;
      break;
    }
    if (warp == 0) {
      sc.finish(tot, a.maxit);
      if (lane == 0) sNext = {sc.alpha, sc.beta, sc.done};
    }
    __syncthreads();
    alpha = sNext.alpha;
    beta = sNext.beta;
    done = sNext.done;
    if (done != kRunning) break;
  }

  // a wait that ran out in any block, be it the last one's, whose brick then lacks its
  // correction, is a failure of the solve (the host clears the flag)
  if (fault && tid == 0) *(volatile int*)&st->fault = 1;
  if (fault) done = kGuard;
  // x64 += correction (the scaled operator's solution times the scale)
  if (done != kNonFinite && done != kGuard && inxy) {
    const double inv = (double)tscale / scale;
#pragma unroll
    for (int k = 0; k < CZ; ++k)
      if (Z0 + k < g.nz) {
        const int64_t c = c0 + g.plane * (Z0 + k);
        a.x64[c] = fma((double)x[k], inv, a.x64[c]);
      }
  }
  if (blk == 0 && tid == 0) {
    sc.report(st, scale, fault);
    *(volatile uint32_t*)a.ctl = epoch;
  }
}

// ---- bricks of up to 32 planes -------------------------------------------------
// The same iteration for grids of up to twice that size (2.5 M cells on GB300).
// r and q are in registers, p, x and Ty in shared memory, with bricks of 24 planes D as
// well; the other coefficients (Tx, Tz and D, or with Jacobi M^-1: 12 bytes per cell) are
// read every iteration from a packed copy, which each thread writes for itself at the
// start and which stays in L2; loads run four planes ahead of the stencil.
//
// The Jacobi variant keeps z = M^-1 r and w = M^-1 q in place of r and q: the step then
// needs no M^-1, the words of the faces carry w, and r'z is the sum of D z^2, formed in
// the stencil, where D is at hand.  The operator is that of the records, as in the
// sweeps.  (CG on S A S with S = M^-1/2, every coefficient rounded again, took 15 to 23 %
// more iterations than the sweep over 24 fields with FP32 records, 50 % more on the worst;
// so it is within 0.6 % of the sweep, 3 % on the worst.)  us per iteration, plain /
// Jacobi, before and now: 100^3 (24 planes) 9.2 / 7.9 and 7.5 / 8.0, 128^3 (32 planes)
// 10.8 / 10.9 and 10.7 / 11.6.  M^-1 is loaded beside D in shared memory (8.0 us against
// 9.5 by reciprocals), and formed where D is loaded (11.7 against 12.3 by a second load).
template <int CZ>
struct BigLayout {
  static constexpr int kP = 0;                                  // [CZ][W + 2][34]
  static constexpr int kX = kP + CZ * (kRW + 2) * 34;           // [CZ][W][32]
  static constexpr int kTy = kX + CZ * kRW * 32;                // [CZ][W + 1][32], row 0: y - 1
  static constexpr int kTx = kTy + CZ * (kRW + 1) * 32;         // [CZ][W]: Tx of x - 1, lane 0
  static constexpr int kFx = CZ * kRW, kFy = CZ * 32, kFz = kRW * 32;
  static constexpr int kFaces = 2 * (kFx + kFy + kFz);
  static constexpr int kNY = CZ / 8, kNX = 2, kNH = 2 + kNY + kNX;  // halo cells per thread
  static constexpr int kRh = kTx + CZ * kRW;                    // r (z) of the y and x halo cells
  static constexpr int kD = kRh + (kNY + kNX) * kRT;            // D [CZ][W][32], where it fits
  static constexpr bool kHasD = CZ <= 24;
  static constexpr int kFloats = kD + (kHasD ? CZ * kRT : 0);
  static_assert(CZ % 8 == 0 && CZ <= 32, "halo rows per warp");
};

template <int CZ, bool JAC>
__global__ void __launch_bounds__(kRT, 1) resident_big_kernel(const __grid_constant__ ResProb a) {
  using LY = BigLayout<CZ>;
  constexpr int NH = LY::kNH;
  extern __shared__ __align__(16) float sm[];
  __shared__ ResShared sh;
  float* sP = sm + LY::kP;
  float* sX = sm + LY::kX;
  float* sTy = sm + LY::kTy;
  float* sTx = sm + LY::kTx;
  float* sRh = sm + LY::kRh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int blk = blockIdx.x;
  const int bx = blk % a.nbx, by = (blk / a.nbx) % a.nby, bz = blk / (a.nbx * a.nby);
  const Grid g = a.g;
  const int64_t gx = 32 * bx + lane, gy = kRW * by + warp, Z0 = (int64_t)CZ * bz;
  const bool inxy = gx < g.nx && gy < g.ny;
  const int64_t c0 = gx + g.nx * gy;
  CgState* st = a.st;
  const double scale = st->rr64 > 0.0 ? 1.0 / sqrt(st->rr64) : 1.0;

  const float4* c32 = static_cast<const float4*>(a.coef);
  const uint2* c16 = static_cast<const uint2*>(a.coef);
  auto inside = [&](int64_t x, int64_t y, int64_t z) {
    return x >= 0 && y >= 0 && z >= 0 && x < g.nx && y < g.ny && z < g.nz;
  };
  auto rec = [&](int64_t x, int64_t y, int64_t z) -> float4 {
    if (!inside(x, y, z)) return make_float4(0.f, 0.f, 0.f, 0.f);
    const int64_t c = x + g.nx * y + g.plane * z;
    if (!a.b16) return __ldg(c32 + c);
    const uint2 u = __ldg(c16 + c);
    return make_float4(bf16_lo(u.x), bf16_hi(u.x), bf16_lo(u.y), bf16_hi(u.y));
  };
  // D of an own cell (BF16 records: formed from the faces as the sweeps do)
  auto diag = [&](int64_t z, const float4& cf) -> float {
    if (!a.b16) return cf.w;
    const float txm = rec(gx - 1, gy, z).x, tym = rec(gx, gy - 1, z).y, tzm = rec(gx, gy, z - 1).z;
    return (((((txm + cf.x) + tym) + cf.y) + tzm) + cf.z) + cf.w;
  };

  // ---- scale, packed coefficients -----------------------------------------------
  uint32_t epoch = *(volatile uint32_t*)a.ctl;
  bool fault = false;
  float tscale = 1.f;
  {
    float dmax = 0.f;
    if (inxy)
      for (int k = 0; k < CZ && Z0 + k < g.nz; ++k)
        dmax = fmaxf(dmax, diag(Z0 + k, rec(gx, gy, Z0 + k)));
    tscale = operator_scale(a, blk, dmax, ++epoch, sh, fault);
  }
  float2* pk = a.packed + ((size_t)blk * CZ * kRW + warp) * 32 + lane;           // (Tx, Tz)
  // D, or M^-1 (Jacobi) where D is in shared memory
  float* pe = reinterpret_cast<float*>(a.packed + (size_t)a.nblk * CZ * kRT) +
              ((size_t)blk * CZ * kRW + warp) * 32 + lane;
  constexpr bool kLoadE = JAC || !LY::kHasD;
  float* sD = sm + LY::kD + tid;
  const float mscale = 1.f / tscale;  // exact: a power of two
  // M^-1 of a cell, 0 outside
  auto minv = [&](int64_t x, int64_t y, int64_t z) -> float {
    if (!inside(x, y, z)) return 0.f;
    const int64_t c = x + g.nx * y + g.plane * z;
    return mscale * (a.b16 ? __ldg(a.dinv + c) : jac_inv(__ldg(c32 + c).w));
  };
  const float tzlo = inxy ? rec(gx, gy, Z0 - 1).z * tscale : 0.f;
#pragma unroll 1
  for (int k = 0; k < CZ; ++k) {
    const int64_t z = Z0 + k;
    const float4 cf = rec(gx, gy, z);
    const bool in = inxy && z < g.nz;
    pk[(size_t)k * kRT] = make_float2(cf.x * tscale, cf.z * tscale);
    const float D = in ? diag(z, cf) * tscale : 0.f;
    if (LY::kHasD) sD[k * kRT] = D;
    if (kLoadE) pe[(size_t)k * kRT] = LY::kHasD ? minv(gx, gy, z) : D;
    sTy[(k * (kRW + 1) + warp + 1) * 32 + lane] = cf.y * tscale;
    if (warp == 0) sTy[k * (kRW + 1) * 32 + lane] = rec(gx, gy - 1, z).y * tscale;
    if (lane == 0) sTx[k * kRW + warp] = rec(gx - 1, gy, z).x * tscale;
    sX[(k * kRW + warp) * 32 + lane] = 0.f;
  }
  for (int i = tid; i < CZ * (kRW + 2) * 34; i += kRT) sP[i] = 0.f;
  __syncthreads();

  // ---- halo cells: 0, 1 below and above; kNY y rows; kNX x cells -------------------
  ResComm<NH, false, 4> cm;
  cm.part = a.part;
  cm.face = a.face;
  cm.nblk = a.nblk;
  cm.blk = blk;
  cm.face_buf = (size_t)a.nblk * LY::kFaces;
  float rz[2] = {0.f, 0.f}, pz[2] = {0.f, 0.f}, qh[NH];
  // y rows: row id warp + 16 j counts (side, k); x cells: tid + 512 j counts (side, w, k)
  // (indices from `ht`, which is made opaque in every iteration: as invariants they
  // would be held in registers)
  int ht = tid;
  auto yk = [&](int j) { return ((ht >> 5) + kRW * j) % CZ; };
  auto yhi = [&](int j) { return (ht >> 5) + kRW * j >= CZ; };
  auto xk = [&](int j) { return (ht + kRT * j) % LY::kFx % CZ; };
  auto xw = [&](int j) { return (ht + kRT * j) % LY::kFx / CZ; };
  auto xhi = [&](int j) { return ht + kRT * j >= LY::kFx; };
  unsigned halo = (bz > 0 ? 1u : 0u) | (bz + 1 < a.nbz ? 2u : 0u);
#pragma unroll
  for (int j = 0; j < LY::kNY; ++j)
    if (yhi(j) ? by + 1 < a.nby : by > 0) halo |= 4u << j;
#pragma unroll
  for (int j = 0; j < LY::kNX; ++j)
    if (tid + kRT * j < 2 * LY::kFx && (xhi(j) ? bx + 1 < a.nbx : bx > 0)) halo |= 4u << (LY::kNY + j);
  auto hoff = [&](int j) {
    constexpr int fy = 2 * LY::kFx, fz = 2 * (LY::kFx + LY::kFy);
    if (j == 0) return (blk - a.nbx * a.nby) * LY::kFaces + fz + LY::kFz + ht;
    if (j == 1) return (blk + a.nbx * a.nby) * LY::kFaces + fz + ht;
    if (j < 2 + LY::kNY) {
      const int w = yk(j - 2) * 32 + (ht & 31);
      return yhi(j - 2) ? (blk + a.nbx) * LY::kFaces + fy + w
                        : (blk - a.nbx) * LY::kFaces + fy + LY::kFy + w;
    }
    const int i = j - 2 - LY::kNY, w = (ht + kRT * i) % LY::kFx;
    return xhi(i) ? (blk + 1) * LY::kFaces + w : (blk - 1) * LY::kFaces + LY::kFx + w;
  };
  auto has = [&](int j) { return ((halo >> j) & 1u) != 0u; };
  const FaceWords<decltype(has), decltype(hoff)> wd{has, hoff};
  // the vector of a cell: r, or z = M^-1 r
  auto halo_r = [&](int64_t x, int64_t y, int64_t z) -> float {
    if (!inside(x, y, z)) return 0.f;
    const float v = (float)(scale * a.r64[x + g.nx * y + g.plane * z]);
    return JAC ? v * minv(x, y, z) : v;
  };
  {
    rz[0] = halo_r(gx, gy, Z0 - 1);
    rz[1] = halo_r(gx, gy, Z0 + CZ);
#pragma unroll
    for (int j = 0; j < LY::kNY; ++j) {
      const int64_t y = kRW * (int64_t)by + (yhi(j) ? kRW : -1), z = Z0 + yk(j);
      sRh[j * kRT + tid] = halo_r(gx, y, z);
    }
#pragma unroll
    for (int j = 0; j < LY::kNX; ++j) {
      const bool use = tid + kRT * j < 2 * LY::kFx;
      const int64_t x = 32 * (int64_t)bx + (xhi(j) ? 32 : -1), y = kRW * (int64_t)by + xw(j),
                    z = Z0 + xk(j);
      sRh[(LY::kNY + j) * kRT + tid] = use ? halo_r(x, y, z) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < NH; ++j) qh[j] = 0.f;
  }

  float r[CZ], q[CZ];
#pragma unroll
  for (int k = 0; k < CZ; ++k) {
    r[k] = halo_r(gx, gy, Z0 + k);
    q[k] = 0.f;
  }

  float alpha = 0.f, beta = 0.f;
  int done = kRunning;
  if (tid == 0) sh.sc.init();
  uint2* fmine = a.face + (size_t)blk * LY::kFaces;

  auto step = [&](bool dir, Acc& s0) {
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      if (!((halo >> j) & 1u)) continue;
      rz[j] = fmaf(-alpha, qh[j], rz[j]);
      if (dir) pz[j] = fmaf(beta, pz[j], rz[j]);
    }
#pragma unroll
    for (int j = 0; j < LY::kNY + LY::kNX; ++j) {
      if (!((halo >> (2 + j)) & 1u)) continue;
      const float rn = fmaf(-alpha, qh[2 + j], sRh[j * kRT + ht]);
      sRh[j * kRT + ht] = rn;
      if (!dir) continue;
      const int i = j - LY::kNY;
      float* ps = j < LY::kNY ? sP + (yk(j) * (kRW + 2) + (yhi(j) ? kRW + 1 : 0)) * 34 + (ht & 31) + 1
                              : sP + (xk(i) * (kRW + 2) + xw(i) + 1) * 34 + (xhi(i) ? 33 : 0);
      *ps = fmaf(beta, *ps, rn);
    }
    float s = 0.f;
#pragma unroll
    for (int k = 0; k < CZ; ++k) {
      float* ps = sP + (k * (kRW + 2) + warp + 1) * 34 + lane + 1;
      float* xs = sX + (k * kRW + warp) * 32 + lane;
      const float p0 = *ps;
      *xs = fmaf(alpha, p0, *xs);
      r[k] = fmaf(-alpha, q[k], r[k]);
      if (dir) *ps = fmaf(beta, p0, r[k]);
      if (JAC && dir) continue;  // r'z is formed with D, in the stencil
      const float D = !JAC ? 1.f : LY::kHasD ? sD[k * kRT] : __ldcg(pe + (size_t)k * kRT);
      s = fmaf(JAC ? r[k] * D : r[k], r[k], s);
      if ((k & 3) == 3) {
        kadd(s0, s);
        s = 0.f;
      }
    }
  };

  while (!fault) {
    asm volatile("" : "+r"(ht));
    Acc acc[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    // the first planes' coefficients, in flight during the step
    constexpr int kPre = 4;
    float2 tc[kPre];
    float ec[kPre];
#pragma unroll
    for (int k = 0; k < kPre; ++k) {
      tc[k] = __ldcg(pk + (size_t)k * kRT);
      if (kLoadE) ec[k] = __ldcg(pe + (size_t)k * kRT);
    }
    step(true, acc[0]);
    __syncthreads();
    ++epoch;
    uint2* fo = fmine + (epoch & 1u) * cm.face_buf;
    float s0 = 0.f, s1 = 0.f, s2 = 0.f, s3 = 0.f;
    float tz0 = tzlo, pm = pz[0];
    float pc = sP[(warp + 1) * 34 + lane + 1];
#pragma unroll
    for (int k = 0; k < CZ; ++k) {
      const float* ps = sP + (k * (kRW + 2) + warp + 1) * 34 + lane + 1;
      const float pp = k + 1 < CZ ? ps[(kRW + 2) * 34] : pz[1];
      const float* ty = sTy + (k * (kRW + 1) + warp) * 32 + lane;
      const float2 t = tc[k % kPre];
      const float D = LY::kHasD ? sD[k * kRT] : ec[k % kPre];
      const float m = !JAC ? 1.f : LY::kHasD ? ec[k % kPre] : jac_inv(D);
      if (k + kPre < CZ) {
        tc[k % kPre] = __ldcg(pk + (size_t)(k + kPre) * kRT);
        if (kLoadE) ec[k % kPre] = __ldcg(pe + (size_t)(k + kPre) * kRT);
      }
      float txm = __shfl_up_sync(kFull, t.x, 1);
      if (lane == 0) txm = sTx[k * kRW + warp];
      const float4 cf = make_float4(t.x, ty[32], t.y, D);
      const float v = stencil7(cf, txm, ty[0], tz0, pc, ps[1], ps[-1], ps[34], ps[-34], pp, pm);
      q[k] = JAC ? v * m : v;
      if (JAC) s0 = fmaf(r[k] * D, r[k], s0);
      s1 = fmaf(pc, v, s1);
      s2 = fmaf(r[k], v, s2);
      s3 = fmaf(v, q[k], s3);
      if ((k & 3) == 3) {
        if (JAC) kadd(acc[0], s0);
        kadd(acc[1], s1);
        kadd(acc[2], s2);
        kadd(acc[3], s3);
        s0 = s1 = s2 = s3 = 0.f;
      }
      tz0 = t.y;
      pm = pc;
      pc = pp;
    }
    if (bz > 0) ll_store(fo + 2 * (LY::kFx + LY::kFy) + tid, q[0], epoch);
    if (bz + 1 < a.nbz) ll_store(fo + 2 * (LY::kFx + LY::kFy) + LY::kFz + tid, q[CZ - 1], epoch);
    if ((warp == 0 && by > 0) || (warp == kRW - 1 && by + 1 < a.nby)) {
      uint2* f = fo + 2 * LY::kFx + (warp == 0 ? 0 : LY::kFy) + lane;
#pragma unroll
      for (int k = 0; k < CZ; ++k) ll_store(f + k * 32, q[k], epoch);
    }
    if (bx > 0 || bx + 1 < a.nbx) {
#pragma unroll
      for (int h = 0; h < CZ; h += 16) {
        float v = 0.f;
#pragma unroll
        for (int k = h; k < h + 16 && k < CZ; ++k) {
          const float t = __shfl_sync(kFull, q[k], lane < 16 ? 0 : 31);
          if ((lane & 15) == k - h) v = t;
        }
        if (h + (lane & 15) < CZ && (lane < 16 ? bx > 0 : bx + 1 < a.nbx))
          ll_store(fo + (lane < 16 ? 0 : LY::kFx) + warp * CZ + h + (lane & 15), v, epoch);
      }
    }
    Dfl mine[4], tot[4];
#pragma unroll
    for (int v = 0; v < 4; ++v) mine[v] = df_fast(acc[v].s, -acc[v].c);
    if (!cm.template exchange<true>(a, mine, epoch, wd, tot, qh, sh)) {
      fault = true;
      break;
    }
    if (warp == 0) {
      ResScalars sc = sh.sc;
      sc.update(tot, a.rtol2, a.maxit);
      if (lane == 0) {
        sh.sc = sc;
        sh.next = {sc.alpha, sc.beta, sc.done};
      }
    }
    __syncthreads();
    alpha = sh.next.alpha;
    beta = sh.next.beta;
    done = sh.next.done;
    if (done == kRunning) continue;
    if (done != kConvEst && done != kMaxit) break;
    // the last step, and the true r'r of the residual it leaves (no face words)
    Acc rr = {0.f, 0.f};
    step(false, rr);
    ++epoch;
    mine[0] = df_fast(rr.s, -rr.c);
    mine[1] = mine[2] = mine[3] = {0.f, 0.f};
    const bool ok = cm.template exchange<false>(a, mine, epoch, wd, tot, qh, sh);
    if (!ok) {
      fault = true;
      break;
    }
    if (warp == 0) {
      ResScalars sc = sh.sc;
      sc.finish(tot, a.maxit);
      if (lane == 0) {
        sh.sc = sc;
        sh.next = {sc.alpha, sc.beta, sc.done};
      }
    }
    __syncthreads();
    alpha = sh.next.alpha;
    beta = sh.next.beta;
    done = sh.next.done;
    if (done != kRunning) break;
  }

  // a wait that ran out in any block, be it the last one's, whose brick then lacks its
  // correction, is a failure of the solve (the host clears the flag)
  if (fault && tid == 0) *(volatile int*)&st->fault = 1;
  if (fault) done = kGuard;
  if (done != kNonFinite && done != kGuard && inxy) {
    const double inv = (double)tscale / scale;
    for (int k = 0; k < CZ && Z0 + k < g.nz; ++k) {
      const int64_t c = c0 + g.plane * (Z0 + k);
      a.x64[c] = fma((double)sX[(k * kRW + warp) * 32 + lane], inv, a.x64[c]);
    }
  }
  if (blk == 0 && tid == 0) {
    sh.sc.report(st, scale, fault);
    *(volatile uint32_t*)a.ctl = epoch;
  }
}

template <int CZ>
cudaError_t launch_big(ResProb& a, bool jac, cudaStream_t s) {
  constexpr int smem = BigLayout<CZ>::kFloats * 4;
  const void* fn = jac ? (const void*)resident_big_kernel<CZ, true>
                       : (const void*)resident_big_kernel<CZ, false>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(fn, dim3(a.nblk), dim3(kRT), args, smem, s);
}
template <int CZ, bool JAC>
__global__ void __launch_bounds__(kRT, 1) resident_kernel(const __grid_constant__ ResProb a) {
  extern __shared__ __align__(16) float sm[];
  __shared__ ResShared sh;
  resident_solve<CZ, JAC, false>(a, blockIdx.x, sm, sh);
}

// ---- many instances in one launch --------------------------------------------
// One block per SM; the instances' inner solves run on teams of blocks.  A team
// needs all its blocks at once, so teams are formed by a scheduler in device
// memory, run under a lock by the first warp of a block whose team has finished
// (at the start: of block 0): it returns the team's blocks to the free list,
// then starts the largest waiting instance that fits the free blocks, and so on
// down the list.  Free blocks wait for a word in their mailbox.  A started team
// always has all its blocks, so every wait ends.
//
// A free block waits for as long as other teams run, which a solve of many
// iterations stretches at will, so its limit is on looks without progress: every
// running team counts up a word once in kBeat iterations, and so does every release.
struct ResSched {
  int lock, nfree, left;   // left: instances not yet started
  uint32_t beat;
};
constexpr uint32_t kExit = 0xffffffffu;

struct ResBatchArgs {
  const ResProb* prob;  // sorted by blocks, largest first
  int nprob, nblocks;
  ResSched* sched;      // zeroed before the launch, like the arrays that follow
  int* started;         // [nprob]
  int* freel;           // [nblocks] free block ids
  uint32_t* sent;       // [nblocks] words sent to a block so far
  unsigned long long* mail;  // [nblocks] {message, sequence number}
  uint32_t* abort;      // the instances' abort flag, shared
  uint32_t look_limit;  // looks of a free block without progress before it gives up
};

// Returns `n` blocks (members, or all blocks when null) to the free list and starts what
// fits.  One whole warp.
__device__ void sched_release(const ResBatchArgs& a, const int* members, int n) {
  const int lane = threadIdx.x & 31;
  if (lane == 0) {
    uint32_t polls = 0;
    while (atomicCAS(&a.sched->lock, 0, 1) != 0) {
      if (++polls >= kResPollLimit) {
        *(volatile uint32_t*)a.abort = 1u;
        break;
      }
    }
    __threadfence();
  }
  __syncwarp();
  if (*(volatile uint32_t*)a.abort != 0u) return;
  volatile int* fl = a.freel;
  volatile int* st = a.started;
  int nfree = *(volatile int*)&a.sched->nfree, left = *(volatile int*)&a.sched->left;
  for (int j = lane; j < n; j += 32) fl[nfree + j] = members != nullptr ? *(volatile const int*)(members + j) : j;
  nfree += n;
  __syncwarp();
  auto send = [&](int id, uint32_t msg) {
    volatile uint32_t* c = a.sent + id;
    const uint32_t q = *c + 1u;
    *c = q;
    const unsigned long long w = (unsigned long long)msg | ((unsigned long long)q << 32);
    asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(a.mail + id), "l"(w) : "memory");
  };
  for (int i0 = 0; i0 < a.nprob && left > 0 && nfree > 0;) {
    const int i = i0 + lane;
    const bool fits = i < a.nprob && st[i] == 0 && a.prob[i].nblk <= nfree;
    const unsigned m = __ballot_sync(kFull, fits);
    if (m == 0u) {
      i0 += 32;
      continue;
    }
    const int p = i0 + __ffs(m) - 1;
    const int need = a.prob[p].nblk;
    int* mem = a.prob[p].team;
    for (int j = lane; j < need; j += 32) *(volatile int*)(mem + j) = fl[nfree - 1 - j];
    __threadfence();  // the team's list before its first block's message
    __syncwarp();
    for (int j = lane; j < need; j += 32)
      send(fl[nfree - 1 - j], ((uint32_t)p << 12) | (uint32_t)j);
    if (lane == 0) st[p] = 1;
    nfree -= need;
    --left;
    __syncwarp();
  }
  if (left == 0) {  // nothing waits any more: the free blocks leave
    for (int j = lane; j < nfree; j += 32) send(fl[j], kExit);
    nfree = 0;
  }
  __syncwarp();
  if (lane == 0) {
    atomicAdd(&a.sched->beat, 1u);
    *(volatile int*)&a.sched->nfree = nfree;
    *(volatile int*)&a.sched->left = left;
    __threadfence();
    atomicExch(&a.sched->lock, 0);
  }
  __syncwarp();
}

// One brick height per launch: with every height in one body the compiler spilled
// 1.2 KB per thread (32 instances with Jacobi: 116 instead of 83 ms).
template <int CZ, bool JAC>
__global__ void __launch_bounds__(kRT, 1) resident_batch_kernel(const __grid_constant__ ResBatchArgs a) {
  extern __shared__ __align__(16) float sm[];
  __shared__ ResShared sh;
  __shared__ ResProb prob;  // shared memory: no registers held for its fields
  __shared__ uint32_t msg;
  const int me = blockIdx.x, warp = threadIdx.x >> 5;
  if (me == 0 && warp == 0) {
    if (threadIdx.x == 0) *(volatile int*)&a.sched->left = a.nprob;
    __syncwarp();
    sched_release(a, nullptr, a.nblocks);
  }
  for (uint32_t seq = 1;; ++seq) {
    if (threadIdx.x == 0) {
      uint32_t got = kExit, beat = 0u;
      for (uint32_t polls = 0;; ++polls) {
        const uint2 w = ll_load(reinterpret_cast<const uint2*>(a.mail + me));
        if (w.y == seq) {
          got = w.x;
          break;
        }
        if (*(volatile uint32_t*)a.abort != 0u) break;
        if (polls >= a.look_limit) {
          const uint32_t now = *(volatile uint32_t*)&a.sched->beat;
          if (now == beat) {
            // a team started from now on could not have this block: none may wait for it
            *(volatile uint32_t*)a.abort = 1u;
            break;
          }
          beat = now;
          polls = 0;
        }
        __nanosleep(200);
      }
      msg = got;
      if (got != kExit) prob = a.prob[got >> 12];
    }
    __syncthreads();
    const uint32_t m = msg;
    if (m == kExit) return;
    const int rank = (int)(m & 4095u);
    resident_solve<CZ, JAC, true>(prob, rank, sm, sh);
    __syncthreads();
    // the blocks of a team end in the same iteration: its first block returns
    // them together, so that a large instance waiting for that many blocks is
    // not starved by small ones
    if (rank == 0 && warp == 0) sched_release(a, prob.team, prob.nblk);
  }
}

template <int CZ, bool JAC>
cudaError_t launch_t(ResProb& a, cudaStream_t s) {
  constexpr int smem = ResLayout<CZ>::floats(JAC) * 4;
  auto fn = resident_kernel<CZ, JAC>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel((const void*)fn, dim3(a.nblk), dim3(kRT), args, smem, s);
}

template <int CZ>
cudaError_t launch_cz(ResProb& a, bool jac, cudaStream_t s) {
  return jac ? launch_t<CZ, true>(a, s) : launch_t<CZ, false>(a, s);
}

template <int CZ>
cudaError_t launch_batch_cz(ResBatchArgs& a, bool jac, cudaStream_t s) {
  const int smem = ResLayout<CZ>::floats(jac) * 4;
  const void* fn = jac ? (const void*)resident_batch_kernel<CZ, true>
                       : (const void*)resident_batch_kernel<CZ, false>;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e != cudaSuccess) return e;
  void* args[] = {&a};
  return cudaLaunchCooperativeKernel(fn, dim3(a.nblocks), dim3(kRT), args, smem, s);
}

size_t sched_words(int nprob, int nblocks) {  // 8-byte words after the sums and faces
  return 4 + (size_t)nblocks + ((size_t)nprob + 2 * (size_t)nblocks + 1) / 2 + 2;
}

}  // namespace

// The lowest brick that gives every brick an SM of its own: time grows with the
// height (0.2 us per plane up to 16, 0.28 above, where the coefficients come from
// L2) and hardly with the number of blocks.  dense: batches, where an SM not taken
// by one instance works on another, so the cost is blocks times their time; one
// kernel per height, hence few of them.  Every grid that fits takes this path: it
// is 2.9 times as fast as the sweeps even at the largest (160x160x96: 10.9 us per
// iteration against 31.8).
bool plan_resident(const Grid& g, int num_sms, bool dense, ResPlan* p) {
  const int64_t bx = (g.nx + 31) / 32, by = (g.ny + kRW - 1) / kRW;
  if (bx * by > num_sms) return false;
  constexpr int fast[] = {1, 2, 4, 6, 8, 12, 16, 24, 32}, packed[] = {4, 8, 16};
  const int* heights = dense ? packed : fast;
  const int nh = dense ? 3 : 9;
  double best = 0.0;
  int cz = 0;
  for (int h = 0; h < nh; ++h) {
    const int64_t n = bx * by * ((g.nz + heights[h] - 1) / heights[h]);
    if (n > num_sms) continue;
    const double cost = dense ? (double)n * (1.9 + 0.21 * heights[h]) : (double)heights[h];
    if (cz == 0 || cost < best) {
      best = cost;
      cz = heights[h];
    }
  }
  if (cz == 0) return false;
  p->cz = cz;
  p->nbx = (int)bx;
  p->nby = (int)by;
  p->nbz = (int)((g.nz + cz - 1) / cz);
  p->nblk = p->nbx * p->nby * p->nbz;
  // control words, sums, faces (two buffers each)
  p->words = 32 + (size_t)2 * p->nblk * 8 +
             (size_t)2 * p->nblk * (2 * ((size_t)cz * kRW + (size_t)cz * 32 + kRW * 32));
  p->packed = cz > 16 ? (size_t)p->nblk * cz * kRT * 12 : 0;
  return true;
}

ResProb make_res_prob(const Grid& g, const ResPlan& p, const void* coef, bool b16,
                      const float* dinv, const double* r64, double* x64, CgState* st, double rtol,
                      long long maxit, unsigned long long* comm) {
  ResProb a;
  a.g = g;
  a.cz = p.cz;
  a.nbx = p.nbx;
  a.nby = p.nby;
  a.nbz = p.nbz;
  a.nblk = p.nblk;
  a.coef = coef;
  a.b16 = b16 ? 1 : 0;
  a.dinv = dinv;
  a.r64 = r64;
  a.x64 = x64;
  a.st = st;
  a.rtol2 = rtol * rtol;
  a.maxit = maxit;
  a.ctl = reinterpret_cast<uint32_t*>(comm);
  a.abort = a.ctl + 1;
  a.part = reinterpret_cast<uint2*>(comm + 32);
  a.face = a.part + (size_t)2 * p.nblk * 8;
  a.team = nullptr;
  a.packed = nullptr;
  a.beat = nullptr;
  a.poll_limit = kResPollLimit;
  return a;
}

cudaError_t launch_resident(const ResProb& prob, bool jac, cudaStream_t s) {
  ResProb a = prob;
  switch (a.cz) {
    case 1: return launch_cz<1>(a, jac, s);
    case 2: return launch_cz<2>(a, jac, s);
    case 4: return launch_cz<4>(a, jac, s);
    case 6: return launch_cz<6>(a, jac, s);
    case 8: return launch_cz<8>(a, jac, s);
    case 12: return launch_cz<12>(a, jac, s);
    case 16: return launch_cz<16>(a, jac, s);
    case 24: return launch_big<24>(a, jac, s);
    case 32: return launch_big<32>(a, jac, s);
    default: return cudaErrorInvalidValue;
  }
}

size_t resident_batch_words(int nprob, int num_sms) { return sched_words(nprob, num_sms); }
uint32_t* resident_batch_abort(unsigned long long* sched) {
  return reinterpret_cast<uint32_t*>(sched + 2);
}
uint32_t* resident_batch_beat(unsigned long long* sched) {
  return &reinterpret_cast<ResSched*>(sched)->beat;
}

cudaError_t launch_resident_batch(const ResProb* prob_dev, int nprob, int cz, int num_sms, bool jac,
                                  unsigned long long* sched, uint32_t look_limit, cudaStream_t s) {
  const size_t words = sched_words(nprob, num_sms);
  cudaError_t e = cudaMemsetAsync(sched, 0, words * 8, s);
  if (e != cudaSuccess) return e;
  ResBatchArgs a;
  a.prob = prob_dev;
  a.nprob = nprob;
  a.nblocks = num_sms;
  a.sched = reinterpret_cast<ResSched*>(sched);
  a.abort = resident_batch_abort(sched);
  a.look_limit = look_limit;
  a.mail = sched + 4;
  a.started = reinterpret_cast<int*>(sched + 4 + num_sms);
  a.freel = a.started + nprob;
  a.sent = reinterpret_cast<uint32_t*>(a.freel + num_sms);
  switch (cz) {
    case 4: return launch_batch_cz<4>(a, jac, s);
    case 8: return launch_batch_cz<8>(a, jac, s);
    case 16: return launch_batch_cz<16>(a, jac, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace tpfa
