// 3x3x3 convolutions of BF16 channels-last volumes on the tcgen05 tensor
// cores (implicit GEMM, FP32 accumulation in tensor memory).
//
// Forward (and input gradient).  The default is conv_fwd_ws_kernel: tiles of 8 x 16
// voxels followed through the planes, whole voxel rows copied in the copy engine's
// swizzle.  Kernels 0 to 2, taken by selection, stage blocks of 8 channels; kernel 0:
//
// An output tile is 128 consecutive voxel indices of the haloed layout (halo
// voxels inside the range are computed and discarded).  For one z-offset dz the three rows dy = -1, 0, 1 of 130
// voxels (the tile plus one voxel either side) are copied to shared memory
// as "row groups" in the K-major core-matrix layout [CIN/8][130][8 channels],
// i.e. 16 bytes per voxel and channel block.  With M-direction stride 128
// bytes per 8 voxels, tap (dy, dx) of the GEMM operand A[m][ci] =
// x[s0 + m + off][ci] is the row group of dy started dx voxels later -- a
// descriptor offset of 16 dx bytes, no data movement.  Each (dz, dy, dx, 16
// channel) step is one tcgen05.mma with M = 128, N = COUT, K = 16 against
// the weights of that tap, which sit in shared memory for the whole
// persistent CTA.  The dz row-group triples are double-buffered: the copy
// of the next one runs while the tensor core works on the current one.
// Epilogue: bias, ReLU or a ReLU-derivative mask, BF16 rounding, halo skip.
// The input gradient of a convolution is the same operation with the taps
// flipped and the weight matrices transposed.
//
// Weight gradient: see conv_wgrad_kernel.
#include <cuda_bf16.h>

#include "net_internal.cuh"
#include "tc_common.cuh"
#include "tpfa_internal.cuh"

namespace tpfa {
namespace net {

// Set (never cleared by a kernel) when a bounded tensor-core wait gave up.
__device__ int g_tc_timeout;

namespace {

constexpr uint32_t kWaitLimit = 1u << 22;  // mbarrier polls before giving up
constexpr int kRG = 130;                   // voxels per staged row group

__device__ __forceinline__ void cp16z(void* dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(tc::smem_addr(dst)),
               "l"(src), "r"(ok ? 16 : 0)
               : "memory");
}
__device__ __forceinline__ void cp_commit_group() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
__device__ __forceinline__ void cp_wait_all() { asm volatile("cp.async.wait_all;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait_groups() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory");
}

__device__ __forceinline__ bool bf16_positive(uint32_t h) {
  return (h & 0x8000u) == 0 && (h & 0x7fffu) != 0;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&v);
}

// stages of the row-group ring: as deep as shared memory allows several CTAs
// per SM for the small layers; the 64-channel layers hold 110 KB of weights
template <int CIN, int COUT>
constexpr int fwd_stages() {
  return (CIN == 16) ? 4 : (CIN == 32 && COUT == 16) ? 3 : 2;
}

template <int CIN, int COUT>
struct FwdCfg {
  static constexpr int kS = fwd_stages<CIN, COUT>();
  static constexpr int kWTap = COUT * CIN * 2;  // bytes of one tap's weight matrix
  static constexpr int kWBytes = 27 * kWTap;
  static constexpr int kRGBytes = kRG * CIN * 2;
  static constexpr int kStage = 3 * kRGBytes;
  static constexpr int kSmem = kWBytes + kS * kStage;
  static constexpr uint32_t kCols = COUT < 32 ? 32 : COUT;
  static_assert(CIN % 16 == 0 && COUT % 16 == 0 && COUT <= 256, "shape");
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(128)
conv_fwd_kernel(const uint16_t* __restrict__ x, const uint16_t* __restrict__ w,
                const float* __restrict__ bias, const uint16_t* __restrict__ mask,
                uint16_t* __restrict__ y, Vol g, int flags, int ntiles) {
  using Cfg = FwdCfg<CIN, COUT>;
  constexpr int kc = CIN / 8;
  constexpr int S = Cfg::kS;
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ __align__(8) uint64_t bars[S];
  __shared__ uint32_t tbase;
  unsigned char* sW = sm;
  unsigned char* sS = sm + Cfg::kWBytes;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  for (int i = tid; i < 27 * COUT * kc; i += 128) {
    const int c = i % kc, r = (i / kc) % COUT, t = i / (kc * COUT);
    const uint4 v = *reinterpret_cast<const uint4*>(w + ((size_t)t * COUT + r) * CIN + c * 8);
    *reinterpret_cast<uint4*>(sW + t * Cfg::kWTap + tc::kmajor_off(r, c * 8, CIN)) = v;
  }
  if (tid == 0)
    for (int b = 0; b < S; ++b) tc::mbar_init(&bars[b], 1);
  if (warp == 0) tc::tmem_alloc(&tbase, Cfg::kCols);
  tc::fence_proxy_async();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t acc = tbase;

  const int my_tiles = (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  const int njobs = 3 * my_tiles;  // job = (tile, dz)

  // copies of job j into buffer j % S; every call commits one group (empty
  // past the last job) so that wait_group counts stay uniform
  auto load_job = [&](int j) {
    if (j < njobs) {
      const int tile = blockIdx.x + (j / 3) * gridDim.x;
      const int dz = j % 3 - 1;
      const int base = g.g0 + tile * 128 + dz * g.pp - g.wp - 1;
      unsigned char* st = sS + (j % S) * Cfg::kStage;
      for (int i = tid; i < 3 * kRG * kc; i += 128) {
        const int c = i % kc, v = (i / kc) % kRG, gi = i / (kc * kRG);
        const int row = base + gi * g.wp + v;
        const bool ok = row >= 0 && row < g.vp;
        cp16z(st + gi * Cfg::kRGBytes + c * (kRG * 16) + v * 16,
              x + (size_t)(ok ? row : 0) * CIN + c * 8, ok);
      }
    }
    cp_commit_group();
  };

  bool abort = false;
  for (int j = 0; j < S - 1; ++j) load_job(j);
  for (int j = 0; j < njobs; ++j) {
    const int buf = j % S;
    cp_wait_groups<S - 2>();  // job j's group is complete
    tc::fence_proxy_async();
    __syncthreads();
    if (tid == 0) {
      tc::fence_after();
      const int dzi = j % 3;
      const uint32_t st = tc::smem_addr(sS + buf * Cfg::kStage);
      const uint32_t wb = tc::smem_addr(sW);
      constexpr uint32_t idesc = tc::idesc_bf16_f32(128, COUT);
#pragma unroll 1
      for (int gi = 0; gi < 3; ++gi) {
#pragma unroll
        for (int dx = 0; dx < 3; ++dx) {
          const int t = dzi * 9 + gi * 3 + dx;
#pragma unroll
          for (int ks = 0; ks < CIN / 16; ++ks) {
            const uint64_t ad = tc::smem_desc(st + gi * Cfg::kRGBytes + dx * 16 + ks * 2 * kRG * 16,
                                              kRG * 16, 128);
            const uint64_t bd = tc::smem_desc(wb + t * Cfg::kWTap + ks * 256, 128, kc * 128);
            tc::mma_bf16(acc, ad, bd, idesc, (dzi | gi | dx | ks) != 0);
          }
        }
      }
      tc::mma_commit(&bars[buf]);
    }
    // job j+S-1 reuses the buffer of job j-1: wait for that job's MMAs
    bool ok = true;
    if (j >= 1 && j + S - 1 < njobs)
      ok = tc::mbar_wait(&bars[(j - 1) % S], ((j - 1) / S) & 1, kWaitLimit);
    if (__syncthreads_or(!ok)) {
      abort = true;
      break;
    }
    load_job(j + S - 1);
    if (j % 3 == 2) {
      const bool done = tc::mbar_wait(&bars[buf], (j / S) & 1, kWaitLimit);
      if (__syncthreads_or(!done)) {
        abort = true;
        break;
      }
      tc::fence_after();
      const int tile = blockIdx.x + (j / 3) * gridDim.x;
      const int idx = g.g0 + tile * 128 + warp * 32 + lane;
      const bool in = vol_interior(g, idx);
#pragma unroll
      for (int c0 = 0; c0 < COUT; c0 += 8) {
        float v[8];
        tc::tmem_ld8(acc + ((uint32_t)(warp * 32) << 16) + c0, v);
        if (in) {
          uint4 mk = make_uint4(0, 0, 0, 0);
          if (flags & kConvMask) mk = *reinterpret_cast<const uint4*>(mask + (size_t)idx * COUT + c0);
          const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
          uint32_t o[4];
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            float a = v[2 * h], b = v[2 * h + 1];
            if (bias) {
              a += bias[c0 + 2 * h];
              b += bias[c0 + 2 * h + 1];
            }
            if (flags & kConvRelu) {
              a = fmaxf(a, 0.f);
              b = fmaxf(b, 0.f);
            }
            if (flags & kConvMask) {
              if (!bf16_positive(mw[h] & 0xffffu)) a = 0.f;
              if (!bf16_positive(mw[h] >> 16)) b = 0.f;
            }
            o[h] = pack_bf16(a, b);
          }
          *reinterpret_cast<uint4*>(y + (size_t)idx * COUT + c0) = make_uint4(o[0], o[1], o[2], o[3]);
        }
      }
      tc::fence_before();
    }
  }
  cp_wait_all();
  if (abort && tid == 0) atomicOr(&g_tc_timeout, 1);
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(acc, Cfg::kCols);
}

// ---- z-marching forward kernel ---------------------------------------------
// A work unit is one 128-voxel segment of a padded plane (offset bi * 128)
// followed through zc consecutive interior planes of one sample.  Output k of
// the unit needs the row-group triples of planes k-1, k, k+1; triple j of the
// unit goes to ring slot j % ST and is loaded once, ST - 3 outputs ahead of its
// first use, instead of three times.  Two TMEM accumulators alternate between
// outputs so that the epilogue of output k-1 runs while the tensor core works
// on output k.
template <int CIN, int COUT>
constexpr int zm_stages() {
  return (CIN == 32 && COUT == 64) ? 4 : (CIN == 16) ? 7 : 5;
}

template <int CIN, int COUT>
struct ZmCfg {
  static constexpr int kST = zm_stages<CIN, COUT>();
  static constexpr int kWTap = COUT * CIN * 2;
  static constexpr int kWBytes = 27 * kWTap;
  static constexpr int kRGBytes = kRG * CIN * 2;
  static constexpr int kTriple = 3 * kRGBytes;
  static constexpr int kSmem = kWBytes + kST * kTriple;
  static constexpr uint32_t kCols = 2 * COUT < 32 ? 32 : 2 * COUT;  // two accumulators
  static_assert(kSmem <= 227 * 1024, "shared memory");
};

struct ZmGrid {
  int nb;   // 128-voxel segments (or tiles, nbx of them along x) per plane
  int nbx;
  int zc;   // interior planes per unit
  int nzc;  // units per sample along z
  int units;
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(128)
conv_fwd_zm_kernel(const uint16_t* __restrict__ x, const uint16_t* __restrict__ w,
                   const float* __restrict__ bias, const uint16_t* __restrict__ mask,
                   uint16_t* __restrict__ y, Vol g, int flags, ZmGrid zg) {
  using Cfg = ZmCfg<CIN, COUT>;
  constexpr int ST = Cfg::kST;
  constexpr int kc = CIN / 8;
  constexpr int kChunks = 3 * kRG * kc;            // 16-byte copies per triple
  constexpr int kPer = (kChunks + 127) / 128;      // per thread
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ uint32_t tbase;
  __shared__ float sbias[COUT];
  unsigned char* sW = sm;
  unsigned char* sR = sm + Cfg::kWBytes;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  for (int i = tid; i < 27 * COUT * kc; i += 128) {
    const int c = i % kc, r = (i / kc) % COUT, t = i / (kc * COUT);
    const uint4 v = *reinterpret_cast<const uint4*>(w + ((size_t)t * COUT + r) * CIN + c * 8);
    *reinterpret_cast<uint4*>(sW + t * Cfg::kWTap + tc::kmajor_off(r, c * 8, CIN)) = v;
  }
  if (tid < COUT) sbias[tid] = bias ? bias[tid] : 0.f;
  if (tid == 0) {
    tc::mbar_init(&bars[0], 1);
    tc::mbar_init(&bars[1], 1);
  }
  if (warp == 0) tc::tmem_alloc(&tbase, Cfg::kCols);
  // this thread's copies of a triple: row offset from the triple's first row,
  // and byte offset inside the ring slot
  int roff[kPer], coff[kPer];
  uint32_t soff[kPer];
#pragma unroll
  for (int m = 0; m < kPer; ++m) {
    const int i = tid + 128 * m;
    const int c = i % kc, v = (i / kc) % kRG, gi = i / (kc * kRG);
    roff[m] = gi * g.wp + v;
    coff[m] = c * 8;
    soff[m] = (uint32_t)(gi * Cfg::kRGBytes + c * (kRG * 16) + v * 16);
  }
  tc::fence_proxy_async();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t acc0 = tbase;
  // descriptors of ring slot 0 (A) and of the weights (B); a byte offset d
  // inside shared memory adds d >> 4 to the start-address field
  const uint64_t adesc0 = tc::smem_desc(tc::smem_addr(sR), kRG * 16, 128);
  const uint64_t bdesc0 = tc::smem_desc(tc::smem_addr(sW), 128, kc * 128);

  bool abort = false;
  int o = 0;  // outputs issued by this CTA (accumulator and barrier phase)
  for (int u = blockIdx.x; u < zg.units && !abort; u += gridDim.x) {
    const int bi = u % zg.nb, cz = u / zg.nb;
    const int sidx = cz / zg.nzc;
    const int z0 = (cz % zg.nzc) * zg.zc;
    const int nout = min(zg.zc, g.nz - z0);
    const int kp0 = sidx * g.dp + 1 + z0;  // padded plane of output 0
    const int seg = bi * 128;              // offset of the segment in its plane
    const int ntrip = nout + 2;            // triples: planes kp0-1 .. kp0+nout
    // this thread's output voxel in the plane: interior in x and y (every
    // plane of a unit is interior in z)
    const int poff = seg + warp * 32 + lane;
    const int px = poff % g.wp, py = poff / g.wp;
    const bool in_xy = poff < g.pp && px >= 1 && px <= g.nx && py >= 1 && py <= g.ny;
    auto load_triple = [&](int j) {
      if (j < ntrip) {
        const int base = seg + (kp0 - 1 + j) * g.pp - g.wp - 1;
        unsigned char* st = sR + (j % ST) * Cfg::kTriple;
#pragma unroll
        for (int m = 0; m < kPer; ++m) {
          if (kChunks % 128 == 0 || tid + 128 * m < kChunks) {
            const int row = base + roff[m];
            const bool ok = row >= 0 && row < g.vp;
            cp16z(st + soff[m], x + (size_t)(ok ? row : 0) * CIN + coff[m], ok);
          }
        }
      }
      cp_commit_group();
    };
    for (int j = 0; j < ST; ++j) load_triple(j);

    auto epilogue = [&](int k, int ok_) {
      const size_t idx = (size_t)(kp0 + k) * g.pp + poff;
      const uint32_t acc = acc0 + (uint32_t)((ok_ & 1) * COUT);
      float va[COUT];
      tc::tmem_ld_cols<COUT>(acc + ((uint32_t)(warp * 32) << 16), va);
#pragma unroll
      for (int c0 = 0; c0 < COUT; c0 += 8) {
        const float* v = va + c0;
        if (in_xy) {
          uint4 mk = make_uint4(0, 0, 0, 0);
          if (flags & kConvMask) mk = *reinterpret_cast<const uint4*>(mask + idx * COUT + c0);
          const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
          uint32_t ov[4];
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            float a = v[2 * h] + sbias[c0 + 2 * h], b = v[2 * h + 1] + sbias[c0 + 2 * h + 1];
            if (flags & kConvRelu) {
              a = fmaxf(a, 0.f);
              b = fmaxf(b, 0.f);
            }
            if (flags & kConvMask) {
              if (!bf16_positive(mw[h] & 0xffffu)) a = 0.f;
              if (!bf16_positive(mw[h] >> 16)) b = 0.f;
            }
            ov[h] = pack_bf16(a, b);
          }
          *reinterpret_cast<uint4*>(y + idx * COUT + c0) = make_uint4(ov[0], ov[1], ov[2], ov[3]);
        }
      }
    };

    for (int k = 0; k < nout; ++k, ++o) {
      cp_wait_groups<ST - 4>();  // triples k .. k+2 are complete
      tc::fence_proxy_async();
      __syncthreads();
      if (tid == 0) {
        tc::fence_after();
        const uint32_t acc = acc0 + (uint32_t)((o & 1) * COUT);
        constexpr uint32_t idesc = tc::idesc_bf16_f32(128, COUT);
        uint64_t slot[3];
#pragma unroll
        for (int dz = 0; dz < 3; ++dz)
          slot[dz] = adesc0 + (uint64_t)(((k + dz) % ST) * (Cfg::kTriple >> 4));
#pragma unroll
        for (int dz = 0; dz < 3; ++dz)
#pragma unroll
          for (int gi = 0; gi < 3; ++gi)
#pragma unroll
            for (int dx = 0; dx < 3; ++dx)
#pragma unroll
              for (int ks = 0; ks < CIN / 16; ++ks) {
                const int t = dz * 9 + gi * 3 + dx;
                const uint64_t ad =
                    slot[dz] + (uint64_t)((gi * Cfg::kRGBytes + dx * 16 + ks * 2 * kRG * 16) >> 4);
                const uint64_t bd = bdesc0 + (uint64_t)((t * Cfg::kWTap + ks * 256) >> 4);
                tc::mma_bf16(acc, ad, bd, idesc, (dz | gi | dx | ks) != 0);
              }
        tc::mma_commit(&bars[o & 1]);
      }
      if (k >= 1) {
        // output k-1 done: its triple k-1 is free and its accumulator is final
        const bool ok = tc::mbar_wait(&bars[(o - 1) & 1], ((o - 1) >> 1) & 1, kWaitLimit);
        if (__syncthreads_or(!ok)) {
          abort = true;
          break;
        }
        load_triple(k - 1 + ST);
        tc::fence_after();
        epilogue(k - 1, o - 1);
        tc::fence_before();
      } else {
        cp_commit_group();
      }
    }
    if (abort) break;
    // last output of the unit
    {
      const bool ok = tc::mbar_wait(&bars[(o - 1) & 1], ((o - 1) >> 1) & 1, kWaitLimit);
      if (__syncthreads_or(!ok)) {
        abort = true;
        break;
      }
      tc::fence_after();
      epilogue(nout - 1, o - 1);
      tc::fence_before();
    }
    cp_wait_all();
    __syncthreads();  // ring slots are rewritten by the next unit
  }
  cp_wait_all();
  if (abort && tid == 0) atomicOr(&g_tc_timeout, 1);
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(acc0, Cfg::kCols);
}

// ---- z-marching forward kernel with the z-taps folded into N ---------------
// Same work units and row-group triples as the z-marching kernel, but the loop
// runs over input planes instead of output planes.  Triple j (planes
// kp0-2+j .. in the unit's numbering) feeds outputs j-2, j-1 and j through the
// taps dz = 2, 1, 0, and for one (dy, dx) row-group offset the three tap
// matrices sit side by side in shared memory, so one tcgen05.mma with
// N = 3 COUT computes all three contributions from one read of the A operand
// (the staged input rows): 9 MMAs of N = 48 per output plane for 16 -> 16
// instead of 27 of N = 16, a third of the operand traffic from shared memory.
// The accumulators of consecutive outputs are consecutive COUT-column slots of
// a TMEM ring of R slots; an output range that wraps around the ring is split
// into two MMAs, and an output's first contribution (triple j = k, first
// (dy, dx, k16) step) is its own MMA with accumulation off.  Output k is final
// after triple k+2: its epilogue runs while the tensor core works on triple
// k+3.
template <int CIN, int COUT>
struct ZfCfg {
  static constexpr int kST = zm_stages<CIN, COUT>();
  static constexpr int kWTap = COUT * CIN * 2;
  static constexpr int kWBytes = 27 * kWTap;
  static constexpr int kRGBytes = kRG * CIN * 2;
  static constexpr int kTriple = 3 * kRGBytes;
  static constexpr int kSmem = kWBytes + kST * kTriple;
  static constexpr int kR = 256 / COUT;  // accumulator slots: 256 TMEM columns
  static constexpr uint32_t kCols = 256;
  static_assert(kSmem <= 227 * 1024, "shared memory");
  static_assert(kR >= 4, "the ring must hold the three outputs in work and one in its epilogue");
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(128)
conv_fwd_zf_kernel(const uint16_t* __restrict__ x, const uint16_t* __restrict__ w,
                   const float* __restrict__ bias, const uint16_t* __restrict__ mask,
                   uint16_t* __restrict__ y, Vol g, int flags, ZmGrid zg) {
  using Cfg = ZfCfg<CIN, COUT>;
  constexpr int ST = Cfg::kST;
  constexpr int R = Cfg::kR;
  constexpr int kc = CIN / 8;
  constexpr int kChunks = 3 * kRG * kc;            // 16-byte copies per triple
  constexpr int kPer = (kChunks + 127) / 128;      // per thread
  extern __shared__ __align__(128) unsigned char sm[];
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ uint32_t tbase;
  __shared__ float sbias[COUT];
  unsigned char* sW = sm;
  unsigned char* sR = sm + Cfg::kWBytes;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  // tap t = dz * 9 + dy * 3 + dx goes to tile (dy * 3 + dx) * 3 + (2 - dz): the
  // taps of one (dy, dx) are consecutive K-major tiles in the order dz = 2, 1, 0,
  // i.e. one B operand of N = 3 COUT rows
  for (int i = tid; i < 27 * COUT * kc; i += 128) {
    const int c = i % kc, r = (i / kc) % COUT, t = i / (kc * COUT);
    const int tt = (t % 9) * 3 + (2 - t / 9);
    const uint4 v = *reinterpret_cast<const uint4*>(w + ((size_t)t * COUT + r) * CIN + c * 8);
    *reinterpret_cast<uint4*>(sW + tt * Cfg::kWTap + tc::kmajor_off(r, c * 8, CIN)) = v;
  }
  if (tid < COUT) sbias[tid] = bias ? bias[tid] : 0.f;
  if (tid == 0) {
    tc::mbar_init(&bars[0], 1);
    tc::mbar_init(&bars[1], 1);
  }
  if (warp == 0) tc::tmem_alloc(&tbase, Cfg::kCols);
  int roff[kPer], coff[kPer];
  uint32_t soff[kPer];
#pragma unroll
  for (int m = 0; m < kPer; ++m) {
    const int i = tid + 128 * m;
    const int c = i % kc, v = (i / kc) % kRG, gi = i / (kc * kRG);
    roff[m] = gi * g.wp + v;
    coff[m] = c * 8;
    soff[m] = (uint32_t)(gi * Cfg::kRGBytes + c * (kRG * 16) + v * 16);
  }
  tc::fence_proxy_async();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t acc0 = tbase;
  const uint64_t adesc0 = tc::smem_desc(tc::smem_addr(sR), kRG * 16, 128);
  const uint64_t bdesc0 = tc::smem_desc(tc::smem_addr(sW), 128, kc * 128);

  bool abort = false;
  int tg = 0;     // triples issued by this CTA (barrier phase)
  int obase = 0;  // outputs of earlier units (accumulator ring position)
  for (int u = blockIdx.x; u < zg.units && !abort; u += gridDim.x) {
    const int bi = u % zg.nb, cz = u / zg.nb;
    const int sidx = cz / zg.nzc;
    const int z0 = (cz % zg.nzc) * zg.zc;
    const int nout = min(zg.zc, g.nz - z0);
    const int kp0 = sidx * g.dp + 1 + z0;  // padded plane of output 0
    const int seg = bi * 128;
    const int ntrip = nout + 2;            // triples: planes kp0-1 .. kp0+nout
    const int poff = seg + warp * 32 + lane;
    const int px = poff % g.wp, py = poff / g.wp;
    const bool in_xy = poff < g.pp && px >= 1 && px <= g.nx && py >= 1 && py <= g.ny;
    auto load_triple = [&](int j) {
      if (j < ntrip) {
        const int base = seg + (kp0 - 1 + j) * g.pp - g.wp - 1;
        unsigned char* st = sR + (j % ST) * Cfg::kTriple;
#pragma unroll
        for (int m = 0; m < kPer; ++m) {
          if (kChunks % 128 == 0 || tid + 128 * m < kChunks) {
            const int row = base + roff[m];
            const bool ok = row >= 0 && row < g.vp;
            cp16z(st + soff[m], x + (size_t)(ok ? row : 0) * CIN + coff[m], ok);
          }
        }
      }
      cp_commit_group();
    };
    for (int j = 0; j < ST; ++j) load_triple(j);

    auto epilogue = [&](int k) {
      const size_t idx = (size_t)(kp0 + k) * g.pp + poff;
      const uint32_t acc = acc0 + (uint32_t)(((obase + k) % R) * COUT);
      float va[COUT];
      tc::tmem_ld_cols<COUT>(acc + ((uint32_t)(warp * 32) << 16), va);
#pragma unroll
      for (int c0 = 0; c0 < COUT; c0 += 8) {
        const float* v = va + c0;
        if (in_xy) {
          uint4 mk = make_uint4(0, 0, 0, 0);
          if (flags & kConvMask) mk = *reinterpret_cast<const uint4*>(mask + idx * COUT + c0);
          const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
          uint32_t ov[4];
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            float a = v[2 * h] + sbias[c0 + 2 * h], b = v[2 * h + 1] + sbias[c0 + 2 * h + 1];
            if (flags & kConvRelu) {
              a = fmaxf(a, 0.f);
              b = fmaxf(b, 0.f);
            }
            if (flags & kConvMask) {
              if (!bf16_positive(mw[h] & 0xffffu)) a = 0.f;
              if (!bf16_positive(mw[h] >> 16)) b = 0.f;
            }
            ov[h] = pack_bf16(a, b);
          }
          *reinterpret_cast<uint4*>(y + idx * COUT + c0) = make_uint4(ov[0], ov[1], ov[2], ov[3]);
        }
      }
    };

    for (int j = 0; j < ntrip; ++j, ++tg) {
      cp_wait_groups<ST - 2>();  // triple j is complete
      tc::fence_proxy_async();
      __syncthreads();
      if (tid == 0) {
        tc::fence_after();
        const int klo = max(0, j - 2), khi = min(nout - 1, j);
        const uint64_t slot = adesc0 + (uint64_t)((j % ST) * (Cfg::kTriple >> 4));
        // outputs ka..kb of this triple, one (dy, dx, k16) step: B tiles
        // consecutive from the tile of output ka, D slots consecutive modulo R
        auto mma_range = [&](int ka, int kb, uint64_t ad, int tile0, int ks, bool accum) {
          int k = ka;
          while (k <= kb) {
            const int sl = (obase + k) % R;
            const int n = min(kb - k + 1, R - sl);
            const uint64_t bd =
                bdesc0 + (uint64_t)(((tile0 + (k - ka)) * Cfg::kWTap + ks * 256) >> 4);
            tc::mma_bf16(acc0 + (uint32_t)(sl * COUT), ad, bd, tc::idesc_bf16_f32(128, n * COUT),
                         accum);
            k += n;
          }
        };
#pragma unroll 1
        for (int gi = 0; gi < 3; ++gi)
#pragma unroll
          for (int dx = 0; dx < 3; ++dx)
#pragma unroll
            for (int ks = 0; ks < CIN / 16; ++ks) {
              const uint64_t ad =
                  slot + (uint64_t)((gi * Cfg::kRGBytes + dx * 16 + ks * 2 * kRG * 16) >> 4);
              // tile of output ka: (dy, dx) group, index 2 - dz with dz = j - ka
              const int grp = (gi * 3 + dx) * 3 + 2 - j;
              const bool first = (gi | dx | ks) == 0;
              if (first && khi == j) {  // output j starts here: accumulation off for it
                if (klo < j) mma_range(klo, j - 1, ad, grp + klo, ks, true);
                mma_range(j, j, ad, grp + j, ks, false);
              } else {
                mma_range(klo, khi, ad, grp + klo, ks, true);
              }
            }
        tc::mma_commit(&bars[tg & 1]);
      }
      if (j >= 1) {
        // triple j-1's MMAs are done: its ring slot is free, and output j-3 is final
        const bool ok = tc::mbar_wait(&bars[(tg - 1) & 1], ((tg - 1) >> 1) & 1, kWaitLimit);
        if (__syncthreads_or(!ok)) {
          abort = true;
          break;
        }
        load_triple(j - 1 + ST);
        if (j >= 3) {
          tc::fence_after();
          epilogue(j - 3);
          tc::fence_before();
        }
      } else {
        cp_commit_group();
      }
    }
    if (abort) break;
    {  // the last output of the unit
      const bool ok = tc::mbar_wait(&bars[(tg - 1) & 1], ((tg - 1) >> 1) & 1, kWaitLimit);
      if (__syncthreads_or(!ok)) {
        abort = true;
        break;
      }
      tc::fence_after();
      epilogue(nout - 1);
      tc::fence_before();
    }
    obase += nout;
    cp_wait_all();
    __syncthreads();  // ring slots are rewritten by the next unit
  }
  cp_wait_all();
  if (abort && tid == 0) atomicOr(&g_tc_timeout, 1);
  tc::fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(acc0, Cfg::kCols);
}

// ---- the folded z-marching kernel with warp-specialised roles -------------
// Folded MMAs (N = 3 cout) and TMEM ring of accumulators as in
// conv_fwd_zf_kernel, over tiles of 8 x 16 voxels (x, y) followed through zc
// planes, with the three kinds of work on warps of their own:
//   warp 5 (one thread) copies the tile's input planes, 10 x 18 voxels with their
//          halo, into a ring of ST slots (one tensor-map copy each, voxels outside
//          the volume filled with zeros), and before them the 27 weight matrices;
//   warp 4 (one elected lane) issues the MMAs of a plane once it is full and the
//          slot of the output it starts is free, and commits to the plane's
//          "empty" barrier and to the "full" barrier of the output the plane
//          completes;
//   warps 0-3 (the four TMEM lane quarters) drain finished accumulators:
//          load, release the slot ("empty"), then bias / ReLU / mask, BF16
//          rounding and the stores.
// Every wait is bounded; a wait that runs out raises a shared abort flag that
// every role checks, and the kernel records the timeout like the others.
//
// Voxels stay whole rows of cin channels in shared memory, in the copy engine's
// swizzle of that width, which the tensor core reads directly: operand row m is
// voxel (m % 8, m / 8) of the tile (row groups of 8 voxels, 10 rows apart), and a
// tap is the same rows started (dy, dx) later.
// Small volumes are bound by launch and pipeline fill (16^3: 5.6 us), larger ones
// by the one warp that issues the MMAs (each runs 32 + N / 4 cycles and takes
// longer than that to issue) and by the voxel rows copied: a linear run of 128
// voxels needs three runs of 130, this tile 180 rows.  16 -> 16, us: 64^3 21.8 in
// 8-channel blocks filled 16 bytes at a time, 16.3 with linear runs of whole
// rows, 14.4 now; 160^3 197, 129, 104 (350 TFLOP/s); 64 -> 32 at 64^3 160 -> 35.
template <int CIN, int COUT>
struct WsCfg {
  static constexpr int kTX = 8, kTY = 16;
  static constexpr int kRow = CIN * 2;
  static constexpr int kPitch = (kTX + 2) * kRow;              // next row of the tile
  static constexpr int kWTap = COUT * kRow;
  static constexpr int kWBytes = 27 * kWTap;
  static constexpr int kTx = (kTY + 2) * kPitch;               // bytes of one plane
  static constexpr int kPlane = (kTx + 1023) / 1024 * 1024;
  // two CTAs per SM where the weights leave room, else one
  static constexpr int kST = CIN == 64 ? 4 : COUT == 64 ? 8 : CIN == 32 ? 6 : 10;
  static constexpr int kSmem = kWBytes + kST * kPlane + 1024;
  static constexpr int kR = 256 / COUT;
  static constexpr uint32_t kCols = 256;
  static_assert(kSmem <= 227 * 1024, "shared memory");
  static_assert(kR >= 4, "accumulator ring");
};

__device__ __forceinline__ void mbar_arrive1(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_addr(bar)) : "memory");
}

struct RowMaps {
  CUtensorMap a, b;
};

template <int CIN, int COUT, int FUSE = kFuseNone>
__global__ void __launch_bounds__(192)
conv_fwd_ws_kernel(const __grid_constant__ RowMaps maps, const float* __restrict__ bias,
                   const uint16_t* __restrict__ mask, uint16_t* __restrict__ y, Vol g, int flags,
                   ZmGrid zg, const ConvFuse fuse) {
  using Cfg = WsCfg<CIN, COUT>;
  constexpr int ST = Cfg::kST;
  constexpr int R = Cfg::kR;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t tfull[ST], tempty[ST], afull[R], aempty[R], wfull, done_bar;
  __shared__ uint32_t tbase;
  __shared__ float sbias[COUT];
  __shared__ volatile int s_abort;
  unsigned char* sR = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* sW = sR + ST * Cfg::kPlane;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  if (tid < COUT) sbias[tid] = bias ? bias[tid] : 0.f;
  if (tid == 0) {
    for (int i = 0; i < ST; ++i) {
      tc::mbar_init(&tfull[i], 1);
      tc::mbar_init(&tempty[i], 1);
    }
    for (int i = 0; i < R; ++i) {
      tc::mbar_init(&afull[i], 1);
      tc::mbar_init(&aempty[i], 4);
    }
    tc::mbar_init(&wfull, 1);
    tc::mbar_init(&done_bar, 1);
    s_abort = 0;
  }
  if (warp == 4) tc::tmem_alloc(&tbase, Cfg::kCols);
  tc::fence_proxy_async();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t acc0 = tbase;

  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    if (s_abort) return false;
    if (tc::mbar_wait(bar, parity, kWaitLimit)) return true;
    s_abort = 1;
    return false;
  };

  if (warp == 5) {
    // ---- copies ---------------------------------------------------------------
    if (lane == 0) {
      // weights in the folded order (see conv_fwd_zf_kernel)
      tc::mbar_expect(&wfull, Cfg::kWBytes);
      for (int t = 0; t < 27; ++t)
        tc::tma_2d(sW + ((t % 9) * 3 + (2 - t / 9)) * Cfg::kWTap, &maps.b, &wfull, 0, t * COUT);
      int tg = 0;
      for (int u = blockIdx.x; u < zg.units && !s_abort; u += gridDim.x) {
        const int bi = u % zg.nb, cz = u / zg.nb;
        const int z0 = (cz % zg.nzc) * zg.zc;
        const int nout = min(zg.zc, g.nz - z0);
        const int p0 = cz / zg.nzc * g.dp + z0;  // padded plane of the first input plane
        const int x0 = bi % zg.nbx * Cfg::kTX, y0 = bi / zg.nbx * Cfg::kTY;  // padded corner
        bool stop = false;
        for (int j = 0; j < nout + 2; ++j, ++tg) {
          const int s = tg % ST;
          if (tg >= ST && !wait(&tempty[s], ((tg / ST) - 1) & 1)) { stop = true; break; }
          tc::mbar_expect(&tfull[s], Cfg::kTx);
          tc::tma_4d(sR + s * Cfg::kPlane, &maps.a, &tfull[s], 0, x0, y0, p0 + j);
        }
        if (stop) break;
      }
      // no copy outlives the block: wait for the last (up to ST) planes and the weights
      tc::mbar_wait(&wfull, 0, kWaitLimit);
      for (int j = tg - 1; j >= 0 && j >= tg - ST; --j)
        if (!tc::mbar_wait(&tfull[j % ST], (j / ST) & 1, kWaitLimit)) s_abort = 1;
    }
  } else if (warp == 4) {
    // ---- MMA warp (one elected lane issues; everything it needs is uniform) ----
    const uint64_t adesc0 = tc::smem_desc_sw(tc::smem_addr(sR), 16, Cfg::kPitch, Cfg::kRow);
    const uint64_t bdesc0 = tc::smem_desc_sw(tc::smem_addr(sW), 16, 8 * Cfg::kRow, Cfg::kRow);
    const uint32_t accu = __shfl_sync(0xffffffffu, acc0, 0);
    auto waitw = [&](uint64_t* bar, uint32_t parity) -> bool {
      if (tc::mbar_wait_warp(bar, parity, kWaitLimit)) return true;
      s_abort = 1;
      return false;
    };
    int tg = 0, obase = 0;
    bool stop = !waitw(&wfull, 0);
    for (int u = blockIdx.x; u < zg.units && !stop; u += gridDim.x) {
      const int cz = u / zg.nb;
      const int z0 = (cz % zg.nzc) * zg.zc;
      const int nout = min(zg.zc, g.nz - z0);
      for (int j = 0; j < nout + 2; ++j, ++tg) {
        const int s = tg % ST;
        if (!waitw(&tfull[s], (tg / ST) & 1)) { stop = true; break; }
        const int klo = max(0, j - 2), khi = min(nout - 1, j);
        if (khi == j) {  // output j starts here: its accumulator slot must be free
          const int oc = obase + j;
          if (oc >= R && !waitw(&aempty[oc % R], ((oc / R) - 1) & 1)) { stop = true; break; }
        }
        tc::fence_after();
        // Accumulator slots, instruction descriptors and operand addresses of
        // the plane are the same for its 9 (dy, dx) x CIN / 16 steps up to
        // constants, and formed once.
        const int sl = (obase + klo) % R;
        const int n1 = min(khi - klo + 1, R - sl), n2 = khi - klo + 1 - n1;
        const uint32_t d1 = accu + (uint32_t)(sl * COUT);
        const uint32_t i1 = tc::idesc_bf16_f32(128, n1 * COUT);
        const uint32_t i2 = tc::idesc_bf16_f32(128, n2 * COUT);
        const uint64_t a0 = adesc0 + (uint32_t)(s * (Cfg::kPlane >> 4));
        const uint64_t b1 = bdesc0 + (uint32_t)((2 - j + klo) * (Cfg::kWTap >> 4));
        const uint64_t b2 = b1 + (uint32_t)(n1 * (Cfg::kWTap >> 4));
        // first step: output j starts with it, the outputs before j go on
        if (khi == j) {
          for (int k = klo; k <= j; ++k)
            tc::mma_bf16_warp(accu + (uint32_t)(((obase + k) % R) * COUT), a0,
                              b1 + (uint32_t)((k - klo) * (Cfg::kWTap >> 4)),
                              tc::idesc_bf16_f32(128, COUT), k < j);
        } else {
          tc::mma_bf16_warp(d1, a0, b1, i1, true);
          if (n2 > 0) tc::mma_bf16_warp(accu, a0, b2, i2, true);
        }
        auto step = [&](int st, bool two) {
          const int gd = st / (CIN / 16), ks = st % (CIN / 16);  // gd = 3 gi + dx
          const uint32_t ao = (gd / 3 * Cfg::kPitch + gd % 3 * Cfg::kRow + ks * 32) >> 4;
          const uint32_t bo = (gd * 3 * Cfg::kWTap + ks * 32) >> 4;
          tc::mma_bf16_warp(d1, a0 + ao, b1 + bo, i1, true);
          if (two) tc::mma_bf16_warp(accu, a0 + ao, b2 + bo, i2, true);
        };
        if (n2 == 0) {
#pragma unroll
          for (int st = 1; st < 9 * (CIN / 16); ++st) step(st, false);
        } else {
#pragma unroll 1
          for (int st = 1; st < 9 * (CIN / 16); ++st) step(st, true);
        }
        tc::mma_commit_warp(&tempty[s]);
        if (j >= 2) tc::mma_commit_warp(&afull[(obase + j - 2) % R]);  // output j-2 is final
      }
      obase += nout;
    }
    // every MMA issued must be complete before the TMEM is released
    tc::mma_commit_warp(&done_bar);
    if (!tc::mbar_wait_warp(&done_bar, 0, kWaitLimit)) s_abort = 1;
  } else {
    // ---- epilogue warps 0-3: TMEM lanes 32 warp .. 32 warp + 31 -------------
    int obase = 0;
    for (int u = blockIdx.x; u < zg.units && !s_abort; u += gridDim.x) {
      const int bi = u % zg.nb, cz = u / zg.nb;
      const int z0 = (cz % zg.nzc) * zg.zc;
      const int nout = min(zg.zc, g.nz - z0);
      const int kp0 = cz / zg.nzc * g.dp + 1 + z0;  // padded plane of output 0
      const int vx = bi % zg.nbx * Cfg::kTX + (lane & 7);
      const int vy = bi / zg.nbx * Cfg::kTY + warp * 4 + (lane >> 3);
      const int poff = (vy + 1) * g.wp + vx + 1;
      const bool in_xy = vx < g.nx && vy < g.ny;
      float psum[FUSE == kFusePool ? COUT : 1];  // pool: sums of the even plane
      (void)psum;
      bool stop = false;
      for (int k = 0; k < nout; ++k) {
        const int oc = obase + k;
        const int sl = oc % R;
        if (!wait(&afull[sl], (oc / R) & 1)) { stop = true; break; }
        tc::fence_after();
        float va[COUT];
        tc::tmem_ld_cols<COUT>(acc0 + ((uint32_t)(warp * 32) << 16) + (uint32_t)(sl * COUT), va);
        tc::fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive1(&aempty[sl]);
        uint32_t ov[COUT / 2];  // the output voxel in BF16
        const size_t idx = (size_t)(kp0 + k) * g.pp + poff;
#pragma unroll
        for (int c0 = 0; c0 < COUT; c0 += 8) {
          const float* v = va + c0;
          uint4 mk = make_uint4(0, 0, 0, 0);
          if (FUSE == kFuseNone && (flags & kConvMask) && in_xy)
            mk = *reinterpret_cast<const uint4*>(mask + idx * COUT + c0);
          const uint32_t mw[4] = {mk.x, mk.y, mk.z, mk.w};
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            float a = v[2 * h] + sbias[c0 + 2 * h], b = v[2 * h + 1] + sbias[c0 + 2 * h + 1];
            if (flags & kConvRelu) {
              a = fmaxf(a, 0.f);
              b = fmaxf(b, 0.f);
            }
            if (FUSE == kFuseNone && (flags & kConvMask)) {
              if (!bf16_positive(mw[h] & 0xffffu)) a = 0.f;
              if (!bf16_positive(mw[h] >> 16)) b = 0.f;
            }
            ov[c0 / 2 + h] = pack_bf16(a, b);
          }
          if (FUSE != kFuseCells && in_xy)
            *reinterpret_cast<uint4*>(y + idx * COUT + c0) =
                make_uint4(ov[c0 / 2], ov[c0 / 2 + 1], ov[c0 / 2 + 2], ov[c0 / 2 + 3]);
        }
        if (FUSE == kFuseCells && in_xy) {
          const int s_ = cz / zg.nzc;
          fuse.z[(((size_t)s_ * g.nz + z0 + k) * g.ny + vy) * g.nx + vx] =
              fuse.rms[s_] * __uint_as_float(ov[0] << 16);
        }
        if (FUSE == kFusePool) {
          // children in the order (dz, dy, dx): x neighbours are lanes 1 apart, y
          // neighbours 8 apart, z neighbours consecutive outputs of the unit
#pragma unroll
          for (int h = 0; h < COUT / 2; ++h) {
            const uint32_t w0 = ov[h];
            const uint32_t w1 = __shfl_down_sync(0xffffffffu, w0, 1);
            const uint32_t w2 = __shfl_down_sync(0xffffffffu, w0, 8);
            const uint32_t w3 = __shfl_down_sync(0xffffffffu, w0, 9);
            float lo = (k & 1) ? psum[2 * h] : 0.f, hi = (k & 1) ? psum[2 * h + 1] : 0.f;
            lo += __uint_as_float(w0 << 16);
            hi += __uint_as_float(w0 & 0xffff0000u);
            lo += __uint_as_float(w1 << 16);
            hi += __uint_as_float(w1 & 0xffff0000u);
            lo += __uint_as_float(w2 << 16);
            hi += __uint_as_float(w2 & 0xffff0000u);
            lo += __uint_as_float(w3 << 16);
            hi += __uint_as_float(w3 & 0xffff0000u);
            psum[2 * h] = lo;
            psum[2 * h + 1] = hi;
          }
          if ((k & 1) && in_xy && (vx & 1) == 0 && (vy & 1) == 0) {
            const Vol& gc = fuse.g2;
            const size_t vc = ((size_t)(cz / zg.nzc * gc.dp + (z0 + k) / 2 + 1) * gc.hp + vy / 2 + 1) *
                                  gc.wp + vx / 2 + 1;
#pragma unroll
            for (int c0 = 0; c0 < COUT; c0 += 8) {
              uint32_t o[4];
#pragma unroll
              for (int h = 0; h < 4; ++h)
                o[h] = pack_bf16(psum[c0 + 2 * h] * 0.125f, psum[c0 + 2 * h + 1] * 0.125f);
              *reinterpret_cast<uint4*>(fuse.out + vc * COUT + c0) = make_uint4(o[0], o[1], o[2], o[3]);
            }
          }
        }
        if (FUSE == kFuseUpadd && in_xy) {
          const Vol& gf = fuse.g2;
          const size_t vf = ((size_t)(cz / zg.nzc * gf.dp + 2 * (z0 + k) + 1) * gf.hp + 2 * vy + 1) *
                                gf.wp + 2 * vx + 1;
#pragma unroll
          for (int dz = 0; dz < 2; ++dz) {
            uint4 sk[4][COUT / 8];  // the four children of a plane: loads first
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
              for (int c = 0; c < COUT / 8; ++c)
                sk[j][c] = __ldg(reinterpret_cast<const uint4*>(
                    fuse.skip + (vf + (size_t)dz * gf.pp + (j >> 1) * gf.wp + (j & 1)) * COUT) + c);
#pragma unroll
            for (int j = 0; j < 4; ++j)
#pragma unroll
              for (int c = 0; c < COUT / 8; ++c) {
                const uint32_t sw[4] = {sk[j][c].x, sk[j][c].y, sk[j][c].z, sk[j][c].w};
                uint32_t o[4];
#pragma unroll
                for (int h = 0; h < 4; ++h) {
                  const uint32_t b = ov[4 * c + h];
                  o[h] = pack_bf16(__uint_as_float(sw[h] << 16) + __uint_as_float(b << 16),
                                   __uint_as_float(sw[h] & 0xffff0000u) +
                                       __uint_as_float(b & 0xffff0000u));
                }
                *(reinterpret_cast<uint4*>(
                      fuse.out + (vf + (size_t)dz * gf.pp + (j >> 1) * gf.wp + (j & 1)) * COUT) + c) =
                    make_uint4(o[0], o[1], o[2], o[3]);
              }
          }
        }
      }
      if (stop) break;
      obase += nout;
    }
  }
  tc::fence_before();
  __syncthreads();
  if (s_abort && tid == 0) atomicOr(&g_tc_timeout, 1);
  if (warp == 4) tc::tmem_dealloc(acc0, Cfg::kCols);
}

// ---- weight gradient ---------------------------------------------------------
// dw[t][co][ci] = sum_u dy[u - dx][co] x[u + (dz, dy)][ci]: a GEMM whose reduction
// runs over voxels.  Rows are (dx, co) and columns (dz, dy, ci), so that one MMA
// covers every tap of its columns.  Both operands are staged by the copy engine
// as they lie in memory, voxel rows of all channels in the swizzle of that width,
// and the tensor core reads them MN-major: a row of the stage is one step of the
// reduction, and the next block of channels (lbo) is the next (dz, dy) row set
// for x, and for dy the same rows started one voxel later, which makes the three
// dx shifts out of one copy of dy.  Row blocks past the third (dx = 2, 3, ..) are
// computed and ignored.
// CTAs split the voxel range, write FP32 partial tiles, and a second kernel adds
// the partials in a fixed order.
// 16 -> 32 on 16 samples of 32^3 (GB300): 41 us (bound by the
// copies: 648 voxel rows per 64 voxels) and
// 12 us for the sum of the partials; 1,008 and 15 us when 8 x 8 blocks went through
// movmatrix.
template <int CIN, int COUT>
struct WgCfg {
  static constexpr int kKV = 64;                   // voxels per stage
  static constexpr int kS = 6;                     // stages
  static constexpr int kRg = CIN == 16 ? 9 : 3;    // (dz, dy) rows per CTA: all, or one dz
  static constexpr int kParts = 9 / kRg;
  static constexpr int kN = kRg * CIN;             // columns of the accumulator
  static constexpr int kRows = 3 * COUT;           // rows that mean something
  static constexpr int kMTiles = (kRows + 127) / 128;
  static constexpr int kARow = COUT * 2, kBRow = CIN * 2;
  static constexpr int kAVox = kKV + 8;            // voxels of dy a stage needs (and reads)
  static constexpr int kABytes = (kAVox * kARow + 1023) / 1024 * 1024;
  static constexpr int kBRg = kKV * kBRow;         // one (dz, dy) row set
  static constexpr int kStage = kABytes + kRg * kBRg;
  static constexpr uint32_t kTx = kAVox * kARow + kRg * kBRg;
  static constexpr int kSmem = kS * kStage + 1024;
  static constexpr int kUse = kMTiles * kN;
  static constexpr uint32_t kCols = kUse <= 64 ? 64 : kUse <= 128 ? 128 : 256;
  // the last voxel read: 63 of the stage, plus the shift of the last row block
  static_assert(kKV - 1 + 128 * kMTiles / COUT - 1 < kAVox, "row blocks stay in the stage");
  static_assert(kBRg % 1024 == 0, "row sets start on a swizzle period");
  static_assert(kN % 16 == 0 && kN <= 256 && kUse <= 256 && kSmem <= 227 * 1024, "shape");
};

template <int CIN, int COUT>
__global__ void __launch_bounds__(192)
conv_wgrad_kernel(const __grid_constant__ RowMaps maps, float* __restrict__ ws, Vol g,
                  int nchunks) {
  using Cfg = WgCfg<CIN, COUT>;
  constexpr int kKV = Cfg::kKV, S = Cfg::kS;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t full[S], empty[S], done_bar;
  __shared__ uint32_t tbase;
  __shared__ volatile int s_abort;
  unsigned char* sm = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int part = blockIdx.x, split = blockIdx.y, nsplit = gridDim.y;
  const int my = (nchunks - split + nsplit - 1) / nsplit;
  const int u00 = g.g0 - 1;  // first voxel u: dy is not zero for u - dx in [g0, g1)

  if (tid == 0) {
    for (int i = 0; i < S; ++i) {
      tc::mbar_init(&full[i], 1);
      tc::mbar_init(&empty[i], 1);
    }
    tc::mbar_init(&done_bar, 1);
    s_abort = 0;
  }
  if (warp == 4) tc::tmem_alloc(&tbase, Cfg::kCols);
  tc::fence_proxy_async();
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t acc = tbase;
  auto wait = [&](uint64_t* bar, uint32_t parity) -> bool {
    if (s_abort) return false;
    if (tc::mbar_wait(bar, parity, kWaitLimit)) return true;
    s_abort = 1;
    return false;
  };

  if (warp == 5) {
    // ---- copies ------------------------------------------------------------------
    if (lane == 0) {
      int issued = 0;
      for (int i = 0; i < my; ++i) {
        const int buf = i % S;
        if (i >= S && !wait(&empty[buf], ((i / S) - 1) & 1)) break;
        const int u0 = u00 + (split + i * nsplit) * kKV;
        unsigned char* st = sm + buf * Cfg::kStage;
        tc::mbar_expect(&full[buf], Cfg::kTx);
        tc::tma_2d(st, &maps.b, &full[buf], 0, u0 - 1);
#pragma unroll
        for (int q = 0; q < Cfg::kRg; ++q) {
          const int rg = part * Cfg::kRg + q;
          tc::tma_2d(st + Cfg::kABytes + q * Cfg::kBRg, &maps.a, &full[buf], 0,
                     u0 + (rg / 3 - 1) * g.pp + (rg % 3 - 1) * g.wp);
        }
        issued = i + 1;
      }
      // no copy outlives the block
      for (int j = issued - 1; j >= 0 && j >= issued - S; --j)
        if (!tc::mbar_wait(&full[j % S], (j / S) & 1, kWaitLimit)) s_abort = 1;
    }
  } else if (warp == 4) {
    // ---- MMA warp (one elected lane issues) ------------------------------------
    const uint32_t accu = __shfl_sync(0xffffffffu, acc, 0);
    for (int i = 0; i < my; ++i) {
      const int buf = i % S;
      if (!tc::mbar_wait_warp(&full[buf], (i / S) & 1, kWaitLimit)) {
        s_abort = 1;
        break;
      }
      tc::fence_after();
      // bits 15, 16: A and B MN-major
      constexpr uint32_t idesc = tc::idesc_bf16_f32(128, Cfg::kN) | (1u << 15) | (1u << 16);
      const uint32_t st = tc::smem_addr(sm + buf * Cfg::kStage);
      const uint64_t ad = tc::smem_desc_sw(st, Cfg::kARow, 8 * Cfg::kARow, Cfg::kARow);
      const uint64_t bd = tc::smem_desc_sw(st + Cfg::kABytes, Cfg::kBRg, 8 * Cfg::kBRow, Cfg::kBRow);
#pragma unroll
      for (int ks = 0; ks < kKV / 16; ++ks)
#pragma unroll
        for (int mt = 0; mt < Cfg::kMTiles; ++mt)
          tc::mma_bf16_warp(accu + mt * Cfg::kN,
                            ad + (uint32_t)(((ks * 16 + mt * (128 / COUT)) * Cfg::kARow) >> 4),
                            bd + (uint32_t)((ks * 16 * Cfg::kBRow) >> 4), idesc, (i | ks) != 0);
      tc::mma_commit_warp(&empty[buf]);
    }
    // every MMA issued must be complete before the accumulator is read or released
    tc::mma_commit_warp(&done_bar);
    if (!tc::mbar_wait_warp(&done_bar, 0, kWaitLimit)) s_abort = 1;
  }
  tc::fence_before();
  __syncthreads();
  const bool abort = s_abort != 0;
  tc::fence_after();
  if (warp < 4) {
#pragma unroll
    for (int mt = 0; mt < Cfg::kMTiles; ++mt) {
      const int row = mt * 128 + warp * 32 + lane;
      const int m = row / COUT, co = row % COUT;  // row block m: voxel u - 1 + m, dx = 1 - m
      float* out = ws + ((size_t)(split * Cfg::kParts + part) * Cfg::kRows + (2 - m) * COUT + co) *
                            Cfg::kN;
#pragma unroll
      for (int c0 = 0; c0 < Cfg::kN; c0 += 16) {
        float v[16];
        if (!abort && my > 0)
          tc::tmem_ld16(acc + ((uint32_t)(warp * 32) << 16) + mt * Cfg::kN + c0, v);
        else
          for (int c = 0; c < 16; ++c) v[c] = 0.f;
        if (m < 3)
#pragma unroll
          for (int c = 0; c < 16; c += 4)
            *reinterpret_cast<float4*>(out + c0 + c) = make_float4(v[c], v[c + 1], v[c + 2], v[c + 3]);
      }
    }
  }
  if (abort && tid == 0) atomicOr(&g_tc_timeout, 1);
  tc::fence_before();
  __syncthreads();
  if (warp == 4) tc::tmem_dealloc(acc, Cfg::kCols);
}

// dw from the partial tiles: 32 outputs per block (consecutive ci), the splits
// dealt to its 16 warps and added in a fixed order in FP64.
template <int CIN, int COUT>
__global__ void __launch_bounds__(512)
wgrad_reduce_kernel(const float* __restrict__ ws, float* __restrict__ dw, int nsplit,
                    int accumulate) {
  using Cfg = WgCfg<CIN, COUT>;
  __shared__ double part[16][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int i = blockIdx.x * 32 + lane;  // 27 COUT CIN is a multiple of 32
  const int ci = i % CIN, co = (i / CIN) % COUT, t = i / (CIN * COUT);
  const int rg = t / 3, d = t % 3;
  const float* src = ws + ((size_t)(rg / Cfg::kRg) * Cfg::kRows + d * COUT + co) * Cfg::kN +
                     (rg % Cfg::kRg) * CIN + ci;
  double s = 0.0;
#pragma unroll 10
  for (int sp = warp; sp < nsplit; sp += 16)
    s += src[(size_t)sp * Cfg::kParts * Cfg::kRows * Cfg::kN];
  part[warp][lane] = s;
  __syncthreads();
  if (warp == 0) {
    for (int w = 1; w < 16; ++w) s += part[w][lane];
    dw[i] = accumulate ? (float)(dw[i] + s) : (float)s;
  }
}

// CTAs per SM from the shared-memory and tensor-memory budgets (the occupancy
// calculator does not see TMEM), with the carveout set to all shared memory
int ctas_per_sm(const void* fn, int smem, uint32_t tmem_cols, int* nsm) {
  int dev = 0, per_sm_smem = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(nsm, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&per_sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  cudaFuncSetAttribute(fn, cudaFuncAttributePreferredSharedMemoryCarveout,
                       cudaSharedmemCarveoutMaxShared);
  int b = per_sm_smem / (smem + 1024);  // 1 KB reserved per CTA
  const int bt = (int)(512 / tmem_cols);
  if (b > bt) b = bt;
  if (b > 8) b = 8;
  return b < 1 ? 1 : b;
}

template <int CIN, int COUT>
int fwd_grid(int ntiles) {
  static int per_sm = -1, nsm = 0;
  if (per_sm < 0)
    per_sm = ctas_per_sm((const void*)conv_fwd_kernel<CIN, COUT>, FwdCfg<CIN, COUT>::kSmem,
                         FwdCfg<CIN, COUT>::kCols, &nsm);
  const int cap = per_sm * nsm;
  return ntiles < cap ? ntiles : cap;
}

template <int CIN, int COUT>
cudaError_t fwd_launch(const uint16_t* x, const uint16_t* w, const float* bias,
                       const uint16_t* mask, uint16_t* y, const Vol& g, int flags,
                       cudaStream_t s) {
  const int ntiles = (g.g1 - g.g0 + 127) / 128;
  if (ntiles <= 0) return cudaSuccess;
  const int grid = fwd_grid<CIN, COUT>(ntiles);
  conv_fwd_kernel<CIN, COUT><<<grid, 128, FwdCfg<CIN, COUT>::kSmem, s>>>(x, w, bias, mask, y, g,
                                                                        flags, ntiles);
  return cudaGetLastError();
}

template <int CIN, int COUT>
cudaError_t zm_launch(const uint16_t* x, const uint16_t* w, const float* bias,
                      const uint16_t* mask, uint16_t* y, const Vol& g, int flags,
                      cudaStream_t s) {
  static int per_sm = -1, nsm = 0;
  if (per_sm < 0)
    per_sm = ctas_per_sm((const void*)conv_fwd_zm_kernel<CIN, COUT>, ZmCfg<CIN, COUT>::kSmem,
                         ZmCfg<CIN, COUT>::kCols, &nsm);
  const int ctas = per_sm * nsm;
  ZmGrid zg;
  zg.nbx = 0;
  zg.nb = (g.pp + 127) / 128;
  zg.zc = g.nz;
  // shorter z runs until there are at least two units per resident CTA
  while (zg.zc > 4 && (long long)zg.nb * g.ns * ((g.nz + zg.zc - 1) / zg.zc) < 2LL * ctas)
    zg.zc = (zg.zc + 1) / 2;
  zg.nzc = (g.nz + zg.zc - 1) / zg.zc;
  zg.units = zg.nb * g.ns * zg.nzc;
  const int grid = zg.units < ctas ? zg.units : ctas;
  conv_fwd_zm_kernel<CIN, COUT><<<grid, 128, ZmCfg<CIN, COUT>::kSmem, s>>>(x, w, bias, mask, y,
                                                                           g, flags, zg);
  return cudaGetLastError();
}

template <int CIN, int COUT>
cudaError_t zf_launch(const uint16_t* x, const uint16_t* w, const float* bias,
                      const uint16_t* mask, uint16_t* y, const Vol& g, int flags,
                      cudaStream_t s) {
  static int per_sm = -1, nsm = 0;
  if (per_sm < 0)
    per_sm = ctas_per_sm((const void*)conv_fwd_zf_kernel<CIN, COUT>, ZfCfg<CIN, COUT>::kSmem,
                         ZfCfg<CIN, COUT>::kCols, &nsm);
  const int ctas = per_sm * nsm;
  ZmGrid zg;
  zg.nbx = 0;
  zg.nb = (g.pp + 127) / 128;
  zg.zc = g.nz;
  // shorter z runs until there are at least two units per resident CTA
  while (zg.zc > 4 && (long long)zg.nb * g.ns * ((g.nz + zg.zc - 1) / zg.zc) < 2LL * ctas)
    zg.zc = (zg.zc + 1) / 2;
  zg.nzc = (g.nz + zg.zc - 1) / zg.zc;
  zg.units = zg.nb * g.ns * zg.nzc;
  const int grid = zg.units < ctas ? zg.units : ctas;
  conv_fwd_zf_kernel<CIN, COUT><<<grid, 128, ZfCfg<CIN, COUT>::kSmem, s>>>(x, w, bias, mask, y,
                                                                           g, flags, zg);
  return cudaGetLastError();
}

// Planes per unit: the split of the planes into runs with the fewest plane steps
// on the busiest CTA (a run of zc outputs takes zc + 2 steps).  Measured, us a call,
// with runs of 4 / 8 / 16 / 24 planes and with the rule's: 16 -> 16 at 64^3 17.1 / 16.5 /
// 18.6 / 24.8, rule 16.6; at 160^3 127 / 115 / 109 / 111, rule 107; 32 -> 64 at 64^3 32.9 /
// 33.0 / 33.0 / 45.3, rule 33.0; 64 -> 32 at 64^3 39.1 / 35.0 / 37.1 / 53.4, rule 37.1; 32 ->
// 16 at 96^3 44.2 / 39.6 / 43.2 / 37.9, rule 38.3.
int ws_run(int nb, int nz, int ns, int ctas) {
  long long best = 0;
  int zc = nz;
  for (int k = 1; k <= nz; ++k) {
    const int z = (nz + k - 1) / k;
    const long long units = (long long)nb * ns * ((nz + z - 1) / z);
    const long long cost = (units + ctas - 1) / ctas * (z + 2);
    if (best == 0 || cost < best) {
      best = cost;
      zc = z;
    }
  }
  return zc;
}

template <int CIN, int COUT, int FUSE = kFuseNone>
cudaError_t ws_launch(const uint16_t* x, const uint16_t* w, const float* bias,
                      const uint16_t* mask, uint16_t* y, const Vol& g, int flags,
                      cudaStream_t s, const ConvFuse& fuse = ConvFuse()) {
  using Cfg = WsCfg<CIN, COUT>;
  const auto fn = conv_fwd_ws_kernel<CIN, COUT, FUSE>;
  static int per_sm = -1, nsm = 0;
  if (per_sm < 0) per_sm = ctas_per_sm((const void*)fn, Cfg::kSmem, Cfg::kCols, &nsm);
  const int ctas = per_sm * nsm;
  ZmGrid zg;
  zg.nbx = (g.nx + Cfg::kTX - 1) / Cfg::kTX;
  zg.nb = zg.nbx * ((g.ny + Cfg::kTY - 1) / Cfg::kTY);
  zg.zc = ws_run(zg.nb, g.nz, g.ns, ctas);
  if (FUSE == kFusePool) zg.zc += zg.zc & 1;  // pairs of planes stay in a unit
  zg.nzc = (g.nz + zg.zc - 1) / zg.zc;
  zg.units = zg.nb * g.ns * zg.nzc;
  const int grid = zg.units < ctas ? zg.units : ctas;
  RowMaps maps;
  if (!encode_volume(&maps.a, x, CIN, g, Cfg::kTX + 2, Cfg::kTY + 2) ||
      !encode_rows(&maps.b, w, CIN, 27 * COUT, COUT))
    return cudaErrorInvalidValue;
  fn<<<grid, 192, Cfg::kSmem, s>>>(maps, bias, mask, y, g, flags, zg, fuse);
  return cudaGetLastError();
}

// one CTA per SM over all parts
int wgrad_splits(int parts, int nchunks) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  int ns = nsm / parts;
  if (ns > nchunks) ns = nchunks;
  return ns < 1 ? 1 : ns;
}

// chunks of 64 voxels u over [g0 - 1, g1 + 1)
int wgrad_chunks(const Vol& g) { return g.g1 > g.g0 ? (g.g1 - g.g0 + 2 + 63) / 64 : 0; }

template <int CIN, int COUT>
cudaError_t wgrad_launch(const uint16_t* x, const uint16_t* dy, float* dw, float* ws,
                         const Vol& g, int accumulate, cudaStream_t s) {
  using Cfg = WgCfg<CIN, COUT>;
  const int nchunks = wgrad_chunks(g);
  const int nsplit = wgrad_splits(Cfg::kParts, nchunks);
  if (nchunks > 0) {
    cudaFuncSetAttribute(conv_wgrad_kernel<CIN, COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                         Cfg::kSmem);
    RowMaps maps;
    if (!encode_rows(&maps.a, x, CIN, g.vp, Cfg::kKV) ||
        !encode_rows(&maps.b, dy, COUT, g.vp, Cfg::kAVox))
      return cudaErrorInvalidValue;
    conv_wgrad_kernel<CIN, COUT>
        <<<dim3(Cfg::kParts, nsplit), 192, Cfg::kSmem, s>>>(maps, ws, g, nchunks);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  wgrad_reduce_kernel<CIN, COUT><<<27 * COUT * CIN / 32, 512, 0, s>>>(
      ws, dw, nchunks > 0 ? nsplit : 0, accumulate);
  return cudaGetLastError();
}

}  // namespace

bool vol_ok(int nx, int ny, int nz, int ns) {
  if (nx < 1 || ny < 1 || nz < 1 || ns < 1) return false;
  const double v = (double)(nx + 2) * (ny + 2) * (nz + 2) * ns;
  return v + 4.0 * (nx + 2) * (ny + 2) < 2147483647.0 / 2;
}

bool conv_shape_ok(int cin, int cout) {
  return (cin == 16 && (cout == 16 || cout == 32)) || (cin == 32 && (cout == 16 || cout == 64)) ||
         (cin == 64 && cout == 32);
}

#define TPFA_CONV_SHAPES(X) X(16, 16) X(16, 32) X(32, 16) X(32, 64) X(64, 32)

// 0: tile kernel, 1: z-marching kernel, 2: z-marching kernel with the z-taps
// folded into N (1 and 2 where their ring fits, else 0), 4: the folded kernel
// with warp-specialised roles, 3: the fastest as measured on GB300 (default: 4)
static int g_conv_kernel = 3;

cudaError_t conv_fwd(const uint16_t* x, const uint16_t* w, const float* bias, const uint16_t* mask,
                     uint16_t* y, const Vol& g, int cin, int cout, int flags, cudaStream_t s) {
  const bool ring = !(cin == 64 && cout == 32);
  const int kern = g_conv_kernel != 3 ? g_conv_kernel : 4;
  if (kern == 4) {
#define X(CI, CO) \
  if (cin == CI && cout == CO) return ws_launch<CI, CO>(x, w, bias, mask, y, g, flags, s);
    TPFA_CONV_SHAPES(X)
#undef X
  }
  if (ring && kern == 2) {
#define X(CI, CO) \
  if (cin == CI && cout == CO) return zf_launch<CI, CO>(x, w, bias, mask, y, g, flags, s);
    X(16, 16) X(16, 32) X(32, 16) X(32, 64)
#undef X
  }
  if (ring && kern == 1) {
#define X(CI, CO) \
  if (cin == CI && cout == CO) return zm_launch<CI, CO>(x, w, bias, mask, y, g, flags, s);
    X(16, 16) X(16, 32) X(32, 16) X(32, 64)
#undef X
  }
#define X(CI, CO) \
  if (cin == CI && cout == CO) return fwd_launch<CI, CO>(x, w, bias, mask, y, g, flags, s);
  TPFA_CONV_SHAPES(X)
#undef X
  return cudaErrorInvalidValue;
}

cudaError_t conv_fwd_fused(const uint16_t* x, const uint16_t* w, const float* bias, uint16_t* y,
                           const Vol& g, int cin, int cout, int flags, const ConvFuse& f,
                           cudaStream_t s) {
  if (g_conv_kernel < 3) return cudaErrorNotSupported;
#define X(CI, CO, F) \
  if (cin == CI && cout == CO && f.mode == F) \
    return ws_launch<CI, CO, F>(x, w, bias, nullptr, y, g, flags, s, f);
  X(16, 16, kFusePool) X(16, 32, kFusePool) X(64, 32, kFuseUpadd) X(32, 16, kFuseUpadd)
  X(16, 16, kFuseCells)
#undef X
  return cudaErrorNotSupported;
}

size_t conv_wgrad_ws_bytes(const Vol& g, int cin, int cout) {
  const int parts = cin == 16 ? 1 : 3;
  const int nchunks = wgrad_chunks(g);
  // 27 cin cout floats per split (all parts together)
  return (size_t)wgrad_splits(parts, nchunks < 1 ? 1 : nchunks) * 27 * cin * cout * sizeof(float);
}

cudaError_t conv_wgrad(const uint16_t* x, const uint16_t* dy, float* dw, float* ws, const Vol& g,
                       int cin, int cout, int accumulate, cudaStream_t s) {
#define X(CI, CO) \
  if (cin == CI && cout == CO) return wgrad_launch<CI, CO>(x, dy, dw, ws, g, accumulate, s);
  TPFA_CONV_SHAPES(X)
#undef X
  return cudaErrorInvalidValue;
}

}  // namespace net
}  // namespace tpfa

using tpfa::net::Vol;

static int conv_args_ok(const void* x, const void* y, int nx, int ny, int nz, int ns, int cin,
                        int cout, int* dev) {
  if (!tpfa::net::vol_ok(nx, ny, nz, ns) || !tpfa::net::conv_shape_ok(cin, cout))
    return TPFA_EINVAL;
  if (cudaGetDevice(dev) != cudaSuccess) return TPFA_ECUDA;
  const Vol g = tpfa::net::make_vol(nx, ny, nz, ns);
  if (!tpfa::dev_ok(x, (size_t)g.vp * cin * 2, 16, *dev) ||
      !tpfa::dev_ok(y, (size_t)g.vp * cout * 2, 16, *dev))
    return TPFA_EINVAL;
  return TPFA_OK;
}

extern "C" int tpfa_conv3d_bf16(const uint16_t* x, const uint16_t* w, const float* bias,
                                const uint16_t* mask, uint16_t* y, int nx, int ny, int nz,
                                int ns, int cin, int cout, int flags, void* stream) {
  int dev = -1;
  int rc = conv_args_ok(x, y, nx, ny, nz, ns, cin, cout, &dev);
  if (rc != TPFA_OK) return rc;
  if (flags & ~3) return TPFA_EINVAL;
  const Vol g = tpfa::net::make_vol(nx, ny, nz, ns);
  if (!tpfa::dev_ok(w, (size_t)27 * cin * cout * 2, 16, dev) ||
      !tpfa::opt_dev_ok(bias, (size_t)cout * 4, 4, dev))
    return TPFA_EINVAL;
  if ((flags & tpfa::net::kConvMask) && !tpfa::dev_ok(mask, (size_t)g.vp * cout * 2, 16, dev))
    return TPFA_EINVAL;
  if (x == y) return TPFA_EINVAL;
  return tpfa::net::conv_fwd(x, w, bias, mask, y, g, cin, cout, flags, (cudaStream_t)stream) ==
                 cudaSuccess
             ? TPFA_OK
             : TPFA_ECUDA;
}

extern "C" int tpfa_conv3d_wgrad_bf16(const uint16_t* x, const uint16_t* dy, float* dw, int nx,
                                      int ny, int nz, int ns, int cin, int cout, int accumulate,
                                      void* stream) {
  int dev = -1;
  int rc = conv_args_ok(x, dy, nx, ny, nz, ns, cin, cout, &dev);
  if (rc != TPFA_OK) return rc;
  if (!tpfa::dev_ok(dw, (size_t)27 * cin * cout * 4, 4, dev)) return TPFA_EINVAL;
  const Vol g = tpfa::net::make_vol(nx, ny, nz, ns);
  cudaStream_t s = (cudaStream_t)stream;
  float* ws = nullptr;
  if (cudaMallocAsync((void**)&ws, tpfa::net::conv_wgrad_ws_bytes(g, cin, cout), s) != cudaSuccess)
    return TPFA_ENOMEM;
  cudaError_t e = tpfa::net::conv_wgrad(x, dy, dw, ws, g, cin, cout, accumulate, s);
  cudaFreeAsync(ws, s);
  return e == cudaSuccess ? TPFA_OK : TPFA_ECUDA;
}

// Selects the forward convolution kernel: 0 = 128-voxel tiles with all nine
// row groups per tile, 1 = z-marching ring where it fits, 2 = z-marching ring
// with the z-taps folded into N, 3 = the default (4), 4 = the folded
// ring with warp-specialised roles.
extern "C" int tpfa_conv3d_select(int kernel) {
  if (kernel < 0 || kernel > 4) return TPFA_EINVAL;
  tpfa::net::g_conv_kernel = kernel;
  return TPFA_OK;
}

namespace tpfa {
namespace net {
// One block waits, with the bounded wait of every tensor-core kernel here, for
// an mbarrier phase that no thread completes (one arrival expected, none
// made): the wait gives up after `polls` polls and records the timeout the way
// a stalled tensor-core kernel does.  No tensor memory, no tensor-core work.
__global__ void wait_probe_kernel(uint32_t polls) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) tc::mbar_init(&bar, 1);
  __syncthreads();
  const bool ok = tc::mbar_wait(&bar, 0, polls);
  if (!ok && threadIdx.x == 0) atomicOr(&g_tc_timeout, 1);
}
}  // namespace net
}  // namespace tpfa

// Test hook for the failure path of the bounded waits (see the header).
extern "C" int tpfa_tc_wait_probe(uint32_t polls, void* stream) {
  if (polls < 1 || polls > tpfa::net::kWaitLimit) return TPFA_EINVAL;
  tpfa::net::wait_probe_kernel<<<1, 32, 0, (cudaStream_t)stream>>>(polls);
  return cudaGetLastError() == cudaSuccess ? TPFA_OK : TPFA_ECUDA;
}

// Waits for the stream, then reports (and clears) a tensor-core wait that
// gave up in any kernel of this library since the last call.
extern "C" int tpfa_net_status(void* stream) {
  if (cudaStreamSynchronize((cudaStream_t)stream) != cudaSuccess) return TPFA_ECUDA;
  int h = 0;
  if (cudaMemcpyFromSymbol(&h, tpfa::net::g_tc_timeout, sizeof(int)) != cudaSuccess)
    return TPFA_ECUDA;
  if (h) {
    const int zero = 0;
    cudaMemcpyToSymbol(tpfa::net::g_tc_timeout, &zero, sizeof(int));
    return TPFA_EINTERNAL;
  }
  return TPFA_OK;
}
