// 3x3x3 convolutions on the fifth-generation tensor cores: tcgen05.mma with
// the accumulator in tensor memory.  Computes the same as the mma.sync
// kernels in cnn.cu (BF16 in, FP32 accumulate), for every layer of the
// network (16 -> 32, 32 -> 32 and 32 -> 16 channels):
//   Y[v][co] = act(bias[co] + sum_t,ci X[v + off(t)][ci] W[t][co][ci] (+ R[v][co]))
// with 'same' zero padding; the data gradient is the same convolution of dY
// with W[26 - t] transposed, read that way when the weights are staged.
//
// The x taps go into the N dimension of the MMA.  A tile is 128 voxels (the
// MMA's M) of one z plane, TY runs of TX along x; for each of the nine (dz,
// dy) the MMAs multiply the tile's voxels moved by (dz, dy) with the weights
// of all three dx at once, N = 3 Cout:
//   D[x][dx][co] = sum_{dz,dy,ci} X[x, y + dy, z + dz][ci] W[dz,dy,dx][co][ci],
// and the epilogue adds out[x] = D[x - 1][0] + D[x][1] + D[x + 1][2] across
// TMEM lanes.  With one tap per MMA (N = 32) an MMA reads 5 KB of operands
// from shared memory for 16 cycles of tensor work; with three it reads 7 KB
// for 48, and a tile takes 18 MMAs instead of 54.  Runs shorter than the
// row give up their two end voxels (TX - 2 outputs a run); a row that fits
// one run loses nothing, its neighbours outside the grid being zero.
// TX in {16, 32, 64, 128} is the one with the fewest tiles for the grid.
//
// Shared memory holds planes of (TY + 2) x TX voxels, a row of channels (64
// or 32 bytes, swizzled over its length) per voxel: one TMA box a plane, which
// is a K-major operand as it lies, and a (dz, dy) tap is a descriptor on plane
// z + dz that starts (dy + 1) runs in (a multiple of the swizzle's period).
// The weights are 9 boxes of 3 Cout rows, or for the data gradient 27 boxes
// in reversed order that are used with N contiguous, so that nothing is
// transposed.  A CTA marches along z through a column of tiles, so each plane
// is loaded once per column and serves three tiles; the tiles of all columns
// are dealt to the CTAs in contiguous ranges of equal length.
//
// One CTA of 18 warps per SM: warp 0 issues the MMAs, warp 1 the TMA copies,
// four groups of four warps form the epilogue, each group of every fourth
// tile; up to ten plane buffers and four TMEM accumulators let all three
// overlap.  Every wait on an mbarrier is bounded: on expiry the CTA records an
// error, finishes its copies and MMAs in flight (again bounded), frees its
// TMEM and returns; the outputs it did not reach are NaN, and the context's
// next call that synchronises returns BO_ERR_TIMEOUT.
// Measured, 64x64x32 voxels x 4 samples, 32 -> 32 channels: forward with
// residual 103 us a call on the first tcgen05 form (a tap per MMA, a 10 x 18 x
// 3 halo a tile in 16-byte TMA rows), 63 with the x taps in N and planes copied
// by cp.async in 16-byte chunks, 40 in this form; data gradient 150, 82 and 57
// (about 20 of it the call's synchronisation).  Per tile of 2250 cycles the
// MMAs take 900 to issue and execute, their commits and waits 900, and the
// epilogue, two shuffles per output, 1150 of its four groups.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>

#include "bo_internal.cuh"

namespace bo {
namespace {

using bf16 = __nv_bfloat16;

constexpr int kGroups = 4;           // groups of four epilogue warps
constexpr int kTcThreads = 64 + 128 * kGroups;  // warp 0: MMA issue; 1: TMA; the others: epilogue
constexpr int kMaxPlanes = 10;       // plane buffers: three of a tile, the others on their way or signalled
constexpr int kAccs = 4;             // accumulators (128 TMEM columns each)
constexpr int kSpinLimit = 1 << 26;
constexpr int kTileM = 128;
constexpr int kTcSmem = 227 * 1024;  // shared memory of a block

__device__ int g_tc_err;  // set by a CTA whose wait expired (read and cleared by bo_tc_status)

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// shared-memory matrix descriptor, version 1.  No swizzle (span 16): lbo and
// sbo are the strides between core matrices (8 rows of 16 bytes) along K and
// along M or N.  Rows of 32 or 64 bytes swizzled over that span, as TMA writes
// them: sbo is the stride between groups of 8 rows; with M or N contiguous lbo
// is the stride between spans along it (else not used).
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo, int span = 16) {
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46) |
         ((uint64_t)(span == 64 ? 4 : span == 32 ? 6 : 0) << 61);
}

// instruction descriptor, kind::f16: D FP32, A and B BF16, M = 128; am, bn:
// A (B) with M (N) contiguous in memory instead of K
__host__ __device__ constexpr uint32_t idesc(int n, bool am, bool bn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (am ? 1u << 15 : 0u) | (bn ? 1u << 16 : 0u) | ((uint32_t)(n >> 3) << 17) |
         ((128u >> 4) << 24);
}

// one thread of a converged warp (always the same)
__device__ __forceinline__ bool elect_one() {
  uint32_t e;
  asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
  return e != 0;
}
// (issued by the thread that elect_one picks, for a whole tile in one branch:
// 45 cycles an MMA.  An elect.sync per MMA took 60, and a branch on lane == 0,
// which the compiler does not know to be one thread, 92.)
__device__ __forceinline__ void umma(uint32_t d, uint64_t a, uint64_t b, uint32_t id, bool acc) {
  asm volatile(
      "{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(id), "r"((uint32_t)acc)
      : "memory");
}

// (stop: where not NULL, the flag of another role's failure, which ends the wait)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, const volatile int* stop = nullptr) {
  uint32_t done = 0;
  for (int it = 0; it < kSpinLimit; ++it) {
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (stop && (it & 255) == 255 && *stop) return false;
  }
  return false;
}
// a wait of this block expired: the block's flag, the process's and the context's
__device__ __forceinline__ void report_timeout(volatile int* sfail, const TcWait& lim) {
  *sfail = 1;
  atomicExch(&g_tc_err, 1);
  if (lim.err) {
    *lim.err = 1;
    __threadfence_system();
  }
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void fence_async_proxy() { asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory"); }
// 16 bytes from global to shared memory, or zeros
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  return (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(lo)) | ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(hi)) << 16);
}
// 32 bytes to global memory: one store where the address allows it (wide),
// which fills a sector, or two of 16 bytes
__device__ __forceinline__ void st32(void* p, bool wide, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e, uint32_t f,
                                     uint32_t g, uint32_t h) {
  if (wide) {
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"l"(p), "r"(a), "r"(b), "r"(c), "r"(d), "r"(e), "r"(f),
                 "r"(g), "r"(h)
                 : "memory");
  } else {
    reinterpret_cast<uint4*>(p)[0] = make_uint4(a, b, c, d);
    reinterpret_cast<uint4*>(p)[1] = make_uint4(e, f, g, h);
  }
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;\n" ::"n"(N) : "memory"); }
__device__ __forceinline__ void named_barrier(int id, int threads) {
  asm volatile("bar.sync %0, %1;\n" ::"r"(id), "r"(threads) : "memory");
}

// N consecutive TMEM columns at each of three addresses
#define BO_R8(o) "=r"(r[o]), "=r"(r[o + 1]), "=r"(r[o + 2]), "=r"(r[o + 3]), "=r"(r[o + 4]), "=r"(r[o + 5]), "=r"(r[o + 6]), "=r"(r[o + 7])
__device__ __forceinline__ void tmem_ld3(uint32_t a0, uint32_t a1, uint32_t a2, float (&v)[3][16]) {
  uint32_t r[48];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%48];\n"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%49];\n"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%32,%33,%34,%35,%36,%37,%38,%39,%40,%41,%42,%43,%44,%45,%46,%47}, [%50];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : BO_R8(0), BO_R8(8), BO_R8(16), BO_R8(24), BO_R8(32), BO_R8(40)
      : "r"(a0), "r"(a1), "r"(a2)
      : "memory");
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 16; ++i) v[k][i] = __uint_as_float(r[16 * k + i]);
}
__device__ __forceinline__ void tmem_ld3(uint32_t a0, uint32_t a1, uint32_t a2, float (&v)[3][8]) {
  uint32_t r[24];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%24];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%25];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%26];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : BO_R8(0), BO_R8(8), BO_R8(16)
      : "r"(a0), "r"(a1), "r"(a2)
      : "memory");
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int i = 0; i < 8; ++i) v[k][i] = __uint_as_float(r[8 * k + i]);
}

// The tiles: nz tiles of a column (z fastest), columns by x tile, y tile, sample
struct ConvGrid {
  int nx, ny, nz, B;
  int ltx;              // log2 TX
  int planes;           // plane buffers
  int ntx, nty;
  int64_t tiles;
};
// A tile's place, stepped from tile to tile (a division once per CTA)
struct March {
  int z, tx, ty, b;
  template <typename Grid>
  __device__ __forceinline__ March(const Grid& g, int64_t t) {
    const int c = (int)(t / g.nz);
    z = (int)(t - (int64_t)c * g.nz);
    tx = c % g.ntx;
    ty = c / g.ntx % g.nty;
    b = c / g.ntx / g.nty;
  }
  template <typename Grid>
  __device__ __forceinline__ void next(const Grid& g) {
    if (++z < g.nz) return;
    z = 0;
    if (++tx < g.ntx) return;
    tx = 0;
    if (++ty < g.nty) return;
    ty = 0;
    ++b;
  }
  __device__ __forceinline__ int x0(const ConvGrid& g) const { return tx * ((1 << g.ltx) - 2); }
  __device__ __forceinline__ int y0(const ConvGrid& g) const { return ty * (kTileM >> g.ltx); }
};
__host__ __device__ __forceinline__ int plane_rows(int ltx) { return kTileM + (2 << ltx); }

template <int CIN, int COUT>
struct ConvLayout {
  static constexpr int NB = 3 * COUT;
  static constexpr int kW = 9 * CIN * NB * 2;
  static constexpr int kEdge = kGroups * 2 * 2 * 4 * 16 * 4;  // [warp group][buffer][side][warp][channel]
  static constexpr int kOffEdge = kW;
  static constexpr int kOffBias = kOffEdge + kEdge;
  static constexpr int kOffBar = kOffBias + 128;
  static constexpr int kOffPlanes = (kOffBar + 256 + 1023) / 1024 * 1024;  // (29 barriers and the TMEM address)
};

__device__ __forceinline__ void expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void tma_rows(const CUtensorMap* map, uint32_t dst, uint32_t bar, int row) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(row), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tma_plane(const CUtensorMap* map, uint32_t dst, uint32_t bar, int x, int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];\n" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(0), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// OUT 0: Y = ReLU(conv + bias (+ R)) in BF16; 1: Yf = conv + bias in FP32;
// 2: Y = conv + bias in BF16 and its channels 0..3 in FP32 (Yf[v][4]).
// TRANSPOSED: the data gradient, W [27][CIN][COUT] (the layer's own output
// channels are this convolution's inputs).
// mbarriers: full[p] plane buffer p holds its plane; empty[p] the MMAs that
// read it are done; accfull[a], accempty[a] (4 warps) as the accumulators pass
// between the MMAs and the epilogue; wfull the weights are there.  The n-th
// completion of a barrier has parity n & 1.
template <int CIN, int COUT, int OUT, bool RES, bool TRANSPOSED>
__global__ void __launch_bounds__(kTcThreads, 1) k_conv3d_tc(const __grid_constant__ ConvGrid g,
                                                           const __grid_constant__ CUtensorMap xmap,
                                                           const __grid_constant__ CUtensorMap wmap,
                                                           const float* __restrict__ bias, const bf16* __restrict__ R,
                                                           bf16* __restrict__ Y, float* __restrict__ Yf, const TcWait lim) {
  using L = ConvLayout<CIN, COUT>;
  constexpr int NB = L::NB;
  constexpr int CH = RES || COUT == 16 ? 8 : 16;  // channels an epilogue thread takes at a time (registers)
  extern __shared__ uint8_t smraw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 1023) & ~uintptr_t(1023));
  float* edge = reinterpret_cast<float*>(sm + L::kOffEdge);
  float* sbias = reinterpret_cast<float*>(sm + L::kOffBias);
  const uint32_t bars = smem_u32(sm + L::kOffBar);
  auto full = [&](int p) { return bars + 8 * p; };
  auto empty = [&](int p) { return bars + 8 * (kMaxPlanes + p); };
  auto accfull = [&](int a) { return bars + 8 * (2 * kMaxPlanes + a); };
  auto accempty = [&](int a) { return bars + 8 * (2 * kMaxPlanes + kAccs + a); };
  const uint32_t wfull = bars + 8 * (2 * kMaxPlanes + 2 * kAccs);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + L::kOffBar + 8 * (2 * kMaxPlanes + 2 * kAccs + 1));
  volatile int* sfail = reinterpret_cast<volatile int*>(tslot + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int p = 0; p < kMaxPlanes; ++p) {
      mbar_init(full(p), 1);
      mbar_init(empty(p), 1);
    }
    for (int a = 0; a < kAccs; ++a) {
      mbar_init(accfull(a), 1);
      mbar_init(accempty(a), 4);
    }
    mbar_init(wfull, 1);
    *sfail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid >= 64 && tid < 64 + COUT) sbias[tid - 64] = bias ? bias[tid - 64] : 0.f;
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tslot;
  const int TX = 1 << g.ltx;
  const uint32_t wbase = smem_u32(sm);
  const uint32_t pbase = smem_u32(sm + L::kOffPlanes), pbytes = (uint32_t)(plane_rows(g.ltx) * CIN * 2);
  const int64_t t0 = g.tiles * blockIdx.x / gridDim.x, t1 = g.tiles * (blockIdx.x + 1) / gridDim.x;
  const int64_t V = (int64_t)g.nx * g.ny * g.nz;
  const bool wide = ((reinterpret_cast<uintptr_t>(Y) | reinterpret_cast<uintptr_t>(Yf)) & 31) == 0;

  if (warp == 1) {
    // ---- TMA: the weights and the planes
    if (elect_one() && t0 < t1) {
      expect_tx(wfull, (uint32_t)L::kW);
      if (!TRANSPOSED) {
        for (int i = 0; i < 9; ++i) tma_rows(&wmap, wbase + (uint32_t)(i * CIN * NB * 2), wfull, i * NB);
      } else {
        for (int i = 0; i < 27; ++i) tma_rows(&wmap, wbase + (uint32_t)(i * CIN * COUT * 2), wfull, (26 - i) * CIN);
      }
      int buf = 0, round = 0, seq = 0;  // the buffer and the round of the next plane; planes issued
      bool ok = true;
      March m(g, t0);
      for (int64_t t = t0; t < t1 && ok; ++t, m.next(g)) {
        const bool start = t == t0 || m.z == 0;
        for (int pz = start ? max(m.z - 1, 0) : m.z + 1; pz <= min(m.z + 1, g.nz - 1); ++pz) {
          if (round > 0) ok = mbar_wait(empty(buf), (round - 1) & 1, sfail);
          if (!ok) break;
          expect_tx(full(buf), pbytes);
          tma_plane(&xmap, pbase + (uint32_t)buf * pbytes, full(buf), m.x0(g), m.y0(g) - 1, m.b * g.nz + pz);
          ++seq;
          if (++buf == g.planes) {
            buf = 0;
            ++round;
          }
        }
      }
      if (!ok) report_timeout(sfail, lim);
      // no copy is in flight when the block ends
      mbar_wait(wfull, 0);
      for (int k = max(0, seq - g.planes); k < seq; ++k) mbar_wait(full(k % g.planes), (k / g.planes) & 1);
    }
    __syncwarp();
  } else if (warp == 0) {
    // ---- MMA issue (the whole warp waits, one thread issues)
    if (t0 < t1) {
      bool ok = __all_sync(0xffffffffu, mbar_wait(wfull, 0, sfail));
      // planes waited for, and the buffer and round of the next one; the
      // buffer of the tile's plane z
      int waited = 0, wbuf = 0, wround = 0, next = 0, cur = 0, issued = 0;
      auto around = [&](int p) { return p < 0 ? p + g.planes : p >= g.planes ? p - g.planes : p; };
      March m(g, t0);
      const int64_t ts = min(t1, t0 + lim.tiles);
      for (int64_t t = t0; t < ts && ok; ++t, m.next(g)) {
        const int k = (int)(t - t0), a = k % kAccs, z = m.z;
        const bool start = t == t0 || z == 0, end = t + 1 == t1 || z == g.nz - 1;
        if (start) {
          next = waited + (z > 0 ? 1 : 0);
          cur = around(wbuf + (z > 0 ? 1 : 0));
        }
        const int need = next + (z < g.nz - 1 ? 1 : 0);
        for (; waited <= need && ok; ++waited) {
          ok = __all_sync(0xffffffffu, mbar_wait(full(wbuf), wround & 1, sfail));
          if (++wbuf == g.planes) {
            wbuf = 0;
            ++wround;
          }
        }
        if (ok && k >= kAccs) ok = __all_sync(0xffffffffu, mbar_wait(accempty(a), (k / kAccs - 1) & 1, sfail));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        if (elect_one()) {
          const uint32_t dacc = tmem + (uint32_t)(a * 128);
          // weights: N rows of CIN channels, or for the data gradient CIN rows
          // of COUT channels per x tap
          const uint64_t db0 = TRANSPOSED ? smem_desc(wbase, CIN * COUT * 2, 16 * COUT, COUT * 2)
                                          : smem_desc(wbase, 16, 16 * CIN, CIN * 2);
          bool acc = false;
          for (int dz = -1; dz <= 1; ++dz) {
            if (z + dz < 0 || z + dz >= g.nz) continue;
            const uint64_t da0 = smem_desc(pbase + (uint32_t)around(cur + dz) * pbytes, 16, 16 * CIN, CIN * 2);
            const uint64_t dbz = db0 + (uint64_t)(((dz + 1) * 3 * CIN * NB * 2) >> 4);
#pragma unroll
            for (int dy = 0; dy < 3; ++dy)
#pragma unroll
              for (int ks = 0; ks < CIN / 16; ++ks) {
                umma(dacc, da0 + (uint64_t)((dy * TX * CIN * 2 + ks * 32) >> 4),
                     dbz + (uint64_t)((dy * CIN * NB * 2 + (TRANSPOSED ? ks * 32 * COUT : ks * 32)) >> 4),
                     idesc(NB, false, TRANSPOSED), acc);
                acc = true;
              }
          }
          if (z > 0) umma_commit(empty(around(cur - 1)));
          if (end) {
            umma_commit(empty(cur));
            if (z < g.nz - 1) umma_commit(empty(around(cur + 1)));
          }
          umma_commit(accfull(a));
        }
        __syncwarp();
        ++issued;
        ++next;
        cur = around(cur + 1);
      }
      if (!ok || ts < t1) report_timeout(sfail, lim);
      // the MMAs in flight finish before shared and tensor memory go away (an
      // epilogue group that gave up has not waited for them)
      for (int k = max(0, issued - kAccs); k < issued; ++k) mbar_wait(accfull(k % kAccs), (k / kAccs) & 1);
    }
    __syncwarp();
  } else {
    {
      // ---- epilogue: the four warps of a group take every fourth tile, each
      // warp the TMEM lane quarter warp % 4, CH channels at a time
      const int quarter = warp & 3, group = (warp - 2) >> 2;
      const int row = quarter * 32 + lane, xl = row & (TX - 1), yl = row >> g.ltx;
      const bool cross = TX > 32;  // runs that span warps
      const bool inner = xl > 0, innerr = xl < TX - 1;
      bool ok = true;
      March at(g, t0);
      bool mine = false;
      size_t o = 0;  // the thread's output in this tile
      uint4 res[RES ? COUT / 8 : 1];
      // the place of tile t, and its residuals (loaded while the tile before is worked on)
      auto place = [&](int64_t t) {
        if (t >= t1) return;
        const int x = at.x0(g) + xl, y = at.y0(g) + yl;
        mine = x < g.nx && y < g.ny && (inner || x == 0) && (innerr || x == g.nx - 1);
        o = ((size_t)at.b * V + x + (size_t)g.nx * (y + (size_t)g.ny * at.z)) * COUT;
        if (RES && mine) {
#pragma unroll
          for (int q = 0; q < COUT / 8; ++q) res[q] = __ldcs(reinterpret_cast<const uint4*>(R + o + 8 * q));
        }
      };
      for (int i = 0; i < group; ++i) at.next(g);
      place(t0 + group);
      for (int64_t t = t0 + group; t < t1; t += kGroups) {
        const int k = (int)(t - t0), a = k % kAccs;
        // (after an expired wait the warp still meets the barriers, and stores nothing)
        if (ok && !mbar_wait(accfull(a), (k / kAccs) & 1, sfail)) {
          ok = false;
          report_timeout(sfail, lim);
        }
        ok = __all_sync(0xffffffffu, ok);
        uint32_t pk[8];  // 16 channels in BF16
#pragma unroll
        for (int part = 0; part < COUT / CH; ++part) {
          const int ch0 = part * CH;
          float d[3][CH];
          if (ok) {
            if (part == 0) asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
            const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(a * 128 + ch0);
            tmem_ld3(ta, ta + COUT, ta + 2 * COUT, d);
            if (part == COUT / CH - 1) {
              asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
              __syncwarp();
              if (lane == 0) mbar_arrive(accempty(a));
            }
          } else {
#pragma unroll
            for (int i = 0; i < CH; ++i) d[0][i] = d[1][i] = d[2][i] = 0.f;
          }
          // the columns beyond the warp's ends, left of lane 0 and right of
          // lane 31 (two buffers: one is rewritten after the other's barrier)
          float* eb = edge + (group * 2 + part % 2) * 2 * 4 * 16;
          if (cross) {
            if (lane == 31) {
#pragma unroll
              for (int i = 0; i < CH; i += 4)
                *reinterpret_cast<float4*>(eb + quarter * 16 + i) = make_float4(d[0][i], d[0][i + 1], d[0][i + 2], d[0][i + 3]);
            }
            if (lane == 0) {
#pragma unroll
              for (int i = 0; i < CH; i += 4)
                *reinterpret_cast<float4*>(eb + 4 * 16 + quarter * 16 + i) =
                    make_float4(d[2][i], d[2][i + 1], d[2][i + 2], d[2][i + 3]);
            }
            named_barrier(2 + group, 128);
          }
          // out = D[x - 1][0] + D[x][1] + D[x + 1][2]
          float out[CH];
#pragma unroll
          for (int i = 0; i < CH; ++i) {
            const float l = __shfl_up_sync(0xffffffffu, d[0][i], 1), r = __shfl_down_sync(0xffffffffu, d[2][i], 1);
            out[i] = (inner && lane > 0 ? l : 0.f) + d[1][i] + (innerr && lane < 31 ? r : 0.f);
          }
          if (cross && ((lane == 0 && inner) || (lane == 31 && innerr))) {
            const float* ep = eb + (lane == 0 ? ((quarter + 3) & 3) * 16 : 4 * 16 + ((quarter + 1) & 3) * 16);
#pragma unroll
            for (int i = 0; i < CH; ++i) out[i] += ep[i];
          }
#pragma unroll
          for (int i = 0; i < CH; i += 4) {
            const float4 b4 = *reinterpret_cast<const float4*>(sbias + ch0 + i);
            out[i] += b4.x, out[i + 1] += b4.y, out[i + 2] += b4.z, out[i + 3] += b4.w;
          }
          if (mine && ok) {
            if (OUT == 1) {
#pragma unroll
              for (int q = 0; q < CH / 8; ++q) {
                const float* v = out + 8 * q;
                st32(Yf + o + ch0 + 8 * q, wide, __float_as_uint(v[0]), __float_as_uint(v[1]), __float_as_uint(v[2]),
                     __float_as_uint(v[3]), __float_as_uint(v[4]), __float_as_uint(v[5]), __float_as_uint(v[6]),
                     __float_as_uint(v[7]));
              }
            } else {
              if (OUT == 2 && part == 0)
                *reinterpret_cast<float4*>(Yf + (o / COUT) * 4) = make_float4(out[0], out[1], out[2], out[3]);
#pragma unroll
              for (int e = 0; e < CH / 2; ++e) {
                float v0 = out[2 * e], v1 = out[2 * e + 1];
                if (RES) {
                  const uint4 r4 = res[RES ? part * (CH / 8) + e / 4 : 0];
                  const uint32_t rw = e % 4 == 0 ? r4.x : e % 4 == 1 ? r4.y : e % 4 == 2 ? r4.z : r4.w;
                  v0 += __uint_as_float(rw << 16);
                  v1 += __uint_as_float(rw & 0xffff0000u);
                }
                if (OUT == 0) {
                  v0 = fmaxf(v0, 0.f);
                  v1 = fmaxf(v1, 0.f);
                }
                pk[ch0 % 16 / 2 + e] = pack_bf16(v0, v1);
              }
              if ((ch0 + CH) % 16 == 0)
                st32(Y + o + ch0 + CH - 16, wide, pk[0], pk[1], pk[2], pk[3], pk[4], pk[5], pk[6], pk[7]);
            }
          }
        }
        for (int i = 0; i < kGroups; ++i) at.next(g);
        place(t + kGroups);
      }
      // a wait of the block expired: NaN on all tiles of the group (a warp that
      // did not give up may have added a column of one that did)
      if (*sfail) {
        at = March(g, t0);
        for (int64_t t = t0; t < t1; ++t, at.next(g)) {
          if ((t - t0) % kGroups != group) continue;
          place(t);
          if (!mine) continue;
          for (int i = 0; i < COUT; ++i) {
            if (OUT != 1) Y[o + i] = __ushort_as_bfloat16(0x7fff);
            if (OUT == 1) Yf[o + i] = __int_as_float(0x7fffffff);
            if (OUT == 2 && i < 4) Yf[(o / COUT) * 4 + i] = __int_as_float(0x7fffffff);
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
  });
  return fn;
}

// tensor map over BF16 rows of c channels (16 or 32, swizzled over the row's
// 32 or 64 bytes), out-of-range coordinates zero
bool encode(CUtensorMap* map, const bf16* p, int rank, int c, const cuuint64_t* rows, const cuuint32_t* box_rows) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = encode_fn();
  if (!enc) return false;
  cuuint64_t dims[4] = {(cuuint64_t)c}, strides[3];
  cuuint32_t box[4] = {(cuuint32_t)c};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  cuuint64_t st = 2 * (cuuint64_t)c;
  for (int d = 1; d < rank; ++d) {
    dims[d] = rows[d - 1];
    box[d] = box_rows[d - 1];
    strides[d - 1] = st;
    st *= rows[d - 1];
  }
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, rank, const_cast<bf16*>(p), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, c == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int CIN, int COUT, int OUT, bool RES, bool TRANSPOSED>
int run_conv(ConvGrid g, const bf16* X, const bf16* W, const float* bias, const bf16* R, bf16* Y, float* Yf,
             const TcWait& lim, cudaStream_t s) {
  using L = ConvLayout<CIN, COUT>;
  CUtensorMap xmap, wmap;
  const cuuint64_t vox[3] = {(cuuint64_t)g.nx, (cuuint64_t)g.ny, (cuuint64_t)g.nz * g.B};
  const cuuint32_t vbox[3] = {1u << g.ltx, (cuuint32_t)(kTileM >> g.ltx) + 2, 1};
  const cuuint64_t wrows = 27 * (TRANSPOSED ? CIN : COUT);
  const cuuint32_t wbox = TRANSPOSED ? CIN : L::NB;
  if (!encode(&xmap, X, 4, CIN, vox, vbox) || !encode(&wmap, W, 2, TRANSPOSED ? COUT : CIN, &wrows, &wbox)) return BO_ERR_ARG;
  auto kern = k_conv3d_tc<CIN, COUT, OUT, RES, TRANSPOSED>;
  const int plane = plane_rows(g.ltx) * CIN * 2;
  g.planes = (kTcSmem - L::kOffPlanes - 1024) / plane;  // (6 at least: TX = 128 with 32 channels)
  if (g.planes > kMaxPlanes) g.planes = kMaxPlanes;
  const int smem = L::kOffPlanes + g.planes * plane + 1024;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return BO_ERR_CUDA;
  const int sms = sm_count();
  const int grid = g.tiles < sms ? (int)g.tiles : sms;
  (kern<<<grid, kTcThreads, smem, s>>>(g, xmap, wmap, bias, R, Y, Yf, lim), note_launch());
  return cudaGetLastError() == cudaSuccess ? BO_OK : BO_ERR_CUDA;
}

}  // namespace

// The tensor-core path of a layer; BO_ERR_ARG where it does not apply (an
// operand off a 16-byte boundary: the caller then uses the mma.sync kernel).
//   mode: 0 ReLU, 1 ReLU with residual, 2 linear FP32 output (Yf), 3 linear
//   with BF16 output and channels 0..3 in FP32; transposed: the data
//   gradient, X = dY and W the layer's own weights [27][cin][cout] (mode 2).
//   bias may be NULL (zero).
int launch_conv_tc(int cin, int cout, int nx, int ny, int nz, int B, const __nv_bfloat16* X, const __nv_bfloat16* W,
                   const float* bias, const __nv_bfloat16* R, __nv_bfloat16* Y, float* Yf, int mode, bool transposed,
                   const TcWait& lim, cudaStream_t s) {
  for (const void* p : {(const void*)X, (const void*)W, (const void*)R, (const void*)Y, (const void*)Yf})
    if (reinterpret_cast<uintptr_t>(p) & 15) return BO_ERR_ARG;
  ConvGrid g{nx, ny, nz, B, 0, 0, 0, 0, 0};
  int64_t best = -1;
  for (int ltx = 4; ltx <= 7; ++ltx) {
    const int TX = 1 << ltx, TY = kTileM >> ltx;
    const int ntx = nx <= TX ? 1 : (nx - TX + TX - 3) / (TX - 2) + 1, nty = (ny + TY - 1) / TY;
    if (best < 0 || (int64_t)ntx * nty < best) {
      best = (int64_t)ntx * nty;
      g.ltx = ltx;
      g.ntx = ntx;
      g.nty = nty;
    }
  }
  g.tiles = best * B * nz;
  if (best * B > INT32_MAX) return BO_ERR_ARG;
  if (transposed) {
    if (mode != 2) return BO_ERR_ARG;
    if (cin == 32 && cout == 32) return run_conv<32, 32, 1, false, true>(g, X, W, bias, R, Y, Yf, lim, s);
    if (cin == 32 && cout == 16) return run_conv<32, 16, 1, false, true>(g, X, W, bias, R, Y, Yf, lim, s);
    if (cin == 16 && cout == 32) return run_conv<16, 32, 1, false, true>(g, X, W, bias, R, Y, Yf, lim, s);
    return BO_ERR_ARG;
  }
  if (cin == 32 && cout == 32) {
    if (mode == 0) return run_conv<32, 32, 0, false, false>(g, X, W, bias, R, Y, Yf, lim, s);
    if (mode == 1) return run_conv<32, 32, 0, true, false>(g, X, W, bias, R, Y, Yf, lim, s);
    if (mode == 2) return run_conv<32, 32, 1, false, false>(g, X, W, bias, R, Y, Yf, lim, s);
  }
  if (cin == 16 && cout == 32) {
    if (mode == 0) return run_conv<16, 32, 0, false, false>(g, X, W, bias, R, Y, Yf, lim, s);
    if (mode == 2) return run_conv<16, 32, 1, false, false>(g, X, W, bias, R, Y, Yf, lim, s);
  }
  if (cin == 32 && cout == 16) {
    if (mode == 2) return run_conv<32, 16, 1, false, false>(g, X, W, bias, R, Y, Yf, lim, s);
    if (mode == 3) return run_conv<32, 16, 2, false, false>(g, X, W, bias, R, Y, Yf, lim, s);
  }
  return BO_ERR_ARG;
}

namespace {

// ---- weight gradient
// dW[t][co][ci] = sum_v dY[v][co] X[v + off(t)][ci] and db[co] = sum_v dY[v][co].
//
// Two tensors meet over voxels: the "halo" tensor (32 channels) at v + off
// and the "core" tensor at v.  The halo tensor is X, or dY for the 16 -> 32
// layer (X then is the core and the taps are mirrored), so that it always
// fills the MMA's M.  An MMA takes 16 consecutive voxels of a grid row as K,
// both operands with their channels contiguous (MN-major): A is four rows of
// the halo plane, y - 1 .. y + 2, times 32 channels (M = 128), B two rows of
// the core plane, y and y + 1, times its channels (N = 64 or 32).  The eight
// (halo row, core row) pairs hold every dy tap of the two core rows and two
// pairs that are not taps and are dropped at the end.  dz picks the halo plane
// and the x tap moves A's start by one voxel, so nine accumulators hold all
// 27 taps; the pairs need 9 x 64 TMEM columns of the 512, so for 32 core
// channels the last two accumulators take one core row per MMA (32 columns;
// A's rows move with it).  A row of a plane is [channel / 8][voxel][8
// channels] with equal strides from chunk to chunk and row to row, which is
// what lets one descriptor span four rows of four chunks.
// The accumulators stay in TMEM over all tiles of a CTA (TX x 4 voxels, a
// march along z as in the convolution above); each CTA writes one partial
// sum, k_wgrad_sum adds them in a fixed order.  dY is read in FP32 by eight
// warps that round it to BF16 on its way to shared memory; X comes by cp.async
// from eight more (with four of each the dY warps took 5800 cycles a tile, the
// MMAs 3900).
// The bias gradient is summed in three FP32 parts, 72 bits, so that it keeps
// what an FP64 sum keeps (two parts took 81 us a call in place of 84, but lose
// to FP64 where large values cancel): by the dY warps as they read it, and
// where dY is the halo tensor by the X warps, which read it again from L2 (16
// -> 32: 103 us a call when the halo warps did it, 85 so).
// What bounds it: the shared-memory operand reads of the MMAs, 6 KB in 46
// cycles for 2 x 16 voxels and a ninth of the taps.
// Measured, 64x64x32 x 4 samples, 32 -> 32: 587 us a call, with scratch
// allocated in it and five launches (mma.sync gradient 144, FP64 bias sums
// 95, reduction 30, conversion 18) -> 164 with MMAs issued in a loop over
// lanes -> 103 with four producer warps a side and FP64 sums -> 84.

struct Sum3 {  // a running sum of FP32 values in three of them: 72 bits
  float a, b, c;
  __device__ __forceinline__ void add(float e) {
    const df t = df_two_sum(a, e), u = df_two_sum(b, t.lo);
    a = t.hi;
    b = u.hi;
    c = __fadd_rn(c, u.lo);
  }
  // (the parts below an infinity are NaN)
  __device__ __forceinline__ double value() const { return isfinite(a) ? (double)a + ((double)b + (double)c) : (double)a; }
};
constexpr int kWgProd = 256;      // threads that fetch halo planes, and as many core planes
constexpr int kWgThreads = 32 + 2 * kWgProd;  // warp 0: MMAs; 1-8: halo producers; 9-16: core producers; 1-16: the end
constexpr int kWgHalo = 5, kWgCore = 3;  // plane buffers
constexpr int kWgTY = 4, kWgHY = kWgTY + 3;

struct WgradGrid {
  int nx, ny, nz, B;
  int tx;  // TX: 16, 32 or 64
  int ntx, nty;
  int64_t tiles;
};

__host__ __device__ __forceinline__ int wg_halo_row(int tx) { return (tx + 2) * 16; }          // one chunk of a row
__host__ __device__ __forceinline__ int wg_core_row(int tx, int kc) { return tx * 16 + 128 / kc; }
__host__ __device__ __forceinline__ int wg_halo_plane(int tx) { return kWgHY * 4 * wg_halo_row(tx); }
__host__ __device__ __forceinline__ int wg_core_plane(int tx, int kc) { return kWgTY * kc * wg_core_row(tx, kc); }
constexpr int kWgOffBar = 0, kWgOffBias = 256, kWgOffPlanes = kWgOffBias + kWgProd * 8 * 8;


// One plane of a tensor into shared memory: NR rows from y0, NX voxels from
// x0, rows [chunk][voxel], a thread every kWgProd / KC voxels of a chunk.
// BF16 by cp.async (the caller commits); FP32 by loads, rounded to BF16,
// `wait` called between the loads and the first store, the values (BIAS)
// added to the thread's bias sums.
struct WgStep {  // voxel index -> (row, place in it), stepped without divisions
  int yl, xl;
  __device__ __forceinline__ WgStep(int i, int NX) : yl(i / NX), xl(i - i / NX * NX) {}
  __device__ __forceinline__ void next(int by, int NX) {
    for (xl += by; xl >= NX; xl -= NX) ++yl;
  }
};
template <int KC, int NR>
__device__ __forceinline__ void wg_plane_bf16(const bf16* T, size_t zb, int nx, int ny, int x0, int y0, int NX, uint32_t dst,
                                              int row_bytes, int pt) {
  const int kc = pt % KC;
  for (WgStep a(pt / KC, NX); a.yl < NR; a.next(kWgProd / KC, NX)) {
    const int x = x0 + a.xl, y = y0 + a.yl;
    const bool in = x >= 0 && x < nx && y >= 0 && y < ny;
    cp16(dst + (uint32_t)((a.yl * KC + kc) * row_bytes + a.xl * 16), T + (in ? (zb + (size_t)y * nx + x) * (KC * 8) : 0) + kc * 8,
         in);
  }
}
template <int KC, int NR, bool BIAS, typename Wait>
__device__ __forceinline__ bool wg_plane_f32(const float* T, size_t zb, int nx, int ny, int x0, int y0, int NX, uint32_t dst,
                                             int row_bytes, int pt, Sum3 (&bias)[8], Wait wait) {
  constexpr int U = 4, kStep = kWgProd / KC;  // U voxels in flight per thread
  const int kc = pt % KC;
  const int n = NR * NX;
  WgStep ld(pt / KC, NX), a = ld;
  bool waited = false;
  for (int base = 0; base < n; base += U * kStep) {  // (the same number of rounds for every thread)
    float4 v[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int x = x0 + ld.xl, y = y0 + ld.yl;
      const bool in = ld.yl < NR && x >= 0 && x < nx && y >= 0 && y < ny;
      const float4* src = reinterpret_cast<const float4*>(T + (in ? (zb + (size_t)y * nx + x) * (KC * 8) : 0) + kc * 8);
      v[u][0] = in ? __ldcs(src) : make_float4(0.f, 0.f, 0.f, 0.f);
      v[u][1] = in ? __ldcs(src + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
      ld.next(kStep, NX);
    }
    if (!waited) {
      waited = true;
      if (!__all_sync(0xffffffffu, wait())) return false;
    }
#pragma unroll
    for (int u = 0; u < U; ++u, a.next(kStep, NX)) {
      if (a.yl >= NR) continue;
      const float e[8] = {v[u][0].x, v[u][0].y, v[u][0].z, v[u][0].w, v[u][1].x, v[u][1].y, v[u][1].z, v[u][1].w};
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(dst + (uint32_t)((a.yl * KC + kc) * row_bytes + a.xl * 16)),
                   "r"(pack_bf16(e[0], e[1])), "r"(pack_bf16(e[2], e[3])), "r"(pack_bf16(e[4], e[5])),
                   "r"(pack_bf16(e[6], e[7]))
                   : "memory");
      if (BIAS) {
#pragma unroll
        for (int q = 0; q < 8; ++q) bias[q].add(e[q]);
      }
    }
  }
  return true;
}
// The bias sums alone: a tile's values, a thread every kWgProd / 4 voxels of a
// chunk of eight channels.
__device__ __forceinline__ void wg_bias_f32(const float* T, size_t zb, int nx, int ny, int x0, int y0, int NX, int pt,
                                            Sum3 (&bias)[8]) {
  constexpr int U = 2, kStep = kWgProd / 4;
  const int kc = pt % 4;
  WgStep a(pt / 4, NX);
  while (a.yl < kWgTY) {
    float4 v[U][2];
#pragma unroll
    for (int u = 0; u < U; ++u, a.next(kStep, NX)) {
      const int x = x0 + a.xl, y = y0 + a.yl;
      const bool in = a.yl < kWgTY && x < nx && y < ny;
      const float4* src = reinterpret_cast<const float4*>(T + (in ? (zb + (size_t)y * nx + x) * 32 : 0) + kc * 8);
      v[u][0] = in ? __ldg(src) : make_float4(0.f, 0.f, 0.f, 0.f);
      v[u][1] = in ? __ldg(src + 1) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const float e[8] = {v[u][0].x, v[u][0].y, v[u][0].z, v[u][0].w, v[u][1].x, v[u][1].y, v[u][1].z, v[u][1].w};
#pragma unroll
      for (int q = 0; q < 8; ++q) bias[q].add(e[q]);
    }
  }
}

template <bool HALO_DY, int CB>
__global__ void __launch_bounds__(kWgThreads, 1) k_wgrad_tc(const __grid_constant__ WgradGrid g, const bf16* __restrict__ X,
                                                          const float* __restrict__ dY, float* __restrict__ part,
                                                          double* __restrict__ bpart, int* __restrict__ odd,
                                                          const TcWait lim) {
  constexpr int KC = CB / 8;          // chunks of the core tensor (the halo tensor has 4)
  constexpr int kPair = CB == 32 ? 7 : 9;  // accumulators that take two core rows per MMA
  constexpr int CY = HALO_DY ? 32 : CB;    // channels of dY
  extern __shared__ uint8_t smraw[];
  uint8_t* sm = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smraw) + 127) & ~uintptr_t(127));
  const uint32_t bars = smem_u32(sm + kWgOffBar);
  auto hfull = [&](int p) { return bars + 8 * p; };
  auto hempty = [&](int p) { return bars + 8 * (kWgHalo + p); };
  auto cfull = [&](int p) { return bars + 8 * (2 * kWgHalo + p); };
  auto cempty = [&](int p) { return bars + 8 * (2 * kWgHalo + kWgCore + p); };
  const uint32_t alldone = bars + 8 * (2 * kWgHalo + 2 * kWgCore);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(sm + kWgOffBar + 8 * (2 * kWgHalo + 2 * kWgCore + 1));
  volatile int* sfail = reinterpret_cast<volatile int*>(tslot + 1);
  volatile uint32_t* sstarted = reinterpret_cast<volatile uint32_t*>(tslot + 2);  // accumulators with a sum in them
  double* sbias = reinterpret_cast<double*>(sm + kWgOffBias);  // [producer][8]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int p = 0; p < kWgHalo; ++p) {
      mbar_init(hfull(p), kWgProd / 32);  // (an arrival per warp)
      mbar_init(hempty(p), 1);
    }
    for (int p = 0; p < kWgCore; ++p) {
      mbar_init(cfull(p), kWgProd / 32);
      mbar_init(cempty(p), 1);
    }
    mbar_init(alldone, 1);
    *sfail = 0;
    *sstarted = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(smem_u32(tslot)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tslot;
  const int TX = g.tx, hrow = wg_halo_row(TX), crow = wg_core_row(TX, KC);
  const uint32_t hbase = smem_u32(sm + kWgOffPlanes), hplane = (uint32_t)wg_halo_plane(TX);
  const uint32_t cbase = hbase + kWgHalo * hplane, cplane = (uint32_t)wg_core_plane(TX, KC);
  const int64_t t0 = g.tiles * blockIdx.x / gridDim.x, t1 = g.tiles * (blockIdx.x + 1) / gridDim.x;
  const int64_t V = (int64_t)g.nx * g.ny * g.nz;
  // a warp's stores to shared memory are visible to the MMAs: one arrival
  auto arrive = [&](uint32_t bar) {
    fence_async_proxy();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar);
  };
  Sum3 bias[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) bias[q] = Sum3{0.f, 0.f, 0.f};
  bool ok = true;
  March m(g, t0);
  if (warp >= 1 + kWgProd / 32) {
    // ---- core planes
    const int pt = tid - 32 - kWgProd;
    for (int64_t t = t0; t < t1 && ok; ++t, m.next(g)) {
      const int k = (int)(t - t0);
      const size_t zb = (size_t)m.b * V + (size_t)m.z * g.nx * g.ny;
      const uint32_t dst = cbase + (uint32_t)(k % kWgCore) * cplane;
      auto wait = [&]() { return k < kWgCore || mbar_wait(cempty(k % kWgCore), (k / kWgCore - 1) & 1, sfail); };
      if constexpr (HALO_DY) {
        ok = __all_sync(0xffffffffu, wait());
        if (!ok) break;
        wg_plane_bf16<KC, kWgTY>(X, zb, g.nx, g.ny, m.tx * TX, m.ty * kWgTY, TX, dst, crow, pt);
        cp_commit();
        wg_bias_f32(dY, zb, g.nx, g.ny, m.tx * TX, m.ty * kWgTY, TX, pt, bias);
        cp_wait<0>();
      } else {
        ok = wg_plane_f32<KC, kWgTY, true>(dY, zb, g.nx, g.ny, m.tx * TX, m.ty * kWgTY, TX, dst, crow, pt, bias, wait);
        if (!ok) break;
      }
      arrive(cfull(k % kWgCore));
    }
  } else if (warp >= 1) {
    // ---- halo planes
    const int pt = tid - 32;
    int seq = 0, done = 0;
    for (int64_t t = t0; t < t1 && ok; ++t, m.next(g)) {
      const int z = m.z, x0 = m.tx * TX - 1, y0 = m.ty * kWgTY - 1;
      const bool start = t == t0 || z == 0;
      for (int pz = start ? max(z - 1, 0) : z + 1; pz <= min(z + 1, g.nz - 1) && ok; ++pz) {
        const size_t zb = (size_t)m.b * V + (size_t)pz * g.nx * g.ny;
        const uint32_t dst = hbase + (uint32_t)(seq % kWgHalo) * hplane;
        auto wait = [&]() { return seq < kWgHalo || mbar_wait(hempty(seq % kWgHalo), (seq / kWgHalo - 1) & 1, sfail); };
        if constexpr (HALO_DY) {
          ok = wg_plane_f32<4, kWgHY, false>(dY, zb, g.nx, g.ny, x0, y0, TX + 2, dst, hrow, pt, bias, wait);
          if (!ok) break;
          arrive(hfull(seq % kWgHalo));
          ++seq;
        } else {
          ok = __all_sync(0xffffffffu, wait());
          if (!ok) break;
          wg_plane_bf16<4, kWgHY>(X, zb, g.nx, g.ny, x0, y0, TX + 2, dst, hrow, pt);
          cp_commit();
          ++seq;
          cp_wait<1>();
          for (; done < seq - 1; ++done) arrive(hfull(done % kWgHalo));
        }
      }
    }
    cp_wait<0>();
    if constexpr (!HALO_DY) {
      if (ok)
        for (; done < seq; ++done) arrive(hfull(done % kWgHalo));
    }
  } else if (t0 < t1) {
    // ---- MMA issue (the whole warp waits, one thread issues)
    uint32_t started = 0;
    int waited = 0, next = 0;
    const int64_t ts = min(t1, t0 + lim.tiles);
    for (int64_t t = t0; t < ts && ok; ++t, m.next(g)) {
      const int k = (int)(t - t0), z = m.z;
      const bool start = t == t0 || z == 0, end = t + 1 == t1 || z == g.nz - 1;
      if (start) next = waited + (z > 0 ? 1 : 0);
      const int need = next + (z < g.nz - 1 ? 1 : 0);
      for (; waited <= need && ok; ++waited)
        ok = __all_sync(0xffffffffu, mbar_wait(hfull(waited % kWgHalo), (waited / kWgHalo) & 1, sfail));
      ok = ok && __all_sync(0xffffffffu, mbar_wait(cfull(k % kWgCore), (k / kWgCore) & 1, sfail));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      if (elect_one()) {
        const uint64_t db0 = smem_desc(cbase + (uint32_t)(k % kWgCore) * cplane, 128, (uint32_t)crow);
#pragma unroll
        for (int dz = 0; dz < 3; ++dz) {
          if (z + dz - 1 < 0 || z + dz - 1 >= g.nz) continue;
          const uint64_t da0 = smem_desc(hbase + (uint32_t)((next + dz - 1) % kWgHalo) * hplane, 128, (uint32_t)hrow);
          bool acc = (started >> (3 * dz)) & 1u;
          for (int kx = 0; kx < TX; kx += 16)
#pragma unroll
            for (int yp = 0; yp < kWgTY; yp += 2) {
              const uint64_t da = da0 + (uint64_t)((yp * 4 * hrow + kx * 16) >> 4);
              const uint64_t db = db0 + (uint64_t)((yp * KC * crow + kx * 16) >> 4);
#pragma unroll
              for (int sx = 0; sx < 3; ++sx) {
                const int i = 3 * dz + sx;
                if (i < kPair) {
                  umma(tmem + (uint32_t)(2 * CB * i), da + (uint64_t)sx, db, idesc(2 * CB, true, true), acc);
                } else {
                  const uint32_t d = tmem + (uint32_t)(2 * CB * kPair + CB * (i - kPair));
                  umma(d, da + (uint64_t)sx, db, idesc(CB, true, true), acc);
                  umma(d, da + (uint64_t)sx + (uint64_t)((4 * hrow) >> 4), db + (uint64_t)((KC * crow) >> 4), idesc(CB, true, true),
                       true);
                }
              }
              acc = true;
            }
        }
        umma_commit(cempty(k % kWgCore));
        if (z > 0) umma_commit(hempty((next - 1) % kWgHalo));
        if (end) {
          umma_commit(hempty(next % kWgHalo));
          if (z < g.nz - 1) umma_commit(hempty((next + 1) % kWgHalo));
        }
      }
      __syncwarp();
      started |= (z > 0 ? 7u : 0u) | 7u << 3 | (z < g.nz - 1 ? 7u << 6 : 0u);
      ++next;
    }
    *sstarted = started;
    if (elect_one()) umma_commit(alldone);
    __syncwarp();
    if (!mbar_wait(alldone, 0) || ts < t1) ok = false;  // every MMA is done before the buffers are used again
  }
  if (!ok) report_timeout(sfail, lim);
  if (warp >= 1 + kWgProd / 32) {
    const int pt = tid - 32 - kWgProd;
#pragma unroll
    for (int q = 0; q < 8; ++q) sbias[pt * 8 + q] = bias[q].value();
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  // ---- sums out: accumulator i, halo row a (lane quarter), core row r holds
  // tap (dz, a - r, sx) of halo channel `lane`; after an expired wait NaN
  float* red = reinterpret_cast<float*>(sm + kWgOffPlanes);
  const uint32_t started = *sstarted;
  const bool fine = !*sfail;
  for (int r = 0; r < 2; ++r) {
    if (warp >= 1) {
      const int a = warp & 3, part2 = (warp - 1) >> 2;  // the warps of a quarter share the accumulators
      for (int i = part2; i < 9; i += kWgProd / 64) {
        const bool pair = i < kPair;
        if (!pair && r == 1) continue;
        const int dy = pair ? a - r : a;
        if (dy < 0 || dy > 2) continue;  // (warp-uniform)
        const uint32_t col = pair ? (uint32_t)(2 * CB * i + CB * r) : (uint32_t)(2 * CB * kPair + CB * (i - kPair));
        const int t = 9 * (i / 3) + 3 * dy + i % 3;
        const int tap = HALO_DY ? 26 - t : t;
        const bool have = (started >> i) & 1u;
        const float none = fine ? 0.f : __int_as_float(0x7fffffff);
#pragma unroll
        for (int c0 = 0; c0 < CB; c0 += 16) {
          uint32_t v[16];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
              "tcgen05.wait::ld.sync.aligned;\n"
              : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
                "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
              : "r"(tmem + ((uint32_t)(a * 32) << 16) + col + (uint32_t)c0)
              : "memory");
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const int o = HALO_DY ? (tap * 32 + lane) * CB + c0 + e : (tap * CB + c0 + e) * 32 + lane;
            const float f = have && fine ? __uint_as_float(v[e]) : none;
            red[o] = r == 0 ? f : red[o] + f;
          }
        }
      }
    }
    __syncthreads();
  }
  const int n = 27 * 32 * CB;
  float* P = part + (size_t)blockIdx.x * n;
  for (int i = tid; i < n / 4; i += kWgThreads) reinterpret_cast<float4*>(P)[i] = reinterpret_cast<const float4*>(red)[i];
  double sum = 0.0;
  if (tid < CY) {
    constexpr int YC = CY / 8;
    for (int p = tid / 8; p < kWgProd; p += YC) sum += sbias[p * 8 + tid % 8];
    if (!fine) sum = (double)__int_as_float(0x7fffffff);
    bpart[(size_t)blockIdx.x * CY + tid] = sum;
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  const int infinite = __syncthreads_or(!isfinite(sum));
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  if (tid == 0) odd[blockIdx.x] = !fine ? 2 : infinite ? 1 : 0;
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;\n" ::"r"(tmem));
}

// Weight i or (bias) channel i of the gradient straight from its definition, the
// voxels whose neighbour lies outside the grid with x = 0 as well: the part of
// slice w of the block's eight, 32 consecutive i side by side.
__device__ __noinline__ double wgrad_direct(const WgradGrid& g, const bf16* X, const float* dY, int cin, int cout, int i,
                                            bool bias, int w) {
  const int64_t rows = (int64_t)g.B * g.nz * g.ny;
  if (bias) {
    double s = 0.0;
    for (int64_t v = w; v < rows * g.nx && !isnan(s); v += 8 * 16) {
      float e[16];
#pragma unroll
      for (int u = 0; u < 16; ++u) e[u] = v + 8 * u < rows * g.nx ? dY[(v + 8 * u) * cout + i] : 0.f;
#pragma unroll
      for (int u = 0; u < 16; ++u) s += e[u];
    }
    return s;
  }
  const int t = i / (cin * cout), co = i / cin % cout, ci = i % cin;
  const int dx = t % 3 - 1, dy = t / 3 % 3 - 1, dz = t / 9 - 1;
  Sum3 s{0.f, 0.f, 0.f};
  for (int64_t r = w; r < rows; r += 8) {
    const int y = (int)(r % g.ny), z = (int)(r / g.ny % g.nz);
    const bool row = y + dy >= 0 && y + dy < g.ny && z + dz >= 0 && z + dz < g.nz;
    const float* D = dY + r * g.nx * cout + co;
    const bf16* N = X + ((r + dy + (int64_t)dz * g.ny) * g.nx + dx) * cin + ci;
    for (int x = 0; x < g.nx; ++x) {
      const float d = __bfloat162float(__float2bfloat16_rn(D[(int64_t)x * cout]));
      const bool in = row && x + dx >= 0 && x + dx < g.nx;
      s.add(d * (in ? __bfloat162float(N[(int64_t)x * cin]) : 0.f));
    }
    if (__all_sync(0xffffffffu, isnan(s.a))) break;
  }
  return s.value();
}

// dW[i] = sum over the chunks' partials in a fixed order, in three FP32 parts
// (4.2 million FP64 additions took 14 of the 20 us of the form that made them);
// 32 outputs by 8 slices of the chunks per block.  The last block
// takes the bias gradient.  odd[chunk]: 1 where one of its bias sums is not
// finite, 2 where it gave up a wait.
// Infinite values: a tile's voxels beyond the grid are zeros, and their
// products with an infinite neighbour that lies in it NaN; conversely planes
// beyond the grid are left out, and the zeros that an infinite dY meets there.
// So a sum that came out as NaN, and all of a channel whose bias is not finite,
// are taken again from the definition (at 64x64x32 x 4, 32 -> 32, 0 to 11 ms,
// the more the later the NaN that ends a sum; finite values: 9.8 -> 10.9 us for
// looking).  Six blocks per SM: the 865 of 32 x 32 channels in one wave.
__global__ void __launch_bounds__(256, 6) k_wgrad_sum(const float* __restrict__ part, const double* __restrict__ bpart,
                                                   const int* __restrict__ odd, const __grid_constant__ WgradGrid g, const bf16* __restrict__ X,
                                                   const float* __restrict__ dY, float* __restrict__ dW,
                                                   float* __restrict__ db, int cin, int cout, int chunks) {
  __shared__ double sh[8][32];
  const int l = threadIdx.x & 31, w = threadIdx.x >> 5, n = 27 * cin * cout;
  const bool last = blockIdx.x == gridDim.x - 1;
  const int i = last ? l : (int)blockIdx.x * 32 + l;  // (n is a multiple of 32)
  double s = 0.0;
  int flag = 0;  // (chunks <= 304)
  if (threadIdx.x < chunks) flag = odd[threadIdx.x];
  if (threadIdx.x + 256 < chunks) flag = max(flag, odd[threadIdx.x + 256]);
  if (last) {
    if (l < cout)
      for (int k = w; k < chunks; k += 8) s += bpart[(size_t)k * cout + l];
  } else {
    const float* p = part + i;
    Sum3 a{0.f, 0.f, 0.f};
    for (int k0 = w; k0 < chunks; k0 += 80) {
      float v[10];
#pragma unroll
      for (int u = 0; u < 10; ++u) v[u] = k0 + 8 * u < chunks ? p[(size_t)(k0 + 8 * u) * n] : 0.f;
#pragma unroll
      for (int u = 0; u < 10; ++u) a.add(v[u]);
    }
    s = a.value();
    if (!isfinite(a.a)) {  // (beyond FP32's range on the way, maybe)
      s = 0.0;
      for (int k = w; k < chunks; k += 8) s += p[(size_t)k * n];
    }
  }
  auto total = [&]() {
    sh[w][l] = s;
    __syncthreads();
    double t = 0.0;
    if (w == 0)  // (FP64 additions are few a clock: one warp's)
      for (int k = 0; k < 8; ++k) t += sh[k][l];
    return t;
  };
  double t = total();
  bool again = last ? l < cout && !isfinite(t) : isnan(t);
  if (__syncthreads_or(again || flag)) {
    if (!last) {  // the block's output channels, 32 / cin from c0 on
      const int per = 32 / cin, c0 = (int)blockIdx.x * per % cout;
      for (int k = threadIdx.x; k < chunks * per; k += 256)
        again = again || !isfinite(bpart[(size_t)(k / per) * cout + c0 + k % per]);
    }
    if (__syncthreads_or(again) && !__syncthreads_or(flag > 1)) {
      s = i < (last ? cout : n) ? wgrad_direct(g, X, dY, cin, cout, i, last, w) : 0.0;
      t = total();
    }
  }
  if (w == 0 && i < (last ? cout : n)) (last ? db : dW)[i] = (float)t;
}

}  // namespace

int wgrad_tc_blocks() { return std::min(sm_count(), kWgradTcBlocks); }

namespace {

template <bool HALO_DY, int CB>
int run_wgrad(const WgradGrid& g, const bf16* X, const float* dY, float* part, double* bpart, float* dW, float* db,
              const TcWait& lim, cudaStream_t s) {
  auto kern = k_wgrad_tc<HALO_DY, CB>;
  const int planes = kWgHalo * wg_halo_plane(g.tx) + kWgCore * wg_core_plane(g.tx, CB / 8);
  const int red = 27 * 32 * CB * 4;
  const int smem = kWgOffPlanes + (planes > red ? planes : red) + 128;
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return BO_ERR_CUDA;
  const int blocks = wgrad_tc_blocks();
  const int grid = g.tiles < blocks ? (int)g.tiles : blocks;
  int* odd = reinterpret_cast<int*>(bpart + grid * (HALO_DY ? 32 : CB));
  (kern<<<grid, kWgThreads, smem, s>>>(g, X, dY, part, bpart, odd, lim), note_launch());
  (k_wgrad_sum<<<27 * CB + 1, 256, 0, s>>>(part, bpart, odd, g, X, dY, dW, db, HALO_DY ? CB : 32, HALO_DY ? 32 : CB, grid),
   note_launch());
  return cudaGetLastError() == cudaSuccess ? BO_OK : BO_ERR_CUDA;
}

}  // namespace

bool wgrad_tc_applies(const __nv_bfloat16* X, const float* dY) {
  return !(reinterpret_cast<uintptr_t>(X) & 15) && !(reinterpret_cast<uintptr_t>(dY) & 15);
}

int launch_wgrad_tc(int cin, int cout, int nx, int ny, int nz, int B, const __nv_bfloat16* X, const float* dY, float* part,
                    double* bpart, float* dW, float* db, const TcWait& lim, cudaStream_t s) {
  if (!wgrad_tc_applies(X, dY)) return BO_ERR_ARG;
  WgradGrid g{nx, ny, nz, B, 0, 0, 0, 0};
  int best = 0;
  for (int tx : {64, 32, 16}) {  // the fewest padded voxels along x; of equals the longest run
    const int w = (nx + tx - 1) / tx * tx;
    if (!best || w < best) {
      best = w;
      g.tx = tx;
    }
  }
  g.ntx = (nx + g.tx - 1) / g.tx;
  g.nty = (ny + kWgTY - 1) / kWgTY;
  if ((int64_t)g.ntx * g.nty * B > INT32_MAX) return BO_ERR_ARG;
  g.tiles = (int64_t)g.ntx * g.nty * B * nz;
  if (cin == 32 && cout == 32) return run_wgrad<false, 32>(g, X, dY, part, bpart, dW, db, lim, s);
  if (cin == 32 && cout == 16) return run_wgrad<false, 16>(g, X, dY, part, bpart, dW, db, lim, s);
  if (cin == 16 && cout == 32) return run_wgrad<true, 16>(g, X, dY, part, bpart, dW, db, lim, s);
  return BO_ERR_ARG;
}

}  // namespace bo

extern "C" int bo_tc_status(void) {
  int h = 0;
  if (cudaMemcpyFromSymbol(&h, bo::g_tc_err, sizeof(int)) != cudaSuccess) return BO_ERR_CUDA;
  if (h) {
    const int z = 0;
    cudaMemcpyToSymbol(bo::g_tc_err, &z, sizeof(int));
    return BO_ERR_TIMEOUT;
  }
  return BO_OK;
}
