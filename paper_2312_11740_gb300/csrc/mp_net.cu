// Learned warm start: BF16 implicit-GEMM 3x3x3 convolutions on the 5th-generation
// tensor cores (tcgen05.mma, operands in shared memory, FP32 accumulator in
// tensor memory), and the U-Net built from them.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/mp_net.h"

namespace mpnet {

using bf16 = __nv_bfloat16;

// ------------------------------------------------------------- tcgen05 helpers
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
// Shared-memory matrix descriptor, no swizzle: start address, leading- and
// stride-dimension byte offsets (all >> 4), descriptor version 1.
__device__ __forceinline__ uint64_t sdesc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | ((uint64_t)1 << 46);
}
// Instruction descriptor, kind::f16: FP32 accumulator, BF16 A and B,
// majorness of A/B (0 = K-major), N >> 3, M >> 4.
__host__ __device__ constexpr uint32_t idesc_bf16(int m, int n, int amaj, int bmaj) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)amaj << 15) | ((uint32_t)bmaj << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t da, uint64_t db, uint32_t id,
                                         uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem),
      "l"(da), "l"(db), "r"(id), "r"(acc));
}
__device__ __forceinline__ void mma_commit(uint64_t *mbar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(mbar)));
}
__device__ __forceinline__ void mbar_init(uint64_t *mbar) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(mbar)));
}
// Bounded wait for the phase of the given parity to complete; false on timeout.
__device__ __forceinline__ bool mbar_wait(uint64_t *mbar, uint32_t parity) {
  uint32_t done = 0;
  for (long it = 0; it < (1L << 24) && !done; ++it) {
    asm volatile(
        "{\n\t.reg .pred P;\n\tmbarrier.try_wait.parity.shared::cta.b64 P, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, P;\n\t}\n"
        : "=r"(done)
        : "r"(smem_u32(mbar)), "r"(parity));
  }
  return done != 0;
}
__device__ __forceinline__ void tmem_alloc(uint32_t *slot, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(slot)),
               "r"(ncols));
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
}
__device__ __forceinline__ void tmem_free(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols));
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float *out) {
  uint32_t v[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
  for (int q = 0; q < 16; ++q) out[q] = __uint_as_float(v[q]);
}
__device__ __forceinline__ void fence_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// ------------------------------------------------------------ convolutions
// Geometry of one 3x3x3 convolution whose input is the channel concatenation
// of xa (optionally at half resolution, read through nearest upsampling)
// and xb.  Smem operand tiles use the no-swizzle K-major core-matrix layout:
// a core matrix is 8 rows x 16 bytes (8 BF16 of K) stored contiguously.
struct ConvGeom {
  int nx, ny, nz;   // output (and full-resolution input) grid
  int ca, cb;       // channels of the two inputs (cb = 0: single input)
  int up_a;         // 1: input a is stored at half resolution
  int cin;          // ca + cb (multiple of 16)
};

constexpr int CONV_THREADS = 128;
constexpr int NSTAGE = 3;
constexpr int STAGE_K = 64;                  // K elements per stage (4 MMAs of K = 16)
// bytes of one row group (8 rows x STAGE_K voxels) of a weight-gradient stage: 64 more
// than its data, so that the two groups a warp writes at once lie in other banks
constexpr int WG_GROUP = STAGE_K * 16 + 64;
constexpr int A_STAGE_BYTES = 16 * WG_GROUP;

// tcgen05.alloc takes a power-of-two column count of at least 32
template <int COUT>
__host__ __device__ constexpr int tmem_cols() {
  return COUT <= 32 ? 32 : (COUT <= 64 ? 64 : (COUT <= 128 ? 128 : 256));
}
template <int COUT>
__host__ __device__ constexpr int b_stage_bytes() {
  return COUT / 8 * WG_GROUP;
}
template <int COUT>
__host__ __device__ constexpr int conv_smem_bytes() {
  return NSTAGE * (A_STAGE_BYTES + b_stage_bytes<COUT>()) + 1024;
}

// ------------------------------------------------ conv forward, halo-tiled
// CTA tile: 8 (x) x 16 (y) x HT_Z (z) output voxels and NC output channels,
// one M = 128 accumulator per z-plane (row r = voxel (r % 8, r / 8) of the
// plane).  For each 16-channel chunk of the input the tile's halo
// (10 x 18 x (HT_Z + 2) voxels) is staged ONCE in shared memory, as two
// 8-channel planes laid out [z][y][x][8 ch] (the box order of a 4D TMA
// load, whose out-of-range fill supplies the zero padding).  An MMA's A
// descriptor starts at a shifted voxel of one input plane: a core matrix
// (8 rows x 16 bytes) is 8 x-consecutive voxels, the next core matrix along
// M is the next y row (stride 10 x 16 bytes), the next along K the other
// 8-channel plane.  For an in-plane tap (dy, dx) the shifted input plane zi
// contributes to output planes zi + 1, zi, zi - 1 through the z-taps -1, 0,
// +1, and those planes' accumulators are adjacent in TMEM: one MMA with the
// three z-taps' weights side by side along N (up to 3 NC) covers them, so the
// 27 taps take 6 MMAs per tap pair instead of 3 x HT_Z, and each A tile is
// read from shared memory once instead of three times (at NC = 16 the A
// reads bound the kernel).  The weights of the chunk arrive as one bulk
// copy of a pre-packed image [dy dx][k/8][z-tap][co/8][co%8][8].
// A persistent CTA walks its tiles chunk by chunk through an NS-deep ring of
// stages (TMA -> mbarrier -> MMA issued by one thread -> commit -> refill),
// with two TMEM accumulator sets so that the epilogue of one tile overlaps
// the MMAs of the next.  Inputs read through nearest upsampling (the
// decoder's up + concat) are gathered by all threads instead of the TMA.
constexpr int HT_Z = 4;
constexpr int HX = 10, HY = 18, HZ = HT_Z + 2;
constexpr int HVOX = HX * HY * HZ;      // halo voxels per tile
constexpr int HPLANE = HVOX * 16;       // bytes of one 8-channel halo plane
constexpr int HALO_BYTES = 2 * HPLANE;  // a 16-channel chunk

template <int NC>
__host__ __device__ constexpr int himg_bytes() {
  return 27 * NC * 32;  // weights of one 16-channel chunk for NC outputs
}
template <int NC>
__host__ __device__ constexpr int h_nstage() {
  return NC == 32 ? 3 : 2;
}
template <int NC>
__host__ __device__ constexpr int h_stage_bytes() {
  return HALO_BYTES + himg_bytes<NC>();
}
template <int NC>
__host__ __device__ constexpr int h_smem_bytes() {
  return h_nstage<NC>() * h_stage_bytes<NC>() + 1024;
}
template <int NC>
__host__ __device__ constexpr int h_tmem_cols() {
  return 2 * HT_Z * NC <= 128 ? 128 : (2 * HT_Z * NC <= 256 ? 256 : 512);
}
template <int NC>
__host__ __device__ constexpr int h_ctas_per_sm() {
  return NC == 16 ? 2 : 1;
}

struct HaloArgs {
  const bf16 *xa;       // first input (read by threads when upsampled)
  const bf16 *wimg;     // packed weights [nsplit][nchunk][27][2][NC/8][8][8]
  const float *bias;    // cout or NULL
  bf16 *y;              // output (BF16) ...
  float *y32;           // ... or FP32 when not NULL
  int nx, ny, nz;       // output grid
  int ca, up_a, cout, relu;
  int tiles_x, tiles_y, ntiles, nsplit, nchunk;
  int fail_first;  // test: treat the first stage wait as timed out (before any MMA)
  int *err;
};

__device__ __forceinline__ void cp_async16(void *smem, const void *gmem) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(smem)), "l"(gmem)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(mbar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void tma_load_4d(void *dst, const CUtensorMap *map, int c0, int c1,
                                            int c2, int c3, uint64_t *mbar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], "
      "[%1, {%2, %3, %4, %5}], [%6];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
      "r"(smem_u32(mbar))
      : "memory");
}
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes,
                                          uint64_t *mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(mbar))
      : "memory");
}

// Threads of a CTA: one issues the TMA loads and the MMAs; all gather upsampled inputs and run
// the epilogue (a warp reads the 32 TMEM lanes of its index mod 4; the two
// halves of the CTA take two output planes each).  256 against 128, with the halo's
// coordinates from a table: 64 + 32 -> 32 at 64^3, first part upsampled, 91 us (107);
// 16 -> 16 at 128^3 unchanged, ~128 cycles an MMA (operand fetch) bound both.
constexpr int HALO_THREADS = 256;
template <int NC>
__global__ void __launch_bounds__(HALO_THREADS, h_ctas_per_sm<NC>())
k_conv3d_halo(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
              const HaloArgs a) {
  constexpr int NS = h_nstage<NC>();
  constexpr int SB = h_stage_bytes<NC>();
  constexpr int WB = himg_bytes<NC>();
  constexpr int TM = h_tmem_cols<NC>();
  constexpr uint32_t IDESC = idesc_bf16(128, NC, 0, 0);
  constexpr uint32_t IDESC2 = idesc_bf16(128, 2 * NC, 0, 0);
  constexpr uint32_t IDESC3 = idesc_bf16(128, 3 * NC, 0, 0);
  static_assert(3 * NC <= 256 && NC % 16 == 0, "N of the folded z-taps: a multiple of 16, <= 256");
  static_assert(HT_Z == 4, "the folded z-tap sequence is written for four output planes");
  extern __shared__ __align__(1024) uint8_t hsm_raw[];
  uint8_t *sm = hsm_raw + ((1024 - (smem_u32(hsm_raw) & 1023)) & 1023);
  __shared__ __align__(8) uint64_t full[NS], done[NS];
  __shared__ uint32_t tslot;
  __shared__ int abort_flag;
  // upsampled inputs: per halo voxel its coordinates in the halo (8 bits each) and its
  // parent's offset from the parent of the tile's origin (tile origins are even)
  __shared__ int2 htab[HVOX];

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (a.up_a)
    for (int v = tid; v < HVOX; v += HALO_THREADS) {
      const int hx = v % HX, hy = (v / HX) % HY, hz = v / (HX * HY);
      htab[v] = make_int2(hx | hy << 8 | hz << 16,
                          (((hz - 1) >> 1) * (a.ny >> 1) + ((hy - 1) >> 1)) * (a.nx >> 1) +
                              ((hx - 1) >> 1));
    }
  if (tid == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s]);
      mbar_init(&done[s]);
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    abort_flag = 0;
  }
  if (warp == 0) tmem_alloc(&tslot, TM);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t taddr = tslot;

  // the grid is a multiple of nsplit: a CTA keeps one output-channel slice
  const int split = blockIdx.x % a.nsplit;
  const int tile0 = blockIdx.x / a.nsplit, tstep = gridDim.x / a.nsplit;
  const int my_tiles = tile0 < a.ntiles ? (a.ntiles - 1 - tile0) / tstep + 1 : 0;
  const int nst = my_tiles * a.nchunk;
  // a stage's weights equal those NS stages earlier when NS % nchunk == 0
  const bool w_reuse = (NS % a.nchunk) == 0;
  const int anx = a.up_a ? a.nx >> 1 : a.nx, any = a.up_a ? a.ny >> 1 : a.ny;

  auto tile_origin = [&](int lt, int &x0, int &y0, int &z0) {
    const int tile = tile0 + lt * tstep;
    const int tx = tile % a.tiles_x, r = tile / a.tiles_x;
    x0 = tx * 8;
    y0 = (r % a.tiles_y) * 16;
    z0 = (r / a.tiles_y) * HT_Z;
  };

  // fill the stage buffer of stage s: TMA (thread 0) and upsampled gathers (all)
  auto produce = [&](int s) {
    const int buf = s % NS, lt = s / a.nchunk, c = s - lt * a.nchunk;
    int x0, y0, z0;
    tile_origin(lt, x0, y0, z0);
    uint8_t *st = sm + buf * SB;
    const bool wload = !(s >= NS && w_reuse);
    if (tid == 0) {
      uint32_t bytes = wload ? (uint32_t)WB : 0u;
      for (int g = 0; g < 2; ++g) {
        const int cc = 16 * c + 8 * g;
        if (!(a.up_a && cc < a.ca)) bytes += HPLANE;
      }
      mbar_expect_tx(&full[buf], bytes);
      for (int g = 0; g < 2; ++g) {
        const int cc = 16 * c + 8 * g;
        if (a.up_a && cc < a.ca) continue;
        if (cc < a.ca)
          tma_load_4d(st + g * HPLANE, &map_a, cc, x0 - 1, y0 - 1, z0 - 1, &full[buf]);
        else
          tma_load_4d(st + g * HPLANE, &map_b, cc - a.ca, x0 - 1, y0 - 1, z0 - 1, &full[buf]);
      }
      if (wload)
        bulk_load(st + HALO_BYTES,
                  a.wimg + ((size_t)split * a.nchunk + c) * (size_t)(WB / 2), (uint32_t)WB,
                  &full[buf]);
    }
    // inputs read through nearest upsampling: one 16-byte cp.async per halo
    // voxel from its parent voxel, zeros outside the grid; all threads, one
    // commit group per stage, complete before the stage's barrier
    for (int g = 0; g < 2; ++g) {
      const int cc = 16 * c + 8 * g;
      if (!(a.up_a && cc < a.ca)) continue;
      uint8_t *dst = st + g * HPLANE;
      const bf16 *src =
          a.xa + (((size_t)(z0 >> 1) * any + (y0 >> 1)) * anx + (x0 >> 1)) * a.ca + cc;
#pragma unroll 3
      for (int v = tid; v < HVOX; v += HALO_THREADS) {
        const int2 h = htab[v];
        const int gx = x0 - 1 + (h.x & 255), gy = y0 - 1 + (h.x >> 8 & 255), gz = z0 - 1 + (h.x >> 16);
        if ((unsigned)gx < (unsigned)a.nx && (unsigned)gy < (unsigned)a.ny &&
            (unsigned)gz < (unsigned)a.nz)
          cp_async16(dst + v * 16, src + (long)h.y * a.ca);
        else
          *reinterpret_cast<uint4 *>(dst + v * 16) = make_uint4(0, 0, 0, 0);
      }
    }
    cp_async_commit();
  };

  auto epilogue = [&](int lt) {
    int x0, y0, z0;
    tile_origin(lt, x0, y0, z0);
    tc_fence_after();
    const int r = (warp & 3) * 32 + lane;
    const int gx = x0 + (r & 7), gy = y0 + (r >> 3);
    const uint32_t acc = (uint32_t)((lt & 1) * HT_Z * NC);
    const int co0 = split * NC, zhalf = (warp >> 2) * (HT_Z / 2);
#pragma unroll 1
    for (int zp = zhalf; zp < zhalf + HT_Z / 2; ++zp) {
      const int gz = z0 + zp;
      const bool inside = gx < a.nx && gy < a.ny && gz < a.nz;
      const size_t vox = ((size_t)gz * a.ny + gy) * a.nx + gx;
#pragma unroll
      for (int c0 = 0; c0 < NC; c0 += 16) {
        float v[16];
        tmem_ld16(taddr + ((uint32_t)((warp & 3) * 32) << 16) + acc + zp * NC + c0, v);
        if (inside) {
#pragma unroll
          for (int q = 0; q < 16; ++q) {
            const float t = v[q] + (a.bias ? a.bias[co0 + c0 + q] : 0.f);
            v[q] = a.relu ? fmaxf(t, 0.f) : t;
          }
          if (a.y32) {
            float4 *o = reinterpret_cast<float4 *>(a.y32 + vox * a.cout + co0 + c0);
#pragma unroll
            for (int q = 0; q < 4; ++q)
              o[q] = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
          } else {
            __align__(16) bf16 hv[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) hv[q] = __float2bfloat16_rn(v[q]);
            uint4 *o = reinterpret_cast<uint4 *>(a.y + vox * a.cout + co0 + c0);
            o[0] = *reinterpret_cast<uint4 *>(&hv[0]);
            o[1] = *reinterpret_cast<uint4 *>(&hv[8]);
          }
        }
      }
    }
    tc_fence_before();
  };

  // one cp.async group per stage slot: NS - 1 in the prologue and one per
  // iteration (empty past the last stage), so that stage s's gathers are the
  // group NS - 2 behind the newest at the top of iteration s
  int produced = 0, waited_full = 0, committed = 0, waited_done = 0;
  // (a single-layer call launches this kernel while its weights are still being packed)
  asm volatile("griddepcontrol.wait;" ::: "memory");
  for (int p = 0; p < NS - 1; ++p) {
    if (produced < nst) {
      produce(produced);
      ++produced;
    } else {
      cp_async_commit();
    }
  }
  for (int s = 0; s < nst; ++s) {
    const int buf = s % NS;
    cp_async_wait<NS - 2>();  // this thread's gathers of stage s have landed ...
    fence_async_smem();       // ... and are visible to the tensor core's reads
    // one thread polls the barriers (255 pollers would load the shared-memory
    // pipe that feeds the tensor core); the others wait at the CTA barrier
    if (tid == 0) {
      if (!(s == 0 && a.fail_first) && mbar_wait(&full[buf], (uint32_t)((s / NS) & 1)))
        waited_full = s + 1;
      else
        abort_flag = 1;
    }
    __syncthreads();  // stage s landed and its gathers are visible; abort is seen by all
    if (abort_flag) break;
    const int lt = s / a.nchunk, c = s - lt * a.nchunk;
    if (tid == 0) {
      tc_fence_after();
      const uint32_t hbase = smem_u32(sm + buf * SB), wbase = hbase + HALO_BYTES;
      const uint32_t acc = taddr + (uint32_t)((lt & 1) * HT_Z * NC);
      // B of tap pair p: rows (b, co), b = 0, 1, 2 for dz = +1, 0, -1
      const uint64_t a0 = sdesc(hbase, HPLANE, HX * 16), b0 = sdesc(wbase, 3 * NC * 16, 128);
      constexpr uint64_t BLK = (uint64_t)(NC * 16) >> 4;  // one z-tap block of B
#pragma unroll 1
      for (int p = 0; p < 9; ++p) {
        const int dy = p / 3, dx = p % 3;
        const uint64_t db = b0 + (uint64_t)((p * 96 * NC) >> 4);
        // A of input plane zi (-1 .. HT_Z: the tile's planes and their halo)
        auto ad = [&](int zi) {
          return a0 + (uint64_t)(((((zi + 1) * HY + dy) * HX + dx) * 16) >> 4);
        };
        // input plane zi feeds output planes zi+1, zi, zi-1 (z-taps -1, 0,
        // +1), whose accumulators are adjacent: one MMA of N = NC per output
        // plane it reaches inside the tile.  Planes 1 and 4 come first: they
        // reach output planes 0-2 and 3, so on a tile's first taps they
        // overwrite every accumulator before the others add to them
        const uint32_t keep = (c > 0 || p > 0) ? 1u : 0u;
        mma_bf16(acc, ad(1), db, IDESC3, keep);
        mma_bf16(acc + 3 * NC, ad(4), db, IDESC, keep);
        mma_bf16(acc, ad(-1), db + 2 * BLK, IDESC, 1u);
        mma_bf16(acc, ad(0), db + BLK, IDESC2, 1u);
        mma_bf16(acc + NC, ad(2), db, IDESC3, 1u);
        mma_bf16(acc + 2 * NC, ad(3), db, IDESC2, 1u);
      }
      mma_commit(&done[buf]);
    }
    committed = s + 1;
    if (s >= 1) {
      // MMAs of stage s-1 are done: its buffer is free and, if it ended a
      // tile, that tile's accumulators are final
      if (tid == 0) {
        if (mbar_wait(&done[(s - 1) % NS], (uint32_t)(((s - 1) / NS) & 1)))
          waited_done = s;
        else
          abort_flag = 1;
      }
      __syncthreads();
    }
    // refill the buffer of stage s-1 (its MMAs are done) before the epilogue
    // of the tile stage s-1 ended, so the copies overlap the epilogue
    if (!abort_flag && produced < nst) {
      produce(produced);
      ++produced;
    } else {
      cp_async_commit();
    }
    if (s >= 1 && !abort_flag && (s - 1) % a.nchunk == a.nchunk - 1) epilogue((s - 1) / a.nchunk);
  }
  cp_async_wait<0>();  // no copy into shared memory outlives the CTA
  if (!abort_flag && nst > 0) {
    if (tid == 0) {
      if (mbar_wait(&done[(nst - 1) % NS], (uint32_t)(((nst - 1) / NS) & 1)))
        waited_done = nst;
      else
        abort_flag = 1;
    }
    __syncthreads();
    if (!abort_flag) epilogue(nst / a.nchunk - 1);
  }
  __syncthreads();
  if (abort_flag && tid == 0) {
    // drain (bounded): copies still in flight into shared memory, MMAs still reading it
    for (int s = waited_full; s < produced; ++s) mbar_wait(&full[s % NS], (uint32_t)((s / NS) & 1));
    for (int s = waited_done; s < committed; ++s) mbar_wait(&done[s % NS], (uint32_t)((s / NS) & 1));
    *(volatile int *)a.err = 1;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(taddr, TM);
}

// packed weight image of a convolution for k_conv3d_halo, the three z-taps
// of each in-plane tap pair p = 3 dy + dx side by side along N:
// img[sp][c][p][kg][b][co/8][co%8][ci%8] = W(co = sp*NC + co_l, t, ci = 16c + 8kg + ci%8)
// with t = 9 (2 - b) + p (block b holds dz = 1 - b) and W(co, t, ci) =
// src[co][t][ci] (src [cout][27][cin]) or, for the input gradient
// (flip != 0), W(co, t, ci) = src[ci][26 - t][co] (src [cin'][27][cout'] of the layer).
template <typename S>
__global__ void k_pack_img(const S *__restrict__ src, int cout, int cin, int flip, int nc,
                           bf16 *__restrict__ img) {
  const int nchunk = cin / 16;
  const size_t total = (size_t)cout * 27 * cin;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    size_t r = e;
    const int cil = (int)(r % 8);
    r /= 8;
    const int col = (int)(r % 8);
    r /= 8;
    const int cog = (int)(r % (nc / 8));
    r /= nc / 8;
    const int b = (int)(r % 3);
    r /= 3;
    const int kg = (int)(r % 2);
    r /= 2;
    const int p = (int)(r % 9);
    r /= 9;
    const int t = 9 * (2 - b) + p;
    const int c = (int)(r % nchunk);
    const int sp = (int)(r / nchunk);
    const int co = sp * nc + cog * 8 + col, ci = 16 * c + 8 * kg + cil;
    const float v = flip ? (float)src[((size_t)ci * 27 + (26 - t)) * cout + co]
                         : (float)src[((size_t)co * 27 + t) * cin + ci];
    img[e] = __float2bfloat16_rn(v);
  }
}


// --------------------------------------------------------- conv weight grad
// D[128 rows (t, ci)][COUT] = sum over a chunk of voxels v of
// X[v + off_t][ci] * G[v][co]: rows are (tap, input channel) pairs, K runs
// over voxels.  Each CTA reduces one chunk of WG_VOX voxels into FP32
// partials; k_wgrad_reduce sums the chunks in a fixed order (split-K,
// deterministic).
//
// Both operands are M/N-major: a core matrix is 8 voxels (K) x 8 channels (16
// bytes), so the 8 channels of a voxel go from global to shared memory as they
// lie, one 16-byte cp.async each (zero-filled outside the grid), [row group][voxel].
// Writing K-major tiles instead took eight 2-byte stores for each of these
// copies and bound the kernel: 32-32 at 64^3 422 us, now 84 (the copies' shared-
// memory wavefronts at 67 % of their rate).
constexpr int WG_VOX = 2048;  // voxels per CTA (32 stages of 64)

__device__ __forceinline__ void cp_async16_zfill(void *smem, const void *gmem, bool in) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(smem)), "l"(gmem),
               "r"(in ? 16 : 0)
               : "memory");
}

template <int COUT>
__global__ void __launch_bounds__(CONV_THREADS)
k_conv3d_wgrad(const bf16 *__restrict__ xa, const bf16 *__restrict__ xb,
               const bf16 *__restrict__ gr, ConvGeom g, float *__restrict__ partial,
               int *__restrict__ err) {
  constexpr int TM = tmem_cols<COUT>();
  constexpr int BST = b_stage_bytes<COUT>();
  constexpr int NG = 8;  // copies of A per thread and stage: one of each pair of row groups
  extern __shared__ __align__(1024) uint8_t conv_smem[];
  uint8_t *sm = conv_smem + ((1024 - (smem_u32(conv_smem) & 1023)) & 1023);
  uint8_t *sA = sm;
  uint8_t *sB = sm + NSTAGE * A_STAGE_BYTES;
  __shared__ __align__(8) uint64_t mbar[NSTAGE];
  __shared__ uint32_t tslot;
  __shared__ int abort_flag;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rows = 27 * g.cin, m0 = blockIdx.x * 128;
  const long nvox = (long)g.nx * g.ny * g.nz;
  const long v0 = (long)blockIdx.y * WG_VOX;
  if (tid == 0) {
    for (int s = 0; s < NSTAGE; ++s) mbar_init(&mbar[s]);
    asm volatile("fence.mbarrier_init.release.cluster;");
    abort_flag = 0;
  }
  if (warp == 0) tmem_alloc(&tslot, TM);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t taddr = tslot;
  constexpr uint32_t IDESC = idesc_bf16(128, COUT, 1, 1);

  // This thread's voxel of a stage is k; its row groups are 2 i + rg.  Two lanes
  // take the 16 channels of a pair of groups (always of one tap and input), so a
  // warp's copies read whole 32-byte sectors.  Per group: the source of this stage's
  // voxel and its advance to the next stage's, and the bits of `edge` that say the
  // tap lies inside the grid.  An upsampled input has no linear source: its
  // groups (step 0) form the parent's address instead.
  static_assert(CONV_THREADS == 2 * STAGE_K, "two threads per voxel of a stage");
  const int k = tid >> 1, rg = tid & 1;
  long v = v0 + k;  // the voxel of the next stage to produce, and its coordinates
  int x = (int)(v % g.nx), y = (int)(v / g.nx % g.ny), z = (int)(v / g.nx / g.ny);
  const bf16 *src[NG];
  int step[NG], need[NG], off[NG];
#pragma unroll
  for (int i = 0; i < NG; ++i) {
    const int m = m0 + (2 * i + rg) * 8, t = m / g.cin, ci = m - t * g.cin;
    const int dx = t % 3 - 1, dy = (t / 3) % 3 - 1, dz = t / 9 - 1;
    need[i] = m < rows ? 1 << (dx + 1) | 8 << (dy + 1) | 64 << (dz + 1) : 1 << 30;
    const bool b = ci >= g.ca;
    const int c = b ? g.cb : g.ca;
    step[i] = !b && g.up_a ? 0 : STAGE_K * c;
    off[i] = ci;
    src[i] = (b ? xb - g.ca : xa) + ci;
    if (step[i]) src[i] += (v + ((long)dz * g.ny + dy) * g.nx + dx) * c;
  }
  const int nst = WG_VOX / STAGE_K;
  auto produce = [&](int s) {
    const int buf = s % NSTAGE;
    const bool in = v < nvox;
    // bit 1 + dx, 4 + dy, 7 + dz: the neighbour of that offset is in range
    const int edge = !in ? 0
                         : (x > 0) | 2 | (x + 1 < g.nx) << 2 | (y > 0) << 3 | 16 |
                               (y + 1 < g.ny) << 5 | (z > 0) << 6 | 128 | (z + 1 < g.nz) << 8;
    uint8_t *a_st = sA + buf * A_STAGE_BYTES + rg * WG_GROUP + k * 16;
#pragma unroll
    for (int i = 0; i < NG; ++i) {
      const bool ok = (edge & need[i]) == need[i];
      const bf16 *p = src[i];
      if (g.up_a && step[i] == 0) {
        const int dx = (need[i] >> 2 & 1) - (need[i] & 1),
                  dy = (need[i] >> 5 & 1) - (need[i] >> 3 & 1),
                  dz = (need[i] >> 8 & 1) - (need[i] >> 6 & 1);
        p = xa + (((size_t)((z + dz) >> 1) * (g.ny >> 1) + ((y + dy) >> 1)) * (g.nx >> 1) +
                  ((x + dx) >> 1)) * g.ca + off[i];
      }
      cp_async16_zfill(a_st + 2 * i * WG_GROUP, ok ? p : xa, ok);
      src[i] += step[i];
    }
    uint8_t *b_st = sB + buf * BST + k * 16;
    const bf16 *pg = in ? gr + v * COUT : gr;
#pragma unroll
    for (int e = 0; e < COUT / 16; ++e)
      cp_async16_zfill(b_st + (2 * e + rg) * WG_GROUP, pg + (2 * e + rg) * 8, in);
    v += STAGE_K;
    x += STAGE_K;
    while (x >= g.nx) {
      x -= g.nx;
      if (++y == g.ny) y = 0, ++z;
    }
  };

  // one cp.async group per stage, NSTAGE - 1 ahead of the MMAs
  int issued = 0, waited = 0;
  for (int p = 0; p < NSTAGE - 1; ++p) {
    produce(p);
    cp_async_commit();
  }
  bool ok = true;
  for (int s = 0; s < nst; ++s) {
    const int buf = s % NSTAGE;
    cp_async_wait<NSTAGE - 2>();  // this thread's copies of stage s have landed ...
    fence_async_smem();           // ... and are visible to the tensor core's reads
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      const uint32_t a0 = smem_u32(sA + buf * A_STAGE_BYTES), b0 = smem_u32(sB + buf * BST);
#pragma unroll
      for (int q = 0; q < STAGE_K / 16; ++q) {
        // K groups of 8 voxels are 128 bytes apart, row groups WG_GROUP
        const uint64_t da = sdesc(a0 + q * 256, 128, WG_GROUP);
        const uint64_t db = sdesc(b0 + q * 256, 128, WG_GROUP);
        mma_bf16(taddr, da, db, IDESC, (s > 0 || q > 0) ? 1u : 0u);
      }
      mma_commit(&mbar[buf]);
    }
    issued = s + 1;
    if (s + NSTAGE - 1 < nst) {
      if (s >= 1) {  // the buffer of stage s - 1 is free once its MMAs are done
        if (tid == 0 && !mbar_wait(&mbar[(s - 1) % NSTAGE], (uint32_t)(((s - 1) / NSTAGE) & 1)))
          abort_flag = 1;
        __syncthreads();
        if (abort_flag) {
          ok = false;
          break;
        }
        waited = s;
      }
      produce(s + NSTAGE - 1);
    }
    cp_async_commit();
  }
  cp_async_wait<0>();  // no copy into shared memory outlives the CTA
  if (tid == 0) {      // every MMA issued is done (after a timeout: bounded, like any wait)
    for (int s = waited; s < issued; ++s)
      if (!mbar_wait(&mbar[s % NSTAGE], (uint32_t)((s / NSTAGE) & 1))) abort_flag = 1;
  }
  __syncthreads();
  tc_fence_after();
  if (abort_flag || !ok) {
    if (tid == 0) *(volatile int *)err = 1;
  } else {
    const int m = m0 + warp * 32 + lane;
    float4 *dst = reinterpret_cast<float4 *>(partial + ((size_t)blockIdx.y * rows + m) * COUT);
#pragma unroll
    for (int c0 = 0; c0 < COUT; c0 += 16) {
      float acc[16];
      tmem_ld16(taddr + ((uint32_t)(warp * 32) << 16) + c0, acc);
      if (m < rows) {
#pragma unroll
        for (int q = 0; q < 4; ++q)
          dst[c0 / 4 + q] = make_float4(acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
      }
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) tmem_free(taddr, TM);
}

// dw[co][t][ci] = sum over chunks (fixed order) of partial[chunk][t*cin + ci][co]: a warp
// reads 32 consecutive entries of one chunk, WR_SEG warps take a segment of the chunks
// each, and the segments' sums are added in order.  (One thread per output walking
// every chunk, outputs strided in memory: 24 us for 128 chunks of 864 x 32.)
constexpr int WR_SEG = 8;
__global__ void __launch_bounds__(32 * WR_SEG)
k_wgrad_reduce(const float *__restrict__ partial, int chunks, int rows, int cout,
               float *__restrict__ dw) {
  __shared__ float part[WR_SEG][32];
  const int lane = threadIdx.x & 31, seg = threadIdx.x >> 5;
  const int n = rows * cout, e = blockIdx.x * 32 + lane;
  const int c1 = (int)((long)(seg + 1) * chunks / WR_SEG);
  float acc = 0.f;
  if (e < n) {
#pragma unroll 8
    for (int c = (int)((long)seg * chunks / WR_SEG); c < c1; ++c) acc += partial[(size_t)c * n + e];
  }
  part[seg][lane] = acc;
  __syncthreads();
  if (seg == 0 && e < n) {
    float s = part[0][lane];
#pragma unroll
    for (int q = 1; q < WR_SEG; ++q) s += part[q][lane];
    dw[(size_t)(e % cout) * rows + e / cout] = s;
  }
}


// ------------------------------------------------------------ small kernels
constexpr int RED_BLOCKS = 1024, RED_THREADS = 256;

__device__ __forceinline__ float warp_sumf(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ double warp_sumd(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
// fixed-order block sum (result in thread 0); blockDim.x == RED_THREADS
__device__ __forceinline__ double block_sumd(double v) {
  __shared__ double red[RED_THREADS / 32];
  v = warp_sumd(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x < 32) {
    s = threadIdx.x < RED_THREADS / 32 ? red[threadIdx.x] : 0.0;
    s = warp_sumd(s);
  }
  return s;
}

// per-block partial sums of f(i) over a fixed grid; mode 0: x, 1: x^2
template <typename T>
__global__ void k_psum(const T *__restrict__ x, size_t n, int mode, double *__restrict__ part) {
  double acc = 0.0;
  for (size_t i = blockIdx.x * (size_t)RED_THREADS + threadIdx.x; i < n;
       i += (size_t)gridDim.x * RED_THREADS) {
    double v = (double)x[i];
    acc += mode ? v * v : v;
  }
  double t = block_sumd(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = t;
}
__global__ void k_pfinal(const double *__restrict__ part, int np, double *__restrict__ out) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < np; i += RED_THREADS) acc += part[i];
  double t = block_sumd(acc);
  if (threadIdx.x == 0) *out = t;
}

// network input: channel 0 = clip(phi / (4h), -1, 1), channel 1 = bt / s, rest 0
__global__ void k_features(const double *__restrict__ phi, const double *__restrict__ bt,
                           size_t n, double inv4h, double inv_s, bf16 *__restrict__ out) {
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < n;
       v += (size_t)gridDim.x * blockDim.x) {
    double f0 = phi[v] * inv4h;
    f0 = f0 > 1.0 ? 1.0 : (f0 < -1.0 ? -1.0 : f0);
    __align__(16) bf16 h[16];
    h[0] = __float2bfloat16_rn((float)f0);
    h[1] = __float2bfloat16_rn((float)(bt[v] * inv_s));
#pragma unroll
    for (int q = 2; q < 16; ++q) h[q] = __float2bfloat16_rn(0.f);
    uint4 *o = reinterpret_cast<uint4 *>(out + v * 16);
    o[0] = *reinterpret_cast<uint4 *>(&h[0]);
    o[1] = *reinterpret_cast<uint4 *>(&h[8]);
  }
}

// Fields of a grid twice as fine as the network's (nxc, nyc, nzc coarse
// cells): the mean of the 8 children of phi and of b, in FP64
__global__ void k_restrict_fields(const double *__restrict__ phi, const double *__restrict__ b,
                                  int nxc, int nyc, int nzc, double *__restrict__ phic,
                                  double *__restrict__ bc) {
  const size_t n = (size_t)nxc * nyc * nzc;
  const size_t fx = 2 * (size_t)nxc, fxy = 4 * (size_t)nxc * nyc;
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < n;
       v += (size_t)gridDim.x * blockDim.x) {
    const size_t I = v % nxc, J = (v / nxc) % nyc, K = v / ((size_t)nxc * nyc);
    const size_t f = 2 * K * fxy + 2 * J * fx + 2 * I;
    double sp = 0.0, sb = 0.0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const size_t e = f + (q & 1) + ((q >> 1) & 1) * fx + (q >> 2) * fxy;
      sp += phi[e];
      sb += b[e];
    }
    phic[v] = 0.125 * sp;
    bc[v] = 0.125 * sb;
  }
}

// qc = q - mean(q) on the network grid: centred in FP64, rounded once to FP32
__global__ void k_center_q(const float *__restrict__ q, const double *__restrict__ sum_q,
                           size_t nc, float *__restrict__ qc) {
  __shared__ double mean;
  if (threadIdx.x == 0) mean = *sum_q / (double)nc;
  __syncthreads();
  const double m = mean;
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < nc;
       v += (size_t)gridDim.x * blockDim.x)
    qc[v] = (float)((double)q[v] - m);
}

// coarse neighbours l0, l1 of fine cell c along one axis and the weight w1 of
// l1 (cell-centred: 3/4 for the nearer coarse cell, 1/4 for the farther one;
// periodic axes wrap, wall axes clamp)
__device__ __forceinline__ void tri_axis(int c, int nc, bool per, int &l0, int &l1, float &w1) {
  const int lo = (c - 1) >> 1;  // coarse cell below the fine centre
  w1 = (c & 1) ? 0.25f : 0.75f;
  l0 = lo;
  l1 = lo + 1;
  if (per) {
    l0 = l0 < 0 ? l0 + nc : l0;
    l1 = l1 >= nc ? l1 - nc : l1;
  } else {
    l0 = l0 < 0 ? 0 : l0;
    l1 = l1 > nc - 1 ? nc - 1 : l1;
  }
}

// p_fine = s * qc interpolated trilinearly from the network grid to the grid
// twice as fine.  The weights and their products are exact in FP32 and qc is
// already centred, so the separable FP32 interpolation loses only a few FP32
// ulps of the centred field; one FP64 multiply per fine cell.
__global__ void k_prolong_tri(const float *__restrict__ qc, int nxc, int nyc, int nzc, int per,
                              double s, double *__restrict__ p) {
  const int nx = 2 * nxc, ny = 2 * nyc, nz = 2 * nzc;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nx) return;
  int i0, i1;
  float wi1;
  tri_axis(i, nxc, per & 1, i0, i1, wi1);
  const float wi0 = 1.f - wi1;
  for (int k = blockIdx.z; k < nz; k += gridDim.z) {
    int k0, k1;
    float wk1;
    tri_axis(k, nzc, per & 4, k0, k1, wk1);
    for (int j = blockIdx.y; j < ny; j += gridDim.y) {
      int j0, j1;
      float wj1;
      tri_axis(j, nyc, per & 2, j0, j1, wj1);
      const float *r00 = qc + ((size_t)k0 * nyc + j0) * nxc;
      const float *r01 = qc + ((size_t)k0 * nyc + j1) * nxc;
      const float *r10 = qc + ((size_t)k1 * nyc + j0) * nxc;
      const float *r11 = qc + ((size_t)k1 * nyc + j1) * nxc;
      const float x00 = wi0 * r00[i0] + wi1 * r00[i1];
      const float x01 = wi0 * r01[i0] + wi1 * r01[i1];
      const float x10 = wi0 * r10[i0] + wi1 * r10[i1];
      const float x11 = wi0 * r11[i0] + wi1 * r11[i1];
      const float y0 = (1.f - wj1) * x00 + wj1 * x01;
      const float y1 = (1.f - wj1) * x10 + wj1 * x11;
      const float v = (1.f - wk1) * y0 + wk1 * y1;
      p[((size_t)k * ny + j) * nx + i] = s * (double)v;
    }
  }
}

// 2x2x2 average pooling (fine nx, ny, nz; C channels)
__global__ void k_pool2(const bf16 *__restrict__ in, bf16 *__restrict__ out, int nx, int ny, int nz,
                        int C) {
  const int cx = nx / 2, cy = ny / 2, cz = nz / 2;
  const size_t total = (size_t)cx * cy * cz * C;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % C);
    const size_t vc = e / C;
    const int X = (int)(vc % cx), Y = (int)((vc / cx) % cy), Z = (int)(vc / ((size_t)cx * cy));
    float acc = 0.f;
    for (int q = 0; q < 8; ++q) {
      const int x = 2 * X + (q & 1), y = 2 * Y + ((q >> 1) & 1), z = 2 * Z + (q >> 2);
      acc += __bfloat162float(in[(((size_t)z * ny + y) * nx + x) * C + c]);
    }
    out[e] = __float2bfloat16_rn(acc * 0.125f);
  }
}

// 1x1x1 head: q[v] = sum_c d[v][c] w[c] + b
__global__ void k_head_fwd(const bf16 *__restrict__ d, const float *__restrict__ w,
                           const float *__restrict__ b, size_t n, int C, float *__restrict__ q) {
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < n;
       v += (size_t)gridDim.x * blockDim.x) {
    float acc = b[0];
    for (int c = 0; c < C; ++c) acc = fmaf(__bfloat162float(d[v * C + c]), w[c], acc);
    q[v] = acc;
  }
}

// gradient through ReLU: gz = gy where y > 0
__global__ void k_relu_mask(const bf16 *__restrict__ gy, const bf16 *__restrict__ y, size_t n,
                            bf16 *__restrict__ gz) {
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < n;
       e += (size_t)gridDim.x * blockDim.x)
    gz[e] = __bfloat162float(y[e]) > 0.f ? gy[e] : __float2bfloat16_rn(0.f);
}

// per-channel partial sums of g (nvox x C) over voxel chunks, fixed order
__global__ void k_chan_psum(const bf16 *__restrict__ g, size_t nvox, int C, int chunk,
                            float *__restrict__ part) {
  const int c = threadIdx.x;  // blockDim.x == C
  const size_t v0 = (size_t)blockIdx.x * chunk;
  float acc = 0.f;
  for (size_t v = v0; v < v0 + chunk && v < nvox; ++v) acc += __bfloat162float(g[v * C + c]);
  part[(size_t)blockIdx.x * C + c] = acc;
}
__global__ void k_chan_final(const float *__restrict__ part, int chunks, int C,
                             float *__restrict__ out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= C) return;
  float acc = 0.f;
  for (int k = 0; k < chunks; ++k) acc += part[(size_t)k * C + c];
  out[c] = acc;
}

// head backward: gd[v][c] = gq[v] w[c]; partials of gq[v] d[v][c] (dw) and gq (db)
__global__ void k_head_bwd(const float *__restrict__ gq, const bf16 *__restrict__ d,
                           const float *__restrict__ w, size_t nvox, int C, int chunk,
                           bf16 *__restrict__ gd, float *__restrict__ part) {
  const int c = threadIdx.x;  // blockDim.x == C + 1 (last lane: bias)
  const size_t v0 = (size_t)blockIdx.x * chunk;
  float acc = 0.f;
  for (size_t v = v0; v < v0 + chunk && v < nvox; ++v) {
    const float g = gq[v];
    if (c < C) {
      gd[v * C + c] = __float2bfloat16_rn(g * w[c]);
      acc = fmaf(g, __bfloat162float(d[v * C + c]), acc);
    } else {
      acc += g;
    }
  }
  part[(size_t)blockIdx.x * (C + 1) + c] = acc;
}

// split the gradient of a concatenated input [up(a) (ca) | b (cb)] at full
// resolution: the a-part goes back through nearest upsampling (a parent
// sums its 8 children) into ga (bf16, half resolution); the b-part is
// stored in FP32 (to be added to the pooling path's contribution)
__global__ void k_split_up(const bf16 *__restrict__ gx, int nx, int ny, int nz, int ca, int cb,
                           bf16 *__restrict__ ga, float *__restrict__ gb32) {
  const int cin = ca + cb;
  const int cx = nx / 2, cy = ny / 2, cz = nz / 2;
  const size_t ncoarse = (size_t)cx * cy * cz;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < ncoarse * cin;
       e += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % cin);
    const size_t vc = e / cin;
    const int X = (int)(vc % cx), Y = (int)((vc / cx) % cy), Z = (int)(vc / ((size_t)cx * cy));
    if (c < ca) {
      float acc = 0.f;
      for (int q = 0; q < 8; ++q) {
        const int x = 2 * X + (q & 1), y = 2 * Y + ((q >> 1) & 1), z = 2 * Z + (q >> 2);
        acc += __bfloat162float(gx[(((size_t)z * ny + y) * nx + x) * cin + c]);
      }
      ga[vc * ca + c] = __float2bfloat16_rn(acc);
    } else {
      for (int q = 0; q < 8; ++q) {
        const int x = 2 * X + (q & 1), y = 2 * Y + ((q >> 1) & 1), z = 2 * Z + (q >> 2);
        const size_t v = ((size_t)z * ny + y) * nx + x;
        gb32[v * cb + (c - ca)] = __bfloat162float(gx[v * cin + c]);
      }
    }
  }
}

// gradient of an encoder output used by both the skip connection (gskip32,
// full resolution, may be null) and 2x2x2 average pooling (gpool, half
// resolution): g = gskip + gpool[parent] / 8
__global__ void k_pool_adjoint_add(const float *__restrict__ gskip32,
                                   const bf16 *__restrict__ gpool, int nx, int ny, int nz, int C,
                                   bf16 *__restrict__ g) {
  const size_t total = (size_t)nx * ny * nz * C;
  for (size_t e = blockIdx.x * (size_t)blockDim.x + threadIdx.x; e < total;
       e += (size_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % C);
    const size_t v = e / C;
    const int x = (int)(v % nx), y = (int)((v / nx) % ny), z = (int)(v / ((size_t)nx * ny));
    const size_t vp = (((size_t)(z >> 1) * (ny >> 1) + (y >> 1)) * (nx >> 1) + (x >> 1));
    float acc = 0.125f * __bfloat162float(gpool[vp * C + c]);
    if (gskip32) acc += gskip32[e];
    g[e] = __float2bfloat16_rn(acc);
  }
}

// gauge-free MSE: e = (q - mean q) - (t - mean t); per-block partial of e^2
// and gradient gq = 2 e / n; means in mq_mt[0], mq_mt[1]
__global__ void k_loss(const float *__restrict__ q, const float *__restrict__ t, size_t n,
                       const double *__restrict__ mq_mt, float *__restrict__ gq,
                       double *__restrict__ part) {
  const double mq = mq_mt[0] / n, mt = mq_mt[1] / n;
  double acc = 0.0;
  for (size_t i = blockIdx.x * (size_t)RED_THREADS + threadIdx.x; i < n;
       i += (size_t)gridDim.x * RED_THREADS) {
    const double e = ((double)q[i] - mq) - ((double)t[i] - mt);
    gq[i] = (float)(2.0 * e / n);
    acc += e * e;
  }
  double s = block_sumd(acc);
  if (threadIdx.x == 0) part[blockIdx.x] = s;
}

// ------------------------------------------------------ energy-norm loss
// A x = sum over faces of beta_f (x_c - x_nb) (positive semidefinite), the
// ghost-fluid faces rebuilt from the input's phi channel f0 = phi / 4h: one
// fluid gives 1/rho, an interface face the series formula with
// theta = |f0_a| / (|f0_a| + |f0_b|) (h cancels).
struct EnergyGeom {
  int nx, ny, nz, per;
  float rl, rg, irl, irg;
};
__device__ __forceinline__ float e_beta(float fa, float fb, const EnergyGeom &e) {
  const bool ga = __float_as_int(fa) > 0, gb = __float_as_int(fb) > 0;
  if (ga == gb) return ga ? e.irg : e.irl;
  const float ra = ga ? e.rg : e.rl, rb = gb ? e.rg : e.rl;
  const float th = fabsf(fa) / (fabsf(fa) + fabsf(fb));
  return 1.f / (th * ra + (1.f - th) * rb);
}

// Aq, At and block partials of q.At, q.Aq, t.At (three arrays of gridDim.x)
__global__ void k_energy_apply(const float *__restrict__ q, const float *__restrict__ t,
                               const bf16 *__restrict__ in16, EnergyGeom e, size_t n,
                               float *__restrict__ aq, float *__restrict__ at,
                               double *__restrict__ part) {
  double sa = 0.0, sc = 0.0, sd = 0.0;
  for (size_t v = blockIdx.x * (size_t)RED_THREADS + threadIdx.x; v < n;
       v += (size_t)gridDim.x * RED_THREADS) {
    const int i = (int)(v % e.nx), j = (int)((v / e.nx) % e.ny), k = (int)(v / ((size_t)e.nx * e.ny));
    const float fc = __bfloat162float(in16[v * 16]), qc = q[v], tc = t[v];
    float sq = 0.f, st = 0.f;
#pragma unroll
    for (int dir = 0; dir < 6; ++dir) {
      const int ax = dir >> 1, hi = dir & 1;
      const int c = ax == 0 ? i : (ax == 1 ? j : k);
      const int m = ax == 0 ? e.nx : (ax == 1 ? e.ny : e.nz);
      const bool wall = !(e.per & (1 << ax)) && (hi ? c == m - 1 : c == 0);
      if (wall) continue;
      const int cn = hi ? (c == m - 1 ? 0 : c + 1) : (c == 0 ? m - 1 : c - 1);
      const int ii = ax == 0 ? cn : i, jj = ax == 1 ? cn : j, kk = ax == 2 ? cn : k;
      const size_t nb = ((size_t)kk * e.ny + jj) * e.nx + ii;
      const float fn = __bfloat162float(in16[nb * 16]);
      const float w = hi ? e_beta(fc, fn, e) : e_beta(fn, fc, e);
      sq = fmaf(w, qc - q[nb], sq);
      st = fmaf(w, tc - t[nb], st);
    }
    aq[v] = sq;
    at[v] = st;
    sa += (double)qc * st;
    sc += (double)qc * sq;
    sd += (double)tc * st;
  }
  double r = block_sumd(sa);
  if (threadIdx.x == 0) part[blockIdx.x] = r;
  r = block_sumd(sc);
  if (threadIdx.x == 0) part[gridDim.x + blockIdx.x] = r;
  r = block_sumd(sd);
  if (threadIdx.x == 0) part[2 * gridDim.x + blockIdx.x] = r;
}

// gq = dL/dq = (2a / (c d)) (alpha Aq - At), alpha = a / c, with
// (a, c, d) = (q.At, q.Aq, t.At) in acd; the loss 1 - a^2 / (c d) -> loss
__global__ void k_energy_grad(const float *__restrict__ aq, const float *__restrict__ at,
                              size_t n, const double *__restrict__ acd, float *__restrict__ gq,
                              double *__restrict__ loss) {
  const double a = acd[0], c = fmax(acd[1], 1e-300), d = fmax(acd[2], 1e-300);
  const float coef = (float)(2.0 * a / (c * d)), alpha = (float)(a / c);
  for (size_t v = blockIdx.x * (size_t)blockDim.x + threadIdx.x; v < n;
       v += (size_t)gridDim.x * blockDim.x)
    gq[v] = coef * fmaf(alpha, aq[v], -at[v]);
  if (blockIdx.x == 0 && threadIdx.x == 0) *loss = 1.0 - a * a / (c * d);
}

// Adam, bias-corrected (step >= 1)
__global__ void k_adam(float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, size_t n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  }
}

// training target q = (p - mean) / rms(p - mean): sums of p and p^2 in sums
__global__ void k_make_target(const double *__restrict__ p, size_t n,
                              const double *__restrict__ sums, float *__restrict__ q) {
  const double m = sums[0] / n;
  const double var = sums[1] / n - m * m;
  const double inv = var > 0.0 ? 1.0 / sqrt(var) : 1.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    q[i] = (float)((p[i] - m) * inv);
}

// p0 = scale * (q - mean q) in FP64 (mean from sum_q)
__global__ void k_to_pressure(const float *__restrict__ q, size_t n, const double *__restrict__ sum_q,
                              double scale, double *__restrict__ p0) {
  const double m = *sum_q / n;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n;
       i += (size_t)gridDim.x * blockDim.x)
    p0[i] = scale * ((double)q[i] - m);
}

}  // namespace mpnet

// =================================================================== host side
#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstring>
#include <mutex>
#include <new>
#include <vector>

using namespace mpnet;

namespace {

#define NCK(call)                                  \
  do {                                             \
    cudaError_t e_ = (call);                       \
    if (e_ != cudaSuccess) return MP_ERR_CUDA;     \
  } while (0)
#define NCKS(call)                  \
  do {                              \
    mp_status s_ = (call);          \
    if (s_ != MP_OK) return s_;     \
  } while (0)

constexpr int NLAYER = 14;
constexpr int CH[4] = {16, 32, 64, 64};

struct Layer {
  int cout, cin, level;  // level: 0 = finest
  int ca, cb, up_a;      // input composition
  size_t woff, boff;     // offsets of weights and bias in the parameter vector
  bf16 *img_f = nullptr;  // packed weights of the forward convolution
  bf16 *img_d = nullptr;  // packed flipped weights (input-gradient convolution)
  bf16 *y = nullptr;     // output activation
  bf16 *gy = nullptr;    // gradient w.r.t. the output
  CUtensorMap map_a, map_b, map_d;  // TMA maps of the inputs and of the masked gradient
};

}  // namespace

struct mp_net {
  int nx[4], ny[4], nz[4];
  size_t nv[4];
  cudaStream_t st = nullptr;
  Layer L[NLAYER];
  size_t nparam = 0, head_w = 0, head_b = 0;
  float *param = nullptr, *grad = nullptr, *adam_m = nullptr, *adam_v = nullptr;
  bf16 *in16 = nullptr;           // network input (16 channels, level 0)
  bf16 *pool[3] = {};             // pooled encoder outputs (levels 1..3)
  float *gskip32[3] = {};         // FP32 skip-path gradients of the encoder outputs, levels 0..2
  bf16 *gz = nullptr;             // ReLU-masked gradient (largest size)
  bf16 *gx = nullptr;             // input gradient of a layer (largest size)
  float *q = nullptr, *gq = nullptr;
  float *qc = nullptr;  // centred output (prolongation to the solver grid)
  float *wpart = nullptr;         // weight-gradient split-K partials
  size_t wpart_n = 0;
  float *cpart = nullptr;         // per-channel partial sums
  double *dpart = nullptr, *dscal = nullptr, *hscal = nullptr;
  int *err = nullptr;
  double *phic = nullptr, *bc = nullptr;  // restricted fields (guess for a 2x finer grid)
  unsigned long long launches = 0;  // kernels launched by the network (all entry points)
  int loss_kind = 0;              // 0: gauge-free MSE; 1: energy norm
  EnergyGeom eg{};                // operator of the energy-norm loss
  float *e_aq = nullptr, *e_at = nullptr;
  std::vector<void *> allocs;
};

namespace {

template <typename T>
mp_status nalloc(mp_net *net, T **p, size_t count) {
  void *v = nullptr;
  if (cudaMalloc(&v, count * sizeof(T) + 64) != cudaSuccess) {
    cudaGetLastError();
    return MP_ERR_OOM;
  }
  net->allocs.push_back(v);
  *p = (T *)v;
  return MP_OK;
}

// Workspace of the single-layer calls (weight image, split-K partials, status
// word): a private stream-ordered pool per device, so calls on any thread and
// stream draw from it safely.  The default pool returns its memory to the
// driver at every synchronisation, and these calls end in one; mapping it again
// took most of a call (a 16-16 layer at 128^3, whose kernel takes 65 us: 287 us
// a call, 102 with this pool).  It keeps up to WS_KEEP bytes (more is returned
// at the next synchronisation) until a network is destroyed.
constexpr uint64_t WS_KEEP = 64ull << 20;
constexpr int WS_DEVICES = 64;
std::mutex ws_mutex;
cudaMemPool_t ws_pools[WS_DEVICES] = {};

mp_status ws_pool(cudaMemPool_t *out) {
  int dev = 0;
  NCK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= WS_DEVICES) return MP_ERR_CUDA;
  std::lock_guard<std::mutex> lock(ws_mutex);
  if (!ws_pools[dev]) {
    cudaMemPoolProps p = {};
    p.allocType = cudaMemAllocationTypePinned;
    p.location.type = cudaMemLocationTypeDevice;
    p.location.id = dev;
    cudaMemPool_t pool = nullptr;
    NCK(cudaMemPoolCreate(&pool, &p));
    uint64_t keep = WS_KEEP;
    if (cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) {
      cudaGetLastError();
      cudaMemPoolDestroy(pool);
      return MP_ERR_CUDA;
    }
    ws_pools[dev] = pool;
  }
  *out = ws_pools[dev];
  return MP_OK;
}
// Status word of a thread's single-layer calls, in mapped host memory: a kernel
// writes it only when a wait gave up, so a call needs neither a memset nor a copy
// (each a few us of a call).  The calls wait for their work, so one per thread does.
// Allocating and freeing it would invalidate a global-mode stream capture of another
// thread (a thread may end at any time), hence the relaxed capture mode around both.
struct RelaxedCapture {
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
  ~RelaxedCapture() { cudaThreadExchangeStreamCaptureMode(&mode); }
};
struct StatusWord {
  int *p = nullptr;
  ~StatusWord() {
    if (!p) return;
    RelaxedCapture relaxed;
    cudaFreeHost(p);
  }
};
mp_status status_word(int **out) {
  static thread_local StatusWord w;
  if (!w.p) {
    RelaxedCapture relaxed;
    if (cudaHostAlloc((void **)&w.p, 64, cudaHostAllocPortable) != cudaSuccess) {
      cudaGetLastError();
      w.p = nullptr;
      return MP_ERR_OOM;
    }
  }
  *(volatile int *)w.p = 0;
  *out = w.p;
  return MP_OK;
}
// return what the current device's pool keeps and no call uses
void ws_trim() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= WS_DEVICES) return;
  std::lock_guard<std::mutex> lock(ws_mutex);
  if (ws_pools[dev]) cudaMemPoolTrimTo(ws_pools[dev], 0);
}

bool cout_ok(int c) { return c == 16 || c == 32 || c == 48 || c == 64 || c == 96 || c == 128; }
// output channels per CTA of k_conv3d_halo (96 and 128 are split in two)
int nc_of(int cout) { return cout <= 64 ? cout : cout / 2; }

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                 const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                 const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                 CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
EncodeTiled encode_fn() {
  static EncodeTiled fn = nullptr;
  if (!fn) {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (EncodeTiled)p;
    else
      cudaGetLastError();
  }
  return fn;
}

// TMA map of a channels-last BF16 tensor (nz, ny, nx, C) with the halo box
// (8 channels, HX, HY, HZ); out-of-range elements read as zero
mp_status make_map(CUtensorMap *m, const bf16 *base, int C, int nx, int ny, int nz) {
  std::memset(m, 0, sizeof(*m));
  if (!base) return MP_OK;  // unused input
  EncodeTiled enc = encode_fn();
  if (!enc) return MP_ERR_CUDA;
  const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)nx, (cuuint64_t)ny, (cuuint64_t)nz};
  const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)nx * C * 2,
                                 (cuuint64_t)ny * nx * C * 2};
  const cuuint32_t box[4] = {8, HX, HY, HZ};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  if (enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, (void *)base, dims, strides, box, es,
          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
          CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return MP_ERR_INVALID_ARG;
  return MP_OK;
}

// maps of a convolution's inputs: xa (unless read through upsampling) and xb
mp_status make_maps(const ConvGeom &g, const bf16 *xa, const bf16 *xb, CUtensorMap *ma,
                    CUtensorMap *mb) {
  NCKS(make_map(ma, g.up_a ? nullptr : xa, g.ca, g.nx, g.ny, g.nz));
  NCKS(make_map(mb, g.cb > 0 ? xb : nullptr, g.cb, g.nx, g.ny, g.nz));
  return MP_OK;
}

int sm_count() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) {
      cudaGetLastError();
      n = 1;
    }
  }
  return n;
}

// Launches that are still to report a timed-out first wait (mp_net_test_wait_timeout).
std::atomic<int> g_wait_failures{0};
int take_wait_failure() {
  int v = g_wait_failures.load();
  while (v > 0 && !g_wait_failures.compare_exchange_weak(v, v - 1)) {
  }
  return v > 0 ? 1 : 0;
}

template <int NC>
mp_status launch_halo(const ConvGeom &g, const CUtensorMap &ma, const CUtensorMap &mb,
                      const bf16 *xa, const bf16 *wimg, const float *bias, int cout, bf16 *y,
                      float *y32, int relu, int *err, cudaStream_t st, bool after_pack) {
  const int smem = h_smem_bytes<NC>();
  static bool attr = false;
  if (!attr) {
    NCK(cudaFuncSetAttribute(k_conv3d_halo<NC>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem));
    attr = true;
  }
  HaloArgs a;
  a.xa = xa;
  a.wimg = wimg;
  a.bias = bias;
  a.y = y;
  a.y32 = y32;
  a.nx = g.nx;
  a.ny = g.ny;
  a.nz = g.nz;
  a.ca = g.ca;
  a.up_a = g.up_a;
  a.cout = cout;
  a.relu = relu;
  a.tiles_x = (g.nx + 7) / 8;
  a.tiles_y = (g.ny + 15) / 16;
  const int tiles_z = (g.nz + HT_Z - 1) / HT_Z;
  a.ntiles = a.tiles_x * a.tiles_y * tiles_z;
  a.nsplit = cout / NC;
  a.nchunk = g.cin / 16;
  a.fail_first = take_wait_failure();
  a.err = err;
  const long items = (long)a.ntiles * a.nsplit;
  long grid = std::min<long>(items, (long)sm_count() * h_ctas_per_sm<NC>());
  grid = std::max<long>(a.nsplit, grid - grid % a.nsplit);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(HALO_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute la[1];
  la[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  la[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = la;
  cfg.numAttrs = after_pack ? 1 : 0;  // after the packing kernel: overlap its end
  NCK(cudaLaunchKernelEx(&cfg, k_conv3d_halo<NC>, ma, mb, a));
  return MP_OK;
}

// forward convolution through k_conv3d_halo; wimg packed by k_pack_img for nc_of(cout)
mp_status conv_fwd(const ConvGeom &g, const CUtensorMap &ma, const CUtensorMap &mb,
                   const bf16 *xa, const bf16 *wimg, const float *bias, int cout, bf16 *y,
                   float *y32, int relu, int *err, cudaStream_t st, bool after_pack = false) {
  switch (nc_of(cout)) {
    case 16:
      return launch_halo<16>(g, ma, mb, xa, wimg, bias, cout, y, y32, relu, err, st, after_pack);
    case 32:
      return launch_halo<32>(g, ma, mb, xa, wimg, bias, cout, y, y32, relu, err, st, after_pack);
    case 48:
      return launch_halo<48>(g, ma, mb, xa, wimg, bias, cout, y, y32, relu, err, st, after_pack);
    case 64:
      return launch_halo<64>(g, ma, mb, xa, wimg, bias, cout, y, y32, relu, err, st, after_pack);
  }
  return MP_ERR_INVALID_ARG;
}

size_t wgrad_chunks(const ConvGeom &g) {
  const size_t nv = (size_t)g.nx * g.ny * g.nz;
  return (nv + WG_VOX - 1) / WG_VOX;
}
size_t wgrad_partial_floats(const ConvGeom &g, int cout) {
  return wgrad_chunks(g) * 27 * (size_t)g.cin * cout;
}

template <int COUT>
mp_status launch_wgrad(const ConvGeom &g, const bf16 *xa, const bf16 *xb, const bf16 *gr,
                       float *part, float *dw, int *err, cudaStream_t st) {
  const int smem = conv_smem_bytes<COUT>();
  static bool attr = false;
  if (!attr) {
    NCK(cudaFuncSetAttribute(k_conv3d_wgrad<COUT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             smem));
    attr = true;
  }
  const int rows = 27 * g.cin;
  const int chunks = (int)wgrad_chunks(g);
  dim3 grid((rows + 127) / 128, chunks);
  k_conv3d_wgrad<COUT><<<grid, CONV_THREADS, smem, st>>>(xa, xb, gr, g, part, err);
  k_wgrad_reduce<<<(rows * COUT + 31) / 32, 32 * WR_SEG, 0, st>>>(part, chunks, rows, COUT, dw);
  NCK(cudaGetLastError());
  return MP_OK;
}

mp_status conv_wgrad(const ConvGeom &g, const bf16 *xa, const bf16 *xb, const bf16 *gr, int cout,
                     float *part, float *dw, int *err, cudaStream_t st) {
  switch (cout) {
    case 16: return launch_wgrad<16>(g, xa, xb, gr, part, dw, err, st);
    case 32: return launch_wgrad<32>(g, xa, xb, gr, part, dw, err, st);
    case 64: return launch_wgrad<64>(g, xa, xb, gr, part, dw, err, st);
  }
  return MP_ERR_INVALID_ARG;
}

mp_status check_err(mp_net *net) {
  int h = 0;
  NCK(cudaMemcpyAsync(&h, net->err, sizeof(int), cudaMemcpyDeviceToHost, net->st));
  NCK(cudaStreamSynchronize(net->st));
  return h ? MP_ERR_TIMEOUT : MP_OK;
}

int grid_for(size_t n, int threads = 256) {
  size_t b = (n + threads - 1) / threads;
  return (int)std::min<size_t>(b, 152 * 32);
}

ConvGeom geom(const mp_net *net, const Layer &l) {
  ConvGeom g;
  g.nx = net->nx[l.level];
  g.ny = net->ny[l.level];
  g.nz = net->nz[l.level];
  g.ca = l.ca;
  g.cb = l.cb;
  g.up_a = l.up_a;
  g.cin = l.cin;
  return g;
}

// inputs (a, b) of layer i
void layer_inputs(const mp_net *net, int i, const bf16 **a, const bf16 **b) {
  const Layer *L = net->L;
  *b = nullptr;
  switch (i) {
    case 0: *a = net->in16; break;
    case 2: *a = net->pool[0]; break;
    case 4: *a = net->pool[1]; break;
    case 6: *a = net->pool[2]; break;
    case 8: *a = L[7].y; *b = L[5].y; break;   // up(e3) | e2
    case 10: *a = L[9].y; *b = L[3].y; break;  // up(d2) | e1
    case 12: *a = L[11].y; *b = L[1].y; break; // up(d1) | e0
    default: *a = L[i - 1].y; break;
  }
}

mp_status pack_all(mp_net *net) {
  for (int i = 0; i < NLAYER; ++i) {
    Layer &l = net->L[i];
    const size_t nw = (size_t)l.cout * 27 * l.cin;
    k_pack_img<float><<<grid_for(nw), 256, 0, net->st>>>(net->param + l.woff, l.cout, l.cin, 0,
                                                         nc_of(l.cout), l.img_f);
    if (i > 0)  // input gradient: output channels l.cin, input channels l.cout
      k_pack_img<float><<<grid_for(nw), 256, 0, net->st>>>(net->param + l.woff, l.cin, l.cout, 1,
                                                           nc_of(l.cin), l.img_d);
  }
  NCK(cudaGetLastError());
  return MP_OK;
}

// TMA maps of every layer's inputs (fixed buffers) and of the masked gradient
mp_status make_all_maps(mp_net *net) {
  for (int i = 0; i < NLAYER; ++i) {
    Layer &l = net->L[i];
    const bf16 *a, *b;
    layer_inputs(net, i, &a, &b);
    NCKS(make_maps(geom(net, l), a, b, &l.map_a, &l.map_b));
    NCKS(make_map(&l.map_d, net->gz, l.cout, net->nx[l.level], net->ny[l.level],
                  net->nz[l.level]));
  }
  return MP_OK;
}

mp_status forward(mp_net *net) {
  NCK(cudaMemsetAsync(net->err, 0, sizeof(int), net->st));
  for (int i = 0; i < NLAYER; ++i) {
    Layer &l = net->L[i];
    if (i == 2 || i == 4 || i == 6) {  // pool the previous level's encoder output
      const int lv = l.level - 1;
      k_pool2<<<grid_for(net->nv[l.level] * l.ca), 256, 0, net->st>>>(
          net->L[i - 1].y, net->pool[l.level - 1], net->nx[lv], net->ny[lv], net->nz[lv], l.ca);
    }
    const bf16 *a, *b;
    layer_inputs(net, i, &a, &b);
    NCKS(conv_fwd(geom(net, l), l.map_a, l.map_b, a, l.img_f, net->param + l.boff, l.cout, l.y,
                  nullptr, 1, net->err, net->st));
  }
  k_head_fwd<<<grid_for(net->nv[0]), 256, 0, net->st>>>(
      net->L[13].y, net->param + net->head_w, net->param + net->head_b, net->nv[0], CH[0],
      net->q);
  NCK(cudaGetLastError());
  net->launches += NLAYER + 3 + 1;  // convolutions, poolings, head
  return MP_OK;
}

// gradients of sum(q * gq) into net->grad (gq in net->gq)
mp_status backward(mp_net *net) {
  const size_t n0 = net->nv[0];
  // head
  {
    const int chunk = 4096;
    const int chunks = (int)((n0 + chunk - 1) / chunk);
    k_head_bwd<<<chunks, CH[0] + 1, 0, net->st>>>(net->gq, net->L[13].y,
                                                  net->param + net->head_w, n0, CH[0], chunk,
                                                  net->L[13].gy, net->cpart);
    k_chan_final<<<1, 32, 0, net->st>>>(net->cpart, chunks, CH[0] + 1, net->grad + net->head_w);
  }
  for (int i = NLAYER - 1; i >= 0; --i) {
    Layer &l = net->L[i];
    const ConvGeom g = geom(net, l);
    const size_t nv = net->nv[l.level];
    k_relu_mask<<<grid_for(nv * l.cout), 256, 0, net->st>>>(l.gy, l.y, nv * l.cout, net->gz);
    {
      const int chunk = 1024;
      const int chunks = (int)((nv + chunk - 1) / chunk);
      k_chan_psum<<<chunks, l.cout, 0, net->st>>>(net->gz, nv, l.cout, chunk, net->cpart);
      k_chan_final<<<1, 128, 0, net->st>>>(net->cpart, chunks, l.cout, net->grad + l.boff);
    }
    const bf16 *a, *b;
    layer_inputs(net, i, &a, &b);
    NCKS(conv_wgrad(g, a, b, net->gz, l.cout, net->wpart, net->grad + l.woff, net->err,
                    net->st));
    if (i == 0) break;
    // input gradient: forward convolution of gz with the flipped, transposed weights
    ConvGeom gd = g;
    gd.ca = l.cout;
    gd.cb = 0;
    gd.up_a = 0;
    gd.cin = l.cout;
    const bool plain = !(i == 2 || i == 4 || i == 6 || i == 8 || i == 10 || i == 12);
    bf16 *dst = plain ? net->L[i - 1].gy : net->gx;
    NCKS(conv_fwd(gd, l.map_d, l.map_d, net->gz, l.img_d, nullptr, l.cin, dst, nullptr, 0,
                  net->err, net->st));
    const int lv = l.level;
    if (i == 12 || i == 10 || i == 8) {  // decoder input: [up(coarse) | skip]
      const int coarse = i == 12 ? 11 : (i == 10 ? 9 : 7);
      k_split_up<<<grid_for(net->nv[lv + 1] * l.cin), 256, 0, net->st>>>(
          net->gx, net->nx[lv], net->ny[lv], net->nz[lv], l.ca, l.cb, net->L[coarse].gy,
          net->gskip32[lv]);
    } else if (i == 6 || i == 4 || i == 2) {  // encoder input = pooled finer output
      const int fine = i - 1, flv = lv - 1;
      k_pool_adjoint_add<<<grid_for(net->nv[flv] * l.cin), 256, 0, net->st>>>(
          net->gskip32[flv], net->gx, net->nx[flv], net->ny[flv], net->nz[flv], l.cin,
          net->L[fine].gy);
    }
  }
  NCK(cudaGetLastError());
  return MP_OK;
}

// Loss of the last forward pass against target and its gradient w.r.t. q
// into net->gq; the loss value lands in net->dscal[2] (MSE: the sum of
// squared errors, divided by n on the host).
mp_status loss_and_grad(mp_net *net, const float *target) {
  const size_t n = net->nv[0];
  // means of prediction and target, then loss and its gradient
  k_psum<float><<<RED_BLOCKS, RED_THREADS, 0, net->st>>>(net->q, n, 0, net->dpart);
  k_pfinal<<<1, RED_THREADS, 0, net->st>>>(net->dpart, RED_BLOCKS, net->dscal);
  k_psum<float><<<RED_BLOCKS, RED_THREADS, 0, net->st>>>(target, n, 0, net->dpart);
  k_pfinal<<<1, RED_THREADS, 0, net->st>>>(net->dpart, RED_BLOCKS, net->dscal + 1);
  if (net->loss_kind == 0) {
    k_loss<<<RED_BLOCKS, RED_THREADS, 0, net->st>>>(net->q, target, n, net->dscal, net->gq,
                                                   net->dpart);
    k_pfinal<<<1, RED_THREADS, 0, net->st>>>(net->dpart, RED_BLOCKS, net->dscal + 2);
  } else {
    k_energy_apply<<<RED_BLOCKS, RED_THREADS, 0, net->st>>>(net->q, target, net->in16, net->eg, n,
                                                           net->e_aq, net->e_at, net->dpart);
    for (int q = 0; q < 3; ++q)
      k_pfinal<<<1, RED_THREADS, 0, net->st>>>(net->dpart + q * RED_BLOCKS, RED_BLOCKS,
                                               net->dscal + 8 + q);
    k_energy_grad<<<grid_for(n), 256, 0, net->st>>>(net->e_aq, net->e_at, n, net->dscal + 8,
                                                    net->gq, net->dscal + 2);
  }
  NCK(cudaGetLastError());
  return MP_OK;
}

}  // namespace

extern "C" {

mp_status mp_conv3d_fwd(int nx, int ny, int nz, const void *xa, int ca, int up_a, const void *xb,
                        int cb, const void *w, const float *bias, int cout, int relu, void *y,
                        float *y32, void *stream) {
  if (nx <= 0 || ny <= 0 || nz <= 0 || nx % 8 || ny % 4 || nz % 4 || !xa || ca <= 0 || ca % 16 ||
      cb < 0 || cb % 16 || (cb > 0 && !xb) || !w || !cout_ok(cout) || (!y && !y32) ||
      (up_a && (nx % 2 || ny % 2 || nz % 2)))
    return MP_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  ConvGeom g{nx, ny, nz, ca, cb, up_a ? 1 : 0, ca + cb};
  CUtensorMap ma, mb;
  NCKS(make_maps(g, (const bf16 *)xa, (const bf16 *)xb, &ma, &mb));
  const size_t nw = (size_t)cout * 27 * g.cin;
  cudaMemPool_t pool;
  int *err = nullptr;
  NCKS(ws_pool(&pool));
  NCKS(status_word(&err));
  bf16 *img = nullptr;  // packed weights
  NCK(cudaMallocFromPoolAsync((void **)&img, nw * sizeof(bf16), pool, st));
  k_pack_img<bf16><<<grid_for(nw), 256, 0, st>>>((const bf16 *)w, cout, g.cin, 0, nc_of(cout), img);
  mp_status s = conv_fwd(g, ma, mb, (const bf16 *)xa, img, bias, cout, (bf16 *)y, y32, relu, err,
                         st, true);
  NCK(cudaFreeAsync(img, st));
  NCK(cudaStreamSynchronize(st));
  if (s != MP_OK) return s;
  return *(volatile int *)err ? MP_ERR_TIMEOUT : MP_OK;
}

mp_status mp_conv3d_wgrad(int nx, int ny, int nz, const void *xa, int ca, int up_a,
                          const void *xb, int cb, const void *g, int cout, float *dw,
                          void *stream) {
  if (nx <= 0 || ny <= 0 || nz <= 0 || !xa || ca <= 0 || ca % 16 || cb < 0 || cb % 16 ||
      (cb > 0 && !xb) || !g || !dw || !(cout == 16 || cout == 32 || cout == 64) ||
      (up_a && (nx % 2 || ny % 2 || nz % 2)))
    return MP_ERR_INVALID_ARG;
  cudaStream_t st = (cudaStream_t)stream;
  ConvGeom geo{nx, ny, nz, ca, cb, up_a ? 1 : 0, ca + cb};
  cudaMemPool_t pool;
  int *err = nullptr;
  NCKS(ws_pool(&pool));
  NCKS(status_word(&err));
  float *part = nullptr;
  NCK(cudaMallocFromPoolAsync((void **)&part, wgrad_partial_floats(geo, cout) * sizeof(float), pool,
                              st));
  mp_status s = conv_wgrad(geo, (const bf16 *)xa, (const bf16 *)xb, (const bf16 *)g, cout, part,
                           dw, err, st);
  NCK(cudaFreeAsync(part, st));
  NCK(cudaStreamSynchronize(st));
  if (s != MP_OK) return s;
  return *(volatile int *)err ? MP_ERR_TIMEOUT : MP_OK;
}

mp_status mp_net_create(mp_net_handle *out, int nx, int ny, int nz, void *stream) {
  if (!out || nx <= 0 || ny <= 0 || nz <= 0 || nx % 32 || ny % 32 || nz % 32)
    return MP_ERR_INVALID_ARG;
  *out = nullptr;
  mp_net *net = new (std::nothrow) mp_net();
  if (!net) return MP_ERR_OOM;
  net->st = (cudaStream_t)stream;
  for (int l = 0; l < 4; ++l) {
    net->nx[l] = nx >> l;
    net->ny[l] = ny >> l;
    net->nz[l] = nz >> l;
    net->nv[l] = (size_t)net->nx[l] * net->ny[l] * net->nz[l];
  }
  // layers in forward order: (cout, cin, level, ca, cb, up_a)
  const int spec[NLAYER][6] = {
      {CH[0], 16, 0, 16, 0, 0},          {CH[0], CH[0], 0, CH[0], 0, 0},
      {CH[1], CH[0], 1, CH[0], 0, 0},    {CH[1], CH[1], 1, CH[1], 0, 0},
      {CH[2], CH[1], 2, CH[1], 0, 0},    {CH[2], CH[2], 2, CH[2], 0, 0},
      {CH[3], CH[2], 3, CH[2], 0, 0},    {CH[3], CH[3], 3, CH[3], 0, 0},
      {CH[2], CH[3] + CH[2], 2, CH[3], CH[2], 1}, {CH[2], CH[2], 2, CH[2], 0, 0},
      {CH[1], CH[2] + CH[1], 1, CH[2], CH[1], 1}, {CH[1], CH[1], 1, CH[1], 0, 0},
      {CH[0], CH[1] + CH[0], 0, CH[1], CH[0], 1}, {CH[0], CH[0], 0, CH[0], 0, 0}};
  size_t off = 0, wpart = 0, maxact = 0;
  mp_status s = MP_OK;
  for (int i = 0; i < NLAYER && s == MP_OK; ++i) {
    Layer &l = net->L[i];
    l.cout = spec[i][0];
    l.cin = spec[i][1];
    l.level = spec[i][2];
    l.ca = spec[i][3];
    l.cb = spec[i][4];
    l.up_a = spec[i][5];
    l.woff = off;
    off += (size_t)l.cout * 27 * l.cin;
    l.boff = off;
    off += l.cout;
    const size_t nv = net->nv[l.level];
    wpart = std::max(wpart, wgrad_partial_floats(geom(net, l), l.cout));
    maxact = std::max(maxact, nv * (size_t)std::max(l.cin, l.cout));
    if ((s = nalloc(net, &l.img_f, (size_t)l.cout * 27 * l.cin)) != MP_OK) break;
    if ((s = nalloc(net, &l.img_d, (size_t)l.cout * 27 * l.cin)) != MP_OK) break;
    if ((s = nalloc(net, &l.y, nv * l.cout)) != MP_OK) break;
    s = nalloc(net, &l.gy, nv * l.cout);
  }
  net->head_w = off;
  off += CH[0];
  net->head_b = off;
  off += 1;
  net->nparam = off;
  net->wpart_n = wpart;
  if (s == MP_OK) s = nalloc(net, &net->param, off);
  if (s == MP_OK) s = nalloc(net, &net->grad, off);
  if (s == MP_OK) s = nalloc(net, &net->adam_m, off);
  if (s == MP_OK) s = nalloc(net, &net->adam_v, off);
  if (s == MP_OK) s = nalloc(net, &net->in16, net->nv[0] * 16);
  for (int l = 0; l < 3 && s == MP_OK; ++l) s = nalloc(net, &net->pool[l], net->nv[l + 1] * CH[l]);
  for (int l = 0; l < 3 && s == MP_OK; ++l) s = nalloc(net, &net->gskip32[l], net->nv[l] * CH[l]);
  if (s == MP_OK) s = nalloc(net, &net->gz, maxact);
  if (s == MP_OK) s = nalloc(net, &net->gx, maxact);
  if (s == MP_OK) s = nalloc(net, &net->q, net->nv[0]);
  if (s == MP_OK) s = nalloc(net, &net->qc, net->nv[0]);
  if (s == MP_OK) s = nalloc(net, &net->gq, net->nv[0]);
  if (s == MP_OK) s = nalloc(net, &net->wpart, wpart);
  if (s == MP_OK) s = nalloc(net, &net->cpart, (net->nv[0] / 1024 + 64) * 130);
  if (s == MP_OK) s = nalloc(net, &net->dpart, 3 * RED_BLOCKS + 8);
  if (s == MP_OK) s = nalloc(net, &net->dscal, 16);
  if (s == MP_OK) s = nalloc(net, &net->e_aq, net->nv[0]);
  if (s == MP_OK) s = nalloc(net, &net->e_at, net->nv[0]);
  if (s == MP_OK) s = nalloc(net, &net->err, 4);
  if (s == MP_OK && cudaMallocHost((void **)&net->hscal, 8 * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    net->hscal = nullptr;
    s = MP_ERR_OOM;
  }
  if (s == MP_OK) {
    if (cudaMemsetAsync(net->param, 0, off * sizeof(float), net->st) != cudaSuccess ||
        cudaMemsetAsync(net->adam_m, 0, off * sizeof(float), net->st) != cudaSuccess ||
        cudaMemsetAsync(net->adam_v, 0, off * sizeof(float), net->st) != cudaSuccess ||
        cudaMemsetAsync(net->in16, 0, net->nv[0] * 16 * sizeof(bf16), net->st) != cudaSuccess)
      s = MP_ERR_CUDA;
  }
  if (s == MP_OK) s = pack_all(net);
  if (s == MP_OK) s = make_all_maps(net);
  if (s == MP_OK && cudaStreamSynchronize(net->st) != cudaSuccess) s = MP_ERR_CUDA;
  if (s != MP_OK) {
    mp_net_destroy(net);
    return s;
  }
  *out = net;
  return MP_OK;
}

size_t mp_net_param_count(mp_net_handle net) { return net ? net->nparam : 0; }

unsigned long long mp_net_launches(mp_net_handle net) { return net ? net->launches : 0; }

mp_status mp_net_dims(mp_net_handle net, int *nx, int *ny, int *nz) {
  if (!net) return MP_ERR_INVALID_ARG;
  if (nx) *nx = net->nx[0];
  if (ny) *ny = net->ny[0];
  if (nz) *nz = net->nz[0];
  return MP_OK;
}

mp_status mp_net_set_params(mp_net_handle net, const float *p) {
  if (!net || !p) return MP_ERR_INVALID_ARG;
  NCK(cudaMemcpyAsync(net->param, p, net->nparam * sizeof(float), cudaMemcpyDeviceToDevice,
                      net->st));
  NCK(cudaMemsetAsync(net->adam_m, 0, net->nparam * sizeof(float), net->st));
  NCK(cudaMemsetAsync(net->adam_v, 0, net->nparam * sizeof(float), net->st));
  NCKS(pack_all(net));
  NCK(cudaStreamSynchronize(net->st));
  return MP_OK;
}

mp_status mp_net_get_params(mp_net_handle net, float *p) {
  if (!net || !p) return MP_ERR_INVALID_ARG;
  NCK(cudaMemcpyAsync(p, net->param, net->nparam * sizeof(float), cudaMemcpyDeviceToDevice,
                      net->st));
  NCK(cudaStreamSynchronize(net->st));
  return MP_OK;
}

mp_status mp_net_get_adam(mp_net_handle net, float *m, float *v) {
  if (!net || !m || !v) return MP_ERR_INVALID_ARG;
  NCK(cudaMemcpyAsync(m, net->adam_m, net->nparam * sizeof(float), cudaMemcpyDeviceToDevice,
                      net->st));
  NCK(cudaMemcpyAsync(v, net->adam_v, net->nparam * sizeof(float), cudaMemcpyDeviceToDevice,
                      net->st));
  NCK(cudaStreamSynchronize(net->st));
  return MP_OK;
}

mp_status mp_net_set_adam(mp_net_handle net, const float *m, const float *v) {
  if (!net || !m || !v) return MP_ERR_INVALID_ARG;
  NCK(cudaMemcpyAsync(net->adam_m, m, net->nparam * sizeof(float), cudaMemcpyDeviceToDevice,
                      net->st));
  NCK(cudaMemcpyAsync(net->adam_v, v, net->nparam * sizeof(float), cudaMemcpyDeviceToDevice,
                      net->st));
  NCK(cudaStreamSynchronize(net->st));
  return MP_OK;
}

mp_status mp_net_set_loss(mp_net_handle net, int kind, double rho_l, double rho_g,
                          const mp_bc bc[3]) {
  if (!net || !(kind == 0 || kind == 1) || !(rho_l > 0.0) || !(rho_g > 0.0) || !bc)
    return MP_ERR_INVALID_ARG;
  int per = 0;
  for (int a = 0; a < 3; ++a) {
    if (bc[a] != MP_BC_PERIODIC && bc[a] != MP_BC_NEUMANN) return MP_ERR_INVALID_ARG;
    if (bc[a] == MP_BC_PERIODIC) per |= 1 << a;
  }
  net->loss_kind = kind;
  net->eg = EnergyGeom{net->nx[0], net->ny[0], net->nz[0], per, (float)rho_l, (float)rho_g,
                       (float)(1.0 / rho_l), (float)(1.0 / rho_g)};
  return MP_OK;
}

mp_status mp_net_set_stream(mp_net_handle net, void *stream) {
  if (!net) return MP_ERR_INVALID_ARG;
  net->st = (cudaStream_t)stream;
  return MP_OK;
}

mp_status mp_net_set_input(mp_net_handle net, const void *x16) {
  if (!net || !x16) return MP_ERR_INVALID_ARG;
  // (a full 16-channel input: channels 2..15 are whatever the caller passes)
  NCK(cudaMemcpyAsync(net->in16, x16, net->nv[0] * 16 * sizeof(bf16), cudaMemcpyDeviceToDevice,
                      net->st));
  NCK(cudaStreamSynchronize(net->st));
  return MP_OK;
}

mp_status mp_net_features(mp_net_handle net, const double *phi, const double *b, double h,
                          double b_scale, double *s_out) {
  if (!net || !phi || !b || !(h > 0.0) || !(b_scale > 0.0)) return MP_ERR_INVALID_ARG;
  const size_t n = net->nv[0];
  k_psum<double><<<RED_BLOCKS, RED_THREADS, 0, net->st>>>(b, n, 1, net->dpart);
  k_pfinal<<<1, RED_THREADS, 0, net->st>>>(net->dpart, RED_BLOCKS, net->dscal);
  NCK(cudaMemcpyAsync(net->hscal, net->dscal, sizeof(double), cudaMemcpyDeviceToHost, net->st));
  NCK(cudaStreamSynchronize(net->st));
  double rb = std::sqrt(net->hscal[0] / (double)n);  // rms(b); f1 = b / rms(b) = bt / s
  if (!(rb > 0.0) || !std::isfinite(rb)) rb = 1.0;
  k_features<<<grid_for(n), 256, 0, net->st>>>(phi, b, n, 0.25 / h, 1.0 / rb, net->in16);
  NCK(cudaGetLastError());
  net->launches += 3;
  NCK(cudaStreamSynchronize(net->st));
  if (s_out) *s_out = b_scale * rb;
  return MP_OK;
}

mp_status mp_net_features_at(mp_net_handle net, int factor, const double *phi, const double *b,
                             double h, double b_scale, double *s_out) {
  if (!net || !(factor == 1 || factor == 2)) return MP_ERR_INVALID_ARG;
  if (factor == 1) return mp_net_features(net, phi, b, h, b_scale, s_out);
  if (!phi || !b || !(h > 0.0) || !(b_scale > 0.0)) return MP_ERR_INVALID_ARG;
  const size_t n = net->nv[0];
  if (!net->phic) {
    NCKS(nalloc(net, &net->phic, n));
    NCKS(nalloc(net, &net->bc, n));
  }
  k_restrict_fields<<<grid_for(n), 256, 0, net->st>>>(phi, b, net->nx[0], net->ny[0], net->nz[0],
                                                      net->phic, net->bc);
  NCK(cudaGetLastError());
  net->launches += 1;
  // the restricted b is the mean of the children: same scale as b
  return mp_net_features(net, net->phic, net->bc, 2.0 * h, b_scale, s_out);
}

mp_status mp_net_pressure_at(mp_net_handle net, int factor, const mp_bc bc[3], double s,
                             double *p_dev) {
  if (!net || !(factor == 1 || factor == 2) || !p_dev || !bc) return MP_ERR_INVALID_ARG;
  if (factor == 1) return mp_net_pressure(net, s, p_dev);
  int per = 0;
  for (int a = 0; a < 3; ++a) {
    if (bc[a] != MP_BC_PERIODIC && bc[a] != MP_BC_NEUMANN) return MP_ERR_INVALID_ARG;
    if (bc[a] == MP_BC_PERIODIC) per |= 1 << a;
  }
  const size_t n = net->nv[0];
  k_psum<float><<<RED_BLOCKS, RED_THREADS, 0, net->st>>>(net->q, n, 0, net->dpart);
  k_pfinal<<<1, RED_THREADS, 0, net->st>>>(net->dpart, RED_BLOCKS, net->dscal);
  k_center_q<<<grid_for(n), 256, 0, net->st>>>(net->q, net->dscal, n, net->qc);
  const dim3 pg((2 * net->nx[0] + 255) / 256, std::min(2 * net->ny[0], 65535),
                std::min(2 * net->nz[0], 65535));
  k_prolong_tri<<<pg, 256, 0, net->st>>>(net->qc, net->nx[0], net->ny[0], net->nz[0], per, s,
                                         p_dev);
  NCK(cudaGetLastError());
  net->launches += 4;
  NCK(cudaStreamSynchronize(net->st));
  return MP_OK;
}

mp_status mp_net_get_input2(mp_net_handle net, void *x2) {
  if (!net || !x2) return MP_ERR_INVALID_ARG;
  NCK(cudaMemcpy2DAsync(x2, 2 * sizeof(bf16), net->in16, 16 * sizeof(bf16), 2 * sizeof(bf16),
                        net->nv[0], cudaMemcpyDeviceToDevice, net->st));
  NCK(cudaStreamSynchronize(net->st));
  return MP_OK;
}

mp_status mp_net_set_input2(mp_net_handle net, const void *x2) {
  if (!net || !x2) return MP_ERR_INVALID_ARG;
  // the other 14 channels stay zero (set at creation, never written)
  NCK(cudaMemcpy2DAsync(net->in16, 16 * sizeof(bf16), x2, 2 * sizeof(bf16), 2 * sizeof(bf16),
                        net->nv[0], cudaMemcpyDeviceToDevice, net->st));
  return MP_OK;
}

mp_status mp_net_forward(mp_net_handle net, float *q_dev) {
  if (!net) return MP_ERR_INVALID_ARG;
  NCKS(forward(net));
  if (q_dev)
    NCK(cudaMemcpyAsync(q_dev, net->q, net->nv[0] * sizeof(float), cudaMemcpyDeviceToDevice,
                        net->st));
  return check_err(net);
}

mp_status mp_net_pressure(mp_net_handle net, double s, double *p_dev) {
  if (!net || !p_dev) return MP_ERR_INVALID_ARG;
  const size_t n = net->nv[0];
  k_psum<float><<<RED_BLOCKS, RED_THREADS, 0, net->st>>>(net->q, n, 0, net->dpart);
  k_pfinal<<<1, RED_THREADS, 0, net->st>>>(net->dpart, RED_BLOCKS, net->dscal);
  k_to_pressure<<<grid_for(n), 256, 0, net->st>>>(net->q, n, net->dscal, s, p_dev);
  NCK(cudaGetLastError());
  net->launches += 3;
  NCK(cudaStreamSynchronize(net->st));
  return MP_OK;
}

mp_status mp_net_make_target(mp_net_handle net, const double *p, float *q) {
  if (!net || !p || !q) return MP_ERR_INVALID_ARG;
  const size_t n = net->nv[0];
  k_psum<double><<<RED_BLOCKS, RED_THREADS, 0, net->st>>>(p, n, 0, net->dpart);
  k_pfinal<<<1, RED_THREADS, 0, net->st>>>(net->dpart, RED_BLOCKS, net->dscal + 4);
  k_psum<double><<<RED_BLOCKS, RED_THREADS, 0, net->st>>>(p, n, 1, net->dpart);
  k_pfinal<<<1, RED_THREADS, 0, net->st>>>(net->dpart, RED_BLOCKS, net->dscal + 5);
  k_make_target<<<grid_for(n), 256, 0, net->st>>>(p, n, net->dscal + 4, q);
  NCK(cudaGetLastError());
  NCK(cudaStreamSynchronize(net->st));
  return MP_OK;
}

mp_status mp_net_backward(mp_net_handle net, const float *gq, float *grad_dev) {
  if (!net || !gq) return MP_ERR_INVALID_ARG;
  NCKS(forward(net));
  NCK(cudaMemcpyAsync(net->gq, gq, net->nv[0] * sizeof(float), cudaMemcpyDeviceToDevice,
                      net->st));
  NCKS(backward(net));
  if (grad_dev)
    NCK(cudaMemcpyAsync(grad_dev, net->grad, net->nparam * sizeof(float),
                        cudaMemcpyDeviceToDevice, net->st));
  return check_err(net);
}

mp_status mp_net_loss_grad(mp_net_handle net, const float *target, float *gq_dev,
                           double *loss_out) {
  if (!net || !target) return MP_ERR_INVALID_ARG;
  NCKS(forward(net));
  NCKS(loss_and_grad(net, target));
  if (gq_dev)
    NCK(cudaMemcpyAsync(gq_dev, net->gq, net->nv[0] * sizeof(float), cudaMemcpyDeviceToDevice,
                        net->st));
  NCK(cudaMemcpyAsync(net->hscal, net->dscal + 2, sizeof(double), cudaMemcpyDeviceToHost,
                      net->st));
  NCKS(check_err(net));
  if (loss_out)
    *loss_out = net->loss_kind == 0 ? net->hscal[0] / (double)net->nv[0] : net->hscal[0];
  return MP_OK;
}

mp_status mp_net_train_step(mp_net_handle net, const float *target, float lr, int step,
                            double *loss_out) {
  if (!net || !target || step < 1 || !(lr > 0.f)) return MP_ERR_INVALID_ARG;
  const size_t n = net->nv[0];
  NCKS(forward(net));
  NCKS(loss_and_grad(net, target));
  NCKS(backward(net));
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)step), c2 = 1.f - std::pow(b2, (float)step);
  k_adam<<<grid_for(net->nparam), 256, 0, net->st>>>(net->param, net->grad, net->adam_m,
                                                     net->adam_v, net->nparam, lr, b1, b2, 1e-8f,
                                                     c1, c2);
  NCKS(pack_all(net));
  NCK(cudaMemcpyAsync(net->hscal, net->dscal + 2, sizeof(double), cudaMemcpyDeviceToHost,
                      net->st));
  NCKS(check_err(net));
  if (loss_out) *loss_out = net->loss_kind == 0 ? net->hscal[0] / (double)n : net->hscal[0];
  return MP_OK;
}

mp_status mp_net_train_step_grad(mp_net_handle net, const float *gq, float lr, int step) {
  if (!net || !gq || step < 1 || !(lr > 0.f)) return MP_ERR_INVALID_ARG;
  NCKS(forward(net));
  NCK(cudaMemcpyAsync(net->gq, gq, net->nv[0] * sizeof(float), cudaMemcpyDeviceToDevice,
                      net->st));
  NCKS(backward(net));
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - std::pow(b1, (float)step), c2 = 1.f - std::pow(b2, (float)step);
  k_adam<<<grid_for(net->nparam), 256, 0, net->st>>>(net->param, net->grad, net->adam_m,
                                                     net->adam_v, net->nparam, lr, b1, b2, 1e-8f,
                                                     c1, c2);
  NCKS(pack_all(net));
  NCK(cudaStreamSynchronize(net->st));
  return check_err(net);
}

mp_status mp_net_test_wait_timeout(int n) {
  if (n < 0) return MP_ERR_INVALID_ARG;
  g_wait_failures.store(n);
  return MP_OK;
}

void mp_net_destroy(mp_net_handle net) {
  if (!net) return;
  cudaStreamSynchronize(net->st);
  for (void *p : net->allocs) cudaFree(p);
  if (net->hscal) cudaFreeHost(net->hscal);
  ws_trim();
  delete net;
}

}  // extern "C"
