// Weight and bias gradient of the learned guess's 3x3x3 convolutions:
//   dw[co][tap cin + ci] += sum_v in[v + tap][ci] dy[v][co],   db[co] += sum_v dy[v][co]
// as products over voxels, straight from staged channels-last blocks.
//
// A CTA walks T^3 blocks of output voxels.  It stages the (T+2)^3 input block
// (up to three groups of 8 channels) and the block's dy (zero on the halo and
// outside the sample) in shared memory, one 16-byte row of 8 channels per
// position in raster order, so that a tap is a constant row shift and the
// whole block is one run of positions p: K.  The rows of the product are
// units of 8 channels of one tap, two units per 16-row tile, read by
// transposing matrix loads where they lie; one more unit of ones gives db.
// The warps share the staged block and split the row tiles.
//
// What bounds it is shared-memory reads: 16 bytes per position and unit.  The
// tensor instructions are warp-level ones: a tcgen05 tile has 64 or 128 rows
// at one stride, of which a tap has 8 per channel group (the three x taps at
// a stride of one row would fill 24 of 128), and its operands would be read
// five times over.  The form before, a 128-row tcgen05 tile gathered element
// by element from global memory, took 1054 us per layer of 8 to 16 output
// channels of a 96^3 pair (all eight layers 5.5 ms, and 138 us for the bias
// gradients); this one takes 62 and 31 us (331 us in all).
#include <cuda_bf16.h>

#include <algorithm>

#include "pm_kernels.cuh"
#include "tc_gemm.cuh"

namespace pm {

namespace {

using bf16 = __nv_bfloat16;
constexpr int WG_T = 8;                        // output block side
constexpr int WG_PX = WG_T + 2;
constexpr int WG_P = WG_PX * WG_PX * WG_PX;    // positions of the padded block
constexpr int WG_P0 = (WG_PX + 1) * WG_PX + 1;  // the first output's
constexpr int WG_LAST = (WG_T * WG_PX + WG_T) * WG_PX + WG_T;
constexpr int WG_CHUNKS = (WG_LAST - WG_P0 + 16) / 16;  // K in steps of 16 positions
// rows staged per channel group: a tap shift of the last step's last position
constexpr int WG_ROWS = (WG_P0 + 16 * WG_CHUNKS + WG_P0 + 7) / 8 * 8;
static_assert(WG_ROWS >= WG_P, "the padded block is staged whole");
constexpr int WG_NT = 256, WG_WARPS = WG_NT / 32;
constexpr int WG_Q = 6;    // row tiles per warp: 27 taps x 3 groups + 1 unit, two per tile
constexpr int WG_CG = 3;   // channel groups of the input a CTA takes at most
static_assert(WG_Q * WG_WARPS * 2 >= 27 * WG_CG + 1, "every unit has a warp");

__device__ __forceinline__ void wg_cp16(uint32_t smem, const void* gmem, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem), "l"(gmem),
               "r"(src_bytes)
               : "memory");
}
__device__ __forceinline__ void wg_ld4(uint32_t a, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void wg_ld2(uint32_t a, uint32_t& r0, uint32_t& r1) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void wg_mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0,
                                       uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// NT: groups of 8 output channels per CTA.  blockIdx.y: the input's channel
// groups [cg0, cg0 + cgp); blockIdx.z: the output's [8 NT z, ...).
template <int NT>
__global__ void __launch_bounds__(WG_NT) k_wgrad(const bf16* __restrict__ in, int B, int S,
                                                 int per, int cin, int cgp,
                                                 const bf16* __restrict__ dy, int cout,
                                                 float* __restrict__ dw,
                                                 float* __restrict__ db) {
  extern __shared__ __align__(16) uint8_t wg_sm[];
  // [cgp groups of the input][NT groups of dy][16 rows of ones]
  const uint32_t s0 = tc::smem_u32(wg_sm), row_bytes = 16u, grp = WG_ROWS * row_bytes;
  const uint32_t sdy = s0 + cgp * grp, sone = sdy + NT * grp;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cg0 = blockIdx.y * cgp, co0 = blockIdx.z * NT * 8;
  const int units = 27 * cgp + 1;  // the last one: ones
  // rows past the padded block (never staged) and the ones
  for (int t = tid; t < (cgp + NT) * (WG_ROWS - WG_P); t += WG_NT) {
    const int g = t / (WG_ROWS - WG_P), r = WG_P + t % (WG_ROWS - WG_P);
    *reinterpret_cast<uint4*>(wg_sm + g * grp + r * 16) = make_uint4(0, 0, 0, 0);
  }
  if (tid < 16) {
    const uint32_t one = 0x3f803f80u;  // two BF16 ones
    *reinterpret_cast<uint4*>(wg_sm + (cgp + NT) * grp + tid * 16) =
        make_uint4(one, one, one, one);
  }
  // this lane's row of the matrix loads: A loads units (2 tile, 2 tile + 1) x
  // positions (0-7, 8-15); their addresses step by 16 positions per K step
  uint32_t abase[WG_Q], ainc[WG_Q];
  bool on[WG_Q];
#pragma unroll
  for (int q = 0; q < WG_Q; ++q) {
    const int tile = warp + WG_WARPS * q;
    on[q] = 2 * tile < units;
    const int u = min(2 * tile + ((lane >> 3) & 1), units - 1);
    const int pos = ((lane >> 4) << 3) + (lane & 7);
    if (u == units - 1) {
      abase[q] = sone + pos * 16;
      ainc[q] = 0;
    } else {
      const int tap = u / cgp, c = u - tap * cgp;
      const int sh = (tap / 9 - 1) * WG_PX * WG_PX + (tap / 3 % 3 - 1) * WG_PX + tap % 3 - 1;
      abase[q] = s0 + c * grp + (WG_P0 + sh + pos) * 16;
      ainc[q] = 256;
    }
  }
  const uint32_t bbase = sdy + (WG_P0 + (lane & 15)) * 16;
  float acc[WG_Q][NT][4];
#pragma unroll
  for (int q = 0; q < WG_Q; ++q)
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[q][n][e] = 0.0f;

  const int tiles = (S + WG_T - 1) / WG_T;
  const long long nblk = (long long)B * tiles * tiles * tiles;
  for (long long blk = blockIdx.x; blk < nblk; blk += gridDim.x) {
    long long b = blk;
    const int tx = (int)(b % tiles); b /= tiles;
    const int ty = (int)(b % tiles); b /= tiles;
    const int tz = (int)(b % tiles);
    const long long sbase = b / tiles * S * S * S;
    const int x0 = tx * WG_T - 1, y0 = ty * WG_T - 1, z0 = tz * WG_T - 1;
    __syncthreads();  // the block before has been read
    for (int p = tid; p < WG_P; p += WG_NT) {
      const int x = p % WG_PX, y = p / WG_PX % WG_PX, z = p / (WG_PX * WG_PX);
      int gx = x0 + x, gy = y0 + y, gz = z0 + z;
      const bool out = x >= 1 && x <= WG_T && y >= 1 && y <= WG_T && z >= 1 && z <= WG_T &&
                       gx < S && gy < S && gz < S;
      if (per) {
        gx = gx < 0 ? gx + S : (gx >= S ? gx - S : gx);
        gy = gy < 0 ? gy + S : (gy >= S ? gy - S : gy);
        gz = gz < 0 ? gz + S : (gz >= S ? gz - S : gz);
      }
      const bool inside = gx >= 0 && gx < S && gy >= 0 && gy < S && gz >= 0 && gz < S;
      const long long v = inside ? sbase + ((long long)gz * S + gy) * S + gx : 0;
      for (int c = 0; c < cgp; ++c)
        wg_cp16(s0 + c * grp + p * 16, in + v * cin + 8 * (cg0 + c), inside ? 16 : 0);
#pragma unroll
      for (int n = 0; n < NT; ++n)
        wg_cp16(sdy + n * grp + p * 16, dy + (out ? v : 0) * cout + co0 + 8 * n, out ? 16 : 0);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_all;" ::: "memory");
    __syncthreads();
    uint32_t a[WG_Q];
#pragma unroll
    for (int q = 0; q < WG_Q; ++q) a[q] = abase[q];
#pragma unroll 2
    for (int k = 0; k < WG_CHUNKS; ++k) {
      uint32_t bf[NT][2];
#pragma unroll
      for (int n = 0; n < NT; ++n) wg_ld2(bbase + n * grp + k * 256, bf[n][0], bf[n][1]);
#pragma unroll
      for (int q = 0; q < WG_Q; ++q) {
        if (!on[q]) continue;  // the same for the whole warp
        uint32_t af[4];
        wg_ld4(a[q], af);
        a[q] += ainc[q];
#pragma unroll
        for (int n = 0; n < NT; ++n) wg_mma(acc[q][n], af, bf[n][0], bf[n][1]);
      }
    }
  }
  const int rows = 27 * cin;
#pragma unroll
  for (int q = 0; q < WG_Q; ++q) {
    if (!on[q]) continue;
#pragma unroll
    for (int n = 0; n < NT; ++n)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int u = 2 * (warp + WG_WARPS * q) + (e >> 1), ch = lane >> 2;
        const int co = co0 + 8 * n + 2 * (lane & 3) + (e & 1);
        if (u < units - 1) {
          const int tap = u / cgp, c = u - tap * cgp;
          atomicAdd(&dw[(long long)co * rows + tap * cin + 8 * (cg0 + c) + ch], acc[q][n][e]);
        } else if (u == units - 1 && ch == 0 && blockIdx.y == 0) {
          atomicAdd(&db[co], acc[q][n][e]);
        }
      }
  }
}

template <int NT>
cudaError_t wg_launch(cudaStream_t st, const void* in, int B, int S, int per, int cin, int cgp,
                      const void* dy, int cout, float* dw, float* db) {
  const int smem = (cgp + NT) * WG_ROWS * 16 + 256;
  // (the most that any launch takes, not this one's: another thread may set it
  // between the setting and the launch)
  const cudaError_t e =
      cudaFuncSetAttribute(k_wgrad<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (WG_CG + NT) * WG_ROWS * 16 + 256);
  if (e != cudaSuccess) return e;
  const long long t = (S + WG_T - 1) / WG_T, nblk = t * t * t * B;
  const int gy = cin / 8 / cgp, gz = cout / 8 / NT;
  // as many CTAs as the staged blocks leave room for (shared memory), at
  // least a block each
  const int per_sm = std::max(1, std::min(6, 220 * 1024 / smem));
  const int gx = (int)std::min<long long>(nblk, std::max(1, 152 * per_sm / (gy * gz)));
  k_wgrad<NT><<<dim3(gx, gy, gz), WG_NT, smem, st>>>((const bf16*)in, B, S, per, cin, cgp,
                                                      (const bf16*)dy, cout, dw, db);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

// cin, cout: multiples of 8 (the network's 8 to 96 and 8 to 64)
cudaError_t launch_wgrad(cudaStream_t st, const void* in, int B, int S, int per, int cin,
                         const void* dy, int cout, float* dw, float* db) {
  const int g = cin / 8, cgp = g % 3 == 0 ? 3 : (g % 2 == 0 ? 2 : 1);
  const int n = cout / 8;
  if (n % 4 == 0) return wg_launch<4>(st, in, B, S, per, cin, cgp, dy, cout, dw, db);
  if (n % 2 == 0) return wg_launch<2>(st, in, B, S, per, cin, cgp, dy, cout, dw, db);
  return wg_launch<1>(st, in, B, S, per, cin, cgp, dy, cout, dw, db);
}

}  // namespace pm
