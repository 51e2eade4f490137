// The 3x3x3 "same" convolutions of the learned guess (forward, and the input
// gradient with the taps reversed) as an implicit
// GEMM on the 5th-generation tensor cores without an im2col copy.
//
// A CTA computes a tx x ty x tz block of output voxels of one sample.  It
// stages the input block with its halo once in shared memory, channel-blocked: block c holds
// channels 8c .. 8c+7 of every position as one 16-byte row, positions in
// raster order of the padded block (x fastest).  In the K-major no-swizzle
// canonical layout an MMA operand of 128 rows x 16 K-elements is two
// 8-element core-matrix columns, each 128 rows of 16 bytes at a common row
// stride of 16 bytes; so the A operand of tap (dz, dy, dx) for 128
// consecutive positions is the staged block itself, started
// ((dz-1) P_y P_x + (dy-1) P_x + (dx-1)) rows further on, with the second core
// column one channel block further (LBO = the block stride), or, for 8
// input channels, at the next tap (LBO = that tap's extra shift).  Every
// (tap, channel pair) is one tcgen05.mma issued straight from the staged
// input; the positions of a 128-row M tile that fall on the block's halo
// or outside the sample are computed and discarded.  All M tiles of the
// block accumulate in tensor memory at once; one commit, one bounded wait,
// then the epilogue (bias, ReLU, BF16 / FP32) reads TMEM row by row.
//
// A decoder layer's input is the coarser level upsampled (nearest, the first
// cup channels) beside the encoder's output: where nothing else needs the
// concatenated tensor, both are staged from where they lie (up, cup; 160^3
// forward: 168 us of upsampling and copies less).
//
// Weights: wf [N][K] BF16, K = 28 taps x 8 (8 input channels: taps in pairs,
// the 28th zero) or 27 taps x cinp (cinp = cin rounded up to 16; channels
// beyond cin zero), tap-major, loaded whole into shared memory.
#include <cuda_bf16.h>

#include <algorithm>

#include "pm_kernels.cuh"
#include "tc_gemm.cuh"

namespace pm {

namespace {

using bf16 = __nv_bfloat16;
constexpr long long CF_WAIT_LIMIT = 20000000;  // mbarrier polls before giving up
// Threads per CTA: two for each TMEM lane.  Staging and the epilogue, not the
// MMAs, take most of a block's time (160^3, 8 -> 8: 98 MMAs, 2700
// instructions a warp), and the layers of many channels have room for one
// CTA per SM (the five layers of 16 columns of a 160^3 forward: 1283 us; 1451
// with 128 threads).
constexpr int CF_NT = 256;
constexpr int CF_SLACK = 128;                  // rows past a block's end an M tile may touch
constexpr int CF_MAXK = 192;                   // K slices of 16 a layer may have

// q = x / d, r = x % d for 0 <= x < 2^22, 1 <= d <= 4096, from a float
// reciprocal (its error is below one, so one correction step suffices)
__device__ __forceinline__ void cf_divmod(int x, int d, float inv_d, int& q, int& r) {
  q = (int)((float)x * inv_d);
  r = x - q * d;
  if (r < 0) { --q; r += d; }
  else if (r >= d) { ++q; r -= d; }
}

// 16-byte asynchronous copy global -> shared; src_bytes 0 fills zeros
__device__ __forceinline__ void cf_cp16(uint8_t* smem, const void* gmem, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(tc::smem_u32(smem)),
               "l"(gmem), "r"(src_bytes)
               : "memory");
}

struct CfShape {
  int tx, ty, tz;  // output block
  int px, py;      // sides of the padded block, tx + 2 and ty + 2
  int P;           // positions of the padded block
  int nbr;         // channel blocks staged (cin / 8)
  int cbs;         // bytes between channel blocks (P + slack rows)
  int mt;          // M tiles of 128 positions
  int p0;          // position of the first output
  int kf;          // K of wf
  int ncols;       // TMEM columns allocated (power of two >= mt N)
  int smem;        // dynamic shared memory bytes
};

__host__ __device__ inline CfShape cf_shape(int tx, int ty, int tz, int cin, int n) {
  CfShape s{};
  const int px = tx + 2, py = ty + 2;
  s.tx = tx;
  s.ty = ty;
  s.tz = tz;
  s.px = px;
  s.py = py;
  s.P = px * py * (tz + 2);
  s.nbr = cin / 8;
  s.cbs = (s.P + CF_SLACK) * 16;
  s.p0 = (py + 1) * px + 1;
  const int last = (tz * py + ty) * px + tx;  // position of the last output
  s.mt = (last - s.p0 + 1 + 127) / 128;
  s.kf = cin == 8 ? 28 * 8 : 27 * ((cin + 15) / 16 * 16);
  int need = s.mt * n, c = 32;
  while (c < need) c *= 2;
  s.ncols = c;
  s.smem = s.nbr * s.cbs + n * s.kf * 2 + 1024;
  return s;
}

template <int N>
__global__ void __launch_bounds__(CF_NT) k_conv_fast(const bf16* __restrict__ in, int B, int S,
                                                     int per, int cin,
                                                     const bf16* __restrict__ wf, CfShape sh,
                                                     const float* __restrict__ bias, int cout,
                                                     int relu, bf16* __restrict__ out_bf,
                                                     float* __restrict__ out_f, int* err,
                                                     const bf16* __restrict__ up, int cup) {
  extern __shared__ __align__(1024) uint8_t cf_sm[];
  __shared__ uint32_t tslot;
  __shared__ __align__(8) uint64_t mbar_s;
  // the A and B descriptors of every K slice for the first M tile (the
  // next tiles start 128 rows, i.e. 2048 bytes = 128 descriptor units, on)
  __shared__ uint64_t adesc[CF_MAXK], bdesc[CF_MAXK];
  __shared__ float sbias[N];
  if (threadIdx.x < N)
    sbias[threadIdx.x] = bias && (int)threadIdx.x < cout ? bias[threadIdx.x] : 0.0f;
  // 1 KB-aligned start of the staged input; the weights follow the blocks
  uint8_t* sA = cf_sm + ((1024 - (tc::smem_u32(cf_sm) & 1023)) & 1023);
  uint8_t* sB = sA + sh.nbr * sh.cbs;
  const int px = sh.px, py = sh.py;
  int bid = blockIdx.x;
  const int nx = (S + sh.tx - 1) / sh.tx, ny = (S + sh.ty - 1) / sh.ty;
  const int nz = (S + sh.tz - 1) / sh.tz;
  // sample coordinates of position 0
  const int x0 = (bid % nx) * sh.tx - 1; bid /= nx;
  const int y0 = (bid % ny) * sh.ty - 1; bid /= ny;
  const int z0 = (bid % nz) * sh.tz - 1;
  const int smp = bid / nz;
  const long long sbase = (long long)smp * S * S * S;

  if (threadIdx.x < 32) tc::tmem_alloc(&tslot, sh.ncols);
  const uint32_t mbar = tc::smem_u32(&mbar_s);
  if (threadIdx.x == 0) tc::mbar_init(mbar, 1);

  // weights: row n, 16-byte group g of K in the canonical layout
  const int kg = sh.kf / 8;
  for (int t = threadIdx.x; t < N * kg; t += CF_NT) {
    const int n = t / kg, g = t - n * kg;
    *reinterpret_cast<uint4*>(sB + (n >> 3) * (sh.kf * 16) + g * 128 + (n & 7) * 16) =
        *reinterpret_cast<const uint4*>(wf + (long long)n * sh.kf + 8 * g);
  }
  // the padded input block, channel-blocked, by asynchronous 16-byte copies
  // (zero-filled outside an open sample, wrapped in a periodic one); the
  // slack rows are zeroed
  const int rows = sh.nbr * sh.P;
  const float inv_px = 1.0f / (float)px, inv_py = 1.0f / (float)py, inv_p = 1.0f / (float)sh.P;
  for (int t = threadIdx.x; t < rows; t += CF_NT) {
    int c, p, x, y, z, r;
    cf_divmod(t, sh.P, inv_p, c, p);
    cf_divmod(p, px, inv_px, r, x);
    cf_divmod(r, py, inv_py, z, y);
    int gx = x0 + x, gy = y0 + y, gz = z0 + z;
    if (per) {
      gx = gx < 0 ? gx + S : (gx >= S ? gx - S : gx);
      gy = gy < 0 ? gy + S : (gy >= S ? gy - S : gy);
      gz = gz < 0 ? gz + S : (gz >= S ? gz - S : gz);
    }
    const bool inside = gx >= 0 && gx < S && gy >= 0 && gy < S && gz >= 0 && gz < S;
    const bf16* src = in;
    if (8 * c < cup) {
      const int h = S >> 1;
      const long long vx = ((long long)(smp * h + (gz >> 1)) * h + (gy >> 1)) * h + (gx >> 1);
      if (inside) src = up + vx * cup + 8 * c;
    } else if (inside) {
      src = in + (sbase + ((long long)gz * S + gy) * S + gx) * (cin - cup) + (8 * c - cup);
    }
    cf_cp16(sA + c * sh.cbs + p * 16, src, inside ? 16 : 0);
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int t = threadIdx.x; t < sh.nbr * CF_SLACK; t += CF_NT) {
    const int c = t / CF_SLACK, r = t - c * CF_SLACK;
    *reinterpret_cast<uint4*>(sA + c * sh.cbs + (sh.P + r) * 16) = make_uint4(0, 0, 0, 0);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  const int nk = sh.kf / 16;  // MMAs per M tile
  {
    const uint32_t a0 = tc::smem_u32(sA), b0 = tc::smem_u32(sB);
    const uint32_t sbo_b = (uint32_t)sh.kf * 16u;
    const int cinp = cin == 8 ? 8 : (cin + 15) / 16 * 16;
    for (int s = threadIdx.x; s < nk; s += CF_NT) {
      uint32_t a, lbo;
      if (cin == 8) {
        // taps 2s and 2s + 1 (the 28th tap has zero weights: any rows)
        const int t0 = 2 * s, t1 = 2 * s + 1;
        const int sh0 = (t0 / 9 - 1) * px * py + ((t0 / 3) % 3 - 1) * px + (t0 % 3 - 1);
        const int sh1 = t1 < 27 ? (t1 / 9 - 1) * px * py + ((t1 / 3) % 3 - 1) * px + (t1 % 3 - 1)
                                : sh0;
        a = a0 + (uint32_t)(sh.p0 + sh0) * 16u;
        lbo = (uint32_t)(sh1 - sh0) * 16u;
      } else {
        // tap s / (cinp / 16), channel blocks 2j and 2j + 1 (a block past the
        // staged ones has zero weights: it re-reads block 2j)
        const int per_tap = cinp / 16;
        const int t = s / per_tap, j = s - t * per_tap;
        const int sht = (t / 9 - 1) * px * py + ((t / 3) % 3 - 1) * px + (t % 3 - 1);
        a = a0 + (uint32_t)(2 * j) * (uint32_t)sh.cbs + (uint32_t)(sh.p0 + sht) * 16u;
        lbo = 2 * j + 1 < sh.nbr ? (uint32_t)sh.cbs : 0u;
      }
      adesc[s] = tc::smem_desc(a, lbo, 128u);
      bdesc[s] = tc::smem_desc(b0 + 256u * (uint32_t)s, 128u, sbo_b);
    }
  }
  tc::fence_async_smem();
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t taddr = tslot;

  if (threadIdx.x == 0) {
    constexpr uint32_t IDESC = tc::idesc_bf16(tc::TM, N);
    for (int m = 0; m < sh.mt; ++m) {
      const uint64_t step = (uint64_t)(128 * m);  // 128 rows of 16 bytes, in 16-byte units
      for (int s = 0; s < nk; ++s)
        tc::mma_bf16(taddr + (uint32_t)(m * N), adesc[s] + step, bdesc[s], IDESC,
                     s > 0 ? 1u : 0u);
    }
    tc::mma_commit(mbar);
  }
  // the block decides together whether the MMAs completed
  const bool ok = __syncthreads_and(tc::mbar_wait(mbar, 0u, CF_WAIT_LIMIT)) != 0;
  if (!ok) {
    if (threadIdx.x == 0) atomicOr(err, 1);
    tc::mbar_wait(mbar, 0u, CF_WAIT_LIMIT);  // one more bounded wait before leaving
  } else {
    tc::tc_fence_after();
    // a warp reads the TMEM lanes 32 (w % 4) .. + 31; the two halves of the
    // CTA take the M tiles in turn
    const int w = (threadIdx.x >> 5) & 3, lane = threadIdx.x & 31;
    const int coutp = (cout + 7) & ~7;
    for (int m = threadIdx.x >> 7; m < sh.mt; m += CF_NT / 128) {
      const int p = sh.p0 + 128 * m + 32 * w + lane;
      int x, y, z, r;
      cf_divmod(p, px, inv_px, r, x);
      cf_divmod(r, py, inv_py, z, y);
      const int gx = x0 + x, gy = y0 + y, gz = z0 + z;
      const bool valid = x >= 1 && x <= sh.tx && y >= 1 && y <= sh.ty && z >= 1 &&
                         z <= sh.tz && gx < S && gy < S && gz < S;
      const long long row = sbase + ((long long)gz * S + gy) * S + gx;
#pragma unroll
      for (int col = 0; col < N; col += 8) {
        if (col >= coutp) break;
        float val[8];
        tc::tmem_ld8(taddr, w, m * N + col, val);
        if (valid) {
          __align__(16) bf16 ob[8];
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            float o = col + q < cout ? val[q] + sbias[col + q] : 0.0f;
            if (relu) o = fmaxf(o, 0.0f);
            ob[q] = __float2bfloat16_rn(o);
            if (out_f && col + q == 0) out_f[row] = o;  // (channel 0 only)
          }
          if (out_bf)
            *reinterpret_cast<uint4*>(out_bf + row * coutp + col) =
                *reinterpret_cast<const uint4*>(ob);
        }
      }
    }
  }
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (threadIdx.x < 32) tc::tmem_free(taddr, sh.ncols);
}

// wf[n][k] from the FP32 masters w[co][tap * cin + ci] (see the file head).
// bwd: the operand of the input gradient, a convolution of the output's
// gradient (co channels in, ci out) with the taps reversed.
__global__ void k_pack_wf(const float* __restrict__ w, int cin, int cout, int n, int kf,
                          bool bwd, bf16* __restrict__ wf) {
  const int c = bwd ? (cout + 7) / 8 * 8 : cin;  // channels of the convolved tensor
  const int cinp = c == 8 ? 8 : (c + 15) / 16 * 16;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * kf; t += gridDim.x * blockDim.x) {
    const int r = t / kf, k = t - r * kf;
    const int tap = k / cinp, ci = k - tap * cinp;
    float v = 0.0f;
    if (!bwd) {
      if (r < cout && tap < 27 && ci < cin) v = w[(long long)r * 27 * cin + tap * cin + ci];
    } else if (r < cin && tap < 27 && ci < cout) {  // (row: input channel, ci: output channel)
      v = w[(long long)ci * 27 * cin + (26 - tap) * cin + r];
    }
    wf[t] = __float2bfloat16_rn(v);
  }
}

constexpr int CF_SMEM_MAX = 200 * 1024;

// the most that any launch takes, not this one's: another thread may set it
// between the setting and the launch
template <int N>
bool cf_set_attr() {
  return cudaFuncSetAttribute(k_conv_fast<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              CF_SMEM_MAX) == cudaSuccess;
}

long long cf_blocks(const CfShape& s, int B, int S) {
  return (long long)B * ((S + s.tx - 1) / s.tx) * ((S + s.ty - 1) / s.ty) *
         ((S + s.tz - 1) / s.tz);
}

// The block for B samples of side S.  An MMA of 128 rows hardly depends on its
// columns (39, 40, 44, 48 cycles an SM for 16, 32, 48, 64 in chains of several
// CTAs, 50 in one CTA alone), and an M tile's rows on the halo are lost: 8^3
// blocks (57 % of the rows are outputs) against 16 x 16 x 2 or 20 x 10 x 2
// (80 %).  So of the blocks that fit, the one whose busiest SM takes the
// fewest cycles by a model of MMAs, staged 16-byte pieces and a start per
// block, the two overlapped where several blocks share an SM.  Its weights
// (64, 1.2, 2000, 0.25) are chosen by whole passes and matter little: from 39
// to 64, 0.8 to 1.8, 1000 to 4000 and 0 to 1 a forward or backward pass at ten
// sides of 32 to 192 moved by 5 % at most.  Every block gives a voxel the same
// MMAs in the same order: the same bits.  160^3 forward, layers of 16 columns:
// 1283 us with 8^3 blocks, 996 so.
CfShape cf_choose(int B, int S, int cin, int n, int T) {
  struct Entry {
    int B, S, cin, n;
    CfShape sh;
  };
  thread_local Entry memo[16];  // (a function of its key alone)
  thread_local int next = 0;
  for (const Entry& e : memo)
    if (e.B == B && e.S == S && e.cin == cin && e.n == n) return e.sh;
  T = std::min(T, S);  // a block never larger than the sample
  CfShape best{};
  double best_cost = 0.0;
  auto offer = [&](int x, int y, int z) {
    const CfShape s = cf_shape(x, y, z, cin, n);
    if (s.smem > CF_SMEM_MAX || s.mt * n > 128) return;
    const int occ = std::min(512 / s.ncols, 227 * 1024 / (s.smem + 5 * 1024));
    const double per_sm = (double)((cf_blocks(s, B, S) + 151) / 152);
    const double mma = 64.0 * s.mt * (s.kf / 16);
    const double stage = 1.2 * s.nbr * s.P + 1.2 * n * (s.kf / 8) + 2000.0;
    const double one = occ >= 2 && per_sm >= 2.0
                           ? std::max(mma, stage) + 0.25 * std::min(mma, stage)
                           : mma + stage;
    if (best.P == 0 || per_sm * one < best_cost) {
      best = s;
      best_cost = per_sm * one;
    }
  };
  offer(T, T, T);
  for (int x : {8, 10, 12, 14, 16, 20, 24, 32})
    for (int y : {4, 6, 8, 10, 12, 14, 16})
      for (int z : {1, 2, 4, 6, 8})
        if (x <= S && y <= S && z <= S) offer(x, y, z);
  memo[next] = Entry{B, S, cin, n, best};
  next = (next + 1) % 16;
  return best;
}

}  // namespace

int conv_fast_kf(int cin);

// The side of a cubic block for a layer (cf_choose starts from it), or 0 when
// the staged block and the weights do not fit in shared memory or the
// accumulators in 128 TMEM columns (four CTAs per SM) at any side >= 4.
int conv_fast_side(int cin, int cout) {
  if (cin % 8 != 0 || conv_fast_kf(cin) / 16 > CF_MAXK) return 0;
  const int n = cout <= 16 ? 16 : (cout + 15) / 16 * 16;
  if (n != 16 && n != 32 && n != 48 && n != 64) return 0;
  for (int T = 14; T >= 4; --T) {
    const CfShape s = cf_shape(T, T, T, cin, n);
    if (s.smem <= CF_SMEM_MAX && s.mt * n <= 128) return T;
  }
  return 0;
}

int conv_fast_kf(int cin) { return cin == 8 ? 28 * 8 : 27 * ((cin + 15) / 16 * 16); }

void launch_pack_wf(cudaStream_t st, const float* w, int cin, int cout, int n, bool bwd,
                    void* wf) {
  const int kf = conv_fast_kf(bwd ? (cout + 7) / 8 * 8 : cin);
  k_pack_wf<<<(n * kf + 255) / 256, 256, 0, st>>>(w, cin, cout, n, kf, bwd, (bf16*)wf);
  note_launch();
}

bool launch_conv_fast(cudaStream_t st, const void* in, int B, int S, int per, int cin,
                      const void* wf, int n, int T, const float* bias, int cout, int relu,
                      void* out_bf, float* out_f, int* err, const void* up, int cup) {
  const CfShape sh = cf_choose(B, S, cin, n, T);
  const dim3 grid((unsigned)cf_blocks(sh, B, S));
#define PM_CF(NN)                                                                       \
  if (!cf_set_attr<NN>()) return false;                                                 \
  k_conv_fast<NN><<<grid, CF_NT, sh.smem, st>>>((const bf16*)in, B, S, per, cin,          \
                                                 (const bf16*)wf, sh, bias, cout, relu,    \
                                                 (bf16*)out_bf, out_f, err,                \
                                                 (const bf16*)up, cup)
  switch (n) {
    case 16: PM_CF(16); break;
    case 32: PM_CF(32); break;
    case 48: PM_CF(48); break;
    case 64: PM_CF(64); break;
    default: return false;
  }
#undef PM_CF
  note_launch();
  return true;
}

}  // namespace pm
