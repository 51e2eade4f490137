// Learned initial guess: BF16 tensor-core (tcgen05, TMEM accumulator)
// kernels of a small 3-D convolutional network and its training.
//
//   * k_gemm_tc      plain C = A B^T (validation of the tile engine)
//   * k_conv_fwd     implicit-GEMM 3x3x3 "same" convolution, channels-last
//                    activations; M = 128 voxels, N = output channels,
//                    K = 27 * input channels (im2col gathered into shared
//                    memory), FP32 accumulation, bias + optional ReLU,
//                    BF16 and/or FP32 output
//   * elementwise    ReLU backward, 2x average pooling / nearest upsampling
//                    (and their backward), channel concatenation, MSE, Adam
// The input-gradient of a convolution is the forward convolution of the
// output-gradient with mirrored, transposed weights (k_pack_w).
#include <cuda_bf16.h>

#include "pm_kernels.cuh"
#include "tc_gemm.cuh"

namespace pm {

using bf16 = __nv_bfloat16;
constexpr long long TC_WAIT_LIMIT = 20000000;  // mbarrier polls before giving up

// ---------------------------------------------------------------------------
// Shared tile loop.  FillA(kt, sA) / FillB(kt, sB) stage K-chunk kt (KC wide)
// of A (128 rows) and B (N rows) into shared memory in the canonical layout;
// the loop issues KC/16 MMAs per chunk from one thread and waits on the
// mbarrier before the next chunk reuses the buffers.  Returns false on a
// timed-out wait (the error word is set; the caller still frees TMEM).
// ---------------------------------------------------------------------------
// the KC / 16 MMAs of one chunk and their commit (one thread)
template <int N, int KC>
__device__ __forceinline__ void tc_chunk(uint32_t taddr, uint8_t* sA, uint8_t* sB, uint32_t mbar,
                                         bool accumulate) {
  constexpr uint32_t IDESC = tc::idesc_bf16(tc::TM, N);
  constexpr uint32_t SBO = KC * 16;
  const uint32_t a0 = tc::smem_u32(sA), b0 = tc::smem_u32(sB);
#pragma unroll
  for (int s = 0; s < KC / 16; ++s) {
    uint64_t ad = tc::smem_desc(a0 + 256u * s, 128u, SBO);
    uint64_t bd = tc::smem_desc(b0 + 256u * s, 128u, SBO);
    tc::mma_bf16(taddr, ad, bd, IDESC, (accumulate || s > 0) ? 1u : 0u);
  }
  tc::mma_commit(mbar);
}

// The block waits for a committed chunk (bounded); false on a timed-out wait.
__device__ __forceinline__ bool tc_chunk_wait(uint32_t mbar, uint32_t& phase, int* err) {
  // every thread polls, but the block decides together: a thread whose
  // polls ran out just before the commit landed must not leave the loop
  // while the others go on (mismatched barriers, a diverged tcgen05.dealloc)
  const bool done = __syncthreads_and(tc::mbar_wait(mbar, phase, TC_WAIT_LIMIT)) != 0;
  phase ^= 1u;
  if (!done) {
    if (threadIdx.x == 0) atomicOr(err, 1);
    // give the MMAs one more bounded wait before the buffers are left
    tc::mbar_wait(mbar, phase ^ 1u, TC_WAIT_LIMIT);
    return false;
  }
  tc::tc_fence_after();
  return true;
}

template <int N, int KC, class FillA, class FillB>
__device__ bool tc_mainloop(FillA fa, FillB fb, int ktiles, uint32_t taddr, uint8_t* sA,
                            uint8_t* sB, uint32_t mbar, uint32_t& phase, int* err) {
  for (int kt = 0; kt < ktiles; ++kt) {
    fa(kt, sA);
    fb(kt, sB);
    tc::fence_async_smem();
    __syncthreads();
    tc::tc_fence_after();
    if (threadIdx.x == 0) tc_chunk<N, KC>(taddr, sA, sB, mbar, kt > 0);
    if (!tc_chunk_wait(mbar, phase, err)) return false;
    __syncthreads();
  }
  return true;
}

// Shared setup/teardown around a tile: TMEM allocation by warp 0, mbarrier.
struct TcCtx {
  uint32_t taddr;
  uint32_t mbar;
};

template <int NCOLS>
__device__ __forceinline__ TcCtx tc_begin(uint32_t* tslot, uint64_t* mbar_slot) {
  if (threadIdx.x < 32) tc::tmem_alloc(tslot, NCOLS);
  if (threadIdx.x == 0) tc::mbar_init(tc::smem_u32(mbar_slot), 1);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  return TcCtx{*tslot, tc::smem_u32(mbar_slot)};
}

template <int NCOLS>
__device__ __forceinline__ void tc_end(const TcCtx& c) {
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  if (threadIdx.x < 32) tc::tmem_free(c.taddr, NCOLS);
}

// Copy rows x (KC/8) 16-byte vectors into the canonical tile; vec(r, v)
// returns the 8 bf16 of row r, K columns [8v, 8v + 8) as a uint4.
template <int KC, class Vec>
__device__ __forceinline__ void fill_tile(uint8_t* s, int rows, Vec vec) {
  constexpr int VPR = KC / 8;
  for (int idx = threadIdx.x; idx < rows * VPR; idx += blockDim.x) {
    int r = idx / VPR, v = idx - r * VPR;
    *reinterpret_cast<uint4*>(s + tc::tile_offset(r, 8 * v, KC)) = vec(r, v);
  }
}

// ---------------------------------------------------------------------------
// Plain GEMM C[M x N] = A[M x K] B[N x K]^T (row-major bf16 inputs, FP32 C).
// M % 128 == 0, K % 64 == 0.
// ---------------------------------------------------------------------------
template <int N>
__global__ void __launch_bounds__(128) k_gemm_tc(const bf16* __restrict__ A,
                                                 const bf16* __restrict__ B,
                                                 float* __restrict__ C, int M, int K,
                                                 int* err) {
  constexpr int KC = 64;
  __shared__ __align__(1024) uint8_t sA[tc::TM * KC * 2];
  __shared__ __align__(1024) uint8_t sB[N * KC * 2];
  __shared__ uint32_t tslot;
  __shared__ __align__(8) uint64_t mbar;
  constexpr int NC = tc::tmem_cols(N);
  TcCtx c = tc_begin<NC>(&tslot, &mbar);
  const int m0 = blockIdx.x * tc::TM;
  uint32_t phase = 0;
  auto fa = [&](int kt, uint8_t* s) {
    fill_tile<KC>(s, tc::TM, [&](int r, int v) {
      return *reinterpret_cast<const uint4*>(A + (long long)(m0 + r) * K + kt * KC + 8 * v);
    });
  };
  auto fb = [&](int kt, uint8_t* s) {
    fill_tile<KC>(s, N, [&](int r, int v) {
      return *reinterpret_cast<const uint4*>(B + (long long)r * K + kt * KC + 8 * v);
    });
  };
  bool ok = tc_mainloop<N, KC>(fa, fb, K / KC, c.taddr, sA, sB, c.mbar, phase, err);
  if (ok) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int row = m0 + 32 * w + lane;
#pragma unroll
    for (int col = 0; col < N; col += 8) {
      float v[8];
      tc::tmem_ld8(c.taddr, w, col, v);
#pragma unroll
      for (int q = 0; q < 8; ++q) C[(long long)row * N + col + q] = v[q];
    }
  }
  tc_end<NC>(c);
}

// Failure-detection self-test of the bounded mbarrier wait the tensor-core
// kernels use: one warp initialises an mbarrier for one arrival; with
// arrive = 1 a thread arrives and the wait completes, otherwise nothing
// arrives and the wait gives up after `limit` polls, setting *gave_up.
// Nothing asynchronous is in flight in either case.
__global__ void k_wait_selftest(int arrive, long long limit, int* gave_up) {
  __shared__ __align__(8) unsigned long long bar;
  const uint32_t mbar = tc::smem_u32(&bar);
  if (threadIdx.x == 0) tc::mbar_init(mbar, 1);
  __syncthreads();
  if (arrive && threadIdx.x == 0) {
    unsigned long long state;
    asm volatile("mbarrier.arrive.shared::cta.b64 %0, [%1];" : "=l"(state) : "r"(mbar) : "memory");
  }
  const bool done = tc::mbar_wait(mbar, 0u, limit);
  if (!done && threadIdx.x == 0) atomicOr(gave_up, 1);
}

void launch_wait_selftest(cudaStream_t st, int arrive, long long limit, int* gave_up) {
  k_wait_selftest<<<1, 32, 0, st>>>(arrive, limit, gave_up);
  note_launch();
}

void launch_gemm_tc(cudaStream_t st, const void* A, const void* B, float* C, int M, int N,
                    int K, int* err) {
  dim3 grid(M / tc::TM);
  switch (N) {
    case 16: k_gemm_tc<16><<<grid, 128, 0, st>>>((const bf16*)A, (const bf16*)B, C, M, K, err); break;
    case 32: k_gemm_tc<32><<<grid, 128, 0, st>>>((const bf16*)A, (const bf16*)B, C, M, K, err); break;
    case 64: k_gemm_tc<64><<<grid, 128, 0, st>>>((const bf16*)A, (const bf16*)B, C, M, K, err); break;
    case 128: k_gemm_tc<128><<<grid, 128, 0, st>>>((const bf16*)A, (const bf16*)B, C, M, K, err); break;
    default: return;
  }
  note_launch();
}

// ---------------------------------------------------------------------------
// Activations: channels-last BF16 tensors [B][D][H][W][C], C % 8 == 0.
// ---------------------------------------------------------------------------
struct Vol {
  int B, D, H, W;  // samples and spatial extent
  int per = 0;     // convolutions wrap around each sample (else zero padding)
  __host__ __device__ long long voxels() const { return (long long)B * D * H * W; }
};

// 3x3x3 "same" convolution, out[v][co] = bias[co] + sum_tap,ci in[v+tap][ci] w[co][tap*cin+ci]
// (zero outside each sample, or periodic when g.per), as a GEMM: rows = 128 voxels, N = output
// columns (>= cout, multiple of 16), K = 27 cin padded to 64.
// wp: [N][kp] BF16, rows >= cout and columns >= 27 cin zero.
//
// It runs for the layers with many channels, on coarse levels with a few
// hundred tiles at most: a tile's chain of K chunks (41 for 96 channels)
// bounds it.  The next chunk's 16-byte pieces are therefore loaded into
// registers while the MMAs of this one run, and eight lanes take eight rows
// of one core matrix (conflict-free stores) with the warp on 64 contiguous
// bytes of each voxel; a thread per voxel had every lane of a load on its own
// line.  96 -> 32 channels at 40^3: 221 -> 114 us.
template <int N>
__global__ void __launch_bounds__(128) k_conv_fwd(const bf16* __restrict__ in, Vol g, int cin,
                                                  const bf16* __restrict__ wp, int kp,
                                                  const float* __restrict__ bias, int cout,
                                                  int relu, bf16* __restrict__ out_bf,
                                                  float* __restrict__ out_f, int* err) {
  constexpr int KC = 64, NB = N / 16;
  __shared__ __align__(1024) uint8_t sA[tc::TM * KC * 2];
  __shared__ __align__(1024) uint8_t sB[N * KC * 2];
  __shared__ int4 srow[tc::TM];  // x, y, z, sample of the tile's rows (sample -1: none)
  __shared__ uint32_t tslot;
  __shared__ __align__(8) uint64_t mbar;
  constexpr int NC = tc::tmem_cols(N);
  const long long nvox = g.voxels();
  const long long m0 = (long long)blockIdx.x * tc::TM;
  {
    const long long v = m0 + threadIdx.x;
    int4 c = make_int4(0, 0, 0, -1);
    if (v < nvox) {
      long long t = v;
      c.x = (int)(t % g.W); t /= g.W;
      c.y = (int)(t % g.H); t /= g.H;
      c.z = (int)(t % g.D);
      c.w = (int)(t / g.D);
    }
    srow[threadIdx.x] = c;
  }
  TcCtx c = tc_begin<NC>(&tslot, &mbar);  // (its barrier covers srow)
  // piece q of a thread: row 8 (4 (q >> 1) + warp) + (lane & 7), 8 K columns
  // from 8 ((q & 1) 4 + (lane >> 3))
  const int warp = threadIdx.x >> 5, lane8 = threadIdx.x & 7, vv0 = (threadIdx.x & 31) >> 3;
  uint4 ra[8], rb[NB];
  auto load = [&](int kt) {
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int k = kt * KC + 8 * (4 * h + vv0);
      const int tap = k / cin, ci = k - tap * cin;
      const int dz = tap / 9 - 1, dy = (tap / 3) % 3 - 1, dx = tap % 3 - 1;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int4 r = srow[8 * (4 * q + warp) + lane8];
        uint4 val = make_uint4(0, 0, 0, 0);
        int zz = r.z + dz, yy = r.y + dy, xx = r.x + dx;
        if (g.per) {
          zz = zz < 0 ? zz + g.D : (zz >= g.D ? zz - g.D : zz);
          yy = yy < 0 ? yy + g.H : (yy >= g.H ? yy - g.H : yy);
          xx = xx < 0 ? xx + g.W : (xx >= g.W ? xx - g.W : xx);
        }
        if (r.w >= 0 && tap < 27 && zz >= 0 && zz < g.D && yy >= 0 && yy < g.H && xx >= 0 &&
            xx < g.W) {
          const long long nv = (((long long)r.w * g.D + zz) * g.H + yy) * g.W + xx;
          val = *reinterpret_cast<const uint4*>(in + nv * cin + ci);
        }
        ra[2 * q + h] = val;
      }
    }
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int idx = threadIdx.x + 128 * q;
      const int r = (idx & 7) + 8 * (idx >> 6), vv = (idx >> 3) & 7;
      rb[q] = *reinterpret_cast<const uint4*>(wp + (long long)r * kp + kt * KC + 8 * vv);
    }
  };
  auto store = [&]() {
#pragma unroll
    for (int q = 0; q < 8; ++q)
      *reinterpret_cast<uint4*>(sA + tc::tile_offset(8 * (4 * (q >> 1) + warp) + lane8,
                                                     8 * (4 * (q & 1) + vv0), KC)) = ra[q];
#pragma unroll
    for (int q = 0; q < NB; ++q) {
      const int idx = threadIdx.x + 128 * q;
      const int r = (idx & 7) + 8 * (idx >> 6), vv = (idx >> 3) & 7;
      *reinterpret_cast<uint4*>(sB + tc::tile_offset(r, 8 * vv, KC)) = rb[q];
    }
  };
  const int ktiles = kp / KC;
  uint32_t phase = 0;
  bool ok = true;
  load(0);
  for (int kt = 0; kt < ktiles; ++kt) {
    store();
    tc::fence_async_smem();
    __syncthreads();
    tc::tc_fence_after();
    if (threadIdx.x == 0) tc_chunk<N, KC>(c.taddr, sA, sB, c.mbar, kt > 0);
    if (kt + 1 < ktiles) load(kt + 1);
    ok = tc_chunk_wait(c.mbar, phase, err);
    if (!ok) break;
  }
  if (ok) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const long long row = m0 + 32 * w + lane;
    const int coutp = (cout + 7) & ~7;
#pragma unroll
    for (int col = 0; col < N; col += 8) {
      float val[8];
      tc::tmem_ld8(c.taddr, w, col, val);
      if (row < nvox && col < coutp) {
        __align__(16) bf16 ob[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          float o = col + q < cout ? val[q] + (bias ? bias[col + q] : 0.0f) : 0.0f;
          if (relu) o = fmaxf(o, 0.0f);
          ob[q] = __float2bfloat16_rn(o);
          if (out_f && col + q == 0) out_f[row] = o;  // (channel 0 only)
        }
        if (out_bf) *reinterpret_cast<uint4*>(out_bf + row * coutp + col) =
                        *reinterpret_cast<const uint4*>(ob);
      }
    }
  }
  tc_end<NC>(c);
}

void launch_conv_fwd(cudaStream_t st, const void* in, int B, int D, int H, int W, int per,
                     int cin, const void* wp, int n, int kp, const float* bias, int cout,
                     int relu, void* out_bf, float* out_f, int* err) {
  Vol g{B, D, H, W, per};
  dim3 grid((unsigned)((g.voxels() + tc::TM - 1) / tc::TM));
  switch (n) {
    case 16: k_conv_fwd<16><<<grid, 128, 0, st>>>((const bf16*)in, g, cin, (const bf16*)wp, kp, bias, cout, relu, (bf16*)out_bf, out_f, err); break;
    case 32: k_conv_fwd<32><<<grid, 128, 0, st>>>((const bf16*)in, g, cin, (const bf16*)wp, kp, bias, cout, relu, (bf16*)out_bf, out_f, err); break;
    case 48: k_conv_fwd<48><<<grid, 128, 0, st>>>((const bf16*)in, g, cin, (const bf16*)wp, kp, bias, cout, relu, (bf16*)out_bf, out_f, err); break;
    case 64: k_conv_fwd<64><<<grid, 128, 0, st>>>((const bf16*)in, g, cin, (const bf16*)wp, kp, bias, cout, relu, (bf16*)out_bf, out_f, err); break;
    case 96: k_conv_fwd<96><<<grid, 128, 0, st>>>((const bf16*)in, g, cin, (const bf16*)wp, kp, bias, cout, relu, (bf16*)out_bf, out_f, err); break;
    default: return;
  }
  note_launch();
}

// ---------------------------------------------------------------------------
// Weight packing.  w: FP32 master [cout][27 cin].  Forward operand
// wp[n][kp] (rows cout.., columns 27 cin.. zero); input-gradient operand
// wt[nt][kpt]: wt[ci][t' cout + co] = w[co][(26 - t') cin + ci].
// ---------------------------------------------------------------------------
__global__ void k_pack_w(const float* __restrict__ w, int cin, int cout, bf16* __restrict__ wp,
                         int n, int kp, bf16* __restrict__ wt, int nt, int kpt) {
  const int K = 27 * cin;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n * kp; t += gridDim.x * blockDim.x) {
    int r = t / kp, k = t - r * kp;
    float v = (r < cout && k < K) ? w[(long long)r * K + k] : 0.0f;
    wp[t] = __float2bfloat16_rn(v);
  }
  const int Kt = 27 * cout;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < nt * kpt; t += gridDim.x * blockDim.x) {
    int ci = t / kpt, k = t - ci * kpt;
    float v = 0.0f;
    if (ci < cin && k < Kt) {
      int tp = k / cout, co = k - tp * cout;
      v = w[(long long)co * K + (26 - tp) * cin + ci];
    }
    wt[t] = __float2bfloat16_rn(v);
  }
}

void launch_pack_w(cudaStream_t st, const float* w, int cin, int cout, void* wp, int n, int kp,
                   void* wt, int nt, int kpt) {
  k_pack_w<<<304, 256, 0, st>>>(w, cin, cout, (bf16*)wp, n, kp, (bf16*)wt, nt, kpt);
  note_launch();
}

// ---------------------------------------------------------------------------
// Elementwise kernels (channels-last BF16 unless stated).
// ---------------------------------------------------------------------------
// dy <- dy * (y > 0), 8 values (16 bytes) per step (n: a multiple of 8)
__global__ void k_relu_bwd(uint4* __restrict__ dy, const uint4* __restrict__ y, long long n8) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n8;
       t += (long long)gridDim.x * blockDim.x) {
    uint4 d = dy[t];
    const uint4 v = y[t];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      if (!(__bfloat162float(reinterpret_cast<const bf16*>(&v)[q]) > 0.0f))
        reinterpret_cast<bf16*>(&d)[q] = __float2bfloat16_rn(0.0f);
    dy[t] = d;
  }
}

// 2x2x2 average pooling: out [B][D/2][H/2][W/2][C], 8 channels (16 bytes) per
// step (C a multiple of 8; I: 32-bit arithmetic below 2^31 pieces of the fine
// grid).  A 160^3 forward's three: 18 us; two bytes per step
// took 53.
template <class I>
__global__ void k_pool2_v8(const uint4* __restrict__ in, Vol g, int C8, uint4* __restrict__ out) {
  const int D2 = g.D / 2, H2 = g.H / 2, W2 = g.W / 2;
  const I n = (I)g.B * D2 * H2 * W2 * C8;
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (I)gridDim.x * blockDim.x) {
    const int c = (int)(t % C8);
    I r = t / C8;
    const int x = (int)(r % W2); r /= W2;
    const int y = (int)(r % H2); r /= H2;
    const int z = (int)(r % D2);
    const I b = r / D2;
    uint4 v[8];
#pragma unroll
    for (int d = 0; d < 8; ++d)
      v[d] = in[(((b * g.D + 2 * z + (d >> 2)) * g.H + 2 * y + ((d >> 1) & 1)) * g.W + 2 * x +
                 (d & 1)) * C8 + c];
    __align__(16) bf16 o[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      float acc = 0.0f;
#pragma unroll
      for (int d = 0; d < 8; ++d) acc += __bfloat162float(reinterpret_cast<const bf16*>(&v[d])[q]);
      o[q] = __float2bfloat16_rn(0.125f * acc);
    }
    out[t] = *reinterpret_cast<const uint4*>(o);
  }
}

// backward of pooling: din[v] = dout[parent] / 8 (din has the fine shape g)
template <class I>
__global__ void k_pool2_bwd_v8(const uint4* __restrict__ dout, Vol g, int C8,
                               uint4* __restrict__ din) {
  const I n = (I)(g.voxels() * C8);
  for (I t = (I)blockIdx.x * blockDim.x + threadIdx.x; t < n; t += (I)gridDim.x * blockDim.x) {
    const int c = (int)(t % C8);
    I r = t / C8;
    const int x = (int)(r % g.W); r /= g.W;
    const int y = (int)(r % g.H); r /= g.H;
    const int z = (int)(r % g.D);
    const I b = r / g.D;
    const I p = ((b * (g.D / 2) + z / 2) * (g.H / 2) + y / 2) * (g.W / 2) + x / 2;
    const uint4 v = dout[p * C8 + c];
    __align__(16) bf16 o[8];
#pragma unroll
    for (int q = 0; q < 8; ++q)
      o[q] = __float2bfloat16_rn(0.125f * __bfloat162float(reinterpret_cast<const bf16*>(&v)[q]));
    din[t] = *reinterpret_cast<const uint4*>(o);
  }
}

// nearest upsampling by 2 into channels [c0, c0 + C) of an output with Cout
// channels (fine shape g); optional accumulate-free backward below
// the same with 8 channels (16 bytes) per step, 32-bit voxel arithmetic (C,
// Cout, c0 multiples of 8; fewer than 2^31 voxels)
__global__ void k_up2_v8(const uint4* __restrict__ in, Vol g, int C8, uint4* __restrict__ out,
                         int Cout8, int c08) {
  const int n = (int)(g.voxels() * C8);
  const int W2 = g.W >> 1, H2 = g.H >> 1, D2 = g.D >> 1;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < n; t += gridDim.x * blockDim.x) {
    const int c = t % C8, v = t / C8;
    int r = v;
    const int x = r % g.W; r /= g.W;
    const int y = r % g.H; r /= g.H;
    const int z = r % g.D;
    const int b = r / g.D;
    const int p = ((b * D2 + (z >> 1)) * H2 + (y >> 1)) * W2 + (x >> 1);
    out[(long long)v * Cout8 + c08 + c] = in[(long long)p * C8 + c];
  }
}

__global__ void k_up2(const bf16* __restrict__ in, Vol g, int C, bf16* __restrict__ out, int Cout,
                      int c0) {
  const long long n = g.voxels() * C;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    int c = (int)(t % C);
    long long v = t / C, r = v;
    int x = (int)(r % g.W); r /= g.W;
    int y = (int)(r % g.H); r /= g.H;
    int z = (int)(r % g.D);
    long long b = r / g.D;
    long long p = ((b * (g.D / 2) + z / 2) * (g.H / 2) + y / 2) * (long long)(g.W / 2) + x / 2;
    out[v * Cout + c0 + c] = in[p * C + c];
  }
}

// backward of upsampling: din[p] = sum of the 8 children of channels
// [c0, c0 + C) of dout (fine shape g, Cout channels)
__global__ void k_up2_bwd(const bf16* __restrict__ dout, Vol g, int Cout, int c0, int C,
                          bf16* __restrict__ din) {
  const int D2 = g.D / 2, H2 = g.H / 2, W2 = g.W / 2;
  const long long n = (long long)g.B * D2 * H2 * W2 * C;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    int c = (int)(t % C);
    long long r = t / C;
    int x = (int)(r % W2); r /= W2;
    int y = (int)(r % H2); r /= H2;
    int z = (int)(r % D2);
    long long b = r / D2;
    float acc = 0.0f;
#pragma unroll
    for (int d = 0; d < 8; ++d) {
      long long v = ((b * g.D + 2 * z + (d >> 2)) * g.H + 2 * y + ((d >> 1) & 1)) * (long long)g.W +
                    2 * x + (d & 1);
      acc += __bfloat162float(dout[v * Cout + c0 + c]);
    }
    din[t] = __float2bfloat16_rn(acc);
  }
}

// copy channels [0, C) of a tensor into channels [c0, c0 + C) of another
// (Cout channels); with `add` the destination is accumulated into
// plain copy of 8-channel groups (C, Csrc, s0, Cdst, c0 multiples of 8)
__global__ void k_chan_copy_v8(const uint4* __restrict__ src, long long nvox, int C8, int Csrc8,
                               int s08, uint4* __restrict__ dst, int Cdst8, int c08) {
  const long long n = nvox * C8;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(t % C8);
    const long long v = t / C8;
    dst[v * Cdst8 + c08 + c] = src[v * Csrc8 + s08 + c];
  }
}

__global__ void k_chan_copy(const bf16* __restrict__ src, long long nvox, int C, int Csrc,
                            int s0, bf16* __restrict__ dst, int Cdst, int c0, int add) {
  const long long n = nvox * C;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    int c = (int)(t % C);
    long long v = t / C;
    bf16 val = src[v * Csrc + s0 + c];
    if (add)
      dst[v * Cdst + c0 + c] =
          __float2bfloat16_rn(__bfloat162float(dst[v * Cdst + c0 + c]) + __bfloat162float(val));
    else
      dst[v * Cdst + c0 + c] = val;
  }
}

// network input: channel 0 = f * scale[b], channel 1 = 1 (the domain mask:
// zero padding turns it into a boundary indicator), channels 2..7 zero
__global__ void k_nn_input(const float* __restrict__ f, long long vps, const float* __restrict__ scale,
                           int B, bf16* __restrict__ x) {
  // a voxel (16 bytes) per thread; blockIdx.y: the sample (160^3: 11.5
  // us; two bytes per thread took 68)
  const float sc = scale[blockIdx.y];
  const long long v0 = blockIdx.y * vps;
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < vps;
       t += (long long)gridDim.x * blockDim.x) {
    __align__(16) bf16 o[8];
    o[0] = __float2bfloat16_rn(f[v0 + t] * sc);
    o[1] = __float2bfloat16_rn(1.0f);
#pragma unroll
    for (int c = 2; c < 8; ++c) o[c] = __float2bfloat16_rn(0.0f);
    *reinterpret_cast<uint4*>(x + (v0 + t) * 8) = *reinterpret_cast<const uint4*>(o);
  }
}

// loss = mean over voxels of (y0 - target * scale_t[b])^2; dy (8 channels)
// = d loss / d y in channel 0; partial sums of the loss per block
__global__ void k_mse(const float* __restrict__ y, const float* __restrict__ target,
                      long long vps, const float* __restrict__ tscale, int B,
                      bf16* __restrict__ dy, double* __restrict__ loss) {
  const long long n = (long long)B * vps;
  const float inv = 1.0f / (float)n;
  double acc = 0.0;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    float d = y[v] - target[v] * tscale[v / vps];
    acc += (double)d * d;
#pragma unroll
    for (int c = 0; c < 8; ++c) dy[v * 8 + c] = __float2bfloat16_rn(c == 0 ? 2.0f * d * inv : 0.0f);
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, acc / (double)n);
}

// Residual-norm loss, in three passes over FP32 fields of B samples:
//   d = y0 - target * tscale[b]           (k_loss_diff)
//   q = A d,  loss = mean q^2             (k_lap_loss; A the 7-point Laplacian
//                                          sum_nb d - 6 d, zero outside a
//                                          sample or periodic)
//   dy0 = 2 A q / n                       (k_lap_grad; A is symmetric)
__global__ void k_loss_diff(const float* __restrict__ y, const float* __restrict__ target,
                            long long vps, const float* __restrict__ tscale, int B,
                            float* __restrict__ d) {
  const long long n = (long long)B * vps;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x)
    d[v] = y[v] - target[v] * tscale[v / vps];
}

__device__ __forceinline__ float lap7(const float* __restrict__ d, const Vol& g, long long v) {
  long long t = v;
  int x = (int)(t % g.W); t /= g.W;
  int y = (int)(t % g.H); t /= g.H;
  int z = (int)(t % g.D);
  const long long sy = g.W, sz = (long long)g.W * g.H;
  float c = d[v], acc = -6.0f * c;
  auto nb = [&](int coord, int ext, long long stride, int dir) {
    int q = coord + dir;
    if (q < 0 || q >= ext) {
      if (!g.per) return 0.0f;
      q = q < 0 ? q + ext : q - ext;
    }
    return d[v + (long long)(q - coord) * stride];
  };
  acc += nb(x, g.W, 1, -1) + nb(x, g.W, 1, 1);
  acc += nb(y, g.H, sy, -1) + nb(y, g.H, sy, 1);
  acc += nb(z, g.D, sz, -1) + nb(z, g.D, sz, 1);
  return acc;
}

__global__ void k_lap_loss(const float* __restrict__ d, Vol g, float* __restrict__ q,
                           double* __restrict__ loss) {
  const long long n = g.voxels();
  double acc = 0.0;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    float a = lap7(d, g, v);
    q[v] = a;
    acc += (double)a * a;
  }
  acc = warp_sum(acc);
  if ((threadIdx.x & 31) == 0) atomicAdd(loss, acc / (double)n);
}

__global__ void k_lap_grad(const float* __restrict__ q, Vol g, bf16* __restrict__ dy) {
  const long long n = g.voxels();
  const float inv = 2.0f / (float)n;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x) {
    float a = lap7(q, g, v) * inv;
#pragma unroll
    for (int c = 0; c < 8; ++c) dy[v * 8 + c] = __float2bfloat16_rn(c == 0 ? a : 0.0f);
  }
}

// Adam on FP32 master parameters
__global__ void k_adam(float* __restrict__ w, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, long long n, float lr, float b1, float b2, float eps,
                       float c1, float c2) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < n;
       t += (long long)gridDim.x * blockDim.x) {
    float gt = g[t];
    float mt = b1 * m[t] + (1.0f - b1) * gt;
    float vt = b2 * v[t] + (1.0f - b2) * gt * gt;
    m[t] = mt;
    v[t] = vt;
    w[t] -= lr * (mt / c1) / (sqrtf(vt / c2) + eps);
  }
}

// network output (FP32, 8 channels) to a potential field: phi = y0 * scale
__global__ void k_nn_output(const float* __restrict__ y, long long vps, const float* __restrict__ scale,
                            int B, float* __restrict__ phi) {
  const long long n = (long long)B * vps;
  for (long long v = blockIdx.x * (long long)blockDim.x + threadIdx.x; v < n;
       v += (long long)gridDim.x * blockDim.x)
    phi[v] = y[v] * scale[v / vps];
}

static inline int ew_grid(long long n) {
  long long b = (n + 255) / 256;
  return (int)(b > 1216 ? 1216 : (b < 1 ? 1 : b));
}

void launch_relu_bwd(cudaStream_t st, void* dy, const void* y, long long n) {
  k_relu_bwd<<<ew_grid(n / 8), 256, 0, st>>>((uint4*)dy, (const uint4*)y, n / 8);
  note_launch();
}
void launch_pool2(cudaStream_t st, const void* in, int B, int D, int H, int W, int C, void* out) {
  Vol g{B, D, H, W};
  const int grid = ew_grid(g.voxels() * C / 64);
  if (g.voxels() * C / 8 < (1LL << 31))
    k_pool2_v8<int><<<grid, 256, 0, st>>>((const uint4*)in, g, C / 8, (uint4*)out);
  else
    k_pool2_v8<long long><<<grid, 256, 0, st>>>((const uint4*)in, g, C / 8, (uint4*)out);
  note_launch();
}
void launch_pool2_bwd(cudaStream_t st, const void* dout, int B, int D, int H, int W, int C,
                      void* din) {
  Vol g{B, D, H, W};
  const int grid = ew_grid(g.voxels() * C / 8);
  if (g.voxels() * C / 8 < (1LL << 31) - (1LL << 20))
    k_pool2_bwd_v8<int><<<grid, 256, 0, st>>>((const uint4*)dout, g, C / 8, (uint4*)din);
  else
    k_pool2_bwd_v8<long long><<<grid, 256, 0, st>>>((const uint4*)dout, g, C / 8, (uint4*)din);
  note_launch();
}
void launch_up2(cudaStream_t st, const void* in, int B, int D, int H, int W, int C, void* out,
                int Cout, int c0) {
  Vol g{B, D, H, W};
  if (C % 8 == 0 && Cout % 8 == 0 && c0 % 8 == 0 && g.voxels() * C / 8 < (1LL << 31))
    k_up2_v8<<<ew_grid(g.voxels() * C / 8), 256, 0, st>>>((const uint4*)in, g, C / 8,
                                                            (uint4*)out, Cout / 8, c0 / 8);
  else
    k_up2<<<ew_grid(g.voxels() * C), 256, 0, st>>>((const bf16*)in, g, C, (bf16*)out, Cout, c0);
  note_launch();
}
void launch_up2_bwd(cudaStream_t st, const void* dout, int B, int D, int H, int W, int Cout,
                    int c0, int C, void* din) {
  Vol g{B, D, H, W};
  k_up2_bwd<<<ew_grid(g.voxels() * C / 8), 256, 0, st>>>((const bf16*)dout, g, Cout, c0, C,
                                                          (bf16*)din);
  note_launch();
}
void launch_chan_copy(cudaStream_t st, const void* src, long long nvox, int C, int Csrc, int s0,
                      void* dst, int Cdst, int c0, bool add) {
  if (!add && C % 8 == 0 && Csrc % 8 == 0 && s0 % 8 == 0 && Cdst % 8 == 0 && c0 % 8 == 0)
    k_chan_copy_v8<<<ew_grid(nvox * C / 8), 256, 0, st>>>((const uint4*)src, nvox, C / 8,
                                                           Csrc / 8, s0 / 8, (uint4*)dst,
                                                           Cdst / 8, c0 / 8);
  else
    k_chan_copy<<<ew_grid(nvox * C), 256, 0, st>>>((const bf16*)src, nvox, C, Csrc, s0,
                                                   (bf16*)dst, Cdst, c0, add ? 1 : 0);
  note_launch();
}
void launch_nn_input(cudaStream_t st, const float* f, long long vps, const float* scale, int B,
                     void* x) {
  k_nn_input<<<dim3(ew_grid(vps), B), 256, 0, st>>>(f, vps, scale, B, (bf16*)x);
  note_launch();
}
void launch_mse(cudaStream_t st, const float* y, const float* target, long long vps,
                const float* tscale, int B, void* dy, double* loss) {
  k_mse<<<ew_grid((long long)B * vps), 256, 0, st>>>(y, target, vps, tscale, B, (bf16*)dy, loss);
  note_launch();
}
void launch_resid_loss(cudaStream_t st, const float* y, const float* target, int B, int S,
                       int per, const float* tscale, float* d, float* q, void* dy, double* loss) {
  Vol g{B, S, S, S, per};
  const long long vps = (long long)S * S * S, n = g.voxels();
  k_loss_diff<<<ew_grid(n), 256, 0, st>>>(y, target, vps, tscale, B, d);
  k_lap_loss<<<ew_grid(n), 256, 0, st>>>(d, g, q, loss);
  k_lap_grad<<<ew_grid(n), 256, 0, st>>>(q, g, (bf16*)dy);
  note_launch();
  note_launch();
  note_launch();
}
void launch_adam(cudaStream_t st, float* w, const float* g, float* m, float* v, long long n,
                 float lr, float b1, float b2, float eps, float c1, float c2) {
  k_adam<<<ew_grid(n), 256, 0, st>>>(w, g, m, v, n, lr, b1, b2, eps, c1, c2);
  note_launch();
}
void launch_nn_output(cudaStream_t st, const float* y, long long vps, const float* scale, int B,
                      float* phi) {
  k_nn_output<<<ew_grid((long long)B * vps), 256, 0, st>>>(y, vps, scale, B, phi);
  note_launch();
}

}  // namespace pm
