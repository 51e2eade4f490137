// Power spectrum of a particle set (Sec. 2.4: power-spectrum calculator with
// a discreteness correction): the first-order form (CIC window deconvolution
// and shot-noise subtraction) and the full alias correction of Jing (2005)
// that the paper names.  The FFT is cuFFT (a library call, off the step's
// hot path).
#include <algorithm>

#include "pm_kernels.cuh"

namespace pm {

// delta = rho / mean - 1 in double-float, rounded to FP32 (four FP64
// operations per cell, at this part's FP64 rate, took 92 us at 256^3 where
// the bytes take 30)
__global__ void __launch_bounds__(256) k_pk_delta(const unsigned long long* __restrict__ rho,
                                                  float* __restrict__ delta, long long total,
                                                  df inv_mean) {
  for (long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x; t < total;
       t += (long long)gridDim.x * blockDim.x)
    delta[t] = df_add(df_mul(df_from_u64(rho[t]), inv_mean), df{-1.0f, 0.0f}).hi;
}

static df df_of(double v) {
  df d;
  d.hi = (float)v;
  d.lo = (float)(v - (double)d.hi);
  return d;
}

void launch_pk_delta(cudaStream_t st, const unsigned long long* rho, float* delta, int n,
                     double inv_mean) {
  const long long total = (long long)n * n * n;
  const int grid = (int)std::min<long long>((total + 255) / 256, 152 * 8);
  k_pk_delta<<<grid, 256, 0, st>>>(rho, delta, total, df_of(inv_mean));
  note_launch();
}

// ---------------------------------------------------------------------------
// Binned modes.  The FFT's output is [kz][ky][kx], kx in 0..n/2; a stored
// mode counts twice where 0 < kx < n/2 (its partner at -k).  Bin b holds
// |k|/k_f in [b + 1/2, b + 3/2).  Per bin, acc[3 b + 0..2] += (modes,
// sum |k|, sum P) with
//   first order (m = 0):   P = P_obs / W^2 - shot,       W = prod_d sinc^2 x_d
//   alias-corrected (m):   P = (P_obs - shot C1) / C2,
//     C1 = prod_d [1 - (2/3) sin^2 x_d],
//     C2 = sum_{v in [-m, m]^3} prod_d sinc^4(x_d + pi v_d) (r_v / r_0)^(nu_b / 2),
// x_d = k_d h / 2, r_v = sum_d (x_d + pi v_d)^2.  The alias terms are FP32
// (factorised per axis), everything else double-float.
//
// FP64 runs at 1/64 of the FP32 rate here: with sin, sqrt and division per
// mode, shared FP64 atomics, and 343 FP64 additions per mode for C2, these
// passes took 1746 us (256^3, m = 0) and 2774 us (128^3, m = 3).  Now
//  - what depends on one axis alone is tabulated once, in FP64 (k_pk_axes);
//  - the up to four stored modes that share |kx|, |ky|, |kz| share W, C1, C2
//    and the bin, so they are added up first;
//  - C2 and the sums of P are double-float (error below 2^-45; the FFT rounds
//    at 2^-24, and P's distance from 64 bits, 2e-7 and up, is what it was with
//    FP64 sums).  |k| knows no FFT: its values and sums are three floats, exact
//    beyond 64 bits (with pairs the mean |k| of a 32^3 mesh's bins was 3.5e-16
//    off in the mean, 2.5 times as far as with FP64 sums);
//  - the bin comes from integers: |k|/k_f >= b + 1/2 iff
//    b (b + 1) < kx^2 + ky^2 + kz^2 in units of k_f;
//  - along a row of kx the bin does not fall, so a warp sums runs of one bin
//    by shuffles and their first lanes add to the warp's own bins without
//    atomics.
// ---------------------------------------------------------------------------
constexpr int PK_MAX_ALIAS = 3;
constexpr int PK_NA = 8;  // table stride (2 PK_MAX_ALIAS + 1, padded)

// per |mode| q of an axis: alias factors f[j] = sinc^4(x + pi (j - m)) and
// y2[j] = (x + pi (j - m))^2, C1's factor, and 1 / sinc^4 x
struct PkAxes {
  float* f;    // [n/2 + 1][PK_NA]
  float* y2;   // [n/2 + 1][PK_NA]
  float2* c1;  // [n/2 + 1] hi, lo
  float2* ti;  // [n/2 + 1] hi, lo
};
static __host__ __device__ PkAxes pk_axes(void* p, int n) {
  const size_t q = (size_t)n / 2 + 1;
  PkAxes a;
  a.f = (float*)p;
  a.y2 = a.f + PK_NA * q;
  a.c1 = (float2*)(a.y2 + PK_NA * q);
  a.ti = a.c1 + q;
  return a;
}
size_t pk_axes_bytes(int n) { return ((size_t)n / 2 + 1) * (2 * PK_NA * 4 + 2 * 8); }

__global__ void __launch_bounds__(32) k_pk_axes(void* tab, int n, double box, int m) {
  const PkAxes a = pk_axes(tab, n);
  const int q = blockIdx.x * 32 + threadIdx.x;
  if (q > n / 2) return;
  const double pi = 3.14159265358979323846;
  const double kf = 2.0 * pi / box, h = box / n;
  const double x = kf * q * h * 0.5, sx = sin(x), s2 = sx * sx;
  auto pair = [](double v) {
    const float hi = (float)v;
    return make_float2(hi, (float)(v - (double)hi));
  };
  const double w = q ? sx / x : 1.0;
  a.c1[q] = pair(1.0 - (2.0 / 3.0) * s2);
  a.ti[q] = pair(1.0 / (w * w * w * w));
  for (int j = 0; j < 2 * m + 1; ++j) {
    const double y = x + pi * (j - m);
    a.y2[q * PK_NA + j] = (float)(y * y);
    a.f[q * PK_NA + j] = y == 0.0 ? 1.0f : (float)((s2 * s2) / (y * y * y * y));
  }
}

__device__ __forceinline__ df df_of2(float2 v) { return df{v.x, v.y}; }
__device__ __forceinline__ df df_scale(df a, float p) {  // by a power of two
  return df{__fmul_rn(a.hi, p), __fmul_rn(a.lo, p)};
}
// hi + lo + c: a pair and a float that takes what a pair rounds away
struct tf {
  float hi, lo, c;
};
__device__ __forceinline__ tf tf_add(tf a, tf b) {
  const df s = two_sum(a.hi, b.hi), t = two_sum(a.lo, b.lo), m = two_sum(s.lo, t.hi);
  const df r = fast_two_sum(s.hi, m.hi);
  return tf{r.hi, r.lo, __fadd_rn(__fadd_rn(a.c, b.c), __fadd_rn(m.lo, t.lo))};
}
__device__ __forceinline__ tf tf_scale(tf a, float p) {  // by a power of two
  return tf{__fmul_rn(a.hi, p), __fmul_rn(a.lo, p), __fmul_rn(a.c, p)};
}
__device__ __forceinline__ tf tf_shfl_down(tf a, int o) {
  return tf{__shfl_down_sync(0xffffffffu, a.hi, o), __shfl_down_sync(0xffffffffu, a.lo, o),
            __shfl_down_sync(0xffffffffu, a.c, o)};
}
// the root of an integer q = s^2 (1 + d) < 2^24 from its FP32 root s: two
// corrections, whose remainders are exact (errors of order d^2, then d^3)
__device__ __forceinline__ tf tf_sqrt(float q, float s) {
  const float d2 = 2.0f * s;
  const float r = __fmaf_rn(-s, s, q), c = __fdiv_rn(r, d2);
  const float e = __fdiv_rn(__fmaf_rn(-c, c, __fmaf_rn(-d2, c, r)), d2);
  const df h = fast_two_sum(s, c);
  return tf{h.hi, h.lo, e};
}
__device__ __forceinline__ df df_div(df a, df b) {
  const float q = __fdiv_rn(a.hi, b.hi);
  const df r = df_add(a, df_mul(df{-q, 0.0f}, b));
  return fast_two_sum(q, __fdiv_rn(r.hi, b.hi));
}
__device__ __forceinline__ df df_shfl_down(df a, int o) {
  return df{__shfl_down_sync(0xffffffffu, a.hi, o), __shfl_down_sync(0xffffffffu, a.lo, o)};
}

constexpr int PK_NT = 256, PK_WARPS = PK_NT / 32;
constexpr size_t PK_SMEM = 200 * 1024;  // at most; one warp's part of 2048 bins is 66 KB
// shared floats of a warp: per bin the count, sum |k| (three floats), sum P
// (and sum C1/C2) as pairs; with aliases each lane's x factors
__host__ __device__ constexpr int pk_warp_floats(int n_bins, int m) {
  return n_bins * (m ? 8 : 6) + (m ? 2 * (2 * m + 1) * 32 : 0);
}

template <int m>
__global__ void __launch_bounds__(PK_NT) k_pk_modes(const float2* __restrict__ dk, int n,
                                                    double box, double shot, int n_bins,
                                                    const void* __restrict__ tab,
                                                    const double* __restrict__ nu,
                                                    double* __restrict__ acc) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int NA = 2 * m + 1, NF = m ? 8 : 6;
  extern __shared__ float sm[];
  const PkAxes T = pk_axes(const_cast<void*>(tab), n);
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nw = blockDim.x >> 5;
  float* bins = sm + (size_t)wib * pk_warp_floats(n_bins, m);
  float *xf = bins + n_bins * NF, *xy = xf + NA * 32;  // [j][lane] (m > 0)
  for (int e = lane; e < n_bins * NF; e += 32) bins[e] = 0.0f;
  __syncwarp();
  const int h = n / 2, nx = h + 1, rows = nx * nx;
  const int top = n_bins + 1;  // bins need kx^2 + ky^2 + kz^2 <= top (top - 1)
  const long long lim = (long long)top * (top - 1);
  for (int row = blockIdx.x * nw + wib; row < rows; row += gridDim.x * nw) {
    const int jy = row % nx, jz = row / nx;
    const long long r2 = (long long)jy * jy + (long long)jz * jz;
    if (r2 > lim) continue;
    const int ny = (jy == 0 || 2 * jy == n) ? 1 : 2, nz = (jz == 0 || 2 * jz == n) ? 1 : 2;
    const float2* im[4];  // the rows of the modes that share |ky|, |kz|
    im[0] = dk + ((long long)jz * n + jy) * nx;
    im[1] = dk + ((long long)jz * n + (n - jy)) * nx;
    im[2] = dk + ((long long)(n - jz) * n + jy) * nx;
    im[3] = dk + ((long long)(n - jz) * n + (n - jy)) * nx;
    df tyz{0.0f, 0.0f}, cyz{0.0f, 0.0f};
    float f2[NA], z2[NA];
    if (m == 0) {
      tyz = df_mul(df_of2(T.ti[jy]), df_of2(T.ti[jz]));
    } else {
      cyz = df_mul(df_of2(T.c1[jy]), df_of2(T.c1[jz]));
#pragma unroll
      for (int l = 0; l < NA; ++l) {
        f2[l] = T.f[jz * PK_NA + l];
        z2[l] = T.y2[jz * PK_NA + l];
      }
    }
    for (int x0 = 0; x0 < nx; x0 += 32) {
      if (r2 + (long long)x0 * x0 > lim) break;
      const int ix = x0 + lane;
      const long long m2 = r2 + (long long)ix * ix;
      const bool in = ix < nx && m2 > 0 && m2 <= lim;
      // r = the integer with r (r - 1) < m2 <= r (r + 1)
      float sq = sqrtf((float)m2);
      int r = (int)(sq + 0.5f);
      while ((long long)r * (r - 1) >= m2 && r > 0) --r;
      while ((long long)r * (r + 1) < m2) ++r;
      const int key = in ? r - 1 : -1;
      if (!__any_sync(FULL, in)) continue;
      float cnt = 0.0f;
      tf K{0.0f, 0.0f, 0.0f};
      df A{0.0f, 0.0f}, C{0.0f, 0.0f};
      if (in) {
        const float w = (ix == 0 || 2 * ix == n) ? 1.0f : 2.0f;
        cnt = w * (float)(ny * nz);
        // (m2 <= 3 (n/2)^2 < 2^24 is exact in FP32 up to n = 4729, past any mesh
        // that fits in memory)
        K = tf_sqrt((float)m2, sq);
        df o{0.0f, 0.0f};
        for (int q = 0; q < 4; ++q) {
          if ((q & 1) >= ny || (q >> 1) >= nz) continue;
          const float2 c = im[q][ix];
          const df a = two_prod(c.x, c.x), b = two_prod(c.y, c.y);
          o = df_add(o, df_add(a, b));
        }
        if (m == 0) {
          A = df_mul(o, df_mul(tyz, df_of2(T.ti[ix])));
        } else {
          float x2m = 0.0f;
#pragma unroll
          for (int j = 0; j < NA; ++j) {
            xf[j * 32 + lane] = T.f[ix * PK_NA + j];
            const float v = T.y2[ix * PK_NA + j];
            xy[j * 32 + lane] = v;
            if (j == m) x2m = v;
          }
          const float r0 = x2m + T.y2[jy * PK_NA + m] + z2[m];
          const float hnu = 0.5f * (float)nu[key];
          df c2{0.0f, 0.0f};
#pragma unroll 1
          for (int i = 0; i < NA; ++i) {
            const float fx = xf[i * 32 + lane], yx = xy[i * 32 + lane];
#pragma unroll 1
            for (int j = 0; j < NA; ++j) {
              const float fxy = fx * T.f[jy * PK_NA + j];
              const float rxy = yx + T.y2[jy * PK_NA + j];
              if (fxy == 0.0f) continue;
#pragma unroll
              for (int l = 0; l < NA; ++l) {
                const float wv = fxy * f2[l];
                if (wv == 0.0f) continue;
                const float t = wv * exp2f(hnu * log2f((rxy + z2[l]) / r0));
                const df s = two_sum(c2.hi, t);
                c2.hi = s.hi;
                c2.lo = __fadd_rn(c2.lo, s.lo);
              }
            }
          }
          c2 = fast_two_sum(c2.hi, c2.lo);
          A = df_div(o, c2);
          C = df_scale(df_div(df_mul(cyz, df_of2(T.c1[ix])), c2), cnt);
        }
        A = df_scale(A, w);
        K = tf_scale(K, cnt);
      }
      // sum each run of one bin onto its first lane
      const int prev = __shfl_up_sync(FULL, key, 1);
      const bool same = lane > 0 && in && prev == key;
      const unsigned cont = __ballot_sync(FULL, same);
      const unsigned brk = ~cont & (0xfffffffeu << lane);
      const int rend = brk ? __ffs(brk) - 2 : 31;
      for (int o = 1; o < 32; o <<= 1) {
        const bool add = lane + o <= rend;
        if (!__any_sync(FULL, add)) break;
        const float ct = __shfl_down_sync(FULL, cnt, o);
        const tf kt = tf_shfl_down(K, o);
        const df at = df_shfl_down(A, o);
        df cc{0.0f, 0.0f};
        if (m) cc = df_shfl_down(C, o);
        if (add) {
          cnt += ct;
          K = tf_add(K, kt);
          A = df_add(A, at);
          if (m) C = df_add(C, cc);
        }
      }
      if (in && !same) {  // the runs of a row have different bins
        float* e = bins + key * NF;
        e[0] += cnt;
        const tf k = tf_add(tf{e[1], e[2], e[3]}, K);
        const df a = df_add(df{e[4], e[5]}, A);
        e[1] = k.hi;
        e[2] = k.lo;
        e[3] = k.c;
        e[4] = a.hi;
        e[5] = a.lo;
        if (m) {
          const df c = df_add(df{e[6], e[7]}, C);
          e[6] = c.hi;
          e[7] = c.lo;
        }
      }
      __syncwarp();
    }
  }
  __syncthreads();
  const double kf = 2.0 * 3.14159265358979323846 / box;
  const double norm = box * box * box / ((double)n * n * n * (double)n * n * n);
  for (int b = threadIdx.x; b < n_bins; b += blockDim.x) {
    double c = 0.0, k = 0.0, p = 0.0, q = 0.0;
    for (int w = 0; w < nw; ++w) {
      const float* e = sm + (size_t)w * pk_warp_floats(n_bins, m) + b * NF;
      if (e[0] == 0.0f) continue;
      c += (double)e[0];
      k += (double)e[1] + ((double)e[2] + (double)e[3]);
      p += (double)e[4] + (double)e[5];
      if (m) q += (double)e[6] + (double)e[7];
    }
    if (c == 0.0) continue;
    atomicAdd(&acc[3 * b + 0], c);
    atomicAdd(&acc[3 * b + 1], kf * k);
    atomicAdd(&acc[3 * b + 2], norm * p - shot * (m ? q : c));
  }
}

template <int m>
static cudaError_t pk_launch(cudaStream_t st, const float2* dk, int n, double box, double shot,
                             int n_bins, const void* tab, const double* nu, double* acc) {
  const size_t per = sizeof(float) * pk_warp_floats(n_bins, m);
  const int nw = (int)std::max<size_t>(1, std::min<size_t>(PK_WARPS, PK_SMEM / per));
  if (per * nw > 48 * 1024) {
    // (the most that any launch takes, not this one's: another thread may set
    // it between the setting and the launch)
    const cudaError_t e = cudaFuncSetAttribute(
        k_pk_modes<m>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)PK_SMEM);
    if (e != cudaSuccess) return e;
  }
  const long long rows = (long long)(n / 2 + 1) * (n / 2 + 1);
  const int grid = (int)std::min<long long>((rows + nw - 1) / nw, 152 * 4);
  k_pk_modes<m><<<grid, 32 * nw, per * nw, st>>>(dk, n, box, shot, n_bins, tab, nu, acc);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_pk_axes(cudaStream_t st, void* tab, int n, double box, int m) {
  k_pk_axes<<<(n / 2 + 32) / 32, 32, 0, st>>>(tab, n, box, m);
  note_launch();
  return cudaGetLastError();
}

cudaError_t launch_pk_modes(cudaStream_t st, const float2* dk, int n, double box, double shot,
                            int n_bins, int m, const void* tab, const double* nu, double* acc) {
  switch (m) {
    case 0: return pk_launch<0>(st, dk, n, box, shot, n_bins, tab, nu, acc);
    case 1: return pk_launch<1>(st, dk, n, box, shot, n_bins, tab, nu, acc);
    case 2: return pk_launch<2>(st, dk, n, box, shot, n_bins, tab, nu, acc);
    default: return pk_launch<PK_MAX_ALIAS>(st, dk, n, box, shot, n_bins, tab, nu, acc);
  }
}

}  // namespace pm
