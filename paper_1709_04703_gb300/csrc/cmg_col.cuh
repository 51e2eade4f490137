// The bottom of the multigrid V-cycle (Sec. 2.1, Eq. 3) in one CTA, for
// unmasked tops of even side 6 to 16.
//
// It is a chain of about 40 dependent one-colour passes over at most 4096
// cells in one SM: what bounds it is the latency and the instructions of a
// pass, and, since other kernels evict it between two V-cycles, fetching its
// code (a straight-line form of this solver took 16 us when repeated and 36 us
// inside a V-cycle).  So the code is small and shared by the levels: sides
// are run-time values, a thread owns two x-adjacent cells (one of each
// colour) on two planes, every index is an offset computed once per level,
// the two colours live in separate padded arrays (conflict-free reads), and
// each level is a named barrier over the warps it needs.  The bottom itself
// (side <= 4 or odd) belongs to one warp, where it is open and of side 5 or 7
// to a thread per cell of a colour (one warp took 11 trips a pass for the 343
// cells: inside open steps a top of 14 37.4 us, of 10 20.7; so 14.1 and 13.0);
// its lexicographic sweep on odd periodic sides runs the diagonal fronts in
// parallel.  The operations and their order are those of cmg_fast.cuh, through
// mg_arith.cuh: the same bits.
#pragma once
#include "cmg_fast.cuh"

namespace pm {

namespace {

__host__ __device__ constexpr bool cl_supported(int S) { return S % 2 == 0 && S >= 6 && S <= 16; }
// floats of one colour's planes of side S (one ghost cell all round, two
// cells of a row per element pair) and threads of a level
__host__ __device__ constexpr int cl_col(int S) { return (S + 2) * (S + 2) * (S / 2 + 2); }
__host__ __device__ constexpr int cl_threads(int S) { return (S * S * S / 4 + 31) / 32 * 32; }
// shared floats: the odd rows' residuals; per level its two colours' values
// and right-hand sides, and (second level) its result in x order; the
// bottom's padded values, right-hand side and result
__host__ __device__ constexpr int cl_floats(int S) {
  int f = S * S * S / 2 + 4 * cl_col(S), C = S / 2;
  if (fc_next(C) != 0) {
    f += 4 * cl_col(C) + C * C * C;
    C /= 2;
  }
  return f + (C + 2) * (C + 2) * (C + 2) + 2 * C * C * C;
}
constexpr int CL_NT = cl_threads(16);  // 1024
constexpr int CL_SMEM = cl_floats(16);

__device__ __forceinline__ void cl_bar(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

// whether a thread per cell of a colour works on the bottom under a top of side
// S (open, the bottom's side 5 or 7; else one warp), and its threads then
__host__ __device__ constexpr bool cl_wide(int S, int periodic) {
  return !periodic && (S == 5 || S == 7 || S == 10 || S == 14);
}
__host__ __device__ constexpr int cl_wide_threads(int S) {
  return (S * S * S / 2 + 1 + 31) / 32 * 32;
}

// the cells lane, lane + 32, ... of an S^3 level in x order, by their
// coordinates
template <int S>
struct ClCells {
  int t, i, j, k;
  __device__ __forceinline__ explicit ClCells(int lane)
      : t(lane), i(lane % S), j(lane / S % S), k(lane / (S * S)) {}
  __device__ __forceinline__ bool ok() const { return t < S * S * S; }
  __device__ __forceinline__ void next() {
    t += 32;
    i += 32 % S;
    j += 32 / S % S;
    k += 32 / (S * S);
    if (i >= S) { i -= S; ++j; }
    if (j >= S) { j -= S; ++k; }
  }
  __device__ __forceinline__ int p() const { return fc_p<S>(i, j, k); }
};

// the bottom by one warp: cmg_fast.cuh's, on its padded u (zero) and b; the
// result to lin in x order
template <int S, bool PER>
__device__ __noinline__ void cl_bottom(float* u, const FcLev& L, int sweeps, float sig0) {
  constexpr int N = S * S * S, P = S + 2, P2 = P * P, Q = (N + 31) / 32;
  float *b = u + P * P2, *lin = b + N;
  const int lane = (int)(threadIdx.x & 31);
  const bool proj = PER && sig0 == 0.0f;
  auto mean = [&](const float* v, bool padded) {
    float m = 0.0f;
    ClCells<S> e(lane);
#pragma unroll 1
    for (int w = 0; w < Q; ++w, e.next()) {  // warp w of the fixed order
      float a = 0.0f;
      if (e.ok()) a += padded ? v[e.p()] : v[e.t];
      m += warp_sumf_all(a);
    }
    return m / (float)N;
  };
  if (proj) {
    const float m = mean(b, false);
    for (int t = lane; t < N; t += 32) b[t] -= m;
    __syncwarp();
  }
  int s1 = S + 1;
  asm volatile("" : "+r"(s1));  // (sinf of a run-time value, as in the other forms)
  const float omega = PER ? 1.0f : 2.0f / (1.0f + sinf(3.14159265f / (float)s1));
  auto cell = [&](int i, int j, int k) {
    const int p = fc_p<S>(i, j, k);
    int xm = p - 1, xp = p + 1, ym = p - P, yp = p + P, zm = p - P2, zp = p + P2;
    if (PER) {
      if (i == 0) xm += S;
      if (i == S - 1) xp -= S;
      if (j == 0) ym += S * P;
      if (j == S - 1) yp -= S * P;
      if (k == 0) zm += S * P2;
      if (k == S - 1) zp -= S * P2;
    }
    const float old = u[p];
    const float gs = gs_value(nb6(u[xm], u[xp], u[ym], u[yp], u[zm], u[zp]), b[fc_d<S>(i, j, k)], L.h2,
                              L.simple, L.simple ? 6.0f : mg_diag(i, j, k, S, PER, L.gam, L.d0));
    u[p] = omega == 1.0f ? gs : __fmaf_rn(omega, __fsub_rn(gs, old), old);
  };
#pragma unroll 1
  for (int w = 0; w < sweeps; ++w) {
    if ((S & 1) && PER) {
      // lexicographic order: the cells of a diagonal i + j + k = d depend
      // only on others, and every neighbour, the wrapped ones included, lies
      // on the same side of d as of the cell in that order
#pragma unroll 1
      for (int d = 0; d <= 3 * (S - 1); ++d) {
#pragma unroll 1
        for (ClCells<S> e(lane); e.ok(); e.next())
          if (e.i + e.j + e.k == d) cell(e.i, e.j, e.k);
        __syncwarp();
      }
    } else {
#pragma unroll 1
      for (int colour = 0; colour < 2; ++colour) {
        if (S % 2 == 0) {  // a lane's cells all in the colour
#pragma unroll
          for (int e = lane; e < N / 2; e += 32) {
            const int j = (e / (S / 2)) % S, k = e / (S * S / 2);
            cell(2 * (e % (S / 2)) + ((j + k + colour) & 1), j, k);
          }
        } else {
#pragma unroll 1
          for (ClCells<S> e(lane); e.ok(); e.next())
            if (((e.i + e.j + e.k) & 1) == colour) cell(e.i, e.j, e.k);
        }
        __syncwarp();
      }
    }
  }
  const float m = proj ? mean(u, true) : 0.0f;
#pragma unroll 1
  for (ClCells<S> e(lane); e.ok(); e.next()) {
    const float v = u[e.p()];
    lin[e.t] = proj ? v - m : v;
  }
}

// an open bottom of odd side: colour c holds the cells c, c + 2, ... in x
// order, thread e the e-th of each, with their values in registers.  The
// barrier is the bottom's own (3).
__device__ __noinline__ void cl_bottom_wide(int S, float* u, const FcLev& L, int sweeps) {
  const int P = S + 2, P2 = P * P, N = S * S * S, n = cl_wide_threads(S);
  float *b = u + P * P2, *lin = b + N;
  int at[2];
  bool on[2];
  float v[2], f[2], r[2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const int t = 2 * (int)threadIdx.x + c;
    on[c] = t < N;
    const int q = on[c] ? t : 0, i = q % S, j = q / S % S, k = q / (S * S);
    at[c] = ((k + 1) * P + j + 1) * P + i + 1;
    v[c] = u[at[c]];
    f[c] = b[q];
    r[c] = L.simple ? 1.0f / 6.0f : __frcp_rn(mg_diag(i, j, k, S, 0, L.gam, L.d0));
  }
  const float omega = 2.0f / (1.0f + sinf(3.14159265f / (float)(S + 1)));
  cl_bar(3, n);  // every value read
#pragma unroll 1
  for (int w = 0; w < sweeps; ++w) {
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      if (on[c]) {
        const float* p = u + at[c];
        const float gs = gs_scaled(nb6(p[-1], p[1], p[-P], p[P], p[-P2], p[P2]), f[c], L.h2, r[c]);
        v[c] = omega == 1.0f ? gs : __fmaf_rn(omega, __fsub_rn(gs, v[c]), v[c]);
        u[at[c]] = v[c];
      }
      cl_bar(3, n);
    }
  }
#pragma unroll
  for (int c = 0; c < 2; ++c)
    if (on[c]) lin[2 * threadIdx.x + c] = v[c];
}

__device__ void cl_bottom_s(int S, int periodic, float* u, const FcLev& L, int sweeps,
                            float sig0) {
  if (periodic) {
    if (S == 4) cl_bottom<4, true>(u, L, sweeps, sig0);
    else if (S == 3) cl_bottom<3, true>(u, L, sweeps, sig0);
    else if (S == 5) cl_bottom<5, true>(u, L, sweeps, sig0);
    else if (S == 7) cl_bottom<7, true>(u, L, sweeps, sig0);
    else cl_bottom<2, true>(u, L, sweeps, sig0);
  } else {
    if (S == 4) cl_bottom<4, false>(u, L, sweeps, sig0);
    else if (S == 3) cl_bottom<3, false>(u, L, sweeps, sig0);
    else cl_bottom<2, false>(u, L, sweeps, sig0);
  }
}
__device__ __forceinline__ FcLev cl_lev(int level, int periodic, float sig0) {
  FcLev L;
  const float Hs = (float)(1 << level);
  L.h2 = Hs * Hs;
  L.inv_h2 = 1.0f / L.h2;
  L.gam = (Hs - 1.0f) / (Hs + 1.0f);
  L.d0 = 6.0f + sig0 * L.h2;
  L.simple = mg_simple(periodic, L.gam, L.d0);
  return L;
}

// a top that is a bottom itself (side 2 to 5 or 7): one warp, or WIDE
// cl_wide_threads
template <bool WIDE>
__device__ __noinline__ void cl_only_bottom(float* sm, const Grid& gu, const Grid& gb, int level,
                                            int periodic, int sweeps, int zero_top,
                                            float sig0) {
  const int S = gu.s, P = S + 2, N = S * S * S, t0 = (int)threadIdx.x;
  const int n = WIDE ? cl_wide_threads(S) : 32;
  float *b = sm + P * P * P, *lin = b + N;
  for (int t = t0; t < P * P * P; t += n) {
    const int i = t % P - 1, j = (t / P) % P - 1, k = t / (P * P) - 1;
    const int out = (i < 0 || i >= S) + (j < 0 || j >= S) + (k < 0 || k >= S);
    const bool rd = out == 0 ? !zero_top : (out == 1 && !periodic);
    sm[t] = rd ? gu.base[gidx(gu, i, j, k)] : 0.0f;
  }
  for (int t = t0; t < N; t += n)
    b[t] = gb.base[gidx(gb, t % S, (t / S) % S, t / (S * S))];
  cl_bar(3, n);
  if (WIDE) cl_bottom_wide(S, sm, cl_lev(level, periodic, sig0), sweeps);
  else cl_bottom_s(S, periodic, sm, cl_lev(level, periodic, sig0), sweeps, sig0);
  cl_bar(3, n);
  for (int t = t0; t < N; t += n)
    gu.base[gidx(gu, t % S, (t / S) % S, t / (S * S))] = lin[t];
}

// the V-cycle from an unmasked even top of side S0 (cl_supported) in one CTA
// of at least cl_threads(S0) threads; sm holds cl_floats(S0) floats.  WIDE as
// cl_wide(S0): a form of its own, since the test in the other one's code cost
// every V-cycle 0.8 us.
template <bool WIDE>
__device__ __forceinline__ void cl_vcycle(float* sm, const Grid& gu, const Grid& gb, int level,
                                          int periodic, int sweeps, int zero_top, float sig0) {
  const int t = (int)threadIdx.x;
  const int S0 = gu.s, C0 = S0 / 2;
  const bool two = !(C0 <= 4 || (C0 & 1));  // a second level above the bottom
  const int Sb = two ? C0 / 2 : C0;         // the bottom's side
  float2* res = reinterpret_cast<float2*>(sm);
  float* lev0 = sm + S0 * S0 * S0 / 2;
  float* lev1 = lev0 + 4 * cl_col(S0);
  float* bot = two ? lev1 + 4 * cl_col(C0) + C0 * C0 * C0 : lev1;

  // this thread's place on the current level
  int S, xp, j, k0, M, PM, c, oym, oyp, ozm, ozp, sA, sB, n, id;
  bool on, odd;
  float h2, inv_h2, dR0, dR1, dB0, dB1, rR0, rR1, rB0, rB1;
  float *uR, *uB, *bR, *bB;
  auto place = [&](int q) {
    S = q ? C0 : S0;
    n = cl_threads(S);
    id = 1 + q;
    // lanes along x, then along z (two planes each): the shared rows of a
    // warp then fall on different banks (16^3: 2 planes are 360 words, 8
    // banks apart; along y the rows of 10 words would overlap)
    const int H = S >> 1, r = t / H, seg = r % H;
    on = t < S * S * S / 4;
    xp = t - r * H;
    j = r / H;
    k0 = 2 * seg;
    odd = j & 1;
    M = H + 2;
    PM = (S + 2) * M;
    c = (k0 + 1) * PM + (j + 1) * M + xp + 1;
    const bool per = periodic != 0;
    oym = (per && j == 0) ? (S - 1) * M : -M;
    oyp = (per && j == S - 1) ? -(S - 1) * M : M;
    ozm = (per && k0 == 0) ? (S - 1) * PM : -PM;          // from plane k0
    ozp = (per && k0 == S - 2) ? -(S - 1) * PM : PM;      // from plane k0 + 1
    const int sm_ = (per && xp == 0) ? H - 1 : -1, sp_ = (per && xp == H - 1) ? -(H - 1) : 1;
    // plane k0 (even): the red cell is the pair's cell `odd`; the pair beside
    // a cell at x offset 1 is the next one, else the one before
    sA = odd ? sp_ : sm_;  // red on plane k0, black on k0 + 1
    sB = odd ? sm_ : sp_;
    const float Hs = (float)(1 << (level + q));
    h2 = Hs * Hs;
    inv_h2 = 1.0f / h2;
    const float gam = (Hs - 1.0f) / (Hs + 1.0f), d0 = 6.0f + sig0 * h2;
    const bool simple = mg_simple(periodic, gam, d0);
    const int fy = (j == 0) + (j == S - 1), f0 = fy + (xp == 0), f1 = fy + (xp == H - 1);
    const int z0 = k0 == 0, z1 = k0 == S - 2;
    auto dg = [&](int nb) { return simple ? 6.0f : (per ? d0 : d0 + gam * (float)nb); };
    dR0 = dg((odd ? f1 : f0) + z0);
    dB0 = dg((odd ? f0 : f1) + z0);
    dR1 = dg((odd ? f0 : f1) + z1);
    dB1 = dg((odd ? f1 : f0) + z1);
    auto rc = [&](float d) { return simple ? 1.0f / 6.0f : __frcp_rn(d); };
    rR0 = rc(dR0);
    rB0 = rc(dB0);
    rR1 = rc(dR1);
    rB1 = rc(dB1);
    uR = q ? lev1 : lev0;
    uB = uR + cl_col(S);
    bR = uB + cl_col(S);
    bB = bR + cl_col(S);
  };
  // neighbour sums of the two cells of one colour: partners p0, p1 in
  // registers, the rest from the other colour's planes
  auto sums = [&](const float* src, float p0, float p1, int a, int b, float& s0, float& s1) {
    const float* q = src + c;
    s0 = nb6(p0, q[a], q[oym], q[oyp], q[ozm], p1);
    s1 = nb6(p1, q[PM + b], q[PM + oym], q[PM + oyp], p0, q[PM + ozp]);
  };
  // two sweeps from the stored values; r, b: the final values
  auto smooth = [&](float& r0, float& r1, float& b0, float& b1) {
    float fR0 = 0.0f, fR1 = 0.0f, fB0 = 0.0f, fB1 = 0.0f;
    if (on) {
      r0 = uR[c]; r1 = uR[c + PM]; b0 = uB[c]; b1 = uB[c + PM];
      fR0 = bR[c]; fR1 = bR[c + PM]; fB0 = bB[c]; fB1 = bB[c + PM];
    }
#pragma unroll 1
    for (int w = 0; w < 2; ++w) {
      float s0, s1;
      if (on) {
        sums(uB, b0, b1, sA, sB, s0, s1);
        r0 = sor_value(r0, gs_scaled(s0, fR0, h2, rR0));
        r1 = sor_value(r1, gs_scaled(s1, fR1, h2, rR1));
        uR[c] = r0;
        uR[c + PM] = r1;
      }
      cl_bar(id, n);
      if (on) {
        sums(uR, r0, r1, sB, sA, s0, s1);
        b0 = sor_value(b0, gs_scaled(s0, fB0, h2, rB0));
        b1 = sor_value(b1, gs_scaled(s1, fB1, h2, rB1));
        uB[c] = b0;
        uB[c + PM] = b1;
      }
      cl_bar(id, n);
    }
  };

  float r0 = 0.0f, r1 = 0.0f, b0 = 0.0f, b1 = 0.0f;
  place(0);
  {
    float w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = 0.0f;
    if (on) {
      const float* p = gb.base + gidx(gb, 2 * xp, j, k0);
      w[0] = p[0]; w[1] = p[1]; w[2] = p[gb.sz]; w[3] = p[gb.sz + 1];
      if (!zero_top) {
        const float* v = gu.base + gidx(gu, 2 * xp, j, k0);
        w[4] = v[0]; w[5] = v[1]; w[6] = v[gu.sz]; w[7] = v[gu.sz + 1];
      }
    }
    const int nth = (int)blockDim.x;
    for (int e = t; e < 2 * cl_col(S0); e += nth) lev0[e] = 0.0f;
    if (two)
      for (int e = t; e < 2 * cl_col(C0); e += nth) lev1[e] = 0.0f;
    for (int e = t; e < (Sb + 2) * (Sb + 2) * (Sb + 2); e += nth) bot[e] = 0.0f;
    __syncthreads();
    if (on) {
      bR[c] = odd ? w[1] : w[0];
      bB[c] = odd ? w[0] : w[1];
      bR[c + PM] = odd ? w[2] : w[3];
      bB[c + PM] = odd ? w[3] : w[2];
      if (!zero_top) {
        uR[c] = odd ? w[5] : w[4];
        uB[c] = odd ? w[4] : w[5];
        uR[c + PM] = odd ? w[6] : w[7];
        uB[c + PM] = odd ? w[7] : w[6];
      }
    }
    if (!periodic) {  // the top's ghost faces (Dirichlet data), by colour
      for (int e = t; e < 6 * S0 * S0; e += nth) {
        const int f = e / (S0 * S0), a = e % S0, o = (e / S0) % S0, g = (f & 1) ? S0 : -1;
        const int gi = f < 2 ? g : a, gj = f < 2 ? a : (f < 4 ? g : o), gk = f < 4 ? o : g;
        const int at = (gk + 1) * PM + (gj + 1) * M + ((gi + 2) >> 1);
        (((gi + gj + gk) & 1) ? uB : uR)[at] = gu.base[gidx(gu, gi, gj, gk)];
      }
    }
  }
  __syncthreads();
  if (t >= n) return;  // (launched with more threads than this top needs)
  // down: a level's warps smooth and restrict; those the next level does not
  // need wait for the way up
  const int nl = two ? 2 : 1;
  int q = 0;
#pragma unroll 1
  for (;;) {
    smooth(r0, r1, b0, b1);
    const int H = S >> 1, rc = (j >> 1) * H + xp;
    float x0 = 0.0f, x1 = 0.0f, x2 = 0.0f, x3 = 0.0f;
    if (on) {
      float s0, s1;
      sums(uB, b0, b1, sA, sB, s0, s1);
      const float a0 = resid_value(s0, r0, bR[c], dR0, inv_h2);
      const float a1 = resid_value(s1, r1, bR[c + PM], dR1, inv_h2);
      sums(uR, r0, r1, sB, sA, s0, s1);
      const float e0 = resid_value(s0, b0, bB[c], dB0, inv_h2);
      const float e1 = resid_value(s1, b1, bB[c + PM], dB1, inv_h2);
      x0 = odd ? e0 : a0;  // x order: plane k0, then k0 + 1
      x1 = odd ? a0 : e0;
      x2 = odd ? a1 : e1;
      x3 = odd ? e1 : a1;
      if (odd) {
        res[k0 * H * H + rc] = make_float2(x0, x1);
        res[(k0 + 1) * H * H + rc] = make_float2(x2, x3);
      }
    }
    cl_bar(id, n);
    if (on && !odd) {
      const float2 y0 = res[k0 * H * H + rc], y1 = res[(k0 + 1) * H * H + rc];
      float acc = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(0.0f, x0), x1), y0.x), y0.y);
      acc = __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(acc, x2), x3), y1.x), y1.y);
      const float v = __fmul_rn(0.125f, acc);
      const int J = j >> 1, K = k0 >> 1;
      if (q + 1 < nl) {  // into the second level's colours
        float* d = lev1 + 2 * cl_col(H) + (((xp + J + K) & 1) ? cl_col(H) : 0);
        d[((K + 1) * (H + 2) + J + 1) * (H / 2 + 2) + (xp >> 1) + 1] = v;
      } else {
        bot[(H + 2) * (H + 2) * (H + 2) + (K * H + J) * H + xp] = v;
      }
    }
    cl_bar(id, n);
    if (q + 1 == nl || t >= cl_threads(C0)) break;
    place(++q);
  }
  if (WIDE) {
    if (q + 1 == nl && t < cl_wide_threads(Sb))
      cl_bottom_wide(Sb, bot, cl_lev(level + nl, periodic, sig0), sweeps);
  } else if (q + 1 == nl && t < 32) {
    cl_bottom_s(Sb, periodic, bot, cl_lev(level + nl, periodic, sig0), sweeps, sig0);
  }
  // up: the level below has left its result in x order
#pragma unroll 1
  for (;; place(--q)) {
    cl_bar(id, n);
    if (on) {
      const int C = S >> 1, J = j >> 1, K = k0 >> 1;
      const float* lin = (q + 1 < nl) ? lev1 + 4 * cl_col(C)
                                      : bot + (C + 2) * (C + 2) * (C + 2) + C * C * C;
      const float Hc = (float)(1 << (level + q + 1)), gc = (Hc - 1.0f) / (Hc + 1.0f);
      int xm = xp - 1, xq = xp + 1, J2 = odd ? J + 1 : J - 1, Km = K - 1, Kp = K + 1;
      float fxm = 1.0f, fxp = 1.0f, fy = 1.0f, fzm = 1.0f, fzp = 1.0f;
      if (periodic) {
        xm = xm < 0 ? C - 1 : xm;
        xq = xq >= C ? 0 : xq;
        J2 = J2 < 0 ? C - 1 : (J2 >= C ? 0 : J2);
        Km = Km < 0 ? C - 1 : Km;
        Kp = Kp >= C ? 0 : Kp;
      } else {
        if (xm < 0) { xm = xp; fxm = -gc; }
        if (xq >= C) { xq = xp; fxp = -gc; }
        if (J2 < 0 || J2 >= C) { J2 = J; fy = -gc; }
        if (Km < 0) { Km = K; fzm = -gc; }
        if (Kp >= C) { Kp = K; fzp = -gc; }
      }
      // prolong_mix: x and y interpolations per coarse plane (its z factor
      // fz multiplied in), then z
      float A0[3], A1[3];
#pragma unroll 1
      for (int e = 0; e < 3; ++e) {
        const int kk = e == 0 ? Km : (e == 1 ? K : Kp);
        const float fz = e == 0 ? fzm : (e == 1 ? 1.0f : fzp);
        const float *l0 = lin + (kk * C + J) * C, *l1 = lin + (kk * C + J2) * C;
        const float v0 = __fmul_rn(fz, l0[xp]), w0 = __fmul_rn(__fmul_rn(fy, fz), l1[xp]);
        const float vm = __fmul_rn(__fmul_rn(fxm, fz), l0[xm]);
        const float vp = __fmul_rn(__fmul_rn(fxp, fz), l0[xq]);
        const float wm = __fmul_rn(__fmul_rn(__fmul_rn(fxm, fy), fz), l1[xm]);
        const float wp = __fmul_rn(__fmul_rn(__fmul_rn(fxp, fy), fz), l1[xq]);
        const float g0 = lerp34(lerp34(v0, vm), lerp34(w0, wm));
        const float g1 = lerp34(lerp34(v0, vp), lerp34(w0, wp));
        if (e == 0) { A0[0] = g0; A1[0] = g1; }
        else if (e == 1) { A0[1] = g0; A1[1] = g1; }
        else { A0[2] = g0; A1[2] = g1; }
      }
      const float p00 = lerp34(A0[1], A0[0]), p01 = lerp34(A1[1], A1[0]);
      const float p10 = lerp34(A0[1], A0[2]), p11 = lerp34(A1[1], A1[2]);
      uR[c] = __fadd_rn(uR[c], odd ? p01 : p00);
      uB[c] = __fadd_rn(uB[c], odd ? p00 : p01);
      uR[c + PM] = __fadd_rn(uR[c + PM], odd ? p10 : p11);
      uB[c + PM] = __fadd_rn(uB[c + PM], odd ? p11 : p10);
    }
    cl_bar(id, n);
    smooth(r0, r1, b0, b1);
    const float v0 = odd ? b0 : r0, v1 = odd ? r0 : b0;
    const float v2 = odd ? r1 : b1, v3 = odd ? b1 : r1;
    if (q == 0) {
      if (on) {
        float* p = gu.base + gidx(gu, 2 * xp, j, k0);
        p[0] = v0;
        p[1] = v1;
        p[gu.sz] = v2;
        p[gu.sz + 1] = v3;
      }
      break;
    }
    if (on) {
      float* l = lev1 + 4 * cl_col(S) + (k0 * S + j) * S + 2 * xp;
      l[0] = v0;
      l[1] = v1;
      l[S * S] = v2;
      l[S * S + 1] = v3;
    }
  }
}

}  // namespace

}  // namespace pm
