// Fused legs of the multigrid V-cycle for the levels between the one-CTA
// bottom and the z-marching smoother (Sec. 2.1, Eq. 3, cell units): one
// launch per level on the way down (two red-black SOR sweeps from zero,
// residual, restriction) and one on the way up (prolongation, two sweeps),
// each over tiles held on chip with a halo of four cells.
//
// What bounds these levels is not bytes (the arrays sit in L2) but the chain
// of dependent passes: a leg as four one-colour passes and a transfer is five
// launches and five sweeps over L2.  A tile recomputes its halo instead: 24 x
// 24 x 16 cells for a 16 x 16 x 8 tile, 4.5 times the updates, but one pass.
//
// Microseconds per leg inside a graph, separate passes -> fused (the tiles of
// tile_small below; periodic, and open on a coarse level):
//   side   down           up             down, open     up, open
//     32   8.3 ->  3.1    9.1 ->  5.0    8.9 ->  4.3    9.0 ->  7.2
//     48   9.5 ->  3.6   11.3 ->  5.8   10.3 ->  4.4   10.9 ->  7.6
//     64  11.2 ->  4.0   13.8 ->  6.3   11.9 ->  5.1   13.7 -> 10.6
//     96  16.9 ->  8.2   20.2 -> 13.5   17.3 -> 11.2   20.3 -> 19.3
//    128  27.1 -> 16.6   35.2 -> 27.2   28.0 -> 20.3   35.7 -> 35.9
// Above, the leg down still gains on the z-marching pass and a restriction
// (its best of nine tile shapes; 160 open: 39.2 -> 33.6, 192: 55.9 -> 52.0,
// 256: 149 -> 124).  The leg up loses to the prolongation and that pass, which
// updates less halo (192: 63.4 against 87.4, 256: 152 against 202; so it would
// at 160 in its best shape, 44.3 against 58.5, but only levels of side 192 and
// up are timed for one, and in its default shape it takes 54.6).
#include "mg_arith.cuh"
#include "pm_kernels.cuh"

namespace pm {

// ---------------------------------------------------------------------------
// Tile TX x TY x TZ plus a halo of 4.  A thread owns a pair of x-adjacent
// columns of the region (one cell of each colour per plane) and keeps their
// values and right-hand sides on all RZ planes in registers, in colour
// order: R the red cell ((x + y + z) even), B the black one.  The red cell
// of plane z sits at x offset (y + z) & 1 of the pair (tiles start at even
// cells).  A cell's z neighbours are the other register of the planes above
// and below, one x neighbour is its partner in the pair; the other x
// neighbour and the y neighbours are read from shared memory, where every
// thread exposes its newly updated colour, conflict-free (thread-linear
// planes).  The ring of valid cells shrinks by one per one-colour pass; what
// lies outside it is computed from stale neighbours and never used.  Cells
// outside an open domain stay zero (the ghosts of a correction), periodic
// coordinates wrap.  The updates are those of the one-colour passes
// (mg_arith.cuh) on the values they would meet: the same bits.
// ---------------------------------------------------------------------------
namespace {

constexpr int TL_H = 4;

template <int TX_, int TY_, int TZ_>
struct TileShape {
  static constexpr int TX = TX_, TY = TY_, TZ = TZ_;
  static constexpr int HX = (TX + 2 * TL_H) / 2;  // pairs per region row
  static constexpr int RY = TY + 2 * TL_H, RZ = TZ + 2 * TL_H;
  static constexpr int NT = HX * RY;
  // shared floats: the two colours' planes, each with a guard row on both
  // sides (reads of the region's rim), and the odd rows' residuals (down) or
  // the coarse patch (up)
  static constexpr int COL = RZ * NT + 2 * HX;
  static constexpr int CX = HX + 2, CY = RY / 2 + 2, CZ = RZ / 2 + 2;
  static constexpr int RES = TZ * (TY / 2) * TX, PATCH = CX * CY * CZ;
  static constexpr int SMEM = 2 * COL + (RES > PATCH ? RES : PATCH);
};

template <class T, bool PER, bool SIMPLE>
struct TilePass {
  const TileArgs& a;
  int s, t, xp, y, x0, y0, z0, gx, gy;
  bool in, odd;
  int de;        // side offset of a red update on an even plane
  int f0, f1;    // ghost faces along x and y of the pair's two cells
  // reciprocal diagonals of the two cells, off the z faces and on them
  float rd0, rd1, rz0, rz1;
  float *sR, *sB;

  __device__ __forceinline__ TilePass(const TileArgs& a_, int bx, int by, int bz, float* sm)
      : a(a_) {
    s = a.b.s;
    t = (int)threadIdx.x;
    xp = t % T::HX;
    y = t / T::HX;
    x0 = bx * T::TX - TL_H + 2 * xp;
    y0 = by * T::TY - TL_H + y;
    z0 = bz * T::TZ - TL_H;
    gx = x0;
    gy = y0;
    in = true;
    if (PER) {
      gx = gx < 0 ? gx + s : (gx >= s ? gx - s : gx);
      gy = gy < 0 ? gy + s : (gy >= s ? gy - s : gy);
    } else {
      in = x0 >= 0 && x0 < s && y0 >= 0 && y0 < s;
    }
    odd = y & 1;
    de = odd ? 1 : -1;
    const int fy = (gy == 0) + (gy == s - 1);
    f0 = fy + (gx == 0);
    f1 = fy + (gx + 1 == s - 1);
    if (!SIMPLE) {
      rd0 = __frcp_rn(PER ? a.d0 : a.d0 + a.gam * (float)f0);
      rd1 = __frcp_rn(PER ? a.d0 : a.d0 + a.gam * (float)f1);
      rz0 = __frcp_rn(a.d0 + a.gam * (float)(f0 + 1));
      rz1 = __frcp_rn(a.d0 + a.gam * (float)(f1 + 1));
    }
    sR = sm + T::HX;
    sB = sR + T::COL;
  }
  // plane z of the region: its cell along z, and whether it is in the domain
  __device__ __forceinline__ int gz(int z) const {
    const int k = z0 + z;
    return PER ? (k < 0 ? k + s : (k >= s ? k - s : k)) : k;
  }
  __device__ __forceinline__ bool zin(int z) const {
    return PER || (z0 + z >= 0 && z0 + z < s);
  }
  // x offset of the red cell of plane z in the pair
  __device__ __forceinline__ bool red1(int z) const { return odd != ((z & 1) != 0); }
  __device__ __forceinline__ float diag(int z, bool red) const {
    if (SIMPLE) return 6.0f;
    if (PER) return a.d0;
    const int k = z0 + z;
    const int nb = (red == red1(z) ? f1 : f0) + (k == 0) + (k == s - 1);
    return a.d0 + a.gam * (float)nb;
  }
  // the Gauss-Seidel value of a cell of plane z (gs_value)
  __device__ __forceinline__ float gs(float s0, float bv, int z, bool red) const {
    if (SIMPLE) return gs_value(s0, bv, a.h2, true, 6.0f);
    const bool one = red == red1(z);
    float r = one ? rd1 : rd0;
    if (!PER && (z0 + z == 0 || z0 + z == s - 1)) r = one ? rz1 : rz0;
    return gs_scaled(s0, bv, a.h2, r);
  }
  __device__ __forceinline__ void load_pair(const Grid& g, int z, float& v0, float& v1) const {
    v0 = 0.0f;
    v1 = 0.0f;
    if (in && zin(z)) {
      const float* p = g.base + (gx + gy * g.sy + gz(z) * g.sz);
      v0 = p[0];
      v1 = p[1];
    }
  }
  // one cell's neighbour sum: partner p, the exposed plane q of the other
  // colour, side offset d, z neighbours zm, zp
  __device__ __forceinline__ float nbs(const float* q, int z, int d, float p, float zm,
                                       float zp) const {
    const float* c = q + z * T::NT + t;
    return nb6(p, c[d], c[-T::HX], c[T::HX], zm, zp);
  }
  __device__ __forceinline__ int side(int z, bool red) const {
    return ((z & 1) != 0) == red ? -de : de;
  }
  // one-colour pass over planes [ZA, RZ - ZA): cells `mine`, neighbours `oth`
  // (registers and exposed planes q), right-hand sides bm; exposes to `me`
  template <int ZA, bool RED, bool ZERO, bool EXPOSE>
  __device__ __forceinline__ void pass(float (&mine)[T::RZ], const float (&oth)[T::RZ],
                                       const float (&bm)[T::RZ], const float* q, float* me) {
#pragma unroll
    for (int z = ZA; z < T::RZ - ZA; ++z) {
      const float s0 = nbs(q, z, side(z, RED), oth[z], oth[z - 1], oth[z + 1]);
      const float v = sor_value(ZERO ? 0.0f : mine[z], gs(s0, bm[z], z, RED));
      mine[z] = (PER || (in && zin(z))) ? v : 0.0f;
      if (EXPOSE) me[z * T::NT + t] = mine[z];
    }
  }
  // the thread's pair lies in the tile (and, ragged, in the domain)
  __device__ __forceinline__ bool interior() const {
    return xp >= TL_H / 2 && xp < T::HX - TL_H / 2 && y >= TL_H && y < T::RY - TL_H && x0 < s &&
           y0 < s;
  }
  __device__ __forceinline__ void store_pair(const Grid& g, int z, float r, float b) const {
    const bool o = red1(z);
    float* p = g.base + (x0 + y0 * g.sy + (z0 + z) * g.sz);
    p[0] = o ? b : r;
    p[1] = o ? r : b;
  }
};

// Down leg of one level: w = two sweeps from zero on A w = b, and the coarse
// right-hand side bc = the 8-cell mean of the residual.
template <class T, bool PER, bool SIMPLE>
__device__ __forceinline__ void tile_down(const TileArgs& a, int bx, int by, int bz, float* sm) {
  TilePass<T, PER, SIMPLE> p(a, bx, by, bz, sm);
  float R[T::RZ], B[T::RZ], bR[T::RZ], bB[T::RZ];
#pragma unroll
  for (int z = 0; z < T::RZ; ++z) {
    float v0, v1;
    p.load_pair(a.b, z, v0, v1);
    const bool o = p.red1(z);
    bR[z] = o ? v1 : v0;
    bB[z] = o ? v0 : v1;
  }
  // red from zero: no neighbours (outside an open domain b is 0, so 0)
#pragma unroll
  for (int z = 0; z < T::RZ; ++z) {
    R[z] = sor_value(0.0f, p.gs(0.0f, bR[z], z, true));
    B[z] = 0.0f;
    p.sR[z * T::NT + p.t] = R[z];
  }
  __syncthreads();
  p.template pass<1, false, true, true>(B, R, bB, p.sR, p.sB);
  __syncthreads();
  p.template pass<2, true, false, true>(R, B, bR, p.sB, p.sR);
  __syncthreads();
  p.template pass<3, false, false, true>(B, R, bB, p.sR, p.sB);
  __syncthreads();
  // residuals of the pair; the odd row of each coarse cell hands its own to
  // the even row's thread, which adds the eight in the restriction's order
  float2* res = reinterpret_cast<float2*>(sm + 2 * T::COL);
  const bool mine = p.interior();
  float r0[T::TZ], r1[T::TZ];
  const int rcol = ((p.y - TL_H) >> 1) * (T::TX / 2) + (p.xp - TL_H / 2);
  if (mine) {
#pragma unroll
    for (int q = 0; q < T::TZ; ++q) {
      const int z = q + TL_H;
      if (p.z0 + z >= p.s) break;
      const float sr = p.nbs(p.sB, z, p.side(z, true), B[z], B[z - 1], B[z + 1]);
      const float sb = p.nbs(p.sR, z, p.side(z, false), R[z], R[z - 1], R[z + 1]);
      const float rr = resid_value(sr, R[z], bR[z], p.diag(z, true), a.inv_h2);
      const float rb = resid_value(sb, B[z], bB[z], p.diag(z, false), a.inv_h2);
      const bool o = p.red1(z);
      r0[q] = o ? rb : rr;
      r1[q] = o ? rr : rb;
      if (p.odd) res[q * (T::TY / 2 * (T::TX / 2)) + rcol] = make_float2(r0[q], r1[q]);
      p.store_pair(a.w, z, R[z], B[z]);
    }
  }
  __syncthreads();
  if (mine && !p.odd) {
    float* bc = a.bc.base + ((p.x0 >> 1) + (p.y0 >> 1) * a.bc.sy);
#pragma unroll
    for (int q = 0; q < T::TZ; q += 2) {
      const int k = p.z0 + TL_H + q;
      if (k >= p.s) break;
      float acc = 0.0f;
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        const float2 o = res[(q + d) * (T::TY / 2 * (T::TX / 2)) + rcol];
        acc = __fadd_rn(acc, r0[q + d]);
        acc = __fadd_rn(acc, r1[q + d]);
        acc = __fadd_rn(acc, o.x);
        acc = __fadd_rn(acc, o.y);
      }
      bc[(k >> 1) * a.bc.sz] = __fmul_rn(0.125f, acc);
    }
  }
}

// Up leg of one level: u = two sweeps on A u = b from w + P uc.
template <class T, bool PER, bool SIMPLE>
__device__ __forceinline__ void tile_up(const TileArgs& a, int bx, int by, int bz, float* sm) {
  TilePass<T, PER, SIMPLE> p(a, bx, by, bz, sm);
  float R[T::RZ], B[T::RZ], bR[T::RZ], bB[T::RZ];
#pragma unroll
  for (int z = 0; z < T::RZ; ++z) p.load_pair(a.w, z, R[z], B[z]);  // x order for now
#pragma unroll
  for (int z = 0; z < T::RZ; ++z) {
    float v0, v1;
    p.load_pair(a.b, z, v0, v1);
    const bool o = p.red1(z);
    bR[z] = o ? v1 : v0;
    bB[z] = o ? v0 : v1;
  }
  // the coarse cells under the region and one around it
  float* pc = sm + 2 * T::COL;
  const int sc = a.uc.s;
  const int cx0 = bx * (T::TX / 2) - TL_H / 2 - 1, cy0 = by * (T::TY / 2) - TL_H / 2 - 1;
  const int cz0 = bz * (T::TZ / 2) - TL_H / 2 - 1;
  for (int e = p.t; e < T::PATCH; e += T::NT) {
    int I = cx0 + e % T::CX, J = cy0 + (e / T::CX) % T::CY, K = cz0 + e / (T::CX * T::CY);
    if (PER) {
      I = I < 0 ? I + sc : (I >= sc ? I - sc : I);
      J = J < 0 ? J + sc : (J >= sc ? J - sc : J);
      K = K < 0 ? K + sc : (K >= sc ? K - sc : K);
    }
    const bool ok = PER || (I >= 0 && I < sc && J >= 0 && J < sc && K >= 0 && K < sc);
    pc[e] = ok ? a.uc.base[I + J * a.uc.sy + K * a.uc.sz] : 0.0f;
  }
  __syncthreads();
  {
    // prolong_mix for the pair's two cells: its x and y interpolations per
    // coarse plane, each used for the four fine planes around it
    const int gI = p.x0 >> 1, gJ = p.y0 >> 1;
    const int gJ2 = p.odd ? gJ + 1 : gJ - 1;
    int oxm = -1, oxp = 1, oy = p.odd ? T::CX : -T::CX;
    float fxm = 1.0f, fxp = 1.0f, fy = 1.0f;
    if (!PER) {
      if (gI - 1 < 0) { oxm = 0; fxm = -a.gam_c; }
      if (gI + 1 >= sc) { oxp = 0; fxp = -a.gam_c; }
      if (gJ2 < 0 || gJ2 >= sc) { oy = 0; fy = -a.gam_c; }
    }
    const float* c0 = pc + ((p.y >> 1) + 1) * T::CX + (p.xp + 1);
    auto plane = [&](int K, float fz, float& A0, float& A1) {
      const float* c = c0 + K * (T::CX * T::CY);
      float q0 = c[0], q0m = c[oxm], q0p = c[oxp];
      float q1 = c[oy], q1m = c[oy + oxm], q1p = c[oy + oxp];
      if (!PER) {
        const float fxy = __fmul_rn(fxm, fy), gxy = __fmul_rn(fxp, fy);
        q0m = __fmul_rn(__fmul_rn(fxm, fz), q0m);
        q0p = __fmul_rn(__fmul_rn(fxp, fz), q0p);
        q1 = __fmul_rn(__fmul_rn(fy, fz), q1);
        q1m = __fmul_rn(__fmul_rn(fxy, fz), q1m);
        q1p = __fmul_rn(__fmul_rn(gxy, fz), q1p);
        q0 = __fmul_rn(fz, q0);
      }
      A0 = lerp34(lerp34(q0, q0m), lerp34(q1, q1m));
      A1 = lerp34(lerp34(q0, q0p), lerp34(q1, q1p));
    };
    float Am0, Am1, Ac0, Ac1, An0, An1;
    plane(0, 1.0f, Am0, Am1);
    plane(1, 1.0f, Ac0, Ac1);
#pragma unroll
    for (int K = 1; K <= T::RZ / 2; ++K) {
      plane(K + 1, 1.0f, An0, An1);
      const int gK = cz0 + K;
      float lo0 = Am0, lo1 = Am1, hi0 = An0, hi1 = An1;
      if (!PER) {
        if (gK == 0) plane(K, -a.gam_c, lo0, lo1);
        if (gK == sc - 1) plane(K, -a.gam_c, hi0, hi1);
      }
#pragma unroll
      for (int d = 0; d < 2; ++d) {
        const int z = 2 * (K - 1) + d;
        const float v0 = __fadd_rn(R[z], lerp34(Ac0, d ? hi0 : lo0));
        const float v1 = __fadd_rn(B[z], lerp34(Ac1, d ? hi1 : lo1));
        const bool o = p.red1(z), ok = PER || (p.in && p.zin(z));
        R[z] = ok ? (o ? v1 : v0) : 0.0f;
        B[z] = ok ? (o ? v0 : v1) : 0.0f;
        p.sB[z * T::NT + p.t] = B[z];
      }
      Am0 = Ac0; Am1 = Ac1; Ac0 = An0; Ac1 = An1;
    }
  }
  __syncthreads();
  p.template pass<1, true, false, true>(R, B, bR, p.sB, p.sR);
  __syncthreads();
  p.template pass<2, false, false, true>(B, R, bB, p.sR, p.sB);
  __syncthreads();
  p.template pass<3, true, false, true>(R, B, bR, p.sB, p.sR);
  __syncthreads();
  p.template pass<4, false, false, false>(B, R, bB, p.sR, p.sB);
  if (p.interior()) {
#pragma unroll
    for (int q = 0; q < T::TZ; ++q) {
      if (p.z0 + TL_H + q >= p.s) break;
      p.store_pair(a.u, q + TL_H, R[q + TL_H], B[q + TL_H]);
    }
  }
}

template <class T, bool UP, bool PER, bool SIMPLE>
__device__ __forceinline__ void tile_one(const TileArgs& a, int bx, int by, int bz, float* sm) {
  if (UP) tile_up<T, PER, SIMPLE>(a, bx, by, bz, sm);
  else tile_down<T, PER, SIMPLE>(a, bx, by, bz, sm);
}

// A tile of an open domain whose region stays a coarse cell away from its
// faces meets no ghost, no ghost-face diagonal and no prolongation ghost: it
// takes the periodic form (nothing wraps), without the per-cell tests and
// factors (128^3 up leg: 33.2 us, 35.7 with the tests in every tile).
template <class T, bool UP, bool SIMPLE>
__device__ __forceinline__ void tile_open(const TileArgs& a, int bx, int by, int bz, float* sm) {
  static_assert(T::TX >= TL_H + 2 && T::TY >= TL_H + 2 && T::TZ >= TL_H + 2, "see inside");
  const int s = a.b.s;
  auto inside = [&](int b, int t) { return b > 0 && (b + 1) * t + TL_H + 2 <= s; };
  if (inside(bx, T::TX) && inside(by, T::TY) && inside(bz, T::TZ))
    tile_one<T, UP, true, SIMPLE>(a, bx, by, bz, sm);
  else
    tile_one<T, UP, false, SIMPLE>(a, bx, by, bz, sm);
}

template <class T, bool UP, bool PER, bool SIMPLE>
__global__ void __launch_bounds__(T::NT, T::NT > 256 ? 2 : 4) k_tile(TileArgs a) {
  __shared__ __align__(16) float sm[T::SMEM];
  pdl_wait();
  pdl_release();
  if (PER) tile_one<T, UP, true, SIMPLE>(a, blockIdx.x, blockIdx.y, blockIdx.z, sm);
  else tile_open<T, UP, SIMPLE>(a, blockIdx.x, blockIdx.y, blockIdx.z, sm);
}

template <class T, bool UP>
__global__ void __launch_bounds__(T::NT, T::NT > 256 ? 2 : 4) kb_tile(const TileDesc* d,
                                                                      const BTable* tab,
                                                                      const int* active) {
  __shared__ __align__(16) float sm[T::SMEM];
  int q;
  BI bi;
  if (!batch_map(d, tab, active, q, bi)) return;
  TileArgs a = d[q].a;  // (a batch solves Poisson's equation: d0 = 6)
  for (Grid* g : {&a.u, &a.b, &a.w, &a.uc, &a.bc}) *g = in_global(*g);
  if (a.periodic) tile_one<T, UP, true, true>(a, bi.x, bi.y, bi.z, sm);
  else if (a.gam == 0.0f) tile_open<T, UP, true>(a, bi.x, bi.y, bi.z, sm);
  else tile_open<T, UP, false>(a, bi.x, bi.y, bi.z, sm);
}

using TileL = TileShape<16, 16, 8>;
using TileS = TileShape<8, 8, 8>;

template <class T>
dim3 grid_of(int s) {
  return dim3((unsigned)((s + T::TX - 1) / T::TX), (unsigned)((s + T::TY - 1) / T::TY),
              (unsigned)((s + T::TZ - 1) / T::TZ));
}

template <class T, bool UP>
void launch_t(cudaStream_t st, const TileArgs& a) {
  const dim3 g = grid_of<T>(a.b.s), b(T::NT);
  const bool simple = (a.periodic || a.gam == 0.0f) && a.d0 == 6.0f;
  if (a.periodic) {
    if (simple) launch_pdl(k_tile<T, UP, true, true>, g, b, 0, st, a);
    else launch_pdl(k_tile<T, UP, true, false>, g, b, 0, st, a);
  } else {
    if (simple) launch_pdl(k_tile<T, UP, false, true>, g, b, 0, st, a);
    else launch_pdl(k_tile<T, UP, false, false>, g, b, 0, st, a);
  }
  note_launch();
}

}  // namespace

// A launch takes as long as its busiest SM: a leg down with 1, 2, 3, 4, 5, 7
// small tiles on an SM 3.7, 4.3, 5.1, 6.1, 8.4, 10.5 us, with 1, 2, 3 large
// ones (four times the cells) 4.9, 6.5, 9.8 us.  So the small shape is taken
// while it puts at most twice the large one's tiles on an SM.  us per leg,
// small / large (periodic, boxes of one side in one launch; 152 SMs):
//   boxes   side  tiles       per SM  down          up
//     1      48   216 /  54   2 / 1   3.6 /  3.9    5.8 /  6.2
//     1      64   512 / 128   4 / 1   6.0 /  5.0    9.3 /  7.3
//     2      48   432 / 108   3 / 1   5.2 /  5.0    7.8 /  7.2
//     4      40   500 / 180   4 / 2   5.8 /  6.4    8.9 /  9.5
//     2      56   686 / 224   5 / 2   8.4 /  6.4   13.0 /  9.5
//    16      24   432 / 192   3 / 2   5.2 /  6.4    7.9 /  9.1
//    16      32  1024 / 256   7 / 2  10.8 /  6.6   16.8 /  9.6
// Over 224 such launches (1 to 32 boxes of side 20 to 128, mixed ones, both
// boundaries) it is 0.2 % from the better shape in the mean, 10 % at worst.
// For one box it draws the line between the sides 48 and 56.
bool tile_small(long long small_tiles, long long large_tiles) {
  constexpr long long SMS = 152;
  return (small_tiles + SMS - 1) / SMS <= 2 * ((large_tiles + SMS - 1) / SMS);
}
bool tile_small(int s) {
  auto count = [&](bool small) {
    const dim3 g = tile_grid(s, small);
    return (long long)g.x * g.y * g.z;
  };
  return tile_small(count(true), count(false));
}

dim3 tile_grid(int s, bool small) { return small ? grid_of<TileS>(s) : grid_of<TileL>(s); }

void launch_tile(cudaStream_t st, const TileArgs& a, bool up, bool small) {
  if (up) {
    if (small) launch_t<TileS, true>(st, a);
    else launch_t<TileL, true>(st, a);
  } else {
    if (small) launch_t<TileS, false>(st, a);
    else launch_t<TileL, false>(st, a);
  }
}

void launch_tile_b(cudaStream_t st, int grid, const TileDesc* d, const BTable* t,
                   const int* active, bool up, bool small) {
  if (grid <= 0) return;
  if (up) {
    if (small) kb_tile<TileS, true><<<grid, TileS::NT, 0, st>>>(d, t, active);
    else kb_tile<TileL, true><<<grid, TileL::NT, 0, st>>>(d, t, active);
  } else {
    if (small) kb_tile<TileS, false><<<grid, TileS::NT, 0, st>>>(d, t, active);
    else kb_tile<TileL, false><<<grid, TileL::NT, 0, st>>>(d, t, active);
  }
  note_launch();
}

}  // namespace pm
