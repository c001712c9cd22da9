// Staggered MAC-grid stencils (Sec. 3.1): the Neumann Laplacian L = G^T G of
// Eq. (Saddle), the gradient G and its transpose G^T = -div, and the pieces of
// the BDF2 momentum predictor of Eq. (ustar) (Helmholtz operator, explicit
// convective term, right-hand side).
//
// Thread layout: one thread per grid point, blocks of 32 x 8 in (x, y) and one
// z-plane per blockIdx.z, so that a warp reads 32 consecutive x values of each
// neighbour row (coalesced; the y/z neighbours hit L1/L2).
#include <algorithm>
#include <cstring>
#include <type_traits>

#include "ds.cuh"
#include "ibm_internal.cuh"

namespace ibm {

namespace {

constexpr int BX = 32, BY = 8;

// Geometry of the packed face vector: comp c has n[c][axis] points per axis.
struct FaceGeom {
  int n[3][3];
  int64_t off[3];
  int64_t sy[3], sz[3];
};

FaceGeom make_face_geom(Dims d) {
  FaceGeom g;
  FaceDims f = face_dims(d);
  int base[3] = {d.nx, d.ny, d.nz};
  for (int c = 0; c < 3; ++c) {
    for (int a = 0; a < 3; ++a) g.n[c][a] = base[a] + (a == c ? 1 : 0);
    g.sy[c] = g.n[c][0];
    g.sz[c] = (int64_t)g.n[c][0] * g.n[c][1];
  }
  g.off[0] = 0;
  g.off[1] = f.nfx;
  g.off[2] = f.nfx + f.nfy;
  return g;
}


dim3 cell_grid(Dims d) { return dim3(div_up(d.nx, BX), div_up(d.ny, BY), d.nz); }

// ---------------------------------------------------------------------------
// L v = G^T G v: sum over existing neighbours of (v_c - v_n) / h^2.
template <typename T>
__global__ void __launch_bounds__(BX * BY) k_laplacian(Dims d, const T* __restrict__ v,
                                                       T* __restrict__ out, T inv_h2) {
  const int i = blockIdx.x * BX + threadIdx.x;
  const int j = blockIdx.y * BY + threadIdx.y;
  const int k = blockIdx.z;
  if (i >= d.nx || j >= d.ny) return;
  const int64_t sy = d.nx, sz = (int64_t)d.nx * d.ny;
  const int64_t c = k * sz + j * sy + i;
  const T vc = __ldg(v + c);
  T r;
  if (i > 0 && i < d.nx - 1 && j > 0 && j < d.ny - 1 && k > 0 && k < d.nz - 1) {
    const T s = ((__ldg(v + c - 1) + __ldg(v + c + 1)) + (__ldg(v + c - sy) + __ldg(v + c + sy))) +
                (__ldg(v + c - sz) + __ldg(v + c + sz));
    r = fma((T)6, vc, -s);
  } else {
    T s = 0;
    int nn = 0;
    if (i > 0) { s += __ldg(v + c - 1); ++nn; }
    if (i < d.nx - 1) { s += __ldg(v + c + 1); ++nn; }
    if (j > 0) { s += __ldg(v + c - sy); ++nn; }
    if (j < d.ny - 1) { s += __ldg(v + c + sy); ++nn; }
    if (k > 0) { s += __ldg(v + c - sz); ++nn; }
    if (k < d.nz - 1) { s += __ldg(v + c + sz); ++nn; }
    r = fma((T)nn, vc, -s);
  }
  out[c] = r * inv_h2;
}

// ---------------------------------------------------------------------------
// FP64 Laplacian with the stencil sum formed exactly in integers.  GB300
// issues FP64 arithmetic at about 1/58 of its FP32 rate, so the seven-term
// FP64 sum bounds k_laplacian<double> far below the HBM rate.  Here each
// value v = m 2^(e - 1075) (m the signed 53-bit significand, e the biased
// exponent; a subnormal has e = 1 and no implicit bit) is aligned to the
// largest exponent E of the seven with kLapGuard extra low bits, and
// S = nn m_c - sum_nb m_nb is summed in 64-bit integers: the bits dropped
// below 2^(E - 1075 - kLapGuard) amount to at most 7 2^-kLapGuard units in
// the last place of the largest term, less than the rounding error of the
// FP64 sum.  Then out = (double)S 2^(E - 1075 - kLapGuard) / h^2 with two
// roundings (the conversion and one multiplication; the scale is 1/h^2 with
// E - 1080 added to its exponent field).  Non-finite values, and sums whose
// scale would leave the normal range, take the FP64 formula.
constexpr int kLapGuard = 5;

struct FxVal {
  int e;
  long long m;
};

__device__ __forceinline__ FxVal fx_unpack(double v) {
  const long long u = __double_as_longlong(v);
  int e = (int)((u >> 52) & 0x7ff);
  long long m = u & 0xFFFFFFFFFFFFFLL;
  if (e != 0)
    m |= 1LL << 52;
  else
    e = 1;
  return {e, u < 0 ? -m : m};
}

// m 2^kLapGuard shifted down to exponent E (|m| < 2^56, so no overflow)
__device__ __forceinline__ long long fx_align(long long m, int e, int E) {
  return (m * (1LL << kLapGuard)) >> min(E - e, 63);
}

// (nn v_c - sum of the six neighbour values) / h^2; an absent neighbour is 0
__device__ __forceinline__ double lap_fx(double vc, double xm, double xp, double ym, double yp,
                                         double zm, double zp, int nn, long long inv_h2_bits,
                                         int e_min, int e_max) {
  const FxVal c = fx_unpack(vc), a0 = fx_unpack(xm), a1 = fx_unpack(xp), a2 = fx_unpack(ym),
              a3 = fx_unpack(yp), a4 = fx_unpack(zm), a5 = fx_unpack(zp);
  const int E = max(max(max(c.e, a0.e), max(a1.e, a2.e)), max(max(a3.e, a4.e), a5.e));
  if (E < e_min || E > e_max) {
    const double s = ((xm + xp) + (ym + yp)) + (zm + zp);
    return fma((double)nn, vc, -s) * __longlong_as_double(inv_h2_bits);
  }
  long long S = fx_align(c.m * nn, c.e, E);
  S -= fx_align(a0.m, a0.e, E) + fx_align(a1.m, a1.e, E);
  S -= fx_align(a2.m, a2.e, E) + fx_align(a3.m, a3.e, E);
  S -= fx_align(a4.m, a4.e, E) + fx_align(a5.m, a5.e, E);
  const double scale =
      __longlong_as_double(inv_h2_bits + (long long)(E - 1075 - kLapGuard) * (1LL << 52));
  return __ll2double_rn(S) * scale;
}

// One cell per thread, blocks of 32 x 8 cells over zc z-planes: x-neighbours
// by shuffles (loads at the warp edges), z-neighbours from the registers of
// the march, y-neighbours through L1.
__global__ void __launch_bounds__(BX * BY) k_laplacian_fx(Dims d, const double* __restrict__ v,
                                                          const double* __restrict__ bsub,
                                                          double* __restrict__ out,
                                                          long long inv_h2_bits, int e_min,
                                                          int e_max, int zc) {
  const int lane = threadIdx.x;
  const int i = blockIdx.x * BX + lane;
  const int j = blockIdx.y * BY + threadIdx.y;
  const bool act = i < d.nx && j < d.ny;
  const int z0 = blockIdx.z * zc;
  const int z1 = min(z0 + zc, d.nz);
  const int64_t sy = d.nx, sz = (int64_t)d.nx * d.ny;
  int64_t c = (int64_t)z0 * sz + (int64_t)j * sy + i;
  const bool hxm = i > 0, hxp = i < d.nx - 1, hym = j > 0, hyp = j < d.ny - 1;
  const int nxy = (int)hxm + (int)hxp + (int)hym + (int)hyp;
  double vp = (act && z0 > 0) ? __ldg(v + c - sz) : 0.0;
  double vc = act ? __ldg(v + c) : 0.0;
  for (int z = z0; z < z1; ++z, c += sz) {
    double vn = 0.0, ym = 0.0, yp = 0.0;
    if (act) {
      if (z + 1 < d.nz) vn = __ldg(v + c + sz);
      if (hym) ym = __ldg(v + c - sy);
      if (hyp) yp = __ldg(v + c + sy);
    }
    double xm = __shfl_up_sync(0xffffffffu, vc, 1);
    double xp = __shfl_down_sync(0xffffffffu, vc, 1);
    if (lane == 0) xm = (act && hxm) ? __ldg(v + c - 1) : 0.0;
    if (lane == 31) xp = (act && hxp) ? __ldg(v + c + 1) : 0.0;
    if (!hxm) xm = 0.0;
    if (!hxp) xp = 0.0;
    const int nn = nxy + (z > 0) + (z < d.nz - 1);
    if (act) {
      const double lv = lap_fx(vc, xm, xp, ym, yp, vp, vn, nn, inv_h2_bits, e_min, e_max);
      out[c] = bsub ? __ldg(bsub + c) - lv : lv;   // b - L v for the true residual
    }
    vp = vc;
    vc = vn;
  }
}

// Scale limits for a fixed-point sum scaled by `scale` (as in lap_fx): the
// scale 2^(E - 1075 - kLapGuard) * scale is formed by adding E - 1075 -
// kLapGuard to the exponent field of `scale`, which must stay in [1, 2046];
// anything else (a non-finite value; a scale that is zero, subnormal or not
// finite) takes the FP64 formula.
struct FxLimits {
  long long bits;
  int e_min, e_max;
};

FxLimits fx_limits(double scale) {
  FxLimits L;
  std::memcpy(&L.bits, &scale, sizeof(L.bits));
  const int e_h = (int)((L.bits >> 52) & 0x7ff);
  L.e_min = std::max(1075 + kLapGuard + 1 - e_h, 1);
  L.e_max = std::min(2046 + 1075 + kLapGuard - e_h, 2046);
  if (e_h == 0 || e_h == 0x7ff) L.e_min = 2047;
  return L;
}

// alpha ((a0 - a1) + (a2 - a3) + (a4 - a5)) with the sum formed exactly in
// 64-bit integers as in lap_fx (|S| < 6 2^58)
__device__ __forceinline__ double div_fx(double a0, double a1, double a2, double a3, double a4,
                                         double a5, FxLimits L) {
  const FxVal v0 = fx_unpack(a0), v1 = fx_unpack(a1), v2 = fx_unpack(a2), v3 = fx_unpack(a3),
              v4 = fx_unpack(a4), v5 = fx_unpack(a5);
  const int E = max(max(max(v0.e, v1.e), max(v2.e, v3.e)), max(v4.e, v5.e));
  if (E < L.e_min || E > L.e_max)
    return __longlong_as_double(L.bits) * (((a0 - a1) + (a2 - a3)) + (a4 - a5));
  long long S = fx_align(v0.m, v0.e, E) - fx_align(v1.m, v1.e, E);
  S += fx_align(v2.m, v2.e, E) - fx_align(v3.m, v3.e, E);
  S += fx_align(v4.m, v4.e, E) - fx_align(v5.m, v5.e, E);
  const double scale =
      __longlong_as_double(L.bits + (long long)(E - 1075 - kLapGuard) * (1LL << 52));
  return __ll2double_rn(S) * scale;
}

// out = alpha * G^T u + beta * cin (cin may be null), (G^T u)_c = sum_d
// (u_{c-1/2} - u_{c+1/2}) over interior faces (wall faces read as 0), the
// sum formed exactly (div_fx).  One cell per thread, blocks of 32 x 8 cells
// over zc planes: the upper x-face from the next lane, the lower z-face from
// the march, the y-faces through L1.  NORM: instead of out, the block's sum
// of the squared values (FP64, fixed order) goes to sq_part[block].
template <bool NORM>
__global__ void __launch_bounds__(BX * BY) k_gradt_fx(Dims d, FaceGeom g,
                                                      const double* __restrict__ u, FxLimits L,
                                                      const double* __restrict__ cin,
                                                      double beta, double* __restrict__ out,
                                                      double* __restrict__ sq_part, int zc) {
  const int lane = threadIdx.x;
  const int i = blockIdx.x * BX + lane;
  const int j = blockIdx.y * BY + threadIdx.y;
  const bool act = i < d.nx && j < d.ny;
  const int z0 = blockIdx.z * zc;
  const int z1 = min(z0 + zc, d.nz);
  const double* ux = u + g.off[0];
  const double* uy = u + g.off[1];
  const double* uz = u + g.off[2];
  // interior faces: x-faces 1..nx-1, y-faces 1..ny-1, z-faces 1..nz-1
  const bool xlo = i > 0, xhi = i + 1 < d.nx, ylo = j > 0, yhi = j + 1 < d.ny;
  double zlo = (act && z0 > 0) ? __ldg(uz + (int64_t)z0 * g.sz[2] + (int64_t)j * g.sy[2] + i) : 0.0;
  double sq = 0.0;
  for (int z = z0; z < z1; ++z) {
    const int64_t fx = (int64_t)z * g.sz[0] + (int64_t)j * g.sy[0] + i;
    const int64_t fy = (int64_t)z * g.sz[1] + (int64_t)j * g.sy[1] + i;
    double a0 = 0.0, a2 = 0.0, a3 = 0.0, zhi = 0.0;
    if (act) {
      if (xlo) a0 = __ldg(ux + fx);
      if (ylo) a2 = __ldg(uy + fy);
      if (yhi) a3 = __ldg(uy + fy + g.sy[1]);
      if (z + 1 < d.nz) zhi = __ldg(uz + (int64_t)(z + 1) * g.sz[2] + (int64_t)j * g.sy[2] + i);
    }
    // the upper x-face of cell i is the lower one of cell i + 1
    double a1 = __shfl_down_sync(0xffffffffu, a0, 1);
    if (lane == 31) a1 = (act && xhi) ? __ldg(ux + fx + 1) : 0.0;
    if (!xhi) a1 = 0.0;
    if (act) {
      const double v = div_fx(a0, a1, a2, a3, zlo, zhi, L);
      if constexpr (NORM) {
        sq = fma(v, v, sq);
      } else {
        const int64_t c = ((int64_t)z * d.ny + j) * d.nx + i;
        out[c] = cin ? fma(beta, __ldg(cin + c), v) : v;
      }
    }
    zlo = zhi;
  }
  if constexpr (NORM) {
    __shared__ double sh[BY];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_down_sync(0xffffffffu, sq, o);
    if (lane == 0) sh[threadIdx.y] = sq;
    __syncthreads();
    if (lane == 0 && threadIdx.y == 0) {
      double t = 0.0;
#pragma unroll
      for (int w = 0; w < BY; ++w) t += sh[w];
      sq_part[((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x] = t;
    }
  }
}

// u = u_in + alpha * G p on interior faces, 0 on wall faces (u_in may be
// null; it may be u).  Thread (i, j) marches over the z-planes 0..nz and
// writes the x-, y- and z-faces at (i, j, k) that exist: p(i-1) comes from
// the previous lane, p(k-1) from the march, p(j-1) through L1.
__global__ void __launch_bounds__(BX * BY) k_grad_axpy(Dims d, FaceGeom g,
                                                       const double* __restrict__ u_in,
                                                       const double* __restrict__ p,
                                                       double alpha, double* __restrict__ u,
                                                       int zc) {
  const int lane = threadIdx.x;
  const int i = blockIdx.x * BX + lane;
  const int j = blockIdx.y * BY + threadIdx.y;
  const bool col = i <= d.nx && j <= d.ny;      // some face of this column exists
  const bool cell = i < d.nx && j < d.ny;       // the cell column exists
  const int z0 = blockIdx.z * zc;
  const int z1 = min(z0 + zc, d.nz + 1);
  const int64_t sy = d.nx, sz = (int64_t)d.nx * d.ny;
  auto pc_at = [&](int k) { return (int64_t)k * sz + (int64_t)j * sy + i; };
  double pzm = (cell && z0 > 0 && z0 - 1 < d.nz) ? __ldg(p + pc_at(z0 - 1)) : 0.0;
  for (int k = z0; k < z1; ++k) {
    const bool kin = k < d.nz;
    const double pc = (cell && kin) ? __ldg(p + pc_at(k)) : 0.0;
    double pxm = __shfl_up_sync(0xffffffffu, pc, 1);
    if (lane == 0) pxm = (i > 0 && i - 1 < d.nx && j < d.ny && kin) ? __ldg(p + pc_at(k) - 1) : 0.0;
    if (col) {
      // x-face (i, j, k): i in 0..nx, j < ny, k < nz
      if (j < d.ny && kin) {
        const int64_t f = g.off[0] + (int64_t)k * g.sz[0] + (int64_t)j * g.sy[0] + i;
        double val = 0.0;
        if (i > 0 && i < d.nx) {
          const double gp = pc - pxm;
          val = u_in ? fma(alpha, gp, __ldg(u_in + f)) : alpha * gp;
        }
        u[f] = val;
      }
      // y-face (i, j, k): i < nx, j in 0..ny, k < nz
      if (i < d.nx && kin) {
        const int64_t f = g.off[1] + (int64_t)k * g.sz[1] + (int64_t)j * g.sy[1] + i;
        double val = 0.0;
        if (j > 0 && j < d.ny) {
          const double gp = pc - __ldg(p + pc_at(k) - sy);
          val = u_in ? fma(alpha, gp, __ldg(u_in + f)) : alpha * gp;
        }
        u[f] = val;
      }
      // z-face (i, j, k): i < nx, j < ny, k in 0..nz
      if (cell) {
        const int64_t f = g.off[2] + (int64_t)k * g.sz[2] + (int64_t)j * g.sy[2] + i;
        double val = 0.0;
        if (k > 0 && k < d.nz) {
          const double gp = pc - pzm;
          val = u_in ? fma(alpha, gp, __ldg(u_in + f)) : alpha * gp;
        }
        u[f] = val;
      }
    }
    pzm = pc;
  }
}

// Predictor Helmholtz operator on the d-faces, A = a I - nu Lap_h with the
// no-slip ghosts: A e = diag e_c - (nu / h^2) * (sum of neighbours), where the
// face-normal axis reads the wall faces (which hold 0) and each cell-centred
// axis adds nu / h^2 to diag for every missing neighbour (ghost = -e_c).
// Kernels below march along z over zc planes; blockIdx.z = comp * zchunks +
// chunk, so one launch covers the three face grids.
// x[c] for a runtime c in 0..2 without dynamic indexing (which would copy a
// kernel-parameter struct to local memory)
template <typename T>
__device__ __forceinline__ T sel3(int c, T a, T b, T d) {
  return c == 0 ? a : (c == 1 ? b : d);
}


// u_E at (x, y, z) of its own face grid, split into an FP32 pair
template <int E>
__device__ __forceinline__ dsf ldu(const FaceGeom& g, const double* __restrict__ u, int x, int y,
                                   int z) {
  return split_exact(__ldg(u + g.off[E] + (int64_t)z * g.sz[E] + (int64_t)y * g.sy[E] + x));
}

// Convective flux on the edge between the C-face at (x, y, z) and the E-face
// index q along E (E != C): (sum of the two u_E adjacent along C) times
// (sum of the two u_C adjacent along E); 0 on the walls (q = 0 or the last
// E-face).  For an interior C-face every value read is an interior face.
template <int C, int E>
__device__ __forceinline__ dsf edge_flux_ds(const FaceGeom& g, const double* __restrict__ u,
                                            int x, int y, int z, int q) {
  if (q <= 0 || q >= g.n[E][E] - 1) return dsf{0.f, 0.f};
  const int ax = E == 0 ? q : x, ay = E == 1 ? q : y, az = E == 2 ? q : z;
  const dsf ue = ds_add_d(ldu<E>(g, u, ax - (C == 0), ay - (C == 1), az - (C == 2)),
                        ldu<E>(g, u, ax, ay, az));
  const dsf uc = ds_add_d(ldu<C>(g, u, ax - (E == 0), ay - (E == 1), az - (E == 2)),
                        ldu<C>(g, u, ax, ay, az));
  return ds_mul(ue, uc);
}

// The same flux in FP64 straight from the FP64 values (no splits): the
// kernel below forms one pair of fluxes per face this way, on the FP64
// pipe, which its double-single arithmetic leaves idle.
template <int C, int E>
__device__ __forceinline__ double edge_flux_f64(const FaceGeom& g, const double* __restrict__ u,
                                                int x, int y, int z, int q) {
  if (q <= 0 || q >= g.n[E][E] - 1) return 0.0;
  const int ax = E == 0 ? q : x, ay = E == 1 ? q : y, az = E == 2 ? q : z;
  auto at = [&](int e, int xx, int yy, int zz) {
    return __ldg(u + g.off[e] + (int64_t)zz * g.sz[e] + (int64_t)yy * g.sy[e] + xx);
  };
  const double ue = at(E, ax - (C == 0), ay - (C == 1), az - (C == 2)) + at(E, ax, ay, az);
  const double uc = at(C, ax - (E == 0), ay - (E == 1), az - (E == 2)) + at(C, ax, ay, az);
  return ue * uc;
}

// Right-hand side of the predictor, Eq. (ustar), with the convective term
// fused in, for the C-faces:
//   rhs = (4 u^n - u^{n-1}) / (2 dt) - G p^n + f - A(u^n) on interior faces
// (0 on wall faces).  A is the central divergence form on the MAC grid (the
// cell-centred square of u_C averaged along C, and on the edges the product
// of u_E averaged along C with u_C averaged along E, 0 on walls) with the 1/2
// averages folded into one factor 1/4:
//   4 A = [ (u_+ + u_0)^2 - (u_0 + u_-)^2 ] along C
//       + sum over the two other axes of (flux at the upper edge - lower edge).
// The march runs along z; the flux through the lower z-edge (or, for u_z, the
// lower cell-centred square) is the previous face's upper one and is reused.
// The FP64 pipe of GB300 is ~58x slower than its FP32 pipes, so the FP64
// inputs are split into FP32 pairs (split_exact, integer operations, 2^-46
// relative) and the formula is evaluated in double-single arithmetic; its
// sums take Dekker's addition (ds_add_d), whose error, a few units of 2^-46
// of the operands, is of the order the inputs' splits already carry.  One
// pair of edge fluxes per face (the y-edges of u_x and u_z, the x-edges of
// u_y) is formed in FP64 from the FP64 values instead, which keeps the
// otherwise idle FP64 pipe busy and saves their splits; their difference
// joins the sum as a pair.  The FP64 result is the exact sum of the pair
// (one FP64 add).
// Templating on C makes every stride and boundary test a compile-time case.
// (The pointers' __restrict__ is the kernels': repeated here it cost 5%.)
template <int C>
__device__ __forceinline__ void predictor_rhs(const Dims& d, const FaceGeom& g, const double* un,
                                              const double* unm1, const double* pn,
                                              const double* fb, int with_adv, dsf c4, dsf c1,
                                              dsf cp_h, dsf ca, double* rhs, int z0, int planes) {
  const int lane = threadIdx.x;
  const int i = blockIdx.x * BX + lane;
  const int j = blockIdx.y * BY + threadIdx.y;
  const int n0 = g.n[C][0], n1 = g.n[C][1], n2 = g.n[C][2];
  // u_y and u_z faces share their x-edge fluxes between neighbouring lanes,
  // so lanes past the last face stay in the march (without loads or stores);
  // a row past the last one leaves as a whole warp
  const bool act = i < n0;
  if (j >= n1 || (C == 0 && !act)) return;
  const int z1 = min(z0 + planes, n2);
  const int64_t sy = g.sy[C], sz = g.sz[C];
  int64_t f = g.off[C] + (int64_t)z0 * sz + (int64_t)j * sy + i;
  const bool col_wall = (C == 0 && (i == 0 || i == n0 - 1)) || (C == 1 && (j == 0 || j == n1 - 1));
  if (col_wall) {
    if (act)
      for (int z = z0; z < z1; ++z, f += sz) rhs[f] = 0.0;
    return;
  }
  const int64_t csy = d.nx, csz = (int64_t)d.nx * d.ny;
  const int64_t cstr = C == 0 ? 1 : (C == 1 ? csy : csz);
  const dsf Z = {0.f, 0.f};
  auto sq = [](dsf x) { return ds_mul(x, x); };
  // lower z-flux (C = 0, 1) or lower cell-centred square (C = 2)
  dsf carry = Z;
  if (with_adv && act) {
    if (C == 2) {
      const dsf lo = (z0 - 1 >= 1) ? ldu<2>(g, un, i, j, z0 - 1) : Z;
      const dsf mid = (z0 >= 1 && z0 <= n2 - 2) ? ldu<2>(g, un, i, j, z0) : Z;
      carry = sq(ds_add_d(lo, mid));
    } else {
      carry = edge_flux_ds<C, 2>(g, un, i, j, z0, z0);
    }
  }
  // the flux through the x-edge at q = i + 1 of this lane is the flux
  // through the x-edge at q = i of the next lane (the same values, the same
  // operations); lane 0 forms its lower one itself
  auto xflux_pair = [&](auto fn, dsf& lower) {
    const dsf up = act ? fn(i + 1) : Z;
    lower.hi = __shfl_up_sync(0xffffffffu, up.hi, 1);
    lower.lo = __shfl_up_sync(0xffffffffu, up.lo, 1);
    if (lane == 0) lower = act ? fn(i) : Z;
    return up;
  };
  for (int z = z0; z < z1; ++z, f += sz) {
    if (C == 2 && (z == 0 || z == n2 - 1)) {
      if (!act) continue;
      rhs[f] = 0.0;
      if (with_adv) {
        const dsf mid = (z >= 1 && z <= n2 - 2) ? ldu<2>(g, un, i, j, z) : Z;
        const dsf hi = (z + 1 <= n2 - 2) ? ldu<2>(g, un, i, j, z + 1) : Z;
        carry = sq(ds_add_d(mid, hi));
      }
      continue;
    }
    // x-edge fluxes (shared between lanes: every lane takes part); for u_y
    // in FP64 (its pair of fluxes on the FP64 pipe)
    dsf fx_lo = Z, fx_up = Z;
    double fx64_lo = 0.0, fx64_up = 0.0;
    if (with_adv && C == 2) {
      fx_up = xflux_pair([&](int q) { return edge_flux_ds<2, 0>(g, un, i, j, z, q); }, fx_lo);
    } else if (with_adv && C == 1) {
      fx64_up = act ? edge_flux_f64<1, 0>(g, un, i, j, z, i + 1) : 0.0;
      fx64_lo = __shfl_up_sync(0xffffffffu, fx64_up, 1);
      if (lane == 0) fx64_lo = act ? edge_flux_f64<1, 0>(g, un, i, j, z, i) : 0.0;
    }
    if (!act) continue;
    const int64_t cp = (int64_t)z * csz + (int64_t)j * csy + i;   // cell on the + side
    const dsf u0 = split_exact(__ldg(un + f));
    // 4/(2dt) u^n - 1/(2dt) u^{n-1} - (p_+ - p_-)/h (+ f)
    dsf v = ds_add_d(ds_mul(c4, u0), ds_neg(ds_mul(c1, split_exact(__ldg(unm1 + f)))));
    const dsf dp = ds_add_d(split_exact(__ldg(pn + cp)), ds_neg(split_exact(__ldg(pn + cp - cstr))));
    v = ds_add_d(v, ds_neg(ds_mul(cp_h, dp)));
    if (fb) v = ds_add_d(v, split_exact(__ldg(fb + f)));
    if (with_adv) {
      dsf acc;
      if (C == 2) {
        const dsf up = (z + 1 <= n2 - 2) ? ldu<2>(g, un, i, j, z + 1) : Z;
        const dsf up2 = sq(ds_add_d(u0, up));
        acc = ds_add_d(up2, ds_neg(carry));
        carry = up2;
        acc = ds_add_d(acc, ds_add_d(fx_up, ds_neg(fx_lo)));
        // y-edges in FP64
        acc = ds_add_d(acc, split_exact(edge_flux_f64<2, 1>(g, un, i, j, z, j + 1) -
                                        edge_flux_f64<2, 1>(g, un, i, j, z, j)));
      } else {
        // own axis: (u_+ - u_-)(u_+ + 2 u_0 + u_-), wall faces read as 0
        constexpr int O = 1 - C;   // the other in-plane axis
        const int pc = C == 0 ? i : j, nc = C == 0 ? n0 : n1;
        const dsf up = (pc + 1 <= nc - 2) ? ldu<C>(g, un, i + (C == 0), j + (C == 1), z) : Z;
        const dsf um = (pc - 1 >= 1) ? ldu<C>(g, un, i - (C == 0), j - (C == 1), z) : Z;
        const dsf two_u0 = {2.f * u0.hi, 2.f * u0.lo};
        acc = ds_mul(ds_add_d(up, ds_neg(um)), ds_add_d(ds_add_d(up, um), two_u0));
        // the other in-plane axis's pair of fluxes in FP64 (x for u_y, y for u_x)
        if (O == 0) {
          acc = ds_add_d(acc, split_exact(fx64_up - fx64_lo));
        } else {
          acc = ds_add_d(acc, split_exact(edge_flux_f64<C, O>(g, un, i, j, z, j + 1) -
                                          edge_flux_f64<C, O>(g, un, i, j, z, j)));
        }
        const dsf fz = edge_flux_ds<C, 2>(g, un, i, j, z, z + 1);
        acc = ds_add_d(acc, ds_add_d(fz, ds_neg(carry)));
        carry = fz;
      }
      v = ds_add_d(v, ds_neg(ds_mul(ca, acc)));
    }
    rhs[f] = f2d_exact(v.hi) + f2d_exact(v.lo);
  }
}

// One component per launch, marches of kRhsPlanes planes.
constexpr int kRhsPlanes = 16;

template <int C>
__global__ void __launch_bounds__(BX * BY) k_predictor_rhs_ds(
    Dims d, FaceGeom g, const double* __restrict__ un, const double* __restrict__ unm1,
    const double* __restrict__ pn, const double* __restrict__ fb, int with_adv, dsf c4, dsf c1,
    dsf cp_h, dsf ca, double* __restrict__ rhs) {
  predictor_rhs<C>(d, g, un, unm1, pn, fb, with_adv, c4, c1, cp_h, ca, rhs,
                   blockIdx.z * kRhsPlanes, kRhsPlanes);
}

// The three components in one launch (blockIdx.z = component * zchunks + chunk),
// for grids that do not fill the chip with marches of 16 planes: one launch per
// component took 160 us at 32^3 and 243 us at 128^3, where their few blocks left
// it idle; together, with fewer planes, 9 and 215.
__global__ void __launch_bounds__(BX * BY) k_predictor_rhs_all(
    Dims d, FaceGeom g, const double* __restrict__ un, const double* __restrict__ unm1,
    const double* __restrict__ pn, const double* __restrict__ fb, int with_adv, dsf c4, dsf c1,
    dsf cp_h, dsf ca, double* __restrict__ rhs, int zc, int zchunks) {
  const int c = blockIdx.z / zchunks;
  const int z0 = (blockIdx.z - c * zchunks) * zc;
  const int n0 = sel3(c, g.n[0][0], g.n[1][0], g.n[2][0]);
  const int n2 = sel3(c, g.n[0][2], g.n[1][2], g.n[2][2]);
  if (z0 >= n2 || (int)blockIdx.x * BX >= n0) return;   // block-uniform
  if (c == 0)
    predictor_rhs<0>(d, g, un, unm1, pn, fb, with_adv, c4, c1, cp_h, ca, rhs, z0, zc);
  else if (c == 1)
    predictor_rhs<1>(d, g, un, unm1, pn, fb, with_adv, c4, c1, cp_h, ca, rhs, z0, zc);
  else
    predictor_rhs<2>(d, g, un, unm1, pn, fb, with_adv, c4, c1, cp_h, ca, rhs, z0, zc);
}

// The predictor's FP32 work arrays hold the faces of a component by colour
// (i + j + k even: colour 0, odd: colour 1), so that one colour of the
// red-black Chebyshev steps below is contiguous: [component][colour][k][j][q],
// q = i / 2, rows padded to a multiple of 4 values (16-byte alignment).  The
// x-neighbours of element q of one colour are the elements q and q - 1 (i
// even) or q and q + 1 (i odd) of the other colour's row, the y- and
// z-neighbours its elements q of the rows beside.  Padding, and the wall face
// i = nx of u_x when nx is odd, hold 0 (also where faces hold infinities or
// NaN); when nx is even that face has no place.
struct HelmGeom {
  int nx;
  int nq;              // elements per row and colour, ceil(nx / 2)
  int n[3][3];         // faces per axis of each component
  int64_t off[3], cs[3], sz[3];   // component, colour and plane strides
  int64_t sy;          // row stride
};

HelmGeom make_helm_geom(Dims d) {
  const FaceGeom g = make_face_geom(d);
  HelmGeom p;
  p.nx = d.nx;
  p.nq = (d.nx + 1) / 2;
  p.sy = (p.nq + 3) / 4 * 4;
  int64_t off = 0;
  for (int c = 0; c < 3; ++c) {
    for (int a = 0; a < 3; ++a) p.n[c][a] = g.n[c][a];
    p.sz[c] = p.sy * g.n[c][1];
    p.cs[c] = p.sz[c] * g.n[c][2];
    p.off[c] = off;
    off += 2 * p.cs[c];
  }
  return p;
}

constexpr unsigned kFullMask = 0xffffffffu;
constexpr int kHelmThreads = 256;

// One of four weights by the number of ghost neighbours (0..3)
__device__ __forceinline__ float by_ghosts(float4 w, int g) {
  return g == 0 ? w.x : (g == 1 ? w.y : (g == 2 ? w.z : w.w));
}

// Ghost neighbours of a component's row or plane: a cell-centred axis has one
// at each wall, the face-normal axis none.
__device__ __forceinline__ int ghosts(bool centred, int x, int n) {
  return centred ? (x == 0) + (x == n - 1) : 0;
}

// One half-step of the cyclic (red-black) Chebyshev iteration for A e = r:
// the faces of colour col are updated in place from the other colour,
//   e <- e + omega (D^{-1} (r + N e_other) - e),   A = D - N,
// as e = w (r + nu s) + (1 - omega) e with s the neighbour sum and
// w = omega / D (by ghost count).  The iterates of both colours at steps n and
// n + 1 are those of the full Chebyshev iteration on D^{-1} A (half of its
// values each), so a full iteration's convergence takes half its work
// (Golub and Varga's cyclic Chebyshev semi-iterative method).
// Four elements per thread (float4), LX threads per row, z-neighbours from the
// march, x by one shuffle, y through L1.  old_zero: e of this colour is zero
// and not read.  Weights are 0 at wall faces, where e is and stays 0.  FULL: nx is
// a multiple of 8, so rows have no padding and only the first and last element
// of a row can differ from the row's others.  Bound by HBM and instruction
// issue: 16 B per updated face, 8 B per face of the grid.
template <int LX, bool FULL>
__global__ void __launch_bounds__(kHelmThreads) k_helm_half(HelmGeom p, int zc, int zchunks,
                                                            int col, float* e,
                                                            const float* __restrict__ r, float nu,
                                                            float4 w, float omw, int old_zero,
                                                            int rev) {
  pdl_wait();
  pdl_trigger();
  constexpr int kRows = kHelmThreads / LX;
  const int bz = z_block(rev);
  const int c = bz / zchunks;
  const int z0 = (bz - c * zchunks) * zc;
  const int n1 = sel3(c, p.n[0][1], p.n[1][1], p.n[2][1]);
  const int n2 = sel3(c, p.n[0][2], p.n[1][2], p.n[2][2]);
  if (z0 >= n2 || (int)blockIdx.y * kRows >= n1) return;   // block-uniform
  const int z1 = min(z0 + zc, n2);
  const int tx = threadIdx.x;
  const int j = blockIdx.y * kRows + threadIdx.y;
  const int q0 = 4 * (blockIdx.x * LX + tx);
  const bool act = q0 < p.nq && j < n1;
  const int64_t cs = sel3(c, p.cs[0], p.cs[1], p.cs[2]), sz = sel3(c, p.sz[0], p.sz[1], p.sz[2]);
  const int64_t base = sel3(c, p.off[0], p.off[1], p.off[2]) + (int64_t)z0 * sz +
                       (int64_t)j * p.sy + q0;
  const float* eo = e + base + (1 - col) * cs;
  float* ec = e + base + col * cs;
  const float* rc = r + base + col * cs;
  const float4 Z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  auto ld = [](const float* q) { return *reinterpret_cast<const float4*>(q); };
  const bool hym = act && j > 0, hyp = act && j < n1 - 1;
  const bool old_in = act && !old_zero;
  // weights off and on the z-walls, of ordinary faces and of those with an
  // x-ghost
  const int gy = ghosts(c != 1, j, n1);
  const bool wally = c == 1 && (j == 0 || j == n1 - 1);
  const float w_in = wally ? 0.f : by_ghosts(w, gy), w_in_x = wally ? 0.f : by_ghosts(w, gy + 1);
  const float w_z = (wally || c == 2) ? 0.f : by_ghosts(w, gy + 1);
  const float w_z_x = (wally || c == 2) ? 0.f : by_ghosts(w, gy + 2);
  // per parity s of i the elements with an x-ghost and the dead ones
  int ghost = 0, dead = 0;
#pragma unroll
  for (int b = 0; b < 8; ++b) {
    const int i = 2 * (q0 + (b & 3)) + (b >> 2);
    if (c != 0 && (i == 0 || i == p.nx - 1)) ghost |= 1 << b;
    if (i >= p.nx || (c == 0 && i == 0)) dead |= 1 << b;
  }
  int s = (col + j + z0) & 1;   // i = 2 q + s
  float4 om = (act && z0 > 0) ? ld(eo - sz) : Z4;
  float4 oc = act ? ld(eo) : Z4;
  for (int z = z0; z < z1; ++z) {
    const float4 on = (act && z + 1 < n2) ? ld(eo + sz) : Z4;
    const float4 ym = hym ? ld(eo - p.sy) : Z4;
    const float4 yp = hyp ? ld(eo + p.sy) : Z4;
    const float4 rr = act ? ld(rc) : Z4;
    const float4 old = old_in ? ld(ec) : Z4;
    // the x-neighbour outside the group: below (s = 0) or above (s = 1)
    float side = __shfl_sync(kFullMask, s ? oc.x : oc.w, s ? tx + 1 : tx - 1, LX);
    if (tx == (s ? LX - 1 : 0))
      side = (act && (s ? q0 + 4 < p.nq : q0 > 0)) ? eo[s ? 4 : -1] : 0.f;
    const bool zw = z == 0 || z == n2 - 1;
    const float w0 = zw ? w_z : w_in, wx = zw ? w_z_x : w_in_x;
    const int sp = s ? 4 : 0;
    float wt[4] = {w0, w0, w0, w0};
    auto special = [&](int t) {
      if ((ghost >> (sp + t)) & 1) wt[t] = wx;
      if ((dead >> (sp + t)) & 1) wt[t] = 0.f;
    };
    if (FULL) {
      special(0);
      special(3);
    } else {
#pragma unroll
      for (int t = 0; t < 4; ++t) special(t);
    }
    float4 o;
    o.x = fmaf(wt[0], fmaf(nu, (oc.x + (s ? oc.y : side)) + (ym.x + yp.x) + (om.x + on.x), rr.x),
               omw * old.x);
    o.y = fmaf(wt[1], fmaf(nu, (oc.y + (s ? oc.z : oc.x)) + (ym.y + yp.y) + (om.y + on.y), rr.y),
               omw * old.y);
    o.z = fmaf(wt[2], fmaf(nu, (oc.z + (s ? oc.w : oc.y)) + (ym.z + yp.z) + (om.z + on.z), rr.z),
               omw * old.z);
    o.w = fmaf(wt[3], fmaf(nu, (oc.w + (s ? side : oc.z)) + (ym.w + yp.w) + (om.w + on.w), rr.w),
               omw * old.w);
    if (!FULL) {
      // The row's padding stays 0 whatever its neighbours hold (a zero weight
      // times an infinity would not): later solves read it and never write it.
      if ((dead >> sp) & 1) o.x = 0.f;
      if ((dead >> (sp + 1)) & 1) o.y = 0.f;
      if ((dead >> (sp + 2)) & 1) o.z = 0.f;
      if ((dead >> (sp + 3)) & 1) o.w = 0.f;
    }
    if (act) *reinterpret_cast<float4*>(ec) = o;
    om = oc;
    oc = on;
    eo += sz;
    ec += sz;
    rc += sz;
    s ^= 1;
  }
}

// Start of the solve: the residual r^ = scale r (scale a power of two: exact)
// of the FP64 right-hand side as FP32 pairs (split_exact) by colour, and the
// first half-step e_0 = D^{-1} r^ of colour 0.  One face per thread, so that a
// warp reads 32 consecutive FP64 values and writes two whole 64-byte pieces.
__global__ void __launch_bounds__(kHelmThreads) k_helm_start(FaceGeom g, HelmGeom p, int zc,
                                                             int zchunks,
                                                             const double* __restrict__ r64,
                                                             float scale, float4 dinv,
                                                             float* __restrict__ rhi,
                                                             float* __restrict__ rlo,
                                                             float* __restrict__ e) {
  const int c = blockIdx.z / zchunks;
  const int z0 = (blockIdx.z - c * zchunks) * zc;
  const int n1 = sel3(c, p.n[0][1], p.n[1][1], p.n[2][1]);
  const int n2 = sel3(c, p.n[0][2], p.n[1][2], p.n[2][2]);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= 2 * p.nq || j >= n1) return;
  const int z1 = min(z0 + zc, n2);
  const int64_t cs = sel3(c, p.cs[0], p.cs[1], p.cs[2]), sz = sel3(c, p.sz[0], p.sz[1], p.sz[2]);
  const int64_t sz64 = sel3(c, g.sz[0], g.sz[1], g.sz[2]);
  const double* src = r64 + sel3(c, g.off[0], g.off[1], g.off[2]) +
                      (int64_t)j * sel3(c, g.sy[0], g.sy[1], g.sy[2]) + i;
  const int64_t base = sel3(c, p.off[0], p.off[1], p.off[2]) + (int64_t)j * p.sy + (i >> 1);
  const bool live = i < p.nx && !(c == 0 && i == 0) && !(c == 1 && (j == 0 || j == n1 - 1));
  const int gxy = ghosts(c != 0, i, p.nx) + ghosts(c != 1, j, n1);
#pragma unroll 4
  for (int z = z0; z < z1; ++z) {
    dsf v = {0.f, 0.f};
    if (live && !(c == 2 && (z == 0 || z == n2 - 1)))
      v = split_exact(__ldg(src + (int64_t)z * sz64));
    v.hi *= scale;
    v.lo *= scale;
    const int col = (i + j + z) & 1;
    const int64_t f = base + (int64_t)z * sz + col * cs;
    rhi[f] = v.hi;
    rlo[f] = v.lo;
    if (col == 0) e[f] = by_ghosts(dinv, gxy + ghosts(c != 2, z, n2)) * v.hi;
  }
}

// (rhi, rlo) <- (rhi, rlo) - A e in double-single arithmetic on the FP32
// pipes: after the FP32 correction e the new residual q = r^ - A e, formed
// exactly enough (A e with error-free sums and products, the last two sums by
// Dekker's addition: a few units of 2^-46 relative to r^); the block's sum of
// q.hi^2 goes to part[block] (every block writes one).  The first half-step of
// the next correction, D^{-1} q on colour 0, goes to en.  Two elements of each
// colour per thread.  The FP64 pipe is not used.
template <int LX>
__global__ void __launch_bounds__(kHelmThreads) k_helm_resid(
    HelmGeom p, int zc, int zchunks, const float* __restrict__ e, float* __restrict__ rhi,
    float* __restrict__ rlo, dsf A, dsf NU, float4 dinv, float* __restrict__ en,
    double* __restrict__ part) {
  constexpr int kRows = kHelmThreads / LX;
  const int c = blockIdx.z / zchunks;
  const int z0 = (blockIdx.z - c * zchunks) * zc;
  const int n1 = sel3(c, p.n[0][1], p.n[1][1], p.n[2][1]);
  const int n2 = sel3(c, p.n[0][2], p.n[1][2], p.n[2][2]);
  const int64_t blk = ((int64_t)blockIdx.z * gridDim.y + blockIdx.y) * gridDim.x + blockIdx.x;
  if (z0 >= n2 || (int)blockIdx.y * kRows >= n1) {   // block-uniform
    if (threadIdx.x == 0 && threadIdx.y == 0) part[blk] = 0.0;
    return;
  }
  const int z1 = min(z0 + zc, n2);
  const int tx = threadIdx.x;
  const int j = blockIdx.y * kRows + threadIdx.y;
  const int q0 = 2 * (blockIdx.x * LX + tx);
  const bool act = q0 < p.nq && j < n1;
  const int64_t cs = sel3(c, p.cs[0], p.cs[1], p.cs[2]), sz = sel3(c, p.sz[0], p.sz[1], p.sz[2]);
  const int64_t base = sel3(c, p.off[0], p.off[1], p.off[2]) + (int64_t)j * p.sy + q0;
  const bool hym = act && j > 0, hyp = act && j < n1 - 1;
  const int gy = ghosts(c != 1, j, n1);
  const bool wally = c == 1 && (j == 0 || j == n1 - 1);
  const float2 Z2 = make_float2(0.f, 0.f);
  auto ld = [](const float* q) { return *reinterpret_cast<const float2*>(q); };
  const dsf D6 = ds_add(A, ds_mul_f(NU, 6.f));
  float acc = 0.f;
  int64_t f = base + (int64_t)z0 * sz;
  // both colours at the planes below, at and above
  float2 em[2], ec[2], ez[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    em[k] = (act && z0 > 0) ? ld(e + f + k * cs - sz) : Z2;
    ec[k] = act ? ld(e + f + k * cs) : Z2;
  }
  for (int z = z0; z < z1; ++z, f += sz) {
    float2 ym[2], yp[2], rh[2], rl[2];
    float side[2];   // x-neighbour of the colour's own group among the other's
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int64_t fk = f + k * cs;
      ez[k] = (act && z + 1 < n2) ? ld(e + fk + sz) : Z2;
      ym[k] = hym ? ld(e + fk - p.sy) : Z2;
      yp[k] = hyp ? ld(e + fk + p.sy) : Z2;
      rh[k] = act ? ld(rhi + fk) : Z2;
      rl[k] = act ? ld(rlo + fk) : Z2;
      const int o = 1 - k, s = (k + j + z) & 1;
      side[k] = __shfl_sync(kFullMask, s ? ec[o].x : ec[o].y, s ? tx + 1 : tx - 1, LX);
      if (tx == (s ? LX - 1 : 0))
        side[k] = (act && (s ? q0 + 2 < p.nq : q0 > 0)) ? e[f + o * cs + (s ? 2 : -1)] : 0.f;
    }
    const bool wall = wally || (c == 2 && (z == 0 || z == n2 - 1));
    const int gyz = gy + ghosts(c != 2, z, n2);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int o = 1 - k, s = (k + j + z) & 1;
      const float2 xb = make_float2(s ? ec[o].y : side[k], s ? side[k] : ec[o].x);
      dsf2 sm = two_sum2(ec[o], xb);
      sm = ds_add_f2(sm, ym[o]);
      sm = ds_add_f2(sm, yp[o]);
      sm = ds_add_f2(sm, em[o]);
      sm = ds_add_f2(sm, ez[o]);
      const int i0 = 2 * q0 + s, i1 = i0 + 2;
      const int g0 = gyz + ghosts(c != 0, i0, p.nx), g1 = gyz + ghosts(c != 0, i1, p.nx);
      dsf d0 = D6, d1 = D6;
      if (g0 > 0) d0 = ds_add(A, ds_mul_f(NU, (float)(6 + g0)));
      if (g1 > 0) d1 = ds_add(A, ds_mul_f(NU, (float)(6 + g1)));
      const dsf2 diag = {make_float2(d0.hi, d1.hi), make_float2(d0.lo, d1.lo)};
      const dsf2 Ae = ds_add_d2(ds_mul_f2(diag, ec[k]), ds_neg2(ds_mul2(sm, NU)));
      dsf2 v = ds_add_d2(dsf2{rh[k], rl[k]}, ds_neg2(Ae));
      if (wall || i0 >= p.nx || (c == 0 && i0 == 0)) v.hi.x = v.lo.x = 0.f;
      if (wall || i1 >= p.nx) v.hi.y = v.lo.y = 0.f;
      acc = fmaf(v.hi.x, v.hi.x, acc);
      acc = fmaf(v.hi.y, v.hi.y, acc);
      if (act) {
        const int64_t fk = f + k * cs;
        *reinterpret_cast<float2*>(rhi + fk) = v.hi;
        *reinterpret_cast<float2*>(rlo + fk) = v.lo;
        if (k == 0)
          *reinterpret_cast<float2*>(en + fk) =
              make_float2(by_ghosts(dinv, g0) * v.hi.x, by_ghosts(dinv, g1) * v.hi.y);
      }
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      em[k] = ec[k];
      ec[k] = ez[k];
    }
  }
  // block reduction (FP64, fixed order)
  double v = (double)acc;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(kFullMask, v, o);
  __shared__ double sh[kHelmThreads / 32];
  const int tid = threadIdx.y * LX + tx;
  if ((tid & 31) == 0) sh[tid >> 5] = v;
  __syncthreads();
  if (tid == 0) {
    double t = 0.0;
    for (int k = 0; k < kHelmThreads / 32; ++k) t += sh[k];
    part[blk] = t;
  }
}

// v 2^k by its exponent field (v 0 or normal, and so the result)
__device__ __forceinline__ double scale_exp(double v, int k) {
  return v == 0.0 ? v : __longlong_as_double(__double_as_longlong(v) + ((long long)k << 52));
}

// Corrections into the FP64 iterate on the faces' own layout: u = 2^k (pe + e)
// (pe null: 2^k e), 0 on the wall faces; ADD: u += 2^k e on the interior
// faces.  The FP32 values are widened with integer operations and the scale
// moves exponents only, so a face costs the FP64 pipe one addition.
// One face per thread (as k_helm_start).
template <bool ADD>
__global__ void __launch_bounds__(kHelmThreads) k_helm_flush(FaceGeom g, HelmGeom p, int zc,
                                                             int zchunks,
                                                             const float* __restrict__ e,
                                                             const float* __restrict__ pe, int k,
                                                             double* __restrict__ u) {
  const int c = blockIdx.z / zchunks;
  const int z0 = (blockIdx.z - c * zchunks) * zc;
  const int n1 = sel3(c, p.n[0][1], p.n[1][1], p.n[2][1]);
  const int n2 = sel3(c, p.n[0][2], p.n[1][2], p.n[2][2]);
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  if (i >= p.nx || j >= n1) return;
  const int z1 = min(z0 + zc, n2);
  const int64_t cs = sel3(c, p.cs[0], p.cs[1], p.cs[2]), sz = sel3(c, p.sz[0], p.sz[1], p.sz[2]);
  const int64_t sz64 = sel3(c, g.sz[0], g.sz[1], g.sz[2]);
  double* dst = u + sel3(c, g.off[0], g.off[1], g.off[2]) +
                (int64_t)j * sel3(c, g.sy[0], g.sy[1], g.sy[2]) + i;
  const int64_t base = sel3(c, p.off[0], p.off[1], p.off[2]) + (int64_t)j * p.sy + (i >> 1);
  const bool live = !(c == 0 && i == 0) && !(c == 1 && (j == 0 || j == n1 - 1));
  const bool wall_next = c == 0 && i == p.nx - 1;   // u_x's wall face i = nx
#pragma unroll 4
  for (int z = z0; z < z1; ++z) {
    const int64_t f = base + (int64_t)z * sz + ((i + j + z) & 1) * cs;
    double* d = dst + (int64_t)z * sz64;
    const bool in = live && !(c == 2 && (z == 0 || z == n2 - 1));
    if (ADD) {
      if (in) *d += scale_exp(f2d_exact(e[f]), k);
    } else {
      double v = f2d_exact(e[f]);
      if (pe) v += f2d_exact(pe[f]);
      *d = in ? scale_exp(v, k) : 0.0;
      if (wall_next) d[1] = 0.0;
    }
  }
}

}  // namespace

int march_zc(Dims d);

template <typename T>
void launch_laplacian(Dims d, const T* v, T* out, double inv_h2, cudaStream_t s) {
  count_launch();
  if constexpr (std::is_same<T, double>::value) {
    const int zc = march_zc(d);
    const FxLimits L = fx_limits(inv_h2);
    k_laplacian_fx<<<dim3(div_up(d.nx, BX), div_up(d.ny, BY), div_up(d.nz, zc)), dim3(BX, BY), 0,
                     s>>>(d, v, nullptr, out, L.bits, L.e_min, L.e_max, zc);
  } else {
    k_laplacian<T><<<cell_grid(d), dim3(BX, BY), 0, s>>>(d, v, out, (T)inv_h2);
  }
}
void launch_laplacian_sub(Dims d, const double* v, const double* b, double* out, double inv_h2,
                          cudaStream_t s) {
  count_launch();
  const int zc = march_zc(d);
  const FxLimits L = fx_limits(inv_h2);
  k_laplacian_fx<<<dim3(div_up(d.nx, BX), div_up(d.ny, BY), div_up(d.nz, zc)), dim3(BX, BY), 0,
                   s>>>(d, v, b, out, L.bits, L.e_min, L.e_max, zc);
}

template void launch_laplacian<float>(Dims, const float*, float*, double, cudaStream_t);
template void launch_laplacian<double>(Dims, const double*, double*, double, cudaStream_t);

dim3 grad_grid(Dims d, int zc) {
  return dim3(div_up(d.nx + 1, BX), div_up(d.ny + 1, BY), div_up(d.nz + 1, zc));
}

void launch_gradient(Dims d, const double* p, double* u, double inv_h, cudaStream_t s) {
  count_launch();
  const int zc = march_zc(d);
  k_grad_axpy<<<grad_grid(d, zc), dim3(BX, BY), 0, s>>>(d, make_face_geom(d), nullptr, p, inv_h,
                                                         u, zc);
}

void launch_grad_axpy(Dims d, const double* u_in, const double* p, double alpha, double* u_out,
                      cudaStream_t s) {
  count_launch();
  const int zc = march_zc(d);
  k_grad_axpy<<<grad_grid(d, zc), dim3(BX, BY), 0, s>>>(d, make_face_geom(d), u_in, p, alpha,
                                                         u_out, zc);
}

// planes per thread of the one-cell z-march kernels: about eight blocks per
// SM over the grid, at most 4
int march_zc(Dims d) {
  const int64_t bxy = (int64_t)div_up(d.nx, BX) * div_up(d.ny, BY);
  return (int)std::min<int64_t>(4, std::max<int64_t>(1, d.nz * bxy / (152 * 8)));
}

void launch_gradt_axpby(Dims d, const double* u, double alpha, const double* c, double beta,
                        double* out, cudaStream_t s) {
  count_launch();
  const int zc = march_zc(d);
  k_gradt_fx<false><<<dim3(div_up(d.nx, BX), div_up(d.ny, BY), div_up(d.nz, zc)), dim3(BX, BY),
                      0, s>>>(d, make_face_geom(d), u, fx_limits(alpha), c, beta, out, nullptr, zc);
}

int64_t gradt_norm2_blocks(Dims d) {
  const int zc = march_zc(d);
  return (int64_t)div_up(d.nx, BX) * div_up(d.ny, BY) * div_up(d.nz, zc);
}

int64_t launch_gradt_norm2(Dims d, const double* u, double alpha, double* part, cudaStream_t s) {
  count_launch();
  const int zc = march_zc(d);
  k_gradt_fx<true><<<dim3(div_up(d.nx, BX), div_up(d.ny, BY), div_up(d.nz, zc)), dim3(BX, BY), 0,
                     s>>>(d, make_face_geom(d), u, fx_limits(alpha), nullptr, 0.0, nullptr, part,
                          zc);
  return gradt_norm2_blocks(d);
}

void launch_gradient_t(Dims d, const double* u, double* out, double inv_h, cudaStream_t s) {
  launch_gradt_axpby(d, u, inv_h, nullptr, 0.0, out, s);
}

// dsf of an FP64 constant (host)
dsf host_ds(double x) {
  const float hi = (float)x;
  return dsf{hi, (float)(x - (double)hi)};
}

int64_t helm_fp32_size(Dims d) {
  const HelmGeom p = make_helm_geom(d);
  return p.off[2] + 2 * p.cs[2];
}

// Launch shape for `groups` threads' worth of a row: LX (32, 16 or 8) threads
// per row so that few of them lie past its end, and planes per thread so that
// there are about eight blocks per SM, at most 8 (several waves of blocks).
struct HelmShape {
  int lx, zc, zch;
  dim3 grid, block;
};

HelmShape helm_shape(Dims d, int groups) {
  HelmShape h;
  h.lx = 32;
  for (int lx : {16, 8})
    if (div_up(groups, lx) * lx < div_up(groups, h.lx) * h.lx) h.lx = lx;
  const int gx = div_up(groups, h.lx), gy = div_up(d.ny + 1, kHelmThreads / h.lx);
  h.zc = (int)std::min<int64_t>(8, std::max<int64_t>(1, (int64_t)gx * gy * 3 * (d.nz + 1) / (152 * 8)));
  h.zch = div_up(d.nz + 1, h.zc);
  h.grid = dim3(gx, gy, 3 * h.zch);
  h.block = dim3(h.lx, kHelmThreads / h.lx);
  return h;
}

// 1 / (a + (6 + g) nu), g = 0..3 ghosts, times f
float4 helm_weights(double a, double nu_h2, double f) {
  auto w = [&](int g) { return (float)(f / (a + (6 + g) * nu_h2)); };
  return make_float4(w(0), w(1), w(2), w(3));
}

void launch_helm_start(Dims d, const double* r64, float scale, double a, double nu_h2, float* rhi,
                       float* rlo, float* e, cudaStream_t s) {
  const HelmShape h = helm_shape(d, 2 * div_up(d.nx, 2));
  count_launch();
  k_helm_start<<<h.grid, h.block, 0, s>>>(make_face_geom(d), make_helm_geom(d), h.zc, h.zch, r64,
                                          scale, helm_weights(a, nu_h2, 1.0), rhi, rlo, e);
}

void launch_helm_half(Dims d, int col, float* e, const float* r, double a, double nu_h2,
                      double omega, bool old_zero, cudaStream_t s) {
  const HelmShape h = helm_shape(d, div_up(d.nx, 8));
  count_launch();
  const bool full = d.nx % 8 == 0;
  const auto k32 = full ? k_helm_half<32, true> : k_helm_half<32, false>;
  const auto k16 = full ? k_helm_half<16, true> : k_helm_half<16, false>;
  const auto k8 = full ? k_helm_half<8, true> : k_helm_half<8, false>;
  launch_pdl(h.lx == 32 ? k32 : (h.lx == 16 ? k16 : k8), h.grid, h.block, 0, s, make_helm_geom(d),
             h.zc, h.zch, col, e, r, (float)nu_h2, helm_weights(a, nu_h2, omega),
             (float)(1.0 - omega), old_zero ? 1 : 0, col & past_l2(24 * (int64_t)d.nx * d.ny * d.nz));
}

// two elements of each colour per thread
static HelmShape helm_resid_shape(Dims d) { return helm_shape(d, div_up(d.nx, 4)); }

int64_t helm_resid_blocks(Dims d) {
  const HelmShape h = helm_resid_shape(d);
  return (int64_t)h.grid.x * h.grid.y * h.grid.z;
}

int64_t launch_helm_resid(Dims d, const float* e, float* rhi, float* rlo, double a, double nu_h2,
                          float* en, double* part, cudaStream_t s) {
  const HelmShape h = helm_resid_shape(d);
  const auto k = h.lx == 32 ? k_helm_resid<32> : (h.lx == 16 ? k_helm_resid<16> : k_helm_resid<8>);
  count_launch();
  k<<<h.grid, h.block, 0, s>>>(make_helm_geom(d), h.zc, h.zch, e, rhi, rlo, host_ds(a),
                               host_ds(nu_h2), helm_weights(a, nu_h2, 1.0), en, part);
  return helm_resid_blocks(d);
}

void launch_helm_flush(Dims d, const float* e, const float* pe, int k, bool add, double* u,
                       cudaStream_t s) {
  const HelmShape h = helm_shape(d, 2 * div_up(d.nx, 2));
  count_launch();
  if (add)
    k_helm_flush<true><<<h.grid, h.block, 0, s>>>(make_face_geom(d), make_helm_geom(d), h.zc,
                                                  h.zch, e, pe, k, u);
  else
    k_helm_flush<false><<<h.grid, h.block, 0, s>>>(make_face_geom(d), make_helm_geom(d), h.zc,
                                                   h.zch, e, pe, k, u);
}

void launch_predictor_rhs_adv(Dims d, const double* u_n, const double* u_nm1, const double* p_n,
                              const double* f_body, int with_adv, double inv_2dt, double inv_h,
                              double* rhs, cudaStream_t s) {
  const FaceGeom g = make_face_geom(d);
  const dsf c4 = host_ds(4.0 * inv_2dt), c1 = host_ds(inv_2dt), cph = host_ds(inv_h),
            ca = host_ds(0.25 * inv_h);
  const int64_t bxy = (int64_t)div_up(d.nx + 1, BX) * div_up(d.ny + 1, BY);
  // planes per thread: about eight blocks per SM (a march forms its first lower
  // z-flux anew)
  const int zc = (int)std::min<int64_t>(kRhsPlanes,
                                        std::max<int64_t>(1, 3 * bxy * (d.nz + 1) / (152 * 8)));
  const dim3 b(BX, BY);
  if (bxy * (d.nz + 1) < (int64_t)kRhsPlanes * 152 * 8) {   // less than that per component
    const int zch = div_up(d.nz + 1, zc);
    count_launch();
    k_predictor_rhs_all<<<dim3(div_up(d.nx + 1, BX), div_up(d.ny + 1, BY), 3 * zch), b, 0, s>>>(
        d, g, u_n, u_nm1, p_n, f_body, with_adv, c4, c1, cph, ca, rhs, zc, zch);
    return;
  }
  auto run = [&](auto kernel, int nx, int ny, int nz) {
    count_launch();
    kernel<<<dim3(div_up(nx, BX), div_up(ny, BY), div_up(nz, kRhsPlanes)), b, 0, s>>>(
        d, g, u_n, u_nm1, p_n, f_body, with_adv, c4, c1, cph, ca, rhs);
  };
  run(k_predictor_rhs_ds<0>, d.nx + 1, d.ny, d.nz);
  run(k_predictor_rhs_ds<1>, d.nx, d.ny + 1, d.nz);
  run(k_predictor_rhs_ds<2>, d.nx, d.ny, d.nz + 1);
}

}  // namespace ibm
