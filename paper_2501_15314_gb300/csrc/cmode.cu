// C^{-1} with C = R^T R, the (2,2) block of Eq. (Saddle), for the exact
// primal Schur complement S_p = L + B^T C^{-1} B (Eqs. (SchurPrimal)-
// (SchurPrimalF)) and the sign-consistent form L - B^T C^{-1} B.
//
// Conjugate gradients on C (symmetric positive definite when the markers'
// weight vectors are independent).  C's diagonal is the same for every marker
// ((sum phi^2)^3 = 1/8 when no tap is cut off), so Jacobi scaling would not
// change anything.  Its condition number grows quickly with the marker density
// (about 5e2 at Lagrangian spacing h, 2e5 at h / 1.38 for a sphere of radius
// 0.3 on 32^3), which is why the paper uses C^{-1} ~ 2 I in production.
//
// A solve takes hundreds of iterations of microseconds' work each, so a whole
// solve is one cooperative launch of at most one block per SM whose phases are
// separated by grid-wide barriers, which carry the partial sums of the two dot
// products with them.  Three forms:
//   rows: C's rows are formed once per marker set (the overlaps of the markers'
//     supports, about 58 per marker at spacing h) and kept until the markers
//     change; an iteration is one product and two barriers.  The vectors'
//     own values stay in registers.
//   spread: C v = R^T (R v) through the shell faces (written, not accumulated,
//     so the rest of the face scratch is never read); four barriers.  For more
//     markers than the grid's registers hold, or rows longer on average than
//     kRowMax (markers denser than h), which take longer than the spread's
//     64 + 27 weights.
//   launched: the spread form's phases as kernels of full grids, nine per
//     iteration, the residual read by the host every four.  For more than
//     kOneLaunchMax markers, where an iteration waits on memory for longer than
//     nine launches take and one block per SM keeps too few loads in flight.
// Measured on GB300, us per iteration: rows 11.5 at 1158 markers, 14 at 4632,
// 24 at 12000, 41 at 25900 (launched 50, 61 at 6000, 73 at 25900), the two
// barriers with their sums taking about 8 of them.  Spread, on spheres at
// spacing h, with blocks of 512 threads / of 1024 / launched: 57 / 47 / 78 at
// 26100 markers, 139 / 104 / 122 at 60000, 310 / 217 / 217 at 150000, 653 / 445 /
// 401 at 330000; 10^6 markers in a volume 1630 / 1252 / 989.
#include "ibm_internal.cuh"

#include <algorithm>
#include <cmath>
#include <cstdio>

namespace ibm {

namespace {

constexpr int TPB = 256;
constexpr int kCgThreads = 512;
constexpr int kCgWarps = kCgThreads / 32;
constexpr int kCgWide = 1024;  // threads of the spread form's larger blocks
constexpr int64_t kOneLaunchMax = 150000;   // markers of the one-launch forms
constexpr int kCheck = 4;      // the residual is tested every four iterations
constexpr int kRowLanes = 4;   // lanes per row and component
constexpr int kRowUnits = 32 / kRowLanes;   // rows a warp takes at once
constexpr int kRowHeld = 4;    // rows a lane group holds in registers
// Longest average row of the rows form, where each lane group has one row and
// where it has several.  Measured, us per iteration rows / spread: 500 markers
// 14.5 / 18.6 with rows of 98, 19.7 / 19.5 with 148; 4000 markers 17.5 / 20.8 and
// 22.3 / 21.5; 8000 (two rows a group) 29.9 / 29.9 with 60, 31.9 / 24.8 with 98;
// 25000 (four) 37.8 / 46.1 with 58, 62 / 44 with 98, 161 / 48 with 215.
constexpr int kRowMax = 112;
constexpr int kRowMaxMany = 64;
// polls before a barrier gives up (about a second; a barrier takes microseconds)
constexpr int kSpinLimit = 1 << 20;

struct CgArgs {
  Dims d;
  int64_t n;         // markers
  int64_t n_shell, n_ell;
  const int32_t *cell, *base, *len, *key;   // interleaved layout
  const double* sw;
  const uint8_t* any;
  const int32_t *bf, *bc;
  const double *wf, *wc;
  const int32_t *off, *col;   // C's rows, val[component][entry]
  const double* val;
  int64_t n_val;
  const double* t;
  double *s, *r, *p, *q, *face;
  double* part;      // [2][blocks] partial sums
  unsigned* bar;     // [0] arrivals, [1] a barrier timed out
  double* out;       // <t, t>, <r, r>, iterations (mapped host memory)
  double rtol2;
  int maxit;
};

// Grid-wide barrier with the sum of v over the grid's threads, in a fixed order
// (each warp, the block's warps, the blocks).  The blocks' arrivals are counted
// up to round * blocks, modulo 2^32 (14 million iterations of 152 blocks): the
// counts compared differ by less than two rounds, so the sign of their
// difference tells which is ahead.  The partial sums alternate between two
// arrays, as a block may enter the next barrier while others still read this
// one's.  Every block is resident (cooperative launch), so the barrier ends;
// should it not, a limit on the polls sets the error flag and all blocks leave.
// One warp forms the total and, from it and num, the scalar the caller needs:
// total / num (OVER), num / total (else), 0 where the divisor is.  An FP64
// operation has 64 cycles of latency and takes a warp 16 cycles of its SM's
// pipe, so sums are trees and no second warp repeats the division.
// Measured on GB300: 2750 cycles for 152 blocks without the sum (the words of
// every block polled by every block instead of one counter: 7000).
struct GridSum {
  double total, ratio;
};

template <bool OVER>
__device__ bool grid_sum(const CgArgs& a, double v, double num, unsigned& round, GridSum& out) {
  __shared__ double sh[kCgWide / 32];
  __shared__ GridSum all;
  __shared__ int ok;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, warps = blockDim.x >> 5;
  if (__any_sync(0xffffffffu, v != 0.0)) {   // NaN included
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  }
  if (lane == 0) sh[wid] = v;
  __syncthreads();
  ++round;
  if (wid == 0) {
    double* part = a.part + (int64_t)(round & 1) * gridDim.x;
    double t = lane < warps ? sh[lane] : 0.0;
    for (int o = 1; o < warps; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) {
      part[blockIdx.x] = t;
      asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
      const unsigned want = round * gridDim.x;
      unsigned seen;
      int polls = 0;
      do {
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.bar) : "memory");
      } while ((int)(seen - want) < 0 && ++polls < kSpinLimit);
      ok = (int)(seen - want) >= 0;
      if (!ok) atomicExch(a.bar + 1, 1u);
    }
    __syncwarp();
    t = 0.0;
    for (int b = lane; b < (int)gridDim.x; b += 32) t += __ldcg(part + b);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
    if (lane == 0) {
      all.total = t;
      all.ratio = OVER ? (num != 0.0 ? t / num : 0.0) : (t != 0.0 ? num / t : 0.0);
    }
  }
  __syncthreads();
  out = all;
  return ok;
}

// ---- rows of C ----

// overlap of two markers' three taps along one axis, the first of whose taps
// lie at b and b + shift (|shift| <= 3)
__device__ __forceinline__ double tap_overlap(const double* w, const double* v, int64_t n,
                                              int shift) {
  double s = 0.0;
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const int p = q - shift;
    if (p >= 0 && p < 3) s = fma(w[q * n], v[p * n], s);
  }
  return s;
}

// The markers whose 4x4x4 cell boxes overlap marker k's, one warp per marker:
// the cells of k's box in order, in each the entries of the cell's segment (the
// sorted list of markers whose box holds the cell), a pair being taken in the
// lowest cell that both boxes hold.  FILL: the columns and the products of the
// overlaps; else only their number.
template <bool FILL>
__global__ void __launch_bounds__(TPB) k_c_rows(Dims d, int64_t n, int64_t n_entries,
                                                const int32_t* __restrict__ org,
                                                const int32_t* __restrict__ start,
                                                const int32_t* __restrict__ key, CgArgs a,
                                                int32_t* __restrict__ count,
                                                const int32_t* __restrict__ off,
                                                int32_t* __restrict__ col,
                                                double* __restrict__ val) {
  const int64_t k = (blockIdx.x * (int64_t)TPB + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (k >= n) return;   // whole warps leave together
  const int o0 = org[k], o1 = org[n + k], o2 = org[2 * n + k];
  int32_t found = FILL ? off[k] : 0;
  for (int c = 0; c < 64; ++c) {
    const int cx = c & 3, cy = (c >> 2) & 3, cz = c >> 4;
    const int64_t seg = start[((int64_t)(o2 + cz) * d.ny + o1 + cy) * d.nx + o0 + cx];
    for (int64_t e0 = seg;; e0 += 32) {
      const int64_t e = e0 + lane;
      bool in = false, take = false;
      int64_t l = 0;
      if (e < n_entries) {
        const int32_t kk = key[e];
        l = kk >> 6;
        const int sx = kk & 3, sy = (kk >> 2) & 3, sz = (kk >> 4) & 3;
        in = org[l] + sx == o0 + cx && org[n + l] + sy == o1 + cy && org[2 * n + l] + sz == o2 + cz;
        // both boxes hold no lower cell along any axis
        take = in && (cx == 0 || sx == 0) && (cy == 0 || sy == 0) && (cz == 0 || sz == 0);
      }
      const unsigned m = __ballot_sync(0xffffffffu, take);
      if (FILL && take) {
        const int64_t dst = found + __popc(m & ((1u << lane) - 1));
        double of[3], oc[3];
#pragma unroll
        for (int x = 0; x < 3; ++x) {
          of[x] = tap_overlap(a.wf + 3 * x * n + k, a.wf + 3 * x * n + l, n,
                              a.bf[x * n + l] - a.bf[x * n + k]);
          oc[x] = tap_overlap(a.wc + 3 * x * n + k, a.wc + 3 * x * n + l, n,
                              a.bc[x * n + l] - a.bc[x * n + k]);
        }
        col[dst] = (int32_t)l;
        val[dst] = of[0] * oc[1] * oc[2];
        val[a.n_val + dst] = oc[0] * of[1] * oc[2];
        val[2 * a.n_val + dst] = oc[0] * oc[1] * of[2];
      }
      found += __popc(m);
      // the segment goes on while every lane read an entry of this cell
      if (__ballot_sync(0xffffffffu, in) != 0xffffffffu) break;
    }
  }
  if (!FILL && lane == 0) count[k] = found;
}

// s = C^{-1} t with C's rows.  A lane group holds its rows' values of s, r, p
// and q; others read r and the previous p (two buffers, a.p and a.q, written
// alternately) past L1 and form the direction p = r + beta p themselves.
__global__ void __launch_bounds__(kCgThreads, 1) k_cg_rows(const CgArgs a) {
  const int lane = threadIdx.x & 31, sub = lane % kRowLanes;
  const int warps = blockDim.x >> 5;
  const int n = (int)a.n, n3 = 3 * n;
  // consecutive warps' rows on different SMs
  const int w0 = ((threadIdx.x >> 5) * (int)gridDim.x + (int)blockIdx.x) * kRowUnits;
  const int step = (int)gridDim.x * warps * kRowUnits;
  unsigned round = 0;
  int it = 0;
  // first and last entry of the lane's rows, and their component's offsets
  int32_t e0[kRowHeld], e1[kRowHeld], comp[kRowHeld];
  double s[kRowHeld], r[kRowHeld], p[kRowHeld], q[kRowHeld], v = 0.0;
  double* pa = a.p;
  double* pb = a.q;
#pragma unroll
  for (int h = 0; h < kRowHeld; ++h) {
    const int u = w0 + h * step + lane / kRowLanes;
    const bool own = u < n3;
    const int dc = u < n ? 0 : (u < 2 * n ? 1 : 2);
    comp[h] = dc;
    e0[h] = own ? a.off[u - dc * n] + sub : 0;
    e1[h] = own ? a.off[u - dc * n + 1] : 0;
    r[h] = own ? a.t[u] : 0.0;
    s[h] = p[h] = q[h] = 0.0;
    if (own && sub == 0) {
      a.r[u] = r[h];
      pa[u] = 0.0;
      v = fma(r[h], r[h], v);
    }
  }
  GridSum g;
  if (!grid_sum<true>(a, v, 0.0, round, g)) return;
  const double tt = g.total, target = a.rtol2 * tt;
  double rr = tt, beta = 0.0;
  if (isfinite(tt) && tt > 0.0) {
    while (it < a.maxit) {
      v = 0.0;
#pragma unroll
      for (int h = 0; h < kRowHeld; ++h) {
        if (w0 + h * step >= n3) break;   // warp-uniform
        const int u = w0 + h * step + lane / kRowLanes;
        const double* pv = pa + comp[h] * n;
        const double* rv = a.r + comp[h] * n;
        const double* val = a.val + comp[h] * a.n_val;
        double acc = 0.0, acc2 = 0.0;
        int32_t e = e0[h];
#pragma unroll 2
        for (; e + kRowLanes < e1[h]; e += 2 * kRowLanes) {
          const int32_t l = __ldg(a.col + e), m = __ldg(a.col + e + kRowLanes);
          acc = fma(__ldg(val + e), fma(beta, __ldcg(pv + l), __ldcg(rv + l)), acc);
          acc2 = fma(__ldg(val + e + kRowLanes), fma(beta, __ldcg(pv + m), __ldcg(rv + m)), acc2);
        }
        if (e < e1[h]) {
          const int32_t l = __ldg(a.col + e);
          acc = fma(__ldg(val + e), fma(beta, __ldcg(pv + l), __ldcg(rv + l)), acc);
        }
        acc += acc2;
#pragma unroll
        for (int o = 1; o < kRowLanes; o <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
        q[h] = acc;
        p[h] = fma(beta, p[h], r[h]);
        if (u < n3 && sub == 0) {
          pb[u] = p[h];
          v = fma(p[h], q[h], v);
        }
      }
      // alpha = rr / <p, q>
      if (!grid_sum<false>(a, v, rr, round, g)) return;
      const double alpha = g.ratio;
      v = 0.0;
#pragma unroll
      for (int h = 0; h < kRowHeld; ++h) {
        if (w0 + h * step >= n3) break;
        const int u = w0 + h * step + lane / kRowLanes;
        s[h] = fma(alpha, p[h], s[h]);
        r[h] = fma(-alpha, q[h], r[h]);
        if (u < n3 && sub == 0) {
          a.r[u] = r[h];
          v = fma(r[h], r[h], v);
        }
      }
      // beta = <r, r> / rr
      if (!grid_sum<true>(a, v, rr, round, g)) return;
      beta = g.ratio;
      rr = g.total;
      double* x = pa;
      pa = pb;
      pb = x;
      ++it;
      if ((it % kCheck == 0 || it == a.maxit) && !(rr > target)) break;   // small, or not a number
    }
  }
#pragma unroll
  for (int h = 0; h < kRowHeld; ++h) {
    const int u = w0 + h * step + lane / kRowLanes;
    if (u < n3 && sub == 0) a.s[u] = s[h];
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.out[0] = tt;
    a.out[1] = rr;
    a.out[2] = (double)it;
  }
}

// ---- through the faces ----

// face = R p on the shell faces; one warp per group of shell cells (as
// k_shell_spread_ell).  p, written by other blocks, is read past L1.
__device__ void cg_spread(const CgArgs& a) {
  const int lane = threadIdx.x & 31;
  const int64_t ng = ell_groups(a.n_shell);
  const FaceDims fd = face_dims(a.d);
  for (int64_t g = (int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x; g < ng;
       g += (int64_t)gridDim.x * (blockDim.x >> 5)) {
    const int64_t qc = g * kEllCells + lane / kEllLanes;
    const bool live = qc < a.n_shell;
    double acc[3] = {0.0, 0.0, 0.0};
    if (live) {
      int64_t idx = a.base[g] + lane;
      const int L = a.len[g];
#pragma unroll 4
      for (int p = 0; p < L; ++p, idx += 32) {
        const int64_t k = __ldg(a.key + idx) >> 6;
#pragma unroll
        for (int dc = 0; dc < 3; ++dc)
          acc[dc] = fma(__ldg(a.sw + dc * a.n_ell + idx), __ldcg(a.p + dc * a.n + k), acc[dc]);
      }
    }
#pragma unroll
    for (int dc = 0; dc < 3; ++dc) acc[dc] = ell_combine(acc[dc]);
    if (!live || lane % kEllLanes != 0) continue;
    const int64_t c = a.cell[qc];
    const int ci = (int)(c % a.d.nx);
    const int cj = (int)((c / a.d.nx) % a.d.ny);
    const int ck = (int)(c / ((int64_t)a.d.nx * a.d.ny));
    const int any = a.any[qc];
#pragma unroll
    for (int dc = 0; dc < 3; ++dc) {
      if (!(any & (1 << dc))) continue;
      const int64_t off = dc == 0 ? 0 : (dc == 1 ? fd.nfx : fd.nfx + fd.nfy);
      const int64_t sy = a.d.nx + (dc == 0 ? 1 : 0);
      const int64_t sz = sy * (a.d.ny + (dc == 1 ? 1 : 0));
      a.face[off + ck * sz + cj * sy + ci] = acc[dc];
    }
  }
}

// (R^T face) of marker k, component dc (the operations of k_interp)
__device__ __forceinline__ double cg_interp(const CgArgs& a, int dc, int64_t k) {
  const FaceDims fd = face_dims(a.d);
  const int64_t off = dc == 0 ? 0 : (dc == 1 ? fd.nfx : fd.nfx + fd.nfy);
  const int64_t sy = a.d.nx + (dc == 0 ? 1 : 0);
  const int64_t sz = sy * (a.d.ny + (dc == 1 ? 1 : 0));
  int b[3];
  const double* w[3];
#pragma unroll
  for (int e = 0; e < 3; ++e) {
    b[e] = (e == dc) ? a.bf[e * a.n + k] : a.bc[e * a.n + k];
    w[e] = ((e == dc) ? a.wf : a.wc) + e * 3 * a.n + k;
  }
  const double* f = a.face + off + b[2] * sz + b[1] * sy + b[0];
  double acc = 0.0;
#pragma unroll
  for (int c2 = 0; c2 < 3; ++c2) {
    double acc1 = 0.0;
#pragma unroll
    for (int c1 = 0; c1 < 3; ++c1) {
      double acc0 = 0.0;
#pragma unroll
      for (int c0 = 0; c0 < 3; ++c0)
        acc0 = fma(__ldg(w[0] + c0 * a.n), __ldcg(f + c2 * sz + c1 * sy + c0), acc0);
      acc1 = fma(__ldg(w[1] + c1 * a.n), acc0, acc1);
    }
    acc = fma(__ldg(w[2] + c2 * a.n), acc1, acc);
  }
  return acc;
}

// s = C^{-1} t through the faces.  A thread owns the same marker values in
// every phase; the spread alone reads others'.  Blocks of 512 threads where
// these are enough for a warp per group of shell cells (128 registers: more loads
// in flight per warp; 600 markers at spacing h / 4 42 us an iteration, against
// 47 with 64 registers), of 1024 where there is more work than that.
template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1) k_cg_spread(const CgArgs a) {
  const int64_t n3 = 3 * a.n;
  const int64_t first =
      ((int64_t)(threadIdx.x >> 5) * gridDim.x + blockIdx.x) * 32 + (threadIdx.x & 31);
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  unsigned round = 0;
  int it = 0;
  double v = 0.0;
  GridSum g;
  for (int64_t i = first; i < n3; i += step) {
    const double ti = a.t[i];
    a.s[i] = 0.0;
    a.r[i] = ti;
    a.p[i] = ti;
    v = fma(ti, ti, v);
  }
  if (!grid_sum<true>(a, v, 0.0, round, g)) return;
  const double tt = g.total, target = a.rtol2 * tt;
  double rr = tt;
  if (isfinite(tt) && tt > 0.0) {
    while (it < a.maxit) {
      cg_spread(a);
      if (!grid_sum<true>(a, 0.0, 0.0, round, g)) return;
      v = 0.0;
      for (int64_t i = first; i < n3; i += step) {
        const int dc = (int)(i / a.n);
        const double qi = cg_interp(a, dc, i - dc * a.n);
        a.q[i] = qi;
        v = fma(a.p[i], qi, v);
      }
      // alpha = rr / <p, q>
      if (!grid_sum<false>(a, v, rr, round, g)) return;
      const double alpha = g.ratio;
      v = 0.0;
      for (int64_t i = first; i < n3; i += step) {
        a.s[i] = fma(alpha, a.p[i], a.s[i]);
        const double ri = fma(-alpha, a.q[i], a.r[i]);
        a.r[i] = ri;
        v = fma(ri, ri, v);
      }
      // beta = <r, r> / rr
      if (!grid_sum<true>(a, v, rr, round, g)) return;
      const double beta = g.ratio;
      rr = g.total;
      ++it;
      if ((it % kCheck == 0 || it == a.maxit) && !(rr > target)) break;   // small, or not a number
      for (int64_t i = first; i < n3; i += step) a.p[i] = fma(beta, a.p[i], a.r[i]);
      if (!grid_sum<true>(a, 0.0, 0.0, round, g)) return;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.out[0] = tt;
    a.out[1] = rr;
    a.out[2] = (double)it;
  }
}

// ---- launched ----

__global__ void __launch_bounds__(TPB) k_spread_set(const CgArgs a) { cg_spread(a); }

__global__ void k_cg_alpha(const double* __restrict__ rr, const double* __restrict__ pq,
                           double* __restrict__ alpha) {
  alpha[0] = pq[0] != 0.0 ? rr[0] / pq[0] : 0.0;
}

// s += alpha p, r -= alpha q
__global__ void __launch_bounds__(TPB) k_cg_update(const CgArgs a,
                                                   const double* __restrict__ alpha) {
  const double f = alpha[0];
  for (int64_t i = blockIdx.x * (int64_t)TPB + threadIdx.x; i < 3 * a.n;
       i += (int64_t)gridDim.x * TPB) {
    a.s[i] = fma(f, a.p[i], a.s[i]);
    a.r[i] = fma(-f, a.q[i], a.r[i]);
  }
}

// p = r + (rr_new / rr) p
__global__ void __launch_bounds__(TPB) k_cg_direction(const CgArgs a,
                                                      const double* __restrict__ rr,
                                                      const double* __restrict__ rr_new) {
  const double beta = rr[0] > 0.0 ? rr_new[0] / rr[0] : 0.0;
  for (int64_t i = blockIdx.x * (int64_t)TPB + threadIdx.x; i < 3 * a.n;
       i += (int64_t)gridDim.x * TPB)
    a.p[i] = fma(beta, a.p[i], a.r[i]);
}

// The solve kernel by kernel; sc: four device scalars (<r, r> before and after
// the iteration in turn, <p, q>, alpha).  tt = <t, t>, rr = the last <r, r> read.
ibm_status cg_launched(ibm_ctx* c, const CgArgs& a, double* sc, double& tt, double& rr, int& it) {
  cudaStream_t str = c->stream;
  const int64_t n = 3 * a.n;
  const int grid = (int)std::min<int64_t>(div_up(n, TPB), kRedBlocks);
  launch_zero(a.s, sizeof(double) * n, str);
  launch_copy(a.r, a.t, sizeof(double) * n, str);
  launch_copy(a.p, a.t, sizeof(double) * n, str);
  launch_dot(a.t, a.t, n, c->red_part, sc, str, c->host_red_dev);
  IBM_LAUNCH_CHECK(c);
  IBM_CUDA(c, cudaStreamSynchronize(str));
  tt = rr = c->host_red[0];
  if (!std::isfinite(tt) || tt == 0.0) return IBM_OK;
  while (it < a.maxit) {
    double* now = sc + (it & 1);
    double* next = sc + 1 - (it & 1);
    count_launch();
    k_spread_set<<<div_up(32 * ell_groups(a.n_shell), TPB), TPB, 0, str>>>(a);
    launch_interp(c, a.face, a.q);
    launch_dot(a.p, a.q, n, c->red_part, sc + 2, str);
    count_launch();
    k_cg_alpha<<<1, 1, 0, str>>>(now, sc + 2, sc + 3);
    count_launch();
    k_cg_update<<<grid, TPB, 0, str>>>(a, sc + 3);
    ++it;
    const bool test = it % kCheck == 0 || it == a.maxit;
    launch_dot(a.r, a.r, n, c->red_part, next, str, test ? c->host_red_dev : nullptr);
    if (test) {
      IBM_LAUNCH_CHECK(c);
      IBM_CUDA(c, cudaStreamSynchronize(str));
      rr = c->host_red[0];
      if (!(rr > a.rtol2 * tt)) break;   // small, or not a number
    }
    count_launch();
    k_cg_direction<<<grid, TPB, 0, str>>>(a, now, next);
  }
  IBM_LAUNCH_CHECK(c);
  return IBM_OK;
}

// C's rows for the markers set (a.off, a.col, a.val), formed at the first
// solve after they change; rows stays false where the spread form is taken.
ibm_status form_rows(ibm_ctx* c, CgArgs& a, int sms, bool& rows) {
  MarkerData& mk = c->mk;
  rows = false;
  if (3 * mk.n > (int64_t)sms * kCgWarps * kRowUnits * kRowHeld) return IBM_OK;
  if (mk.n > c->m) return IBM_OK;   // the scan's scratch is sized by the cells
  const int64_t row_max =
      3 * mk.n <= (int64_t)sms * kCgWarps * kRowUnits ? kRowMax : kRowMaxMany;
  // a marker's row holds all markers of each of its cells
  if (mk.n_entries > row_max * mk.n_shell) return IBM_OK;
  cudaStream_t str = c->stream;
  const int blocks = div_up(32 * mk.n, TPB);
  if (!mk.c_formed) {
    int32_t* count = c->cell_flag;   // scratch
    a.n_val = 0;
    count_launch();
    k_c_rows<false><<<blocks, TPB, 0, str>>>(c->d, mk.n, mk.n_entries, mk.org, c->cell_start,
                                             mk.entry_key, a, count, nullptr, nullptr, nullptr);
    ibm_status st = exclusive_scan(c, count, mk.c_off, mk.n);
    if (st != IBM_OK) return st;
    launch_to_host(mk.c_off + mk.n, c->host_flag_dev, sizeof(int32_t), str);
    IBM_LAUNCH_CHECK(c);
    IBM_CUDA(c, cudaStreamSynchronize(str));
    int64_t entries = c->host_flag[0];
    mk.c_n = 0;
    if (entries > row_max * mk.n) entries = 0;   // too long: the spread form
    if (entries > mk.c_val_cap) {
      cudaFree(mk.c_val);
      mk.c_val_cap = 0;
      // the values, then the columns
      if (cudaMalloc(&mk.c_val, (3 * sizeof(double) + sizeof(int32_t)) * entries) != cudaSuccess) {
        cudaGetLastError();
        mk.c_val = nullptr;
        entries = 0;   // no room for the rows: the spread form
      } else {
        mk.c_val_cap = entries;
      }
    }
    if (entries > 0) {
      mk.c_col = reinterpret_cast<int32_t*>(mk.c_val + 3 * entries);
      a.n_val = entries;
      count_launch();
      k_c_rows<true><<<blocks, TPB, 0, str>>>(c->d, mk.n, mk.n_entries, mk.org, c->cell_start,
                                              mk.entry_key, a, nullptr, mk.c_off, mk.c_col,
                                              mk.c_val);
      IBM_LAUNCH_CHECK(c);
    }
    mk.c_n = entries;      // rows that were not filled are never taken as formed
    mk.c_formed = true;
  }
  rows = mk.c_n > 0;
  a.off = mk.c_off;
  a.col = mk.c_col;
  a.val = mk.c_val;
  a.n_val = mk.c_n;
  return IBM_OK;
}

}  // namespace

ibm_status c_solve(ibm_ctx* c, const double* t, double* s, double rtol, int maxit,
                   int* iters_out) {
  MarkerData& mk = c->mk;
  const int64_t n = 3 * mk.n;
  cudaStream_t str = c->stream;
  if (iters_out) *iters_out = 0;
  if (n == 0) return IBM_OK;
  if (!c->cg_bar) {
    if (cudaMalloc(&c->cg_bar, 2 * sizeof(unsigned) + 4 * sizeof(double)) != cudaSuccess) {
      cudaGetLastError();
      c->cg_bar = nullptr;
      return set_err(c, IBM_ERR_NOMEM, "CG barrier allocation failed");
    }
  }
  int dev = 0, sms = 0;
  IBM_CUDA(c, cudaGetDevice(&dev));
  IBM_CUDA(c, cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  sms = std::min(sms, kRedBlocks);
  CgArgs a = {};
  a.d = c->d;
  a.n = mk.n;
  a.n_shell = mk.n_shell;
  a.n_ell = mk.n_ell;
  a.cell = mk.ell_cell;
  a.base = mk.ell_base;
  a.len = mk.ell_len;
  a.key = mk.ell_key;
  a.sw = mk.ell_sw;
  a.any = mk.ell_any;
  a.bf = mk.bf;
  a.bc = mk.bc;
  a.wf = mk.wf;
  a.wc = mk.wc;
  a.t = t;
  a.s = s;
  a.r = mk.cg;
  a.p = mk.cg + n;
  a.q = mk.cg + 2 * n;
  a.face = c->f4;
  a.part = c->red_part;
  a.bar = c->cg_bar;
  a.out = c->host_red_dev;
  a.rtol2 = rtol * rtol;
  a.maxit = maxit;
  bool rows;
  const ibm_status st = form_rows(c, a, sms, rows);
  if (st != IBM_OK) return st;
  double tt = 0.0, rr = 0.0;
  int it = 0;
  if (!rows && mk.n > kOneLaunchMax) {
    const ibm_status sl =
        cg_launched(c, a, reinterpret_cast<double*>(c->cg_bar + 2), tt, rr, it);
    if (sl != IBM_OK) return sl;
  } else {
    // at most one block per SM (all resident), and no more warps than the
    // markers give work: an idle warp still takes part in the barriers
    const int64_t warps = rows ? div_up(n, kRowUnits)
                               : std::max<int64_t>(ell_groups(mk.n_shell), div_up(n, 32));
    const int blocks = (int)std::min<int64_t>(warps, sms);
    const int64_t each = div_up(warps, blocks);
    const bool wide = !rows && each > kCgWarps;
    const int threads = 32 * (int)std::min<int64_t>(wide ? kCgWide / 32 : kCgWarps, each);
    const void* kernel = rows ? (const void*)k_cg_rows
                              : (wide ? (const void*)k_cg_spread<kCgWide>
                                      : (const void*)k_cg_spread<kCgThreads>);
    launch_zero(c->cg_bar, 2 * sizeof(unsigned), str);
    count_launch();
    void* args[] = {&a};
    IBM_CUDA(c, cudaLaunchCooperativeKernel(kernel, dim3(blocks), dim3(threads), args, 0, str));
    launch_to_host(a.bar + 1, c->host_flag_dev, sizeof(unsigned), str);
    IBM_LAUNCH_CHECK(c);
    IBM_CUDA(c, cudaStreamSynchronize(str));
    if (c->host_flag[0]) return set_err(c, IBM_ERR_CUDA, "grid barrier of the CG on C timed out");
    tt = c->host_red[0];
    rr = c->host_red[1];
    it = (int)c->host_red[2];
  }
  if (!std::isfinite(tt)) return set_err(c, IBM_ERR_NAN, "non-finite right-hand side of C s = t");
  if (tt == 0.0) return IBM_OK;
  if (!std::isfinite(rr)) return set_err(c, IBM_ERR_NAN, "non-finite CG residual on C");
  if (iters_out) *iters_out = it;
  c->c_iters += it;
  if (rr > rtol * rtol * tt) {
    char buf[160];
    snprintf(buf, sizeof buf, "CG on C = R^T R did not reach c_rtol %.3g in %d iterations (%.3g)",
             rtol, maxit, std::sqrt(rr / tt));
    return set_err(c, IBM_ERR_NOT_CONVERGED, buf);
  }
  return IBM_OK;
}

}  // namespace ibm

using namespace ibm;

extern "C" {

ibm_status ibm_apply_c_inverse(ibm_ctx* c, const double* t, double* s, double c_rtol,
                               int32_t c_maxit, int32_t* iters) {
  if (check_ctx(c) != IBM_OK) return IBM_ERR_ARG;
  const int64_t n = c->mk.n;
  if (n > 0 && (bad_ptr(t) || bad_ptr(s) || t == s))
    return set_err(c, IBM_ERR_ARG, "bad t/s");
  if (!(c_rtol > 0.0) || c_maxit < 1) return set_err(c, IBM_ERR_ARG, "need c_rtol > 0, c_maxit >= 1");
  int it = 0;
  const ibm_status st = c_solve(c, t, s, c_rtol, c_maxit, &it);
  if (iters) *iters = it;
  return st;
}

}  // extern "C"
