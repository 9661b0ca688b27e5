// Krylov vector kernels and per-instance scalar recurrences, all on the device so an iteration
// needs no host round trip.  Sec. 4 of the paper uses MINRES (symmetric A, SPD preconditioner)
// and GMRES; the scalar recurrences are the textbook ones:
//   MINRES  (Paige & Saunders 1975): preconditioned Lanczos, Givens QR, three-term directions;
//   FGMRES  (Saad 1993): right preconditioning with the preconditioned basis stored, Arnoldi by
//           classical Gram-Schmidt applied twice, Givens rotations on the Hessenberg column.
// Reductions are deterministic: each block of an instance writes one partial for a fixed slice
// of the vector, and one block per instance adds the partials in a fixed order, so a result does
// not depend on which other instances share the launch.  (MINRES's r1 . y has two such orders, the vector
// blocks and the tiles of the fused preconditioner passes; which one holds is decided per instance.)
#include <math.h>

#include "pcb_internal.cuh"

namespace pcb {

enum { SS_NONE = 0, SS_MINRES_INIT, SS_MINRES_ALFA, SS_MINRES_GIVENS, SS_NORM, SS_GMRES_ARNOLDI, SS_GMRES_START,
       SS_BNORM };

__device__ __forceinline__ double block_sum(double v) {
  __shared__ double red[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  double r = 0.0;
  if (w == 0) {
    r = lane < (int)(blockDim.x >> 5) ? red[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) r += __shfl_down_sync(0xffffffffu, r, o);
  }
  return r;   // valid in thread 0
}

#define INST_PROLOGUE                                              \
  const int inst = find_inst(off, count, blockIdx.x);             \
  if (active && !active[inst]) return;                            \
  const Geom& g = G[inst];                                         \
  const int lb = blockIdx.x - off[inst];                           \
  const long long len = 2 * g.mn;                                  \
  const long long stride = (long long)g.vec_blocks * blockDim.x;   \
  const long long e0 = (long long)lb * blockDim.x + threadIdx.x;

// partial[blk] = sum a.b over the instance's slice.  skip (k_axpby too): instances to leave out, or null
__global__ void __launch_bounds__(256) k_dot(const Geom* __restrict__ G, const Slots* __restrict__ S,
                                             const int* __restrict__ off, int count, const int* __restrict__ active,
                                             const int* __restrict__ skip, int sa, int sb,
                                             double* __restrict__ partial) {
  INST_PROLOGUE
  if (skip && skip[inst]) return;
  const double* __restrict__ a = S[inst].v[sa];
  const double* __restrict__ b = S[inst].v[sb];
  double acc = 0.0;
  for (long long e = e0; e < len; e += stride) acc = fma(a[e], b[e], acc);
  const double r = block_sum(acc);
  if (threadIdx.x == 0) partial[blockIdx.x] = r;
}

// y = a*x + b*y with (a, b) chosen by `mode` from the instance scalars
enum { AX_COPY = 0, AX_MINRES_R = 1, AX_SCALE_INV_BETA = 2, AX_SCALE_INV_HNORM = 3, AX_ADD = 4, AX_ZERO = 5 };
__global__ void __launch_bounds__(256) k_axpby(const Geom* __restrict__ G, const Slots* __restrict__ S,
                                               const Scal* __restrict__ Sc, const int* __restrict__ off, int count,
                                               const int* __restrict__ active, const int* __restrict__ skip, int mode,
                                               int sx, int sy, int sz) {
  INST_PROLOGUE
  if (skip && skip[inst]) return;
  const Scal& c = Sc[inst];
  const double* __restrict__ x = sx >= 0 ? S[inst].v[sx] : nullptr;
  double* __restrict__ y = S[inst].v[sy];
  if (mode == AX_COPY) {
    for (long long e = e0; e < len; e += stride) y[e] = x[e];
  } else if (mode == AX_MINRES_R) {
    // z = x - (alfa/beta) y  written to slot sz  (x = q, y = r2, z = r1 slot)
    double* __restrict__ z = S[inst].v[sz];
    const double f = c.rf;
    for (long long e = e0; e < len; e += stride) z[e] = fma(f, y[e], x[e]);
  } else if (mode == AX_SCALE_INV_BETA) {
    const double f = 1.0 / c.beta;
    for (long long e = e0; e < len; e += stride) y[e] = x[e] * f;
  } else if (mode == AX_SCALE_INV_HNORM) {
    const double f = 1.0 / c.hnorm;
    for (long long e = e0; e < len; e += stride) y[e] = x[e] * f;
  } else if (mode == AX_ADD) {
    for (long long e = e0; e < len; e += stride) y[e] += x[e];
  } else {   // AX_ZERO
    for (long long e = e0; e < len; e += stride) y[e] = 0.0;
  }
}

// MINRES direction and solution update.  The direction w_k = (y/oldb - oldeps w_{k-2} - delta w_{k-1})/gamma is
// kept without its scale, u = gamma oldb w, so that y enters with coefficient one:
//   u_new = y + c2 u_{k-2} + c1 u_{k-1}  -> slot w2 ;  x += cx u_new
// with the coefficients of the scalar step (Scal::wc1, wc2, wcx): three FP64 operations per value instead
// of four, which leaves the kernel at the HBM limit (48 B per value; N = 511, n = 512: 2.24 -> 2.02 ms).
// Run beside the product and the transforms in a branch of the iteration's graph it gained nothing: every
// variant (1, 2, 3 or all its blocks per SM, with and without priorities) took the others' HBM time.
__global__ void __launch_bounds__(256) k_minres_wx(const Geom* __restrict__ G, const Slots* __restrict__ S,
                                                   const Scal* __restrict__ Sc, const int* __restrict__ off, int count,
                                                   const int* __restrict__ active, int sy, int sw, int sw2, int sx) {
  INST_PROLOGUE
  const Scal& c = Sc[inst];
  const double* __restrict__ y = S[inst].v[sy];
  const double* __restrict__ w = S[inst].v[sw];
  double* __restrict__ w2 = S[inst].v[sw2];
  double* __restrict__ x = S[inst].v[sx];
  const double c1 = c.wc1, c2 = c.wc2, cx = c.wcx;
  long long e = e0;
  for (; e + 3 * stride < len; e += 4 * stride) {       // four values in flight
    double t[4], a[4], b[4], z[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      t[q] = y[e + q * stride];
      a[q] = w2[e + q * stride];
      b[q] = w[e + q * stride];
      z[q] = x[e + q * stride];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      t[q] = fma(c1, b[q], fma(c2, a[q], t[q]));
      w2[e + q * stride] = t[q];
      x[e + q * stride] = fma(cx, t[q], z[q]);
    }
  }
  for (; e < len; e += stride) {
    const double t = fma(c1, w[e], fma(c2, w2[e], y[e]));
    w2[e] = t;
    x[e] = fma(cx, t, x[e]);
  }
}

// The updates of two iterations k, k+1 at once (coefficients wp*: iteration k, w*: k+1):
//   u_k     = y_k     + wpc2 u_{k-2} + wpc1 u_{k-1}   -> slot w2
//   u_{k+1} = y_{k+1} + wc2 u_{k-1} + wc1 u_k         -> slot w;   x += wpcx u_k + wcx u_{k+1}
// 64 B a value for both (five reads, three writes) instead of 96: the update of a single iteration is bound by
// HBM.  Here the six FP64 operations a value are the bound, 0.97 of the measured 529 G/s, and the traffic
// runs at 0.81 of HBM (N = 511, n = 512: two launches of 2.02 ms -> one of 3.12).
__global__ void __launch_bounds__(256) k_minres_wx2(const Geom* __restrict__ G, const Slots* __restrict__ S,
                                                    const Scal* __restrict__ Sc, const int* __restrict__ off, int count,
                                                    const int* __restrict__ active, int sy0, int sy1, int sw, int sw2,
                                                    int sx) {
  INST_PROLOGUE
  const Scal& c = Sc[inst];
  const double* __restrict__ y0 = S[inst].v[sy0];
  const double* __restrict__ y1 = S[inst].v[sy1];
  double* __restrict__ w = S[inst].v[sw];
  double* __restrict__ w2 = S[inst].v[sw2];
  double* __restrict__ x = S[inst].v[sx];
  const double p1 = c.wpc1, p2 = c.wpc2, px = c.wpcx, c1 = c.wc1, c2 = c.wc2, cx = c.wcx;
  long long e = e0;
  for (; e + 3 * stride < len; e += 4 * stride) {       // four values in flight
    double s[4], t[4], a[4], b[4], z[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      s[q] = y0[e + q * stride];
      t[q] = y1[e + q * stride];
      a[q] = w2[e + q * stride];
      b[q] = w[e + q * stride];
      z[q] = x[e + q * stride];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      s[q] = fma(p1, b[q], fma(p2, a[q], s[q]));
      t[q] = fma(c1, s[q], fma(c2, b[q], t[q]));
      w2[e + q * stride] = s[q];
      w[e + q * stride] = t[q];
      x[e + q * stride] = fma(cx, t[q], fma(px, s[q], z[q]));
    }
  }
  for (; e < len; e += stride) {
    const double b = w[e];
    const double u = fma(p1, b, fma(p2, w2[e], y0[e]));
    const double t = fma(c1, u, fma(c2, b, y1[e]));
    w2[e] = u;
    w[e] = t;
    x[e] = fma(cx, t, fma(px, u, x[e]));
  }
}

// Classical Gram-Schmidt over JB basis vectors, two values per thread and step (vectors have even
// length and basis vectors start on 16 bytes).  Both kernels are bound by FP64 issue (one FMA per value
// and vector: 63 us a vector at N = 255, n = 256, against 39 us of HBM) as long as enough loads are in
// flight: the basis values of a step are loaded in groups of eight before they are used, and the blocks
// per SM divide the 16 per SM of a large vector.  JB is the exact count (EXACT; a predicated-off step
// costs its issue slot) or a bound on the per-instance count: 32 Arnoldi steps without a preconditioner at
// N = 255, n = 128 take 78.2 ms with exact counts, 84.1 with bounds 24, 28 and 32 above 20 vectors.  With one
// value per step and the loads left to the compiler, 10, 12, 15 and 17-20 vectors ran 1.2-1.5 times above the
// FP64 rate (12 vectors 1.18 ms).
constexpr int kGroup = 8;
constexpr int gs_blocks(int JB) { return JB <= 8 ? 4 : 2; }

// partial[i tot + blk] = V_i . W over the block's slice, i = 0 .. j
template <int JB, bool EXACT>
__global__ void __launch_bounds__(256, gs_blocks(JB)) k_multidot(const Geom* __restrict__ G, const Slots* __restrict__ S,
                                                  const Scal* __restrict__ Sc, const int* __restrict__ off, int count,
                                                  const int* __restrict__ active, int svbase, int j, int sw,
                                                  double* __restrict__ partial, int tot) {
  INST_PROLOGUE
  if (!EXACT && j < 0) j = Sc[inst].j;   // each instance at its own Arnoldi index
  const long long h = len / 2;
  const double2* __restrict__ V = (const double2*)S[inst].v[svbase];
  const double2* __restrict__ W = (const double2*)S[inst].v[sw];
  double acc[JB];
#pragma unroll
  for (int i = 0; i < JB; ++i) acc[i] = 0.0;
#pragma unroll(JB <= 4 ? 4 : 1)
  for (long long e = e0; e < h; e += stride) {
    const double2 w = W[e];
#pragma unroll
    for (int i0 = 0; i0 < JB; i0 += kGroup) {
      double2 v[kGroup];
#pragma unroll
      for (int i = 0; i < kGroup; ++i)
        if (i0 + i < JB && (EXACT || i0 + i <= j)) v[i] = V[(i0 + i) * h + e];
#pragma unroll
      for (int i = 0; i < kGroup; ++i)
        if (i0 + i < JB && (EXACT || i0 + i <= j)) acc[i0 + i] = fma(v[i].y, w.y, fma(v[i].x, w.x, acc[i0 + i]));
    }
  }
  // block sums, eight at a time: halving the values held per lane at each exchange costs 9 FP64 additions
  // a warp for eight sums instead of 40
  constexpr int NGRP = (JB + 7) / 8;
  __shared__ double red[NGRP][8][8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < NGRP; ++q) {
    double v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = 8 * q + i < JB ? acc[8 * q + i < JB ? 8 * q + i : 0] : 0.0;
#pragma unroll
    for (int w = 4; w >= 1; w >>= 1) {           // lane bit 4 w selects the upper w of 2 w values
      const bool up = lane & (4 * w);
#pragma unroll
      for (int i = 0; i < w; ++i) {
        const double send = up ? v[i] : v[i + w], keep = up ? v[i + w] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * w);
      }
    }
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
    v[0] += __shfl_xor_sync(0xffffffffu, v[0], 1);
    if ((lane & 3) == 0) red[q][warp][lane >> 2] = v[0];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < JB; i += blockDim.x) {
    if (!EXACT && i > j) break;
    double r = 0.0;
#pragma unroll
    for (int w = 0; w < 8; ++w) r += red[i >> 3][w][i & 7];
    partial[(long long)i * tot + blockIdx.x] = r;
  }
}

// W -= sum_i h_i V_i (coef from Scal.H[pass*(MAX+1) + i]) ; or X += sum_i y_i Z_i (pass = -1).  pass 1 (the
// second projection) also leaves partial[blk] = sum of W^2 over the block's slice: the norm of the new
// basis vector without another sweep.  X may be a caller's vector aligned to 8 bytes only.
template <int JB, bool EXACT>
__global__ void __launch_bounds__(256, gs_blocks(JB)) k_multiaxpy(const Geom* __restrict__ G, const Slots* __restrict__ S,
                                                   const Scal* __restrict__ Sc, const int* __restrict__ off, int count,
                                                   const int* __restrict__ active, int svbase, int j, int sw,
                                                   int pass, double* __restrict__ partial) {
  INST_PROLOGUE
  const Scal& c = Sc[inst];
  if (!EXACT && j < 0) j = pass >= 0 ? c.j : c.j - 1;   // per-instance index (after Arnoldi, c.j = columns)
  const long long h = len / 2;
  const double2* __restrict__ V = (const double2*)S[inst].v[svbase];
  double* __restrict__ W = S[inst].v[sw];
  double coef[JB];
#pragma unroll
  for (int i = 0; i < JB; ++i) {
    double k = 0.0;
    if (EXACT || i <= j) k = pass >= 0 ? -c.H[pass * (PCB_MAX_RESTART + 1) + i] : c.y[i];
    coef[i] = k;
  }
  double sq = 0.0;
#pragma unroll(JB <= 4 ? 4 : 1)
  for (long long e = e0; e < h; e += stride) {
    double wx = W[2 * e], wy = W[2 * e + 1];
#pragma unroll
    for (int i0 = 0; i0 < JB; i0 += kGroup) {
      double2 v[kGroup];
#pragma unroll
      for (int i = 0; i < kGroup; ++i)
        if (i0 + i < JB && (EXACT || i0 + i <= j)) v[i] = V[(i0 + i) * h + e];
#pragma unroll
      for (int i = 0; i < kGroup; ++i)
        if (i0 + i < JB && (EXACT || i0 + i <= j)) {
          wx = fma(coef[i0 + i], v[i].x, wx);
          wy = fma(coef[i0 + i], v[i].y, wy);
        }
    }
    W[2 * e] = wx;
    W[2 * e + 1] = wy;
    if (pass == 1) sq = fma(wy, wy, fma(wx, wx, sq));
  }
  if (pass == 1) {
    const double r = block_sum(sq);
    if (threadIdx.x == 0) partial[blockIdx.x] = r;
  }
}

// ------------------------------------------------------------------------------------------
// per-instance reductions + scalar steps (one block per instance)
// ------------------------------------------------------------------------------------------
__device__ void scalar_step(Scal& c, int step, double v, double tol, int j, int restart) {
  switch (step) {
    case SS_BNORM:
      c.bnorm = sqrt(v);
      break;
    case SS_NORM:           // true-residual norm: must not touch the Lanczos scalars
      c.dot1 = v;
      break;
    case SS_MINRES_INIT: {
      c.itn = 0; c.flags = 0; c.active = 1;
      if (!isfinite(v)) { c.flags |= 4; c.active = 0; break; }
      if (v < 0.0) { c.flags |= 2; c.active = 0; break; }
      if (v == 0.0) { c.beta1 = 0.0; c.beta = 0.0; c.est = 0.0; c.flags |= 1; c.active = 0; break; }
      c.beta1 = sqrt(v); c.beta = c.beta1; c.oldb = 0.0; c.dbar = 0.0; c.epsln = 0.0; c.phibar = c.beta1;
      c.cs = -1.0; c.sn = 0.0; c.est = 1.0;
      c.ws1 = c.ws2 = 0.0;
      break;
    }
    case SS_MINRES_ALFA:
      c.alfa = v;
      c.rf = -v / c.beta;
      break;
    case SS_MINRES_GIVENS: {
      c.oldb = c.beta;
      if (!(v >= 0.0)) { c.flags |= isfinite(v) ? 2 : 4; c.active = 0; break; }
      c.beta = sqrt(v);
      c.oldeps = c.epsln;
      c.delta = c.cs * c.dbar + c.sn * c.alfa;
      c.gbar = c.sn * c.dbar - c.cs * c.alfa;
      c.epsln = c.sn * c.beta;
      c.dbar = -c.cs * c.beta;
      c.gamma = hypot(c.gbar, c.beta);
      if (c.gamma == 0.0) { c.flags |= 2; c.active = 0; break; }
      c.cs = c.gbar / c.gamma;
      c.sn = c.beta / c.gamma;
      c.phi = c.cs * c.phibar;
      c.phibar = c.sn * c.phibar;
      // coefficients of k_minres_wx: w_{k-1} = ws1 u_{k-1}, w_{k-2} = ws2 u_{k-2}
      c.wpc1 = c.wc1; c.wpc2 = c.wc2; c.wpcx = c.wcx;
      c.wc1 = -c.oldb * c.delta * c.ws1;
      c.wc2 = -c.oldb * c.oldeps * c.ws2;
      c.ws2 = c.ws1;
      c.ws1 = 1.0 / (c.gamma * c.oldb);
      c.wcx = c.phi * c.ws1;
      c.itn += 1;
      c.est = c.phibar / c.beta1;
      if (c.est <= tol) c.flags |= 1;
      if (!isfinite(c.est)) { c.flags |= 4; c.active = 0; }
      break;
    }
    case SS_GMRES_START: {
      // v = ||r||^2 ; beta = ||r|| ; g = (beta, 0, ...); a new cycle clears the previous flags
      c.flags = 0;
      c.itn = 0;
      c.beta = sqrt(v);
      for (int i = 0; i <= PCB_MAX_RESTART; ++i) c.g[i] = 0.0;
      c.g[0] = c.beta;
      c.j = 0;
      c.est = c.beta / c.bnorm;
      if (!isfinite(v)) { c.flags |= 4; c.active = 0; }
      break;
    }
    default:
      break;
  }
  (void)restart;
}

// Arnoldi column j of FGMRES from the two projections' coefficients and v = ||w||^2: the earlier
// rotations, a new one, the residual estimate.  The block stages the operands in shared memory (one thread
// walking them in global memory took 15-50 us a step, the back substitution it also ran each time included;
// k_backsub now runs that once, when the cycle ends).
__device__ void arnoldi_step(Scal& c, double v, double tol, int j) {
  const int M1 = PCB_MAX_RESTART + 1;
  __shared__ double col[PCB_MAX_RESTART + 1], cs_[PCB_MAX_RESTART], sn_[PCB_MAX_RESTART];
  for (int i = threadIdx.x; i <= j; i += blockDim.x) {
    col[i] = c.H[i] + c.H[M1 + i];
    if (i < j) { cs_[i] = c.gcs[i]; sn_[i] = c.gsn[i]; }
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const double hn = sqrt(v);
    double next = col[0];
    for (int i = 0; i < j; ++i) {
      const double b = col[i + 1];
      col[i] = cs_[i] * next + sn_[i] * b;
      next = -sn_[i] * next + cs_[i] * b;
    }
    double cs = 1.0, sn = 0.0;
    if (hn != 0.0) {
      const double r = hypot(next, hn);
      cs = next / r; sn = hn / r;
    }
    col[j] = cs * next + sn * hn;
    c.hnorm = hn;
    c.gcs[j] = cs; c.gsn[j] = sn;
    const double gj = c.g[j], gn = -sn * gj;
    c.g[j + 1] = gn;
    c.g[j] = cs * gj;
    c.itn += 1;
    c.j = j + 1;
    c.est = fabs(gn) / c.bnorm;
    if (c.est <= tol) c.flags |= 1;
    if (hn == 0.0) c.flags |= 8;        // lucky breakdown: the cycle ends here
    if (!isfinite(c.est)) { c.flags |= 4; c.active = 0; }
  }
  __syncthreads();
  double* R = c.R + (long long)j * M1;
  for (int i = threadIdx.x; i <= j; i += blockDim.x) R[i] = col[i];
  if (threadIdx.x == 0) R[j + 1] = 0.0;
}

// coefficients y of the cycle's update, R y = g: one warp per instance, a column of R per step
__global__ void __launch_bounds__(32) k_backsub(int count, const int* __restrict__ active, Scal* Sc) {
  const int inst = blockIdx.x;
  if (inst >= count || (active && !active[inst])) return;
  Scal& c = Sc[inst];
  const int k = c.j, lane = threadIdx.x, M1 = PCB_MAX_RESTART + 1;
  __shared__ double s[PCB_MAX_RESTART];
  for (int i = lane; i < k; i += 32) s[i] = c.g[i];
  for (int q = k - 1; q >= 0; --q) {
    __syncwarp();
    const double* R = c.R + (long long)q * M1;
    const double y = s[q] / R[q];
    __syncwarp();
    for (int i = lane; i < q; i += 32) s[i] -= R[i] * y;
    if (lane == 0) c.y[q] = y;
  }
}

// Sum the instance's partials (one per block) and run a scalar step.  code2: the instances with a nonzero
// code have theirs at off2, the others at base + off (null: all at off, base 0).
__global__ void __launch_bounds__(512) k_reduce(const int* __restrict__ off, int count, const int* __restrict__ active,
                                                const double* __restrict__ partial, Scal* Sc,
                                                int step, double tol, const double* __restrict__ tols, int j,
                                                int restart, Slots* S, int a0, int s0, int a1, int s1,
                                                const int* __restrict__ off2, const int* __restrict__ code2, int base) {
  const int inst = blockIdx.x;
  if (inst >= count) return;
  if (active && !active[inst]) return;
  const bool second = code2 && code2[inst];
  const int b0 = second ? off2[inst] : base + off[inst], b1 = second ? off2[inst + 1] : base + off[inst + 1];
  // the products leave tens of thousands of partials of a large instance: four loads in flight per thread
  // (N = 511, n = 512: 64 -> 17 us)
  double a4[4] = {0.0, 0.0, 0.0, 0.0};
  int b = b0 + threadIdx.x;
  for (; b + 3 * (int)blockDim.x < b1; b += 4 * blockDim.x) {
#pragma unroll
    for (int q = 0; q < 4; ++q) a4[q] += partial[b + q * blockDim.x];
  }
  for (; b < b1; b += blockDim.x) a4[0] += partial[b];
  const double s = block_sum((a4[0] + a4[1]) + (a4[2] + a4[3]));
  const double tl = tols ? tols[inst] : tol;
  if (step == SS_GMRES_ARNOLDI) {
    __shared__ double total;
    if (threadIdx.x == 0) total = s;
    __syncthreads();
    arnoldi_step(Sc[inst], total, tl, j < 0 ? Sc[inst].j : j);
  } else if (threadIdx.x == 0) {
    scalar_step(Sc[inst], step, s, tl, j, restart);
    if (a0 >= 0) {
      double** v = S[inst].v;
      double* t = v[a0]; v[a0] = v[s0]; v[s0] = t;
      t = v[a1]; v[a1] = v[s1]; v[s1] = t;
    }
  }
}

// multi-reduction for CGS: H[pass][i] = sum of the partials of vector i = blockIdx.y (partial[i tot + b])
__global__ void __launch_bounds__(256) k_reduce_multi(const int* __restrict__ off, int count,
                                                      const int* __restrict__ active,
                                                      const double* __restrict__ partial, int tot, int j, int pass,
                                                      Scal* Sc) {
  const int inst = blockIdx.x, i = blockIdx.y;
  if (inst >= count) return;
  if (active && !active[inst]) return;
  if (i > (j < 0 ? Sc[inst].j : j)) return;
  const int b0 = off[inst], b1 = off[inst + 1];
  double acc = 0.0;
  for (int b = b0 + threadIdx.x; b < b1; b += blockDim.x) acc += partial[(long long)i * tot + b];
  const double s = block_sum(acc);
  if (threadIdx.x == 0) Sc[inst].H[pass * (PCB_MAX_RESTART + 1) + i] = s;
}

// swap slot pointers (per instance, one thread)
__global__ void k_swap(Slots* S, int count, const int* __restrict__ active, int a0, int b0, int a1, int b1, int a2,
                       int b2) {
  const int inst = blockIdx.x * blockDim.x + threadIdx.x;
  if (inst >= count) return;
  if (active && !active[inst]) return;
  double* t;
  if (a0 >= 0) { t = S[inst].v[a0]; S[inst].v[a0] = S[inst].v[b0]; S[inst].v[b0] = t; }
  if (a1 >= 0) { t = S[inst].v[a1]; S[inst].v[a1] = S[inst].v[b1]; S[inst].v[b1] = t; }
  if (a2 >= 0) { t = S[inst].v[a2]; S[inst].v[a2] = S[inst].v[b2]; S[inst].v[b2] = t; }
}

// GMRES basis addressing: slot `dst` = slot `base` + k * 2mn, for up to three (dst, base, k); dst < 0: none
struct SetSlots { int dst[3], base[3], k[3]; };
__global__ void k_setslot(const Geom* __restrict__ G, Slots* S, int count, const int* __restrict__ active, SetSlots q) {
  const int inst = blockIdx.x * blockDim.x + threadIdx.x;
  if (inst >= count) return;
  if (active && !active[inst]) return;
#pragma unroll
  for (int a = 0; a < 3; ++a)
    if (q.dst[a] >= 0) S[inst].v[q.dst[a]] = S[inst].v[q.base[a]] + (long long)q.k[a] * 2 * G[inst].mn;
}

// ------------------------------------------------------------------------------------------
// host launchers
// ------------------------------------------------------------------------------------------
cudaError_t launch_dot(const Batch& B, int sa, int sb) {
  k_dot<<<B.tot_vec, 256, 0, B.stream>>>(B.G, B.S, B.off_vec, B.count, B.active, nullptr, sa, sb, B.partial);
  return cudaGetLastError();
}
// the residual update and the inner product of a MINRES batch's instances without the fused passes (code 0);
// their partials follow those of the fused passes' tiles
cudaError_t launch_minres_rest_residual(const Batch& B, int q, int r2, int r1) {
  k_axpby<<<B.tot_vec, 256, 0, B.stream>>>(B.G, B.S, B.Sc, B.off_vec, B.count, B.active, B.lane_sp[1], AX_MINRES_R, q, r2,
                                           r1);
  return cudaGetLastError();
}
cudaError_t launch_minres_rest_dot(const Batch& B, int sa, int sb) {
  k_dot<<<B.tot_vec, 256, 0, B.stream>>>(B.G, B.S, B.off_vec, B.count, B.active, B.lane_sp[1], sa, sb,
                                         B.partial + B.tot_ls[1]);
  return cudaGetLastError();
}
cudaError_t launch_reduce(const Batch& B, const int* off, int step, double tol, int j, int restart, int a0, int b0,
                          int a1, int b1) {
  // one block size for every instance: the order of its sum must not depend on the batch it is in
  k_reduce<<<B.count, 512, 0, B.stream>>>(off, B.count, B.active, B.partial, B.Sc, step, tol, B.tols, j, restart,
                                          B.S, a0, b0, a1, b1, nullptr, nullptr, 0);
  return cudaGetLastError();
}
// MINRES's scalar step after r1 . y: fused = its partials are the tiles of the preconditioner's passes
// (launch_precond_minres), for the instances that have them
cudaError_t launch_reduce_minres(const Batch& B, bool fused, double tol, int a0, int b0, int a1, int b1) {
  if (!fused) return launch_reduce(B, B.off_vec, SS_MINRES_GIVENS, tol, 0, 0, a0, b0, a1, b1);
  if (B.tot_dst_i[1] == 0) return launch_reduce(B, B.off_ls[1], SS_MINRES_GIVENS, tol, 0, 0, a0, b0, a1, b1);
  k_reduce<<<B.count, 512, 0, B.stream>>>(B.off_vec, B.count, B.active, B.partial, B.Sc, SS_MINRES_GIVENS, tol, B.tols, 0, 0,
                                          B.S, a0, b0, a1, b1, B.off_ls[1], B.lane_sp[1], B.tot_ls[1]);
  return cudaGetLastError();
}
cudaError_t launch_axpby(const Batch& B, int mode, int sx, int sy, int sz) {
  k_axpby<<<B.tot_vec, 256, 0, B.stream>>>(B.G, B.S, B.Sc, B.off_vec, B.count, B.active, nullptr, mode, sx, sy,
                                            sz);
  return cudaGetLastError();
}
cudaError_t launch_minres_wx(const Batch& B, int sy, int sw, int sw2, int sx) {
  k_minres_wx<<<B.tot_vec, 256, 0, B.stream>>>(B.G, B.S, B.Sc, B.off_vec, B.count, B.active, sy, sw, sw2, sx);
  return cudaGetLastError();
}
cudaError_t launch_minres_wx2(const Batch& B, int sy0, int sy1, int sw, int sw2, int sx) {
  k_minres_wx2<<<B.tot_vec, 256, 0, B.stream>>>(B.G, B.S, B.Sc, B.off_vec, B.count, B.active, sy0, sy1, sw, sw2, sx);
  return cudaGetLastError();
}
// Arnoldi index j >= 0 (at most PCB_MAX_RESTART - 1): the kernel of exactly j + 1 vectors.  j < 0 (per-instance
// indices, at most jmax when jmax >= 0): the smallest bound that covers them.
#define PCB_EXACT(X)                                                                                      \
  X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9) X(10) X(11) X(12) X(13) X(14) X(15) X(16) X(17) X(18)     \
  X(19) X(20) X(21) X(22) X(23) X(24) X(25) X(26) X(27) X(28) X(29) X(30) X(31) X(32)
#define PCB_BOUNDS(X) X(2) X(4) X(6) X(8) X(10) X(12) X(14) X(16) X(20) X(24) X(32)
static_assert(PCB_MAX_RESTART == 32, "the lists above cover the largest basis");
cudaError_t launch_multidot(const Batch& B, int svbase, int j, int sw, int jmax) {
#define PCB_ARGS B.G, B.S, B.Sc, B.off_vec, B.count, B.active, svbase, j, sw, B.partial, B.tot_vec
  if (j >= 0) {
    switch (j + 1) {
#define PCB_CASE(JB) case JB: k_multidot<JB, true><<<B.tot_vec, 256, 0, B.stream>>>(PCB_ARGS); break;
      PCB_EXACT(PCB_CASE)
#undef PCB_CASE
      default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
  }
  const int need = jmax < 0 ? PCB_MAX_RESTART : jmax + 1;
#define PCB_CASE(JB) \
  if (need <= JB) { k_multidot<JB, false><<<B.tot_vec, 256, 0, B.stream>>>(PCB_ARGS); return cudaGetLastError(); }
  PCB_BOUNDS(PCB_CASE)
#undef PCB_CASE
#undef PCB_ARGS
  return cudaErrorInvalidValue;
}
// jmax: as for launch_multidot
cudaError_t launch_reduce_multi(const Batch& B, int j, int pass, int jmax) {
  const int rows = j >= 0 ? j + 1 : jmax >= 0 ? jmax + 1 : PCB_MAX_RESTART;
  k_reduce_multi<<<dim3(B.count, rows), 256, 0, B.stream>>>(B.off_vec, B.count, B.active, B.partial, B.tot_vec, j, pass,
                                                           B.Sc);
  return cudaGetLastError();
}
cudaError_t launch_backsub(const Batch& B) {
  k_backsub<<<B.count, 32, 0, B.stream>>>(B.count, B.active, B.Sc);
  return cudaGetLastError();
}
cudaError_t launch_multiaxpy(const Batch& B, int svbase, int j, int sw, int pass, int jmax) {
#define PCB_ARGS B.G, B.S, B.Sc, B.off_vec, B.count, B.active, svbase, j, sw, pass, B.partial
  if (j >= 0) {
    switch (j + 1) {
#define PCB_CASE(JB) case JB: k_multiaxpy<JB, true><<<B.tot_vec, 256, 0, B.stream>>>(PCB_ARGS); break;
      PCB_EXACT(PCB_CASE)
#undef PCB_CASE
      default: return cudaErrorInvalidValue;
    }
    return cudaGetLastError();
  }
  const int need = jmax < 0 ? PCB_MAX_RESTART : jmax + 1;
#define PCB_CASE(JB) \
  if (need <= JB) { k_multiaxpy<JB, false><<<B.tot_vec, 256, 0, B.stream>>>(PCB_ARGS); return cudaGetLastError(); }
  PCB_BOUNDS(PCB_CASE)
#undef PCB_CASE
#undef PCB_ARGS
  return cudaErrorInvalidValue;
}
cudaError_t launch_swap(const Batch& B, int a0, int b0, int a1, int b1, int a2, int b2) {
  k_swap<<<(B.count + 63) / 64, 64, 0, B.stream>>>(B.S, B.count, B.active, a0, b0, a1, b1, a2, b2);
  return cudaGetLastError();
}
cudaError_t launch_setslot(const Batch& B, int dst, int base, int k) {
  const SetSlots q = {{dst, -1, -1}, {base, 0, 0}, {k, 0, 0}};
  k_setslot<<<(B.count + 63) / 64, 64, 0, B.stream>>>(B.G, B.S, B.count, B.active, q);
  return cudaGetLastError();
}
// the three vectors of Arnoldi step j: v_j, z_j, v_{j+1}
cudaError_t launch_setslots(const Batch& B, int vj, int zj, int vj1, int vbase, int zbase, int j) {
  const SetSlots q = {{vj, zj, vj1}, {vbase, zbase, vbase}, {j, j, j + 1}};
  k_setslot<<<(B.count + 63) / 64, 64, 0, B.stream>>>(B.G, B.S, B.count, B.active, q);
  return cudaGetLastError();
}

}  // namespace pcb
