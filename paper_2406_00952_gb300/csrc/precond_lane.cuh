// Preconditioner passes with one line per lane (paper Sec. 3.5): the spatial DST-I / DCT-I passes
// and the time pass of precond_lane_*.cu, in FP32 and FP64.
//
// A line of M = A B points is transformed in two register steps with one exchange through shared
// memory.  With s = t + B q and k = k1 + A k2,
//     X[k1 + A k2] = sum_t W_B^{t k2} W_M^{t k1} U[t][k1],   U[t][k1] = sum_q x[t + B q] W_A^{q k1}.
// Adjacent lanes hold the same step of adjacent lines, so every global access of a pass that
// walks across lines is a contiguous segment, every twiddle is uniform over a group of lanes, no
// value moves between lanes, and no lane index enters the arithmetic.
//
// Spatial lines are the odd (DST-I) or even (DCT-I) extension of L = M/2 -/+ 1 values.  Its
// symmetry x[M - s] = -/+ x[s] is used in both steps, not only in the exchange:
//     U[B - t][k1] = -/+ W_A^{-k1} U[t][-k1],   X[M - k] = -/+ X[k],
// so only t = 0 .. B/2 and k1 = 0 .. A/2 are computed: B/2 + 1 register DFTs of size A and A/2 + 1 of
// size B per line instead of B and A.  That is 17 + 17 DFTs of 32 points for M = 1024, against 32 + 32
// for the transform of the extension as a general line, at the same rounding per value (no running
// sums, no divisions).
//
// What bounds the passes and what they measured (one GB300, ncu durations; in brackets the pipelined
// kernels of precond_pipe.cu, which remain the alternative a caller can pin, and the tile kernels):
//   N = 511, n = 512, FP32: pass 1 0.61 ms (0.83), pass 2 0.32 (0.68; 6.5 TB/s, at the HBM limit), time 0.58
//   (0.83), pass 4 0.35 (0.65; 6.0 TB/s), pass 5 0.65 (0.59); the apply 2.54 ms (3.53).  Passes 1 and 5 wait for
//   the conversion of their FP64 side between load and store, the time pass for its two barriers with
//   only 16 warps a multiprocessor (128 registers).
//   N = 255, n = 256, FP64: spatial passes 1.06 ms each, time 2.03, the apply 6.3 ms (14.7): 89% of the FP64
//   issue rate on the operations of the symmetric transform.
//   N = 383, n = 64, FP32 (tile kernels before): apply 0.21 ms (1.00).
#pragma once
#include "f32_convert.cuh"
#include "fft_reg.cuh"

namespace pcb {
namespace lane {

enum { PK_ABS_PS = 1, PK_PS = 2, PK_PMS = 3 };

// line lengths M = 2 L of the spatial passes and their factors.  Both factors are register DFT sizes.
// GROUPS is the number of lane groups that share the B/2 + 1 and the A/2 + 1 steps of a tile.
template <int M> struct Shape;
template <> struct Shape<32> { static constexpr int A = 8, B = 4, GROUPS = 5; };
template <> struct Shape<48> { static constexpr int A = 8, B = 6, GROUPS = 5; };
template <> struct Shape<64> { static constexpr int A = 8, B = 8, GROUPS = 5; };
template <> struct Shape<96> { static constexpr int A = 12, B = 8, GROUPS = 7; };
template <> struct Shape<128> { static constexpr int A = 16, B = 8, GROUPS = 9; };
template <> struct Shape<192> { static constexpr int A = 16, B = 12, GROUPS = 9; };
template <> struct Shape<256> { static constexpr int A = 16, B = 16, GROUPS = 9; };
template <> struct Shape<384> { static constexpr int A = 24, B = 16, GROUPS = 13; };
template <> struct Shape<512> { static constexpr int A = 32, B = 16, GROUPS = 9; };
template <> struct Shape<768> { static constexpr int A = 32, B = 24, GROUPS = 17; };
template <> struct Shape<1024> { static constexpr int A = 32, B = 32, GROUPS = 17; };

// Lines per tile.  The exchange holds (B/2 + 1) A complex values a line and has to leave room for two or
// more blocks per SM; sixteen FP32 pairs are a full 128-byte line.
template <typename R, int M>
constexpr int spatial_lanes() {
  return sizeof(R) == 4 ? (M >= 512 ? 16 : 32) : (M >= 768 ? 8 : M >= 384 ? 16 : 32);
}

template <typename R> __device__ __forceinline__ const cx<R>* tw_space(const Geom& g);
template <> __device__ __forceinline__ const float2* tw_space<float>(const Geom& g) { return g.twd_f; }
template <> __device__ __forceinline__ const double2* tw_space<double>(const Geom& g) { return g.twd_d; }
template <typename R> __device__ __forceinline__ const cx<R>* tw_time(const Geom& g);
template <> __device__ __forceinline__ const float2* tw_time<float>(const Geom& g) { return g.twt_f; }
template <> __device__ __forceinline__ const double2* tw_time<double>(const Geom& g) { return g.twt_d; }
template <typename R> __device__ __forceinline__ const cx<R>* twist(const Geom& g);
template <> __device__ __forceinline__ const float2* twist<float>(const Geom& g) { return g.pre_f; }
template <> __device__ __forceinline__ const double2* twist<double>(const Geom& g) { return g.pre_d; }
template <typename R> __device__ __forceinline__ const cx<R>* lam_time(const Geom& g);
template <> __device__ __forceinline__ const float2* lam_time<float>(const Geom& g) { return g.mu_f; }
template <> __device__ __forceinline__ const double2* lam_time<double>(const Geom& g) { return g.mu_d; }

template <typename T> __device__ __forceinline__ T mulc(T a, T b) {   // a * conj(b)
  T c;
  c.x = a.x * b.x + a.y * b.y;
  c.y = a.y * b.x - a.x * b.y;
  return c;
}
template <typename T> __device__ __forceinline__ T neg(T a) { a.x = -a.x; a.y = -a.y; return a; }
__device__ __forceinline__ float rsq(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsq(double x) { return rsqrt(x); }

// Where a pass reads or writes.  sel >= 0: a vector slot of the instance (FP64, two halves of mn values:
// rows of N, slices of m).  sel < 0: scratch buffer -1 - sel.  The FP32 scratch holds the two halves of a
// position as one pair, rows of lr pairs, slices of mp pairs: a tile of 16 columns is then a full
// 128-byte line, read and written with half the instructions two separate halves would take.  The
// FP64 scratch is one buffer in the vector layout.
struct View {
  void* base;
  long long hs;      // distance of the second half (vector layout)
  int ts, rs;        // time step, row
};
template <typename R>
__device__ __forceinline__ View view_of(const Geom& g, const Slots& s, int sel) {
  View v;
  v.hs = g.mn;
  if (sel >= 0) {
    v.base = s.v[sel]; v.ts = g.m; v.rs = g.N;
  } else if (sizeof(R) == 8) {
    v.base = g.scratch; v.ts = g.m; v.rs = g.N;
  } else {
    v.ts = (int)g.mp; v.rs = g.lr;
    v.base = (float2*)g.scratch + (sel == -1 ? 0 : (long long)g.n * g.mp);
  }
  return v;
}
// the pair of values at an offset of a view, in the pass's scratch layout
template <typename R> struct Pairs;
template <> struct Pairs<float> {
  float2* p;
  __device__ __forceinline__ Pairs(const View& v, long long at) : p((float2*)v.base + at) {}
  __device__ __forceinline__ float2 get(int at) const { return p[at]; }
  __device__ __forceinline__ float half(int at, int h) const { return h ? p[at].y : p[at].x; }
  __device__ __forceinline__ void put(int at, float2 v) const { p[at] = v; }
};
template <> struct Pairs<double> {
  double *p, *q;
  __device__ __forceinline__ Pairs(const View& v, long long at) : p((double*)v.base + at), q(p + v.hs) {}
  __device__ __forceinline__ double2 get(int at) const { return make_double2(p[at], q[at]); }
  __device__ __forceinline__ double half(int at, int h) const { return h ? q[at] : p[at]; }
  __device__ __forceinline__ void put(int at, double2 v) const { p[at] = v.x; q[at] = v.y; }
};

// What a pass of a MINRES iteration takes over from the vector kernels around the apply (see FUSE)
struct LaneFuse {
  const Scal* Sc;
  double* partial;
  int r2, z;
};

// Bring a line towards L2.  A block asks for the tile `ahead` blocks on, which starts about when it
// ends: HBM then works through the register steps, and the loads of a tile find most of it in L2.
// (N = 511, n = 512: pass 2 0.41 -> 0.39 ms, pass 4 0.42 -> 0.39.  Not for FP64 rows, which start at any
// 8-byte offset: fetching the lines they straddle costs more than it hides, pass 1 0.87 -> 1.05 ms.)
__device__ __forceinline__ void prefetch(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// Input of the first step of one line, t in [0, B/2]: x[t + B q], q < A, of the extension.  get(index)
// returns the pair of values (first half, second half) at `index` of the line.  Neumann inverse passes
// scale the two end values by sqrt 2.
template <typename R, int M, bool EV, typename G>
__device__ __forceinline__ void gather(cx<R>* x, int t, bool inv, G&& get) {
  constexpr int A = Shape<M>::A, B = Shape<M>::B;
#pragma unroll
  for (int q = 0; q < A; ++q) {
    const int s = t + B * q;
    const int at = q < A / 2 ? s : M - s;                 // s = 0 only for q = 0, s = L only for q = A/2
    cx<R> v;
    if constexpr (EV) {
      v = get(at);
      if ((q == 0 || q == A / 2) && t == 0 && inv) v = cscale(v, (R)1.41421356237309504880);
    } else {
      if (q == 0 || q == A / 2) {
        v = get(t == 0 ? 0 : at - 1);
        if (t == 0) v = mk<R>((R)0, (R)0);
      } else {
        v = get(at - 1);
      }
      if (q >= A / 2) v = neg(v);
    }
    x[q] = v;
  }
}

// Second step, k1 in [0, A/2]: v[t] = W_M^{t k1} U[t][k1] for all t from the stored half, then the
// B-point DFT.  u(t, k) reads the exchange.
template <typename R, int M, bool EV, typename U>
__device__ __forceinline__ void second_step(cx<R>* v, int k1, const cx<R>* __restrict__ w, U&& u) {
  constexpr int A = Shape<M>::A, B = Shape<M>::B;
  const int km = k1 ? A - k1 : 0;
  v[0] = u(0, k1);
  v[B / 2] = cmul(u(B / 2, k1), __ldg(&w[B / 2 * k1]));
#pragma unroll
  for (int t = 1; t < B / 2; ++t) {
    const cx<R> wt = __ldg(&w[t * k1]);
    v[t] = cmul(u(t, k1), wt);
    const cx<R> m = mulc(u(t, km), wt);
    v[B - t] = EV ? m : neg(m);
  }
  reg_dft<cx<R>, R, B>(v, false);
}

// Write the outputs of one k1: put(index, first half, second half).  FP64 passes leave the four
// spatial scales to the time pass's weights; FP32 passes scale here (sc), which keeps the range.
template <typename R, int M, bool EV, typename P>
__device__ __forceinline__ void put_outputs(const cx<R>* v, int k1, bool inv, R sc, P&& put) {
  constexpr int A = Shape<M>::A, B = Shape<M>::B, L = M / 2;
  const bool edge = k1 == 0 || k1 == A / 2;               // k and M - k both in this row
#pragma unroll
  for (int k2 = 0; k2 < B; ++k2) {
    const int k = k1 + A * k2;
    cx<R> Y = v[pos<B>(k2)];
    if (k2 >= B / 2 && edge && !(EV && k2 == B / 2 && k1 == 0)) continue;
    const int p = k2 < B / 2 ? k : M - k;
    if constexpr (EV) {
      if (sizeof(R) == 4) Y = cscale(Y, sc);
      if ((k2 == 0 || k2 == B / 2) && k1 == 0 && !inv) Y = cscale(Y, (R)0.70710678118654752440);
      put(p, Y.x, Y.y);
    } else {
      if (k2 == 0 && k1 == 0) continue;
      if (sizeof(R) == 4) Y = cscale(Y, sc);
      if (k2 < B / 2) put(p - 1, -Y.y, Y.x);
      else put(p - 1, Y.y, -Y.x);
    }
  }
}

template <typename R, int M>
constexpr size_t spatial_smem() {
  return (size_t)(Shape<M>::B / 2 + 1) * Shape<M>::A * spatial_lanes<R, M>() * sizeof(cx<R>);
}
template <typename R, int M>
constexpr int spatial_threads() { return Shape<M>::GROUPS * spatial_lanes<R, M>(); }
// resident blocks the compiler budgets registers for
template <typename R, int M>
constexpr int spatial_blocks() {
  if (sizeof(R) == 8) return 2;
  return M >= 768 ? 2 : M >= 512 ? 4 : M >= 384 ? 1 : 4;
}

// ------------------------------------------------------------------------------------------
// Transform along the row index (the strided axis): lines (t, c), c = c0 .. c0 + LT - 1, values at row
// r of the slice; in place or to a second view of the same orientation.  Loads go straight to
// registers and stores straight from them: LT adjacent columns are one contiguous segment.
// USER: the input is a vector slot.  An FP32 pass converts it on its way to the exchange memory first:
// 2 A FP64 values in registers would spill.
// FUSE (FP32, USER): the input is MINRES's residual r1 = q + rf r2 (q = in_sel, rf = -alfa/beta from the
// scalar step), formed here and written to slot fuse.z, instead of by a kernel of its own that this pass
// would read again: 28 B a value in one launch instead of 24 + 12 (N = 511, n = 512: 0.94 + 0.61 -> 1.26 ms).
// ------------------------------------------------------------------------------------------
template <typename R, int M, bool EV, bool USER, bool FUSE>
__global__ void __launch_bounds__(spatial_threads<R, M>(), spatial_blocks<R, M>())
    k_lane_rows(const Geom* __restrict__ G, const Slots* __restrict__ S, const int* __restrict__ off, int count, Sel sel,
                int in_sel, int out_sel, int inv, LaneFuse fuse, int ahead) {
  using T = cx<R>;
  constexpr int A = Shape<M>::A, B = Shape<M>::B, NG = Shape<M>::GROUPS, LT = spatial_lanes<R, M>();
  constexpr bool STAGED = USER && sizeof(R) == 4;
  static_assert(NG > B / 2, "one first step per group");
  extern __shared__ __align__(16) unsigned char lane_smem[];
  const int inst = find_inst(off, count, blockIdx.x);
  if (sel.skip(inst)) return;
  const Geom& g = G[inst];
  const int N = g.N, nb = (N + LT - 1) / LT;
  const int lt = blockIdx.x - (count > 1 ? __ldg(off + inst) : 0);
  const int ts = lt / nb, c0 = (lt - ts * nb) * LT;
  const int l = threadIdx.x % LT, grp = threadIdx.x / LT;
  T* ex = (T*)lane_smem + l;
  const bool ok = c0 + l < N;
  const bool first = grp <= B / 2;
  T x[A];
  {
    const View v = view_of<R>(g, S[inst], in_sel);
    const long long at0 = (long long)ts * v.ts + (ok ? c0 + l : N - 1);
    const int rs = v.rs;
    if constexpr (STAGED) {
      // U rows per batch: their loads are in flight together, then all are converted without a branch.
      // (N = 511, n = 512: apply 2.73 ms with 4 rows, 2.61 with 8, 2.55 with 16; shorter lines lose with
      // 16, most of a second batch being past the end.)  A value the integer conversion does not cover
      // sends the thread through its rows once more.
      const double* __restrict__ in0 = (const double*)v.base + at0;
      const double* __restrict__ in1 = in0 + v.hs;
      constexpr int U = FUSE ? (M >= 512 ? 8 : 4) : M >= 1024 ? 16 : 8;
      unsigned rare = 0;
      const double rf = FUSE ? fuse.Sc[inst].rf : 0.0;
      const double* __restrict__ r0 = FUSE ? S[inst].v[fuse.r2] + at0 : nullptr;
      double* __restrict__ z0 = FUSE ? S[inst].v[fuse.z] + at0 : nullptr;
      for (int r = grp; r < N; r += U * NG) {
        double a[U], b[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int at = min(r + u * NG, N - 1) * rs;
          a[u] = in0[at];
          b[u] = in1[at];
        }
        if constexpr (FUSE) {
          double c[U], d[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int at = min(r + u * NG, N - 1) * rs;
            c[u] = r0[at];
            d[u] = r0[v.hs + at];
          }
#pragma unroll
          for (int u = 0; u < U; ++u) {
            a[u] = fma(rf, c[u], a[u]);
            b[u] = fma(rf, d[u], b[u]);
            if (ok && r + u * NG < N) {
              z0[(r + u * NG) * rs] = a[u];
              z0[v.hs + (r + u * NG) * rs] = b[u];
            }
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const T z = mk<R>((R)d2f_plain(a[u], rare), (R)d2f_plain(b[u], rare));
          if (r + u * NG < N) ex[(r + u * NG) * LT] = z;
        }
      }
      if (rare) {
#pragma unroll 1
        for (int r = grp; r < N; r += NG) {
          double a = in0[r * rs], b = in1[r * rs];
          if (FUSE) {
            a = fma(rf, r0[r * rs], a);
            b = fma(rf, r0[v.hs + r * rs], b);
          }
          ex[r * LT] = mk<R>((R)a, (R)b);
        }
      }
      __syncthreads();
      if (first) gather<R, M, EV>(x, grp, inv != 0, [&](int at) { return ex[at * LT]; });
    } else {
      if (sizeof(R) == 4 && lt + ahead < g.n * nb) {
        const int t2 = (lt + ahead) / nb, c2 = (lt + ahead - t2 * nb) * LT;
        const T* p = (const T*)v.base + (long long)t2 * v.ts + c2;
        for (int r = threadIdx.x; r < N; r += spatial_threads<R, M>()) prefetch(p + r * rs);
      }
      const Pairs<R> in(v, at0);
      if (first) gather<R, M, EV>(x, grp, inv != 0, [&](int at) { return in.get(at * rs); });
    }
    if (first) reg_dft<T, R, A>(x, false);
    if (STAGED) __syncthreads();                       // every staged value has been read
    if (first) {
#pragma unroll
      for (int k = 0; k < A; ++k) ex[(grp * A + k) * LT] = x[pos<A>(k)];
    }
  }
  __syncthreads();
  const View v = view_of<R>(g, S[inst], out_sel);
  const Pairs<R> out(v, (long long)ts * v.ts + c0 + l);
  const int rs = v.rs;
  const T* __restrict__ w = tw_space<R>(g);
  const R sc = sizeof(R) == 4 ? (R)__frsqrt_rn((float)M) : (R)1;     // 0.5 sqrt(2 / L)
  for (int k1 = grp; k1 <= A / 2; k1 += NG) {
    T y[B];
    second_step<R, M, EV>(y, k1, w, [&](int t, int k) { return ex[(t * A + k) * LT]; });
    if (ok) put_outputs<R, M, EV>(y, k1, inv != 0, sc, [&](int p, R a, R b) { out.put(p * rs, mk<R>(a, b)); });
  }
}

// ------------------------------------------------------------------------------------------
// Transform along the contiguous index with a transposed result: lines are rows r0 .. r0 + LT - 1 of
// a slice; value p of row r goes to out[p rs + r].  The rows come in with 8-byte asynchronous copies
// (coalesced along the row) and are read back one line per lane (odd pitch); the exchange reuses that
// memory.  USER: the output is a vector slot.
// FUSE (FP32, USER): also leaves partial[block] = sum of the output times slot fuse.z over the tile, the
// inner product r1 . y of MINRES, whose kernel would read the output again: 20 B a value instead of
// 12 + 16 (N = 511, n = 512: 0.65 + 0.60 -> 1.07 ms).
// ------------------------------------------------------------------------------------------
template <int M, bool EV>
constexpr int cols_pitch() { return (EV ? M / 2 + 1 : M / 2 - 1) | 1; }
template <typename R, int M, bool EV>
constexpr size_t cols_smem() {
  constexpr size_t rows = (size_t)2 * spatial_lanes<R, M>() * cols_pitch<M, EV>() * sizeof(R);
  return rows > spatial_smem<R, M>() ? rows : spatial_smem<R, M>();
}

// partial[block] = the sum of the block's dots.  Sixteen lanes at a time: the last warp of a block may be half a
// warp.
template <int NT>
__device__ __forceinline__ void tile_sum(double dot, double* __restrict__ partial) {
  __shared__ double red[NT / 16];
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) dot += __shfl_xor_sync(threadIdx.x & 16 ? 0xffff0000u : 0x0000ffffu, dot, o, 16);
  if (threadIdx.x % 16 == 0) red[threadIdx.x / 16] = dot;
  __syncthreads();
  if (threadIdx.x == 0) {
    double sum = 0.0;
    for (int k = 0; k < NT / 16; ++k) sum += red[k];
    partial[blockIdx.x] = sum;
  }
}

template <typename R, int M, bool EV, bool USER, bool FUSE>
__global__ void __launch_bounds__(spatial_threads<R, M>(), spatial_blocks<R, M>())
    k_lane_cols(const Geom* __restrict__ G, const Slots* __restrict__ S, const int* __restrict__ off, int count, Sel sel,
                int in_sel, int out_sel, int inv, LaneFuse fuse, int ahead) {
  using T = cx<R>;
  constexpr int A = Shape<M>::A, B = Shape<M>::B, NG = Shape<M>::GROUPS, LT = spatial_lanes<R, M>();
  constexpr int N = EV ? M / 2 + 1 : M / 2 - 1, PITCH = cols_pitch<M, EV>(), NT = spatial_threads<R, M>();
  constexpr bool STAGED = USER && sizeof(R) == 4;
  static_assert(NG > B / 2, "one first step per group");
  extern __shared__ __align__(16) unsigned char lane_smem[];
  const int inst = find_inst(off, count, blockIdx.x);
  if (sel.skip(inst)) return;
  const Geom& g = G[inst];
  constexpr int nb = (N + LT - 1) / LT;
  const int lt = blockIdx.x - (count > 1 ? __ldg(off + inst) : 0);
  const int ts = lt / nb, r0 = (lt - ts * nb) * LT;
  const int l = threadIdx.x % LT, grp = threadIdx.x / LT;
  {
    // FP32: LT rows of pairs; FP64: LT rows of the first half, then LT of the second
    const View v = view_of<R>(g, S[inst], in_sel);
    constexpr int H = sizeof(R) == 4 ? 1 : 2;
    const long long at0 = (long long)ts * v.ts + (long long)r0 * v.rs;
    const int nr = min(LT, N - r0);
    constexpr int CL = 16;                         // sixteen threads a row: 128 contiguous bytes per step
    const int cl = threadIdx.x % CL;
    for (int row = threadIdx.x / CL; row < H * LT; row += NT / CL) {
      const int h = row >= LT, r = row - h * LT;
      if (r >= nr) continue;
      const unsigned sa = (unsigned)__cvta_generic_to_shared(lane_smem + ((size_t)row * PITCH + cl) * 8);
      const double* src = (const double*)v.base + at0 + (h ? v.hs : 0) + (long long)r * v.rs + cl;   // 8-byte units
#pragma unroll
      for (int i = 0; i < (N + CL - 1) / CL; ++i)
        if ((i + 1) * CL <= N || i * CL + cl < N)
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8;\n" ::"r"(sa + i * CL * 8), "l"(src + i * CL) : "memory");
    }
    if (sizeof(R) == 4 && lt + ahead < g.n * nb) {
      const int t2 = (lt + ahead) / nb, r2 = (lt + ahead - t2 * nb) * LT, n2 = min(LT, N - r2);
      const T* p = (const T*)v.base + (long long)t2 * v.ts + (long long)r2 * v.rs;
      constexpr int LN = (N + 15) / 16;            // cache lines a row
      for (int e = threadIdx.x; e < n2 * LN; e += NT) {
        const int row = e / LN, c = e - row * LN;
        prefetch(p + row * v.rs + c * 16);
      }
    }
    asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
  }
  __syncthreads();
  const bool ok = r0 + l < N;
  T* ex = (T*)lane_smem + l;
  const bool first = grp <= B / 2;
  T x[A];
  if (first) {
    if constexpr (sizeof(R) == 4) {
      const T* a = (const T*)lane_smem + (ok ? l : 0) * PITCH;
      gather<R, M, EV>(x, grp, inv != 0, [&](int at) { return a[at]; });
    } else {
      const R* a = (const R*)lane_smem + (ok ? l : 0) * PITCH;
      gather<R, M, EV>(x, grp, inv != 0, [&](int at) { return mk<R>(a[at], a[LT * PITCH + at]); });
    }
    reg_dft<T, R, A>(x, false);
  }
  __syncthreads();                                 // every row has been read: the exchange may overwrite
  if (first) {
#pragma unroll
    for (int k = 0; k < A; ++k) ex[(grp * A + k) * LT] = x[pos<A>(k)];
  }
  __syncthreads();
  const View v = view_of<R>(g, S[inst], out_sel);
  const long long at0 = (long long)ts * v.ts + r0 + l;
  const Pairs<R> out(v, at0);
  const int rs = v.rs;
  const T* __restrict__ w = tw_space<R>(g);
  const R sc = sizeof(R) == 4 ? (R)__frsqrt_rn((float)M) : (R)1;
  for (int k1 = grp; k1 <= A / 2; k1 += NG) {
    T y[B];
    second_step<R, M, EV>(y, k1, w, [&](int t, int k) { return ex[(t * A + k) * LT]; });
    if (ok)
      put_outputs<R, M, EV>(y, k1, inv != 0, sc, [&](int p, R a, R b) {
        // line position p is exchange slot (p / A, p mod A): a slot of row k1 or A - k1, which this
        // thread alone has read
        if constexpr (STAGED) ex[(p + (EV ? 0 : 1)) * LT] = mk<R>(a, b);
        else out.put(p * rs, mk<R>(a, b));
      });
  }
  if constexpr (STAGED) {
    // FP32 -> FP64 on the way out, as on the way in (k_lane_rows)
    __syncthreads();
    double* __restrict__ out0 = (double*)v.base + at0;
    double* __restrict__ out1 = out0 + v.hs;
    const double* __restrict__ z0 = FUSE ? S[inst].v[fuse.z] + at0 : nullptr;
    constexpr int U = FUSE && M >= 512 ? 8 : 4;
    const T* src = ex + (EV ? 0 : LT);
    unsigned rare = 0;
    double dot = 0.0;
    if (ok)
      for (int p = grp; p < N; p += U * NG) {
        double za[U], zb[U];
        if constexpr (FUSE) {
#pragma unroll
          for (int u = 0; u < U; ++u) {
            const int at = min(p + u * NG, N - 1) * rs;
            za[u] = z0[at];
            zb[u] = z0[v.hs + at];
          }
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (p + u * NG < N) {
            const T z = src[(p + u * NG) * LT];
            const double a = f2d_plain(z.x, rare), b = f2d_plain(z.y, rare);
            out0[(p + u * NG) * rs] = a;
            out1[(p + u * NG) * rs] = b;
            if constexpr (FUSE) dot = fma(b, zb[u], fma(a, za[u], dot));
          }
        }
      }
    if (ok && rare) {
      dot = 0.0;
#pragma unroll 1
      for (int p = grp; p < N; p += NG) {
        const double a = src[p * LT].x, b = src[p * LT].y;
        out0[p * rs] = a;
        out1[p * rs] = b;
        if constexpr (FUSE) dot = fma(b, z0[v.hs + p * rs], fma(a, z0[p * rs], dot));
      }
    }
    if constexpr (FUSE) tile_sum<NT>(dot, fuse.partial);
  }
}

// The inner product of the fused pass on its own, tile by tile and value by value in the same order: for
// solves whose preconditioner is timed alone (profile), so that timing does not change the iterates.
template <int M>
__global__ void __launch_bounds__(spatial_threads<float, M>())
    k_lane_dot(const Geom* __restrict__ G, const Slots* __restrict__ S, const int* __restrict__ off, int count, Sel sel,
               int sy, int sz, double* __restrict__ partial) {
  constexpr int NG = Shape<M>::GROUPS, LT = spatial_lanes<float, M>(), N = M / 2 - 1, nb = (N + LT - 1) / LT;
  const int inst = find_inst(off, count, blockIdx.x);
  if (sel.skip(inst)) return;
  const Geom& g = G[inst];
  const int lt = blockIdx.x - (count > 1 ? __ldg(off + inst) : 0);
  const int ts = lt / nb, r0 = (lt - ts * nb) * LT;
  const int l = threadIdx.x % LT, grp = threadIdx.x / LT;
  double dot = 0.0;
  if (r0 + l < N) {
    const long long at0 = (long long)ts * g.m + r0 + l;
    const double* __restrict__ y = S[inst].v[sy] + at0;
    const double* __restrict__ z = S[inst].v[sz] + at0;
    for (int p = grp; p < N; p += NG) dot = fma(y[g.mn + p * N], z[g.mn + p * N], fma(y[p * N], z[p * N], dot));
  }
  tile_sum<spatial_threads<float, M>()>(dot, partial);
}

// ------------------------------------------------------------------------------------------
// Time pass: forward DFT of the twisted lines, the pointwise solve, inverse DFT, untwist.  Columns
// (row p, index c0 .. c0 + LT - 1) per tile; n = A B.
//   zeta = pi: the two halves are one complex line z = h0 + i h1; slots r = k1 + A k2 and n-1-r (the
//   conjugate partner) are rows k1 and A-1-k1 at k2 and B-1-k2, and one thread holds both rows, so
//   the pair shares one weight (lambda_{n-1-r} = conj lambda_r) and P_S couples in registers.  The
//   twist exp(-i pi (t + B q) / n) is a compile-time factor exp(-i pi q / A) before the first step and
//   part of the twiddle after it: exp(-i pi t / n) W_n^{t k1} = exp(-i pi t (2 k1 + 1) / n), a table
//   of 2n entries.
//   General zeta (GZ): the halves are two lines; a thread holds both at the same k1.
// B = 1 (short lines): the whole line sits in one thread.
// ------------------------------------------------------------------------------------------
template <typename R, int n> struct TimeShape { static constexpr int A = n, B = 1; };       // n <= 4
// FP32 lines of 8 and 16 steps stay in one thread; FP64 ones are spread, because a small problem is bound
// by the serial FP64 work of a warp (about 76 cycles an instruction): N = 15, n = 16 26 -> 12 us
template <> struct TimeShape<float, 8> { static constexpr int A = 8, B = 1; };
template <> struct TimeShape<float, 16> { static constexpr int A = 16, B = 1; };
template <> struct TimeShape<double, 8> { static constexpr int A = 4, B = 2; };
template <> struct TimeShape<double, 16> { static constexpr int A = 8, B = 2; };
template <typename R> struct TimeShape<R, 32> { static constexpr int A = 8, B = 4; };
template <typename R> struct TimeShape<R, 64> { static constexpr int A = 8, B = 8; };
template <typename R> struct TimeShape<R, 128> { static constexpr int A = 16, B = 8; };
template <typename R> struct TimeShape<R, 256> { static constexpr int A = 16, B = 16; };
template <typename R> struct TimeShape<R, 512> { static constexpr int A = 32, B = 16; };
template <typename R> struct TimeShape<R, 1024> { static constexpr int A = 32, B = 32; };

// columns per tile: an exchange near 64 KB (two lines a column for general zeta)
template <typename R, int n, bool GZ>
constexpr int time_lanes() {
  constexpr int vals = n * (GZ ? 2 : 1) * (int)(sizeof(R) / 4);
  return TimeShape<R, n>::B == 1 ? 32 : vals <= 128 ? 32 : vals <= 512 ? 16 : vals <= 1024 ? (sizeof(R) == 8 ? 16 : 8) : 8;
}
// lane groups: one per pair of rows (zeta = pi: A/2 pairs) or per row (general zeta: A), at most one per
// first step (B) on long lines; the one-thread lines run four tiles a block
template <typename R, int n, bool GZ>
constexpr int time_groups() {
  constexpr int A = TimeShape<R, n>::A, B = TimeShape<R, n>::B;
  constexpr int rows = GZ ? A : A / 2;
  return B == 1 ? 1 : n <= 16 || rows < B ? rows : B;
}
template <typename R, int n, bool GZ>
constexpr int time_threads() { return time_groups<R, n, GZ>() * time_lanes<R, n, GZ>(); }
template <typename R, int n, bool GZ>
constexpr size_t time_smem() {
  return TimeShape<R, n>::B == 1 ? 0 : (size_t)(GZ ? 2 : 1) * n * time_lanes<R, n, GZ>() * sizeof(cx<R>);
}
template <typename R, int n, bool GZ>
constexpr int time_blocks_per_sm() {
  constexpr int th = TimeShape<R, n>::B == 1 ? 128 : time_threads<R, n, GZ>();
  if (sizeof(R) == 8) return th <= 128 ? 2 : 1;
  return n >= 1024 ? 1 : n <= 64 && th <= 128 ? 8 : th <= 128 || n == 128 ? 4 : th <= 256 ? 2 : 1;
}

// Solve at a slot pair (zeta = pi): Xr at r, Xq at n-1-r, both overwritten.  `scale` carries 1/n (and
// in FP64 the spatial scales).
template <typename R>
__device__ __forceinline__ void solve_pair(int kind, cx<R>& Xr, cx<R>& Xq, cx<R> mr, R c, R a2, R alpha, R scale) {
  using T = cx<R>;
  if (kind == PK_PS) {
    const T lam = mk<R>(mr.x + c, mr.y);
    // 20 operations and a division, where forming F1, F2, U1 and U2 takes 30 (with odd_dft: FP64 time pass at
    // N = 255, n = 256 2.21 -> 2.03 ms): with U1, U2 the solved halves, Xr' = U1 + i U2 and Xq' = conj U1 + i conj U2 collapse to
    //   Xr' = ((a - i alpha) Xr - i b conj Xq) iv,  Xq' = ((a - i alpha) Xq + i b conj Xr) iv,  lambda = a + i b
    const R iv = scale / (lam.x * lam.x + (lam.y * lam.y + a2));
    const R a = lam.x * iv, b = lam.y * iv, al = alpha * iv;
    const T x = Xr, q = Xq;
    Xr.x = a * x.x + (al * x.y - b * q.y);
    Xr.y = a * x.y - (al * x.x + b * q.x);
    Xq.x = a * q.x + (al * q.y + b * x.y);
    Xq.y = a * q.y - (al * q.x - b * x.x);
    return;
  }
  R w;
  if (kind == PK_ABS_PS) {
    const R lx = mr.x + c;
    w = rsq(lx * lx + (mr.y * mr.y + a2)) * scale;
  } else {
    w = scale / ((R)sqrt(mr.x * mr.x + mr.y * mr.y + a2) + c);
  }
  Xr = cscale(Xr, w);
  Xq = cscale(Xq, w);
}
// general zeta: V1, V2 the two halves at one slot
template <typename R>
__device__ __forceinline__ void solve_halves(int kind, cx<R>& V1, cx<R>& V2, cx<R> mr, R c, R a2, R alpha, R scale) {
  using T = cx<R>;
  if (kind == PK_PS) {
    const T lam = mk<R>(mr.x + c, mr.y);
    const R iv = scale / (lam.x * lam.x + (lam.y * lam.y + a2));
    const T U1 = cscale(cadd(cmul(cconj(lam), V1), cscale(V2, alpha)), iv);
    const T U2 = cscale(csub(cmul(lam, V2), cscale(V1, alpha)), iv);
    V1 = U1;
    V2 = U2;
    return;
  }
  R w;
  if (kind == PK_ABS_PS) {
    const R lx = mr.x + c;
    w = rsq(lx * lx + (mr.y * mr.y + a2)) * scale;
  } else {
    w = scale / ((R)sqrt(mr.x * mr.x + mr.y * mr.y + a2) + c);
  }
  V1 = cscale(V1, w);
  V2 = cscale(V2, w);
}

template <typename R, int n, bool GZ>
__global__ void __launch_bounds__((TimeShape<R, n>::B == 1 ? 128 : time_threads<R, n, GZ>()), (time_blocks_per_sm<R, n, GZ>()))
    k_lane_time(const Geom* __restrict__ G, const Slots* __restrict__ S, const int* __restrict__ off, int count, Sel sel,
                int kind, int in_sel, int out_sel, int) {
  using T = cx<R>;
  constexpr int A = TimeShape<R, n>::A, B = TimeShape<R, n>::B, NG = time_groups<R, n, GZ>(), LT = time_lanes<R, n, GZ>();
  constexpr int H = GZ ? 2 : 1;
  extern __shared__ __align__(16) unsigned char lane_smem[];
  const int inst = find_inst(off, count, blockIdx.x);
  if (sel.skip(inst)) return;
  const Geom& g = G[inst];
  const int N = g.N;
  int lt = blockIdx.x - (count > 1 ? __ldg(off + inst) : 0);
  const int l = threadIdx.x % LT, grp = threadIdx.x / LT;
  const int nb = (N + LT - 1) / LT;
  if (B == 1) {
    lt = lt * (128 / LT) + grp;                    // four one-warp tiles a block
    if (lt >= nb * N) return;
  }
  const int row = lt / nb, c0 = (lt - row * nb) * LT;
  const bool ok = c0 + l < N;
  const int ci = ok ? c0 + l : N - 1;
  const View vi = view_of<R>(g, S[inst], in_sel), vo = view_of<R>(g, S[inst], out_sel);
  const long long iat = (long long)row * vi.rs + ci, oat = (long long)row * vo.rs + ci;
  const int its = vi.ts, ots = vo.ts;
  const T* __restrict__ pre = twist<R>(g);
  const T* __restrict__ mu = lam_time<R>(g);
  const R c = (R)(g.tau * (__ldg(&g.kap[ci]) + __ldg(&g.kap[row])));
  const R alpha = (R)g.alpha, a2 = (R)(g.alpha * g.alpha);
  // 1/n, and in FP64 the scale 1/(2L) of each spatial transform pair (forward and inverse, two axes)
  const R scale = sizeof(R) == 8 ? (R)1 / ((R)n * (R)g.M * (R)g.M) : (R)1 / (R)n;

  if constexpr (B == 1) {
    T x[H][A];
#pragma unroll
    for (int t = 0; t < n; ++t) {
      const T a = Pairs<R>(vi, iat).get(t * its);
      const T p = __ldg(&pre[t]);
      if constexpr (GZ) {
        x[0][t] = cscale(p, a.x);
        x[H - 1][t] = cscale(p, a.y);
      } else {
        x[0][t] = cmul(a, p);
      }
    }
#pragma unroll
    for (int h = 0; h < H; ++h) reg_dft<T, R, A>(x[h], false);
    if constexpr (GZ) {
      T z[2][A];
#pragma unroll
      for (int r = 0; r < n; ++r) {
        T V1 = x[0][pos<A>(r)], V2 = x[H - 1][pos<A>(r)];
        solve_halves<R>(kind, V1, V2, __ldg(&mu[r]), c, a2, alpha, scale);
        z[0][r] = V1;
        z[1][r] = V2;
      }
#pragma unroll
      for (int h = 0; h < H; ++h) reg_dft<T, R, A>(z[h], true);
#pragma unroll
      for (int t = 0; t < n; ++t) {
        const T p = __ldg(&pre[t]);
        if (ok)
          Pairs<R>(vo, oat).put(t * ots, mk<R>(z[0][pos<A>(t)].x * p.x + z[0][pos<A>(t)].y * p.y,
                                               z[1][pos<A>(t)].x * p.x + z[1][pos<A>(t)].y * p.y));
      }
    } else {
      T z[A];
#pragma unroll
      for (int r = 0; r < n / 2; ++r) {
        T Xr = x[0][pos<A>(r)], Xq = x[0][pos<A>(n - 1 - r)];
        solve_pair<R>(kind, Xr, Xq, __ldg(&mu[r]), c, a2, alpha, scale);
        z[r] = Xr;
        z[n - 1 - r] = Xq;
      }
      reg_dft<T, R, A>(z, true);
#pragma unroll
      for (int t = 0; t < n; ++t) {
        const T o = mulc(z[pos<A>(t)], __ldg(&pre[t]));
        if (ok) Pairs<R>(vo, oat).put(t * ots, o);
      }
    }
  } else {
    T* ex = (T*)lane_smem + l;                     // line h, position e: ex[(h n + e) LT]
    const T* __restrict__ w = GZ ? tw_time<R>(g) : pre;
    const int istep = B * vi.ts, ostep = B * vo.ts;
    // first step: position t of the line, or of both lines
#pragma unroll 1
    for (int t = grp; t < B; t += NG) {
      const Pairs<R> in(vi, iat + (long long)t * its);
      T x[A];
      if constexpr (GZ) {
#pragma unroll
        for (int q = 0; q < A; ++q) x[q] = cscale(__ldg(&pre[t + B * q]), in.half(q * istep, 0));
        reg_dft<T, R, A>(x, false);
#pragma unroll
        for (int k = 0; k < A; ++k) ex[(t * A + k) * LT] = x[pos<A>(k)];
        asm volatile("" ::: "memory");               // the second half is read again, not kept in registers
#pragma unroll
        for (int q = 0; q < A; ++q) x[q] = cscale(__ldg(&pre[t + B * q]), in.half(q * istep, 1));
      } else {
#pragma unroll
        for (int q = 0; q < A; ++q) x[q] = in.get(q * istep);
      }
      if constexpr (GZ) reg_dft<T, R, A>(x, false);
      else odd_dft<T, R, A>(x);
#pragma unroll
      for (int k = 0; k < A; ++k) ex[((H - 1) * n + t * A + k) * LT] = x[GZ ? pos<A>(k) : k];
    }
    __syncthreads();
    // second step, pointwise solve, inverse second step: rows (k1, A-1-k1), or row k1 of both halves
#pragma unroll 1
    for (int k1 = grp; k1 < (GZ ? A : A / 2); k1 += NG) {
      const int k1b = GZ ? k1 : A - 1 - k1;
      // the twiddle of row A-1-k1 is W_B^t conj(that of row k1), and W_B^t shifts the B-point DFT by one
      // slot: row k1b's value at k2 is output (k2 + 1) mod B of the DFT without it
      const int ka = GZ ? k1 : 2 * k1 + 1;
      T* ra = ex + k1 * LT;
      T* rb = ex + ((GZ ? n : 0) + k1b) * LT;
      T va[B], vb[B];
#pragma unroll
      for (int t = 0; t < B; ++t) {
        va[t] = ra[t * A * LT];
        vb[t] = rb[t * A * LT];
        if (t) {
          const T wa = __ldg(&w[t * ka]);
          va[t] = cmul(va[t], wa);
          vb[t] = GZ ? cmul(vb[t], wa) : mulc(vb[t], wa);
        }
      }
      reg_dft<T, R, B>(va, false);
      reg_dft<T, R, B>(vb, false);
      T za[B], zb[B];
#pragma unroll
      for (int k2 = 0; k2 < B; ++k2) {
        const int k2b = GZ ? k2 : (B - k2) % B;
        T Xa = va[pos<B>(k2)], Xb = vb[pos<B>(k2b)];
        const T mr = __ldg(&mu[k1 + A * k2]);
        if constexpr (GZ) solve_halves<R>(kind, Xa, Xb, mr, c, a2, alpha, scale);
        else solve_pair<R>(kind, Xa, Xb, mr, c, a2, alpha, scale);
        za[k2] = Xa;
        zb[k2b] = Xb;
      }
      reg_dft<T, R, B>(za, true);
      reg_dft<T, R, B>(zb, true);
#pragma unroll
      for (int t = 0; t < B; ++t) {
        T a = za[pos<B>(t)], b = zb[pos<B>(t)];
        if (t) {
          const T wa = __ldg(&w[t * ka]);
          a = mulc(a, wa);
          b = GZ ? mulc(b, wa) : cmul(b, wa);
        }
        ra[t * A * LT] = a;
        rb[t * A * LT] = b;
      }
    }
    __syncthreads();
    // inverse first step and untwist
#pragma unroll 1
    for (int t = grp; t < B; t += NG) {
      const Pairs<R> out(vo, oat + (long long)t * ots);
      T x[A];
#pragma unroll
      for (int k = 0; k < A; ++k) x[k] = ex[(t * A + k) * LT];
      if constexpr (GZ) reg_dft<T, R, A>(x, true);
      else odd_idft<T, R, A>(x);
      if constexpr (GZ) {
        R real[A];
#pragma unroll
        for (int q = 0; q < A; ++q) {
          const T p = __ldg(&pre[t + B * q]), z = x[pos<A>(q)];
          real[q] = z.x * p.x + z.y * p.y;
        }
#pragma unroll
        for (int k = 0; k < A; ++k) x[k] = ex[(n + t * A + k) * LT];
        reg_dft<T, R, A>(x, true);
        if (ok) {
#pragma unroll
          for (int q = 0; q < A; ++q) {
            const T p = __ldg(&pre[t + B * q]), z = x[pos<A>(q)];
            out.put(q * ostep, mk<R>(real[q], z.x * p.x + z.y * p.y));
          }
        }
      } else if (ok) {
#pragma unroll
        for (int q = 0; q < A; ++q) out.put(q * ostep, x[q]);
      }
    }
  }
}

// ------------------------------------------------------------------------------------------
// launches
// ------------------------------------------------------------------------------------------
// `resident`: blocks of the kernel the device holds at once (kept per device)
template <typename K, typename... Args>
cudaError_t launch(K kern, DeviceInt& resident, int blocks, int threads, size_t smem, cudaStream_t st, Args... args) {
  if (blocks <= 0) return cudaSuccess;
  int ahead = 0;
  const cudaError_t e = resident.get(&ahead, [&](int* out) {
    cudaError_t e2 = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e2 != cudaSuccess) return e2;
    int occ = 0, dev = 0, sms = 0;
    if ((e2 = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, threads, smem)) != cudaSuccess) return e2;
    if ((e2 = cudaGetDevice(&dev)) != cudaSuccess) return e2;
    if ((e2 = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e2;
    *out = occ * sms > 0 ? occ * sms : 1;
    return cudaSuccess;
  });
  if (e != cudaSuccess) return e;
  kern<<<blocks, threads, smem, st>>>(args..., ahead);
  return cudaGetLastError();
}

template <typename R, int M, bool EV, bool USER, bool FUSE = false>
cudaError_t rows_pass(const Batch& B, Sel sel, int in_sel, int out_sel, int inv) {
  constexpr int p = sizeof(R) == 4;
  static DeviceInt resident;
  return launch(k_lane_rows<R, M, EV, USER, FUSE>, resident, B.tot_ls[p], spatial_threads<R, M>(), spatial_smem<R, M>(),
                B.stream, B.G, (const Slots*)B.S, B.off_ls[p], B.count, sel, in_sel, out_sel, inv, LaneFuse{B.Sc, B.partial, B.fuse_r2, B.fuse_z});
}
template <typename R, int M, bool EV, bool USER, bool FUSE = false>
cudaError_t cols_pass(const Batch& B, Sel sel, int in_sel, int out_sel, int inv) {
  constexpr int p = sizeof(R) == 4;
  static DeviceInt resident;
  return launch(k_lane_cols<R, M, EV, USER, FUSE>, resident, B.tot_ls[p], spatial_threads<R, M>(), cols_smem<R, M, EV>(),
                B.stream, B.G, (const Slots*)B.S, B.off_ls[p], B.count, sel, in_sel, out_sel, inv, LaneFuse{B.Sc, B.partial, B.fuse_r2, B.fuse_z});
}
template <typename R, int n, bool GZ>
cudaError_t time_pass_n(const Batch& B, Sel sel, int kind, int in_sel, int out_sel) {
  constexpr int p = sizeof(R) == 4;
  static DeviceInt resident;
  return launch(k_lane_time<R, n, GZ>, resident, B.tot_lt[p], TimeShape<R, n>::B == 1 ? 128 : time_threads<R, n, GZ>(),
                time_smem<R, n, GZ>(), B.stream, B.G, (const Slots*)B.S, B.off_lt[p], B.count, sel, kind, in_sel, out_sel);
}

// calls F<M, EV>::run for the line length M
template <bool EV, template <int, bool> class F, typename... Args>
cudaError_t by_length(int M, Args... args) {
  switch (M) {
    case 32: return F<32, EV>::run(args...);
    case 48: return F<48, EV>::run(args...);
    case 64: return F<64, EV>::run(args...);
    case 96: return F<96, EV>::run(args...);
    case 128: return F<128, EV>::run(args...);
    case 192: return F<192, EV>::run(args...);
    case 256: return F<256, EV>::run(args...);
    case 384: return F<384, EV>::run(args...);
    case 512: return F<512, EV>::run(args...);
    case 768: return F<768, EV>::run(args...);
    case 1024: return F<1024, EV>::run(args...);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace lane
}  // namespace pcb
